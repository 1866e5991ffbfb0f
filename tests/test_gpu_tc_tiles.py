"""The 3xTF32 tile shapes and their edges: one dense step per case against numpy in 64 bits.

A-priori bound, relative to the absolute products: the dropped lo.lo and lo's truncation 2^-20;
up to eight truncating additions of a 32-term chunk 2^-20; the chunks' round-to-nearest sum and
the cross terms (k / 32 + 2) 2^-24."""
import numpy as np
import pytest

from tests._lib import ensure_built
from tn_inputs.network import Network, Path

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tn():
    tn = ensure_built()
    old = tn.binding.cost_model()  # narrow tiles would go to the CUDA cores at the peak rates
    tn.binding.set_cost_model(old["hbm_bytes_per_s"], old["simt_flops"], [10 * f for f in old["tc_flops"]])
    yield tn
    tn.binding.set_cost_model(old["hbm_bytes_per_s"], old["simt_flops"], old["tc_flops"])


def check(tn, real, m, n, k, scaled=False, slices=1):
    rng = np.random.default_rng(m + 3 * n + 5 * k)
    shape = lambda x: (slices, x, k) if slices > 1 else (x, k)
    A, B = rng.standard_normal(shape(m)), rng.standard_normal(shape(n))
    if not real:
        A, B = A + 1j * rng.standard_normal(shape(m)), B + 1j * rng.standard_normal(shape(n))
    dt = np.float32 if real else np.complex64
    A, B = A.astype(dt), B.astype(dt)
    lead = (3,) if slices > 1 else ()
    net = Network([A, B], [lead + (0, 2), lead + (1, 2)], {0: m, 1: n, 2: k, 3: slices}, (0, 1))
    plan = tn.Plan(net, Path([(0, 1)]), lead, prec="r32_3xtf32" if real else "3xtf32", exp_scaling=scaled)
    assert plan.step(0)["cls"] == tn.TN_CLASS_TC
    out, ls = np.zeros((m, n), dtype=np.float64 if real else np.complex128), np.zeros(1)
    plan.contract_host([A, B], out, ls)
    plan.destroy()
    out = out * np.exp2(np.round(ls[0] / np.log(2)))
    wide = np.float64 if real else np.complex128
    A, B = (x.reshape(slices, -1, k).astype(wide) for x in (A, B))
    want, size = sum(a @ b.T for a, b in zip(A, B)), sum(np.abs(a) @ np.abs(b).T for a, b in zip(A, B))
    bound = 2 * 2.0 ** -20 + (k / 32 + 2) * 2.0 ** -24
    assert np.all(np.abs(out - want) <= (1 if real else np.sqrt(2)) * bound * size)


# (m, n, k): each tile width of the form chosen (by waves of tiles), sizes just off the tiles, the
# 32-term blocks and whole 32 x 32 store blocks
@pytest.mark.parametrize("m,n,k", [(2049, 5800, 40), (2048, 6144, 32), (1100, 4000, 72), (1024, 4096, 256), (130, 100, 8),
                                   (128, 64, 36), (300, 65, 1000)])
def test_real_tiles(tn, m, n, k):
    check(tn, True, m, n, k)


@pytest.mark.parametrize("m,n,k", [(1000, 1000, 44), (1024, 1024, 64), (129, 2050, 8), (200, 33, 12), (128, 32, 100),
                                   (256, 31, 260)])
def test_complex_tiles(tn, m, n, k):
    check(tn, False, m, n, k)


@pytest.mark.parametrize("real", [True, False])
@pytest.mark.parametrize("m,n,k", [(300, 200, 36), (256, 128, 64)])
def test_scaled_and_batched(tn, real, m, n, k):
    check(tn, real, m, n, k, scaled=True)
    check(tn, real, m, n, k, slices=3)
