"""Large leaves whose planned order is the declared one: a copy. Staged FP32 values are exact: the
leaf meets a factor 1 in a step of depth 1, so the result has to equal the leaf; the split forms
within their one-product bounds."""
import numpy as np
import pytest
import torch

from tests._lib import BF16X3_BOUND, BF16X3M_BOUND, ensure_built
from tn_inputs.network import Network, Path

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tn():
    return ensure_built()


@pytest.mark.parametrize("real", [True, False])
@pytest.mark.parametrize("m", [2048, 2049, 4098, 70001, 1 << 20])
@pytest.mark.parametrize("shift", [0, 1])  # elements by which the source misses 16-byte alignment
def test_exact_copy(tn, real, m, shift):
    dt = torch.float32 if real else torch.complex64
    g = torch.Generator(device="cuda").manual_seed(m)
    leaf = torch.randn(m + shift, dtype=dt, device="cuda", generator=g)[shift:]
    net = Network([None, None], [(0, 1), (1,)], {0: m, 1: 1}, (0,))
    plan = tn.Plan(net, Path([(0, 1)]), prec="r32_fp32" if real else "fp32", exp_scaling=real)
    assert plan.tensor(0)["tiled"] and plan.layout(0) == (0, 1)
    out = torch.zeros(m, dtype=torch.float64 if real else torch.complex128, device="cuda")
    ls = torch.zeros(1, dtype=torch.float64, device="cuda")
    plan.contract([leaf, torch.ones(1, dtype=dt, device="cuda")], out, ls)
    torch.cuda.synchronize()
    plan.destroy()
    out = out * torch.exp2(torch.round(ls / np.log(2)))
    assert torch.equal(out, leaf.to(out.dtype))


def test_sliced_copies(tn):
    """A leaf sliced in its first label: the copies of a pass are contiguous runs of the source."""
    m, s = 3001, 5
    leaf = torch.randn(s, m, dtype=torch.complex64, device="cuda")
    net = Network([None, None], [(2, 0, 1), (2, 1)], {0: m, 1: 1, 2: s}, (0,))
    plan = tn.Plan(net, Path([(0, 1)]), (2,), max_slice_batch=2)
    out = torch.zeros(m, dtype=torch.complex128, device="cuda")
    plan.contract([leaf, torch.ones(s, 1, dtype=torch.complex64, device="cuda")], out)
    torch.cuda.synchronize()
    plan.destroy()
    want = leaf.to(torch.complex128).sum(0)
    assert torch.max(torch.abs(out - want)) <= 1e-14 * s * torch.max(torch.abs(leaf))


@pytest.mark.parametrize("prec,bound", [("bf16x3", BF16X3_BOUND), ("bf16x3m", BF16X3M_BOUND)])
@pytest.mark.parametrize("m,n,k", [(300, 260, 64), (257, 130, 24)])
def test_split_forms(tn, prec, bound, m, n, k):
    rng = np.random.default_rng(k)
    A, B = (rng.standard_normal((x, k)) + 1j * rng.standard_normal((x, k)) for x in (m, n))
    net = Network([A, B], [(0, 2), (1, 2)], {0: m, 1: n, 2: k}, (0, 1))
    plan = tn.Plan(net, Path([(0, 1)]), prec=prec)
    assert plan.step(0)["cls"] == tn.TN_CLASS_TC and plan.tensor(0)["format"] != 0
    out = np.zeros((m, n), dtype=np.complex128)
    plan.contract_host([x.astype(np.complex64) for x in (A, B)], out)
    plan.destroy()
    assert np.all(np.abs(out - A @ B.T) <= 2 * bound * (np.abs(A) @ np.abs(B).T))
