"""The batched kernel's step forms at their edges: register tiles with ragged rows and columns,
loads of 4, 2 and 1 terms, panels
of large steps in shared memory, extents that are not powers of two, leaves staged by groups and by the
whole team, and more steps than the exponents a team keeps. Every launch shape gives the same bits
(one thread runs an output's terms in order), and the value is the direct sum's within FP32's error
bound for the sum: every term is positive (or bounded by its absolute sum), so each of the
k + m n additions and the products add at most one rounding of 2^-24 each."""
import numpy as np
import pytest
import torch

from tests._lib import ensure_built
from tn_inputs import greedy, ising_pf
from tn_inputs.network import Network, Path

pytestmark = pytest.mark.gpu

SIZES = [(1, 1, 1), (4, 4, 2), (5, 7, 3), (16, 16, 8), (17, 33, 4), (64, 33, 6), (37, 130, 4), (100, 101, 1), (130, 3, 16),
         (2, 300, 2), (64, 128, 32), (129, 64, 12), (70, 33, 36), (33, 70, 20), (16, 8, 512), (300, 40, 52), (97, 97, 16)]
# (threads, CTAs per SM, networks per CTA, shared arena): tiles from 256 outputs on in the first, never in the last
SHAPES = [(32, 4, 1), (128, 2, 1, 4096), (256, 1, 1, 8192), (64, 2, 1, 2304), (256, 2, 1), (512, 1, 1), (32, 2, 4), (32, 1, 16)]


@pytest.fixture(scope="module")
def tn():
    return ensure_built()


def triangle(m, n, k, seed, kind):
    """sum_ijk A[i, k] B[j, k] C[j, i]: one m x n x k step, then a closed one."""
    rng = np.random.default_rng(seed)

    def tensor(*shape):
        t = rng.uniform(0.5, 2.0, shape) * 2.0 ** rng.integers(-20, 20)
        if kind == "complex":
            t = t * np.exp(2j * np.pi * rng.random(shape))
        return t if kind != "maxplus" else np.round(16 * t / np.abs(t).max())
    net = Network([tensor(m, k), tensor(n, k), tensor(n, m)], [(0, 2), (1, 2), (1, 0)], {0: m, 1: n, 2: k}, ())
    net.check()
    return net, Path([(0, 1), (2, 3)])


@pytest.mark.parametrize("kind", ["real", "real_scaled", "complex", "complex_scaled", "maxplus"])
def test_step_forms(tn, kind):
    base = kind.split("_")[0]
    pairs = [triangle(m, n, k, 7 * i, base) for i, (m, n, k) in enumerate(SIZES)]
    b = tn.Batch([p[0] for p in pairs], [p[1] for p in pairs], complex_=base == "complex",
                 exp_scaling=kind.endswith("scaled"), semiring="maxplus" if base == "maxplus" else "standard")
    packed = torch.tensor(b.pack([p[0] for p in pairs]), device="cuda")
    first = None
    for shape in SHAPES:
        try:
            b.set_launch_shape(*shape)
        except tn.TnError:
            continue  # the offset tables of that many networks do not fit
        v = torch.zeros((len(pairs), 2), dtype=torch.float64, device="cuda")
        l = torch.zeros(len(pairs), dtype=torch.float64, device="cuda")
        b.contract(packed, v, l)
        got = np.concatenate([v.cpu().numpy(), l.cpu().numpy()[:, None]], axis=1)
        first = got if first is None else first
        assert np.array_equal(got, first), shape
    for (m, n, k), (net, path), (re, im, lg) in zip(SIZES, pairs, first):
        A, B, C = (np.asarray(t) for t in net.tensors)
        if base == "maxplus":
            assert re == np.max(A[:, None, :] + B[None] + C.T[:, :, None])  # small integers: exact
            continue
        terms = np.einsum("ik,jk,ji->", np.abs(A), np.abs(B), np.abs(C))
        want = np.einsum("ik,jk,ji->", A, B, C)
        got = complex(re, im) * np.exp(lg)
        assert abs(got - want) <= (m * n + k + 8) * 2.0 ** -23 * terms, (m, n, k)


def test_more_steps_than_kept_exponents(tn):
    nets = [ising_pf.ring_network(n, 1.0, 1.0) for n in (30, 100, 300, 600)]
    paths = [greedy.greedy_path(net, seed=0) for net in nets]
    b = tn.Batch(nets, paths)
    packed = torch.tensor(b.pack(nets), device="cuda")
    first = None
    for shape in SHAPES:
        b.set_launch_shape(*shape)
        v = torch.zeros((len(nets), 2), dtype=torch.float64, device="cuda")
        l = torch.zeros(len(nets), dtype=torch.float64, device="cuda")
        b.contract(packed, v, l)
        got = np.concatenate([v.cpu().numpy(), l.cpu().numpy()[:, None]], axis=1)
        first = got if first is None else first
        assert np.array_equal(got, first), shape
    for n, (re, _, lg) in zip((30, 100, 300, 600), first):
        want = n * np.log(2 * np.cosh(1.0)) + np.log1p(np.tanh(1.0) ** n)
        assert abs(np.log(re) + lg - want) < 4 * n * 2.0 ** -23
