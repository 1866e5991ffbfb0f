"""A chain's steps at the edges of their loads: rows of 4 n, 2 and other numbers of terms, outputs
interleaved over more merged dims than one 16-byte load of places holds, extents that are not
powers of two. sum A[i.., k] B[j.., k] C[i, j interleaved]: one step of k terms and a closed one,
both in one chain, against the direct sum in 64 bits; an output's error is at most one 2^-24
rounding per product and addition of the terms' absolute sum."""
import numpy as np
import pytest
import torch

from tests._lib import ensure_built
from tn_inputs.network import Network, Path

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["complex", "real", "scaled", "maxplus"])
@pytest.mark.parametrize("rows,cols,k", [((4,), (4,), 1), ((4,), (4,), 2), ((3,), (5,), 3), ((2, 2), (2, 3), 4),
                                         ((5,), (3, 2), 6), ((2,) * 5, (2,) * 4, 2), ((2,) * 4, (2,) * 5, 8),
                                         ((3, 2, 3), (2, 3, 2), 12), ((2, 3), (2,), 64), ((1,), (1,), 129),
                                         ((2, 2, 2, 2, 3), (2, 2, 2, 2), 4)])
def test_terms(kind, rows, cols, k):
    tn = ensure_built()
    rng = np.random.default_rng(len(rows) * 100 + len(cols) * 10 + k)
    R, N = list(range(len(rows))), list(range(50, 50 + len(cols)))
    mix = [x for p in zip(R, N) for x in p] + R[len(N):] + N[len(R):]
    ext = {99: k, **dict(zip(R, rows)), **dict(zip(N, cols))}

    def tensor(modes):
        t = rng.uniform(0.5, 2.0, [ext[x] for x in modes])
        return t * np.exp(2j * np.pi * rng.random(t.shape)) if kind == "complex" else np.round(8 * t)
    modes = [tuple(R) + (99,), tuple(N) + (99,), tuple(mix)]
    tensors = [tensor(m) for m in modes]
    net = Network(tensors, modes, ext, ())
    net.check()
    plan = tn.Plan(net, Path([(0, 1), (2, 3)]), prec="fp32" if kind == "complex" else "r32_fp32",
                   exp_scaling=kind == "scaled", semiring="maxplus" if kind == "maxplus" else "standard")
    assert plan.step(0)["chain"] == 0 and plan.step(1)["chain"] == 0
    inputs = [torch.tensor(t.astype(np.complex64 if kind == "complex" else np.float32), device="cuda") for t in tensors]
    out = torch.zeros(1, dtype=torch.complex128 if kind == "complex" else torch.float64, device="cuda")
    log_scale = torch.zeros(1, dtype=torch.float64, device="cuda")
    plan.contract(inputs, out, log_scale)
    got = out.item() * np.exp(log_scale.item() if kind == "scaled" else 0.0)
    A, B, C = tensors
    m, n = int(np.prod(rows)), int(np.prod(cols))
    C = np.transpose(C, [mix.index(x) for x in R + N]).reshape(m, n)
    A, B = A.reshape(m, k), B.reshape(n, k)
    if kind == "maxplus":
        assert got == np.max(A[:, None, :] + B[None] + C[:, :, None])  # small integers: exact
        return
    terms = np.einsum("ik,jk,ij->", np.abs(A), np.abs(B), np.abs(C))
    assert abs(got - np.einsum("ik,jk,ij->", A, B, C)) <= (m * n + k + 8) * 2.0 ** -23 * terms
