"""The CUDA-core GEMM's tile shapes and edges: one dense step per case, output order natural or
interleaved, against numpy in 64 bits. FP32 sums of t products are held to the a-priori bound
(t + 2) 2^-24 times the sum of the absolute products (t = k real, 2 k complex); max-plus on
integers is exact."""
import numpy as np
import pytest

from tests._lib import ensure_built
from tn_inputs.network import Network, Path

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tn():
    return ensure_built()


# (m, n, k): below, at and above the 32-, 64- and 128-wide tiles, the 16-term blocks and the
# 4-term loads; enough tiles for the large shapes; a k split
SHAPES = [(1, 17, 3), (31, 33, 16), (32, 32, 15), (33, 64, 17), (65, 63, 4), (128, 129, 33), (1000, 1003, 20),
          (1024, 1600, 18), (2049, 1537, 7), (40, 70, 4099)]


@pytest.mark.parametrize("form", ["complex", "real", "maxplus"])
@pytest.mark.parametrize("m,n,k", SHAPES)
def test_tile_edges(tn, form, m, n, k):
    rng = np.random.default_rng(m * 7 + n * 3 + k)
    if form == "maxplus":
        A, B = (rng.integers(-50, 50, size=s).astype(np.float64) for s in ((m, k), (n, k)))
        A[rng.random((m, k)) < 0.2] = -np.inf
        A[0] = -np.inf  # an excluded row stays at the semiring's zero
    else:
        A, B = (rng.standard_normal(s) for s in ((m, k), (n, k)))
        if form == "complex":
            A, B = A + 1j * rng.standard_normal((m, k)), B + 1j * rng.standard_normal((n, k))
        A, B = (x.astype(np.complex64 if form == "complex" else np.float32) for x in (A, B))
    net = Network([A, B], [(0, 2), (1, 2)], {0: m, 1: n, 2: k}, (0, 1))
    plan = tn.Plan(net, Path([(0, 1)]), prec="fp32" if form == "complex" else "r32_fp32",
                   semiring="maxplus" if form == "maxplus" else "standard")
    assert plan.step(0)["cls"] == tn.TN_CLASS_SIMT
    dt = np.complex64 if form == "complex" else np.float32
    out = np.zeros((m, n), dtype=np.complex128 if form == "complex" else np.float64)
    plan.contract_host([np.ascontiguousarray(A, dtype=dt), np.ascontiguousarray(B, dtype=dt)], out)
    plan.destroy()
    if form == "maxplus":
        want = np.full((m, n), -np.inf)
        for t in range(k):
            want = np.maximum(want, A[:, t, None] + B[None, :, t])
        assert np.array_equal(out, want)
        return
    A, B = (x.astype(np.complex128 if form == "complex" else np.float64) for x in (A, B))
    want = A @ B.T
    if form == "real":
        assert np.all(np.abs(out - want) <= (k + 2) * 2.0 ** -24 * (np.abs(A) @ np.abs(B).T))
    else:
        ar, ai, br, bi = (np.abs(x) for x in (A.real, A.imag, B.real, B.imag))
        g = (2 * k + 2) * 2.0 ** -24
        assert np.all(np.abs(out.real - want.real) <= g * (ar @ br.T + ai @ bi.T))
        assert np.all(np.abs(out.imag - want.imag) <= g * (ar @ bi.T + ai @ br.T))


@pytest.mark.parametrize("form", ["complex", "real", "maxplus"])
@pytest.mark.parametrize("m,n,k", [(1, 1, 4096), (4, 4, 16384), (2, 3, 5003), (1, 16, 4097), (1, 1, 2 ** 20 + 2)])
def test_split_k(tn, form, m, n, k):
    """Few outputs, long k: a thread sums at most 16 terms in FP32 (32 products complex), the rest is
    FP64, the result is rounded once: (2 * 16 + 3) 2^-24 of the absolute products for each of the
    real and the imaginary part."""
    rng = np.random.default_rng(k)
    if form == "maxplus":
        A, B = (rng.integers(-9000, 9000, size=s).astype(np.float64) for s in ((m, k), (n, k)))
    else:
        A, B = (rng.standard_normal(s) for s in ((m, k), (n, k)))
        if form == "complex":
            A, B = A + 1j * rng.standard_normal((m, k)), B + 1j * rng.standard_normal((n, k))
    dt = np.complex64 if form == "complex" else np.float32
    A, B = A.astype(dt), B.astype(dt)
    net = Network([A, B], [(0, 2), (1, 2)], {0: m, 1: n, 2: k}, (0, 1))
    plan = tn.Plan(net, Path([(0, 1)]), prec="fp32" if form == "complex" else "r32_fp32",
                   semiring="maxplus" if form == "maxplus" else "standard")
    assert plan.step(0)["cls"] == tn.TN_CLASS_SPLITK
    out = np.zeros((m, n), dtype=np.complex128 if form == "complex" else np.float64)
    plan.contract_host([A, B], out)
    plan.destroy()
    A, B = (x.astype(np.complex128 if form == "complex" else np.float64) for x in (A, B))
    if form == "maxplus":
        assert np.array_equal(out, np.max(A[:, None, :] + B[None, :, :], axis=2))
        return
    want, size = A @ B.T, np.abs(A) @ np.abs(B).T
    assert np.all(np.abs(out - want) <= 2 * 35 * 2.0 ** -24 * size)


@pytest.mark.parametrize("m,n,k", [(32, 64, 5), (256, 512, 40)])
def test_interleaved_scaled(tn, m, n, k):
    """Extent-2 modes with rows and columns interleaved in the output, exponent scaling on: the
    address-ordered stores and the scale record."""
    rng = np.random.default_rng(k)
    bm, bn = int(np.log2(m)), int(np.log2(n))
    M, N, K = list(range(bm)), list(range(bm, bm + bn)), bm + bn
    A, B = (rng.standard_normal((x, k)).astype(np.float32) * 2.0 ** 40 for x in (m, n))
    order = [x for pair in zip(M, N[:bm]) for x in pair] + N[bm:]
    ext = {x: 2 for x in M + N}
    ext[K] = k
    net = Network([A.reshape((2,) * bm + (k,)), B.reshape((2,) * bn + (k,))], [tuple(M) + (K,), tuple(N) + (K,)], ext,
                  tuple(order))
    plan = tn.Plan(net, Path([(0, 1)]), prec="r32_fp32", exp_scaling=True)
    out, ls = np.zeros((2,) * (bm + bn)), np.zeros(1)
    plan.contract_host([A, B], out, ls)
    plan.destroy()
    got = (out * np.exp2(np.round(ls[0] / np.log(2)))).transpose([order.index(x) for x in M + N]).reshape(m, n)
    A, B = A.astype(np.float64), B.astype(np.float64)
    assert np.all(np.abs(got - A @ B.T) <= (k + 2) * 2.0 ** -24 * (np.abs(A) @ np.abs(B).T))
