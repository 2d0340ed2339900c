"""Epilogue of the tcgen05 products at the edges of its 32 x 32 blocks and of the tile families.

Every product runs through the four-element form where rows are 16-byte and the masked form
elsewhere (odd column counts, leading dimensions that are no multiple of 4, unaligned outputs,
blocks on the diagonal), with the C term, gamma I on diagonal blocks, transposed placement, the
symmetric mirror and the fused dot; columns beyond the matrix must stay untouched. Sizes: below
and above one 128-row tile, block remainders of 1, 4, 31, and one with two-SM tiles.
Tolerance, elementwise: 2^-9 (one-pass TF32: both operands rounded to 11 bits) or 2^-19 (split:
dropped lo*lo terms and the truncating accumulation) of |X| |Y|^T, and the FP32 rounding of the
epilogue.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

EPS = {"tf32": 2.0 ** -9, "3xtf32": 2.0 ** -19}


def _call(pkg, engine, X, Y, D, ldd, C, gamma, diag, tb, dot, off=0):
    code = {"tf32": 2, "3xtf32": 3}[engine]
    M, K = X.shape
    N = Y.shape[0]
    st = pkg.lib().cdmpt_gemm_f32(code, M, N, K, X.data_ptr(), X.stride(0), Y.data_ptr(),
                                  Y.stride(0), D.data_ptr() + 4 * off, ldd, 0.5, -1.25,
                                  C.data_ptr(), C.stride(0), gamma, diag, tb, dot.data_ptr(), None,
                                  0, 0)
    assert st == 0


@pytest.mark.parametrize("engine", ["3xtf32", "tf32"])
@pytest.mark.parametrize("M,N,K,pad,off", [
    (33, 33, 40, 3, 0), (128, 100, 64, 28, 0), (130, 131, 96, 1, 0), (160, 159, 40, 1, 0),
    (260, 260, 260, 0, 0), (288, 320, 64, 4, 1), (257, 1001, 100, 23, 0), (2100, 2100, 64, 0, 0)])
@pytest.mark.parametrize("mode", ["plain", "sym", "trans"])
def test_epilogue_blocks(cuda, cdmpt_lib, engine, M, N, K, pad, off, mode):
    import torch
    if mode != "plain" and M != N:
        pytest.skip("square results only")
    g = np.random.default_rng(M * 7 + N + K)
    ldk = (K + 3) // 4 * 4
    dev = lambda a: torch.from_numpy(a).cuda()
    Xp = np.zeros((M, ldk), np.float32)
    Xp[:, :K] = g.standard_normal((M, K))
    Yp = Xp if mode == "sym" else np.zeros((N, ldk), np.float32)
    if mode != "sym":
        Yp[:, :K] = g.standard_normal((N, K))
    C = g.standard_normal((M, N)).astype(np.float32)
    if mode == "sym":
        C = 0.5 * (C + C.T)
    ldd = N + pad
    D = torch.full((M * ldd + off,), 7.5, dtype=torch.float32, device="cuda")
    dot = torch.zeros(1, dtype=torch.float64, device="cuda")
    X, Y = dev(Xp)[:, :K], dev(Yp)[:, :K]
    _call(cdmpt_lib, engine, X, Y, D, ldd, dev(C), 0.375, min(M, N),
          {"plain": 0, "sym": -1, "trans": N}[mode], dot, off)
    X64, Y64 = Xp[:, :K].astype(np.float64), Yp[:, :K].astype(np.float64)
    P, mag = X64 @ Y64.T, np.abs(X64) @ np.abs(Y64).T
    eye = 0.375 * ((np.arange(M)[:, None] % min(M, N)) == np.arange(N)[None, :])
    if mode == "trans":
        P, mag, eye = P.T, mag.T, eye.T
    ref = 0.5 * P - 1.25 * C + eye
    out = D[off:].cpu().numpy().reshape(M, ldd)
    assert np.all(out[:, N:] == 7.5) and (off == 0 or D[0].item() == 7.5)
    got = out[:, :N].astype(np.float64)
    tol = EPS[engine] * mag + 2.0 ** -21 * (np.abs(ref) + 1.25 * np.abs(C) + 0.375 + mag / K)
    assert np.all(np.abs(got - ref) <= tol), np.max(np.abs(got - ref) / tol)
    s = (got * got).sum()
    assert abs(dot.item() - s) <= 1e-5 * s
    if mode == "sym":
        assert np.array_equal(out[:, :N], out[:, :N].T)


@pytest.mark.parametrize("engine", ["3xtf32", "tf32"])
@pytest.mark.parametrize("diag", [1, 2, 3, 4, 5, 31])
@pytest.mark.parametrize("N", [32, 64, 260])
def test_small_diagonal_blocks(cuda, cdmpt_lib, engine, diag, N):
    """gamma I on diagonal blocks below, at and above the four rows of one vector step: gamma
    stands at [m % diag == n], with products and C small against it."""
    import torch
    g = np.random.default_rng(N + diag)
    X = g.standard_normal((N, 32)).astype(np.float32)
    C = g.standard_normal((N, N)).astype(np.float32)
    dev = lambda a: torch.from_numpy(a).cuda()
    D = torch.empty(N * N, dtype=torch.float32, device="cuda")
    dot = torch.zeros(1, dtype=torch.float64, device="cuda")
    _call(cdmpt_lib, engine, dev(X), dev(X), D, N, dev(C), 1000.0, diag, 0, dot)
    X64 = X.astype(np.float64)
    P, mag = X64 @ X64.T, np.abs(X64) @ np.abs(X64).T
    eye = 1000.0 * ((np.arange(N)[:, None] % diag) == np.arange(N)[None, :])
    ref = 0.5 * P - 1.25 * C + eye
    got = D.cpu().numpy().reshape(N, N).astype(np.float64)
    tol = EPS[engine] * mag + 2.0 ** -21 * (np.abs(ref) + 1.25 * np.abs(C) + eye + mag / 32)
    assert np.all(np.abs(got - ref) <= tol), np.argwhere(np.abs(got - ref) > tol)[:4]
