"""FP64 products of small matrices (8 x 8 DFMA tiles) against numpy's FP64 product.

Sizes: one tile, tile edges, the 256-wide k chunks and the last size before the 64 x 64 tiles.
Tolerance: the rounding of a K-term FP64 sum, 4 K 2^-53 of |X| |Y|^T elementwise.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (8, 8, 8), (9, 7, 3), (64, 64, 64), (63, 65, 255),
                                   (40, 33, 256), (17, 129, 257), (343, 343, 343), (960, 320, 320),
                                   (1024, 1024, 24)])
@pytest.mark.parametrize("trans", [False, True])
def test_small_fp64_product(cuda, cdmpt_lib, M, N, K, trans):
    import torch
    if trans and M % N:
        pytest.skip("transposed placement needs whole row blocks")
    g = np.random.default_rng(M + 1000 * N + K)
    X, Y, C = g.standard_normal((M, K)), g.standard_normal((N, K)), g.standard_normal((M, N))
    t = lambda a: torch.from_numpy(a).cuda()
    D = torch.empty((M, N), dtype=torch.float64, device="cuda")
    dot = torch.zeros(1, dtype=torch.float64, device="cuda")
    cdmpt_lib.gemm_f64(t(X), t(Y), D, alpha=-0.75, beta=1.5, C=t(C), gamma=0.25, diag_block=N,
                       trans_block=N if trans else 0, dot=dot)
    P = X @ Y.T
    eye = 0.25 * ((np.arange(M)[:, None] % N) == np.arange(N)[None, :])
    if trans:
        sw = lambda a: a.reshape(M // N, N, N).transpose(0, 2, 1).reshape(M, N)
        ref = -0.75 * sw(P) + 1.5 * C + sw(eye)
        mag = sw(np.abs(X) @ np.abs(Y).T)
    else:
        ref = -0.75 * P + 1.5 * C + eye
        mag = np.abs(X) @ np.abs(Y).T
    tol = 4.0 * K * 2.0 ** -53 * mag + 8.0 * 2.0 ** -53 * (np.abs(C) + 1.0)
    out = D.cpu().numpy()
    assert np.all(np.abs(out - ref) <= tol)
    assert abs(dot.item() - (out * out).sum()) <= 1e-12 * (out * out).sum()
