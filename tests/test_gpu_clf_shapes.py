"""The factorisation at shapes where its products take another tile: one or two accumulators of rows, widths of 64 to 320
columns, one or several K ranges, T inside and beyond a tile.  A = X V, orthonormal V and the residual are checked in fp64."""
import pytest
import torch

from tests.test_gpu_clf import _factorize_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,G,d,r,p", [
    (100, 1, 64, 8, 32),           # one tile of everything, l = N = 64
    (257, 1, 192, 64, 32),         # one row beyond a 256-row tile; l = 128
    (1000, 2, 160, 128, 64),       # l = 192; N = 320
    (2049, 4, 128, 200, 40),       # l = 256; two K ranges
    (5003, 3, 128, 264, 40),       # l = 320: 384 columns of tiles; N = 384
])
def test_factors_at_tile_edges(T, G, d, r, p):
    g = torch.Generator().manual_seed(T)
    N = G * d
    s = 1.0 / torch.arange(1, min(N, T) + 1)
    X = ((torch.randn(T, len(s), generator=g) * s) @ torch.randn(len(s), N, generator=g)).to(torch.bfloat16)
    A, B, sig, _ = _factorize_gpu(X, G, d, r, p, 2, seed=5)
    Xd, V = X.cuda().double(), torch.cat([B[i] for i in range(G)], dim=1).double().T          # (N, r)
    sv = torch.linalg.svdvals(Xd)
    assert (V.T @ V - torch.eye(r, device="cuda")).abs().max() <= 2e-2
    proj = Xd @ V
    assert (A.double() - proj).abs().max() <= 2e-2 * proj.abs().max()
    res, rounding = ((Xd - A.double() @ V.T) ** 2).sum(), 2e-5 * (sv ** 2).sum()
    k = min(r, len(sv))
    assert res <= 1.15 * (sv[k:] ** 2).sum() + rounding
    assert ((sig[:k].double() - sv[:k]).abs() <= 2e-2 * sv[:k] + 2e-3 * sv[0]).all()
