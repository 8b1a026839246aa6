"""A = X V where it comes from the Rayleigh-Ritz step's W = X Z (three l-column parts shorter than a row of X), at edges of the
product's tiles and of the rule: against the fp64 product with the B that is handed back, and by the residual."""
import pytest
import torch

from tests.test_gpu_clf import _factorize_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,G,d,r,p", [
    (257, 1, 192, 8, 32),          # 3 l = N = 192: the product with V itself
    (257, 1, 256, 8, 32),          # l = 64, one row beyond a 256-row tile
    (1000, 4, 160, 104, 32),       # l = 192, N = 640; r inside a tile of 128
    (2050, 2, 512, 200, 56),       # l = 256, N = 1024
    (4099, 4, 512, 264, 40),       # l = 320, N = 2048; 384 columns of tiles; pitch of W longer than T
])
def test_coefficients_from_the_ritz_step(T, G, d, r, p):
    g = torch.Generator().manual_seed(T)
    N = G * d
    s = 1.0 / torch.arange(1, min(N, T) + 1)
    X = ((torch.randn(T, len(s), generator=g) * s) @ torch.randn(len(s), N, generator=g)).to(torch.bfloat16)
    A, B, _, _ = _factorize_gpu(X, G, d, r, p, 2, seed=5)
    Xd, V = X.cuda().double(), torch.cat([B[i] for i in range(G)], dim=1).double().T          # (N, r)
    # A is rounded to bf16 (rms 2^-9 / sqrt(3) of an entry), V was for B: a vector of unit length, off by 2^-9 / sqrt(3) of
    # itself at random, moves X v by that part of |X|_F / sqrt(N) < sigma_1 only
    proj = Xd @ V
    assert (A.double() - proj).norm() <= 4e-3 * proj.norm()
    # best coefficients for these B leave the least; A may add its own rounding and that of V
    coef = Xd @ torch.linalg.pinv(V.T)
    least = ((Xd - coef @ V.T) ** 2).sum()
    assert ((Xd - A.double() @ V.T) ** 2).sum() <= 1.02 * least + (4e-3 * proj.norm()) ** 2
