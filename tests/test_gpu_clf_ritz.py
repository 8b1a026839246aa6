"""The Rayleigh-Ritz step of the factorisation: the rows of B are the Ritz vectors of their own span, as good as bf16 can
hold them.  The measure is the off-diagonal part of V^T X^T X V, relative to the diagonal; exact Ritz vectors rounded to bf16
set the scale (a rounded noise direction holds 2^-9 of the largest singular values), and an error of the l x l matrix or of
its eigenvectors adds to it."""
import pytest
import torch

from tests.test_gpu_clf import _factorize_gpu

pytestmark = pytest.mark.gpu


def _off_diagonal(H, V):
    M = V.T @ H @ V
    d = M.diagonal().sqrt()
    M = M / d[:, None] / d[None, :]
    return float((M - torch.diag(M.diagonal())).pow(2).mean().sqrt())


@pytest.mark.parametrize("T,G,d,r", [(4096, 4, 256, 128), (3001, 2, 320, 200), (8191, 2, 1024, 256)])
def test_rows_of_b_are_ritz_vectors_to_bf16(T, G, d, r):
    """Three caches each: one rounding of the same vectors differs from another by up to a quarter in this measure, because a
    few noise directions with a large entry weigh most."""
    N, rho = G * d, r // 2
    got = want = 0.0
    for seed in (1, 2, 3):
        g = torch.Generator(device="cuda").manual_seed(T + seed)
        s = 1.0 / torch.arange(1, rho + 1, device="cuda")
        signal = (torch.randn(T, rho, generator=g, device="cuda") * s) @ torch.randn(rho, N, generator=g, device="cuda")
        X = (signal / signal.std() + 0.01 * torch.randn(T, N, generator=g, device="cuda")).to(torch.bfloat16)
        A, B, sig, _ = _factorize_gpu(X, G, d, r, 32, 2, seed=7 + seed)
        Xd = X.double()
        H = Xd.T @ Xd
        V = torch.cat([B[i] for i in range(G)], dim=1).double().T            # (N, r)
        Q = torch.linalg.qr(V)[0]
        exact = Q @ torch.linalg.eigh(Q.T @ H @ Q)[1]
        got += _off_diagonal(H, V)
        want += _off_diagonal(H, exact.to(torch.bfloat16).double())
    assert got <= 1.25 * want


@pytest.mark.parametrize("T,N,r", [(4096, 640, 608), (2500, 192, 136)])
def test_rotations_keep_the_length(T, N, r):
    """With l = N the sketch holds everything and a flat spectrum takes the most sweeps; the singular values are those of X
    up to the drift of the eigenvectors' length.  A vector takes part in l - 1 rotations of a sweep; with c and s rounded to
    nearest c^2 + s^2 is off by 2^-23 and the length by 2^-24 at most, with no preferred sign: a quarter of that is allowed
    as a bias.  (The rounding of X Z to bf16 has none: 1e-6 in the mean.)"""
    from paper_2503_18893_b200 import xkv
    g = torch.Generator(device="cuda").manual_seed(N)
    X = torch.randn(T, N, generator=g, device="cuda").to(torch.bfloat16)
    cfg = xkv.make_clf_config(T=T, G=1, d=N, r=r, oversample=32, power_iters=1)
    assert xkv.xkv_clf_rank_l(cfg) == N
    omega = torch.randn(N, N, generator=g, device="cuda").to(torch.bfloat16)
    ws = torch.empty(xkv.xkv_clf_workspace_bytes(cfg), dtype=torch.uint8, device="cuda")
    A = torch.empty((T, r), dtype=torch.bfloat16, device="cuda")
    B = torch.empty((1, r, N), dtype=torch.bfloat16, device="cuda")
    sig = torch.empty(r, dtype=torch.float32, device="cuda")
    xkv.xkv_clf_factorize(cfg, X, omega, ws, A, B, sig)
    assert xkv.xkv_clf_status(ws) == (0, 0)
    sweeps = int(ws[44:48].view(torch.int32))
    sv = torch.linalg.svdvals(X.double())[:r]
    drift = (sig.double() / sv - 1).mean().abs()
    assert drift <= (N - 1) * sweeps * 2.0 ** -26 + 2e-6


@pytest.mark.parametrize("T,heavy", [(3000, 1e3), (1200, 30.0), (1, 1.0)])
def test_one_row_holds_the_weight(T, heavy):
    """A row a thousand times the others (or the only one): no error averages out over the rows.  The largest singular value
    is that of X up to the two-part bf16 of Z and W (2^-17 each, on both sides), the length of a vector (see above) and fp32
    sums."""
    from paper_2503_18893_b200 import xkv
    g = torch.Generator(device="cuda").manual_seed(T)
    X = torch.randn(T, 256, generator=g, device="cuda")
    X[T // 2] *= heavy
    X = X.to(torch.bfloat16)
    A, B, sig, _ = _factorize_gpu(X, 2, 128, 64, 32, 2, seed=11)
    sv = torch.linalg.svdvals(X.double())
    l, sweeps = 128, 16
    assert abs(float(sig[0]) / float(sv[0]) - 1) <= 4 * 2.0 ** -17 + (l - 1) * sweeps * 2.0 ** -26 + 1e-6


@pytest.mark.parametrize("which", ["row", "column"])
def test_directions_are_chosen_where_one_holds_the_weight(which):
    """An outlier row or column leaves the off-diagonal weight below any fraction of the total; the r best of the l directions
    have to be found all the same.  Converged, the residual is 1.017 and 1.008 times the optimum here (a sketch of 128 for a
    flat rest of 64 directions); unrotated directions give 1.049 and 1.039."""
    g = torch.Generator(device="cuda").manual_seed(5)
    T, N = (3000, 256) if which == "row" else (700, 512)
    X = torch.randn(T, N, generator=g, device="cuda")
    if which == "row":
        X[7] *= 1e3
    else:
        X[:, 7] *= 1e4
    X = X.to(torch.bfloat16)
    A, B, sig, _ = _factorize_gpu(X, 2, N // 2, 64, 32, 2, seed=13)
    Xd, V = X.double(), torch.cat([B[0], B[1]], dim=1).double()
    res = float(((Xd - A.double() @ V) ** 2).sum())
    assert res <= 1.03 * float((torch.linalg.svdvals(Xd)[64:] ** 2).sum())
