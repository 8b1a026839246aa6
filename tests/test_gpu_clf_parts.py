"""The two parts in which the Ritz step's W = X Z is stored, bf16 H and twice what its rounding leaves out, add up to the fp64
product of X and the two parts of Z, where a CTA walks several tiles and where it has one.

Both products' operands and results are read from the workspace of a finished call: behind the flag block of 256 bytes Z as
two [N][l] matrices, then H and the rest as [l][T rounded up to 8], each aligned to 256 bytes.

Bounds: H + rest is the fp32 sum rounded to twice eight bits, 2^-17 of its value; the fp32 sum of the 2 N products is off by
at most 2 N 2^-24 of the sum of their magnitudes, and by far less in the mean.  H alone, or with the rest of another tile, is
off by 2^-10 in the mean: sixty times the second bound."""
import pytest
import torch

from tests.test_gpu_clf import _factorize_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,G,d,r,p", [
    (80001, 1, 256, 96, 32),         # l = 128: 313 tiles of 256 x 128
    (40003, 2, 160, 128, 64),        # l = 192: 157 of 256 x 192
    (40003, 3, 128, 264, 40),        # l = 320: 314, every second one ragged
    (45000, 2, 128, 200, 40),        # l = 256: 176 of 256 x 256
    (100, 1, 64, 8, 32),             # one accumulator, l = 64: half a tile
    (300, 2, 160, 128, 64),          # three tiles of 128 x 192
])
def test_the_two_parts_are_the_product(T, G, d, r, p, monkeypatch):
    from paper_2503_18893_b200 import xkv
    kept = {}
    call = xkv.xkv_clf_factorize
    monkeypatch.setattr(xkv, "xkv_clf_factorize", lambda cfg, X, omega, ws, *a: (kept.update(ws=ws, X=X, l=omega.shape[1]), call(cfg, X, omega, ws, *a)))
    N = G * d
    g = torch.Generator().manual_seed(T)
    X = torch.randn(T, N, generator=g).to(torch.bfloat16)
    _factorize_gpu(X, G, d, r, p, 1, seed=5)
    ws, l, Tp = kept["ws"], kept["l"], (T + 7) // 8 * 8
    up = lambda n: (n + 255) // 256 * 256
    at_z, at_h = 256, 256 + up(4 * N * l)
    at_rest = at_h + up(2 * l * Tp)
    part = lambda at, rows, cols: ws[at:at + 2 * rows * cols].view(torch.bfloat16).reshape(rows, cols).double()
    Z = part(at_z, N, l) + part(at_z + 2 * N * l, N, l)
    W = (part(at_h, l, Tp) + 0.5 * part(at_rest, l, Tp))[:, :T].T
    Xd = kept["X"].double()
    ref, mag = Xd @ Z, Xd.abs() @ Z.abs()
    err = (W - ref).abs()
    assert (err <= 2.0 ** -17 * ref.abs() + 2 * N * 2.0 ** -24 * mag).all()
    assert float(err.pow(2).mean().sqrt() / ref.pow(2).mean().sqrt()) <= 2.0 ** -16
