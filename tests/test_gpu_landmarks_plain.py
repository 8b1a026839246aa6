"""Landmarks of the default chunk with and without cosines come from two kernels with the same arithmetic on a row, also where
a CTA walks many row blocks, keeps one table or two, or has row groups without a layer of their own: the same bits where
nothing is rotated.  With rotation the two reach a table entry from other fp64 starts by other numbers of steps: after n steps
(at most T) the angles agree to n 2^-53, so a share of n 2^-28 of the fp32 entries is rounded the other way, off by 2^-24.  A
sum of eight such rows then moves by 2^-24 of its terms and changes its bf16 (a spacing of 2^-8) once in 2^15 times, to the
neighbour unless the terms cancel: 8 T 2^-28 2^-15, below 1e-7 of the entries, are expected to differ, and ten times that is
allowed."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,G,H_kv,d_h,base", [
    (40003, 4, 4, 128, 10000.0),     # blocks of 32 rows without cosines, 64 with
    (40003, 1, 2, 128, 500000.0),    # more row groups than layers: blocks of 64 rows for both
    (50001, 3, 2, 64, 10000.0),
    (20001, 2, 16, 128, 10000.0),
    (30007, 2, 8, 128, 0.0),         # no rotation
    (13, 1, 1, 64, 10000.0),
])
def test_same_landmarks(T, G, H_kv, d_h, base):
    from paper_2503_18893_b200 import xkv
    g = torch.Generator(device="cuda").manual_seed(T)
    n_c = -(-T // 8)
    keys = torch.randn((1, G, T, H_kv * d_h), generator=g, device="cuda").to(torch.bfloat16)
    lm = [torch.full((1, G, H_kv, n_c, d_h), float("nan"), dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    mc = torch.empty((G, 1, H_kv, n_c), dtype=torch.float32, device="cuda")
    xkv.xkv_build_landmarks(keys, lm[0], G=G, batch=1, T=T, H_kv=H_kv, d_h=d_h, rope_base=base)
    xkv.xkv_build_landmarks(keys, lm[1], G=G, batch=1, T=T, H_kv=H_kv, d_h=d_h, rope_base=base, min_cos=mc)
    if base == 0:
        assert torch.equal(lm[0].view(torch.int16), lm[1].view(torch.int16))
    else:
        a, b = lm[0].double(), lm[1].double()
        assert int((a != b).sum()) <= 1e-6 * a.numel()
        assert ((a - b).abs() <= 2.0 ** -7 * a.abs() + 2.0 ** -20 * a.abs().max()).all()
    # the last chunk of one head, which may be ragged: its mean and its cosines in fp64
    x = keys[0, G - 1, 8 * (n_c - 1):, :d_h].double()
    if base > 0:
        half = d_h // 2
        at = torch.arange(8 * (n_c - 1), T, dtype=torch.float64, device="cuda")[:, None] * base ** (-torch.arange(half, device="cuda", dtype=torch.float64) / half)
        x = torch.cat([x[:, :half] * at.cos() - x[:, half:] * at.sin(), x[:, half:] * at.cos() + x[:, :half] * at.sin()], 1)
    mean = x.mean(0)
    assert (lm[1][0, G - 1, 0, -1].double() - mean).abs().max() <= 2.0 ** -8 * mean.abs().max()
    cos = (x @ mean / (x.norm(dim=1) * mean.norm())).min()
    assert abs(mc[G - 1, 0, 0, -1].item() - cos.item()) <= 32 * 2.0 ** -24   # sums of 16 terms per lane, folds, roots, a quotient
