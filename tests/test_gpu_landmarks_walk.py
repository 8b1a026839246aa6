"""Landmarks of the default chunk where a CTA walks many row blocks and carries the rotation from one to the next, against
fp64 with bounds from the operation counts (the shapes of the other tests end within a CTA's first or second block)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,G,H_kv,d_h,base", [
    (40003, 1, 32, 128, 500000.0),       # one chunk per block: 17 blocks a CTA
    (131072, 2, 8, 128, 10000.0),        # four chunks per block
    (150001, 2, 4, 64, 10000.0),         # eight chunks per block and row groups on other layers
    (40003, 1, 32, 128, 0.0),            # no rotation
])
def test_many_blocks_per_cta(T, G, H_kv, d_h, base):
    from paper_2503_18893_b200 import xkv
    g = torch.Generator(device="cuda").manual_seed(T)
    n_c, half = -(-T // 8), d_h // 2
    common = torch.randn((G, n_c, H_kv * d_h), generator=g, device="cuda").repeat_interleave(8, 1)[:, :T]
    keys = (common + 0.5 * torch.randn((G, T, H_kv * d_h), generator=g, device="cuda")).to(torch.bfloat16).unsqueeze(0)
    del common
    lm = torch.empty((1, G, H_kv, n_c, d_h), dtype=torch.bfloat16, device="cuda")
    mc = torch.empty((G, 1, H_kv, n_c), dtype=torch.float32, device="cuda")
    xkv.xkv_build_landmarks(keys, lm, G=G, batch=1, T=T, H_kv=H_kv, d_h=d_h, rope_base=base, min_cos=mc)
    rows = torch.full((n_c, 1), 8.0, device="cuda", dtype=torch.float64)
    rows[-1] = T - 8 * (n_c - 1)
    pad = torch.zeros((8 * n_c - T, d_h), device="cuda", dtype=torch.float64)
    chunks = lambda x: torch.cat([x, pad]).view(n_c, 8, d_h)
    if base > 0:
        theta = torch.tensor(base, dtype=torch.float64, device="cuda") ** (-torch.arange(half, device="cuda", dtype=torch.float64) / half)
        angle = torch.arange(T, device="cuda", dtype=torch.float64)[:, None] * theta
        c, s = angle.cos(), angle.sin()
    for l, h in {(0, 0), (G - 1, H_kv - 1), (0, H_kv // 2)}:
        x = keys[0, l, :, h * d_h:(h + 1) * d_h].double()
        size = x.abs()
        if base > 0:
            x1, x2 = x[:, :half], x[:, half:]
            size = torch.cat([x1.abs() + x2.abs()] * 2, 1)
            x = torch.cat([x1 * c - x2 * s, x2 * c + x1 * s], 1)
        x = chunks(x)
        mean = x.sum(1) / rows
        # a term: table entry, product, difference; then at most eight sums and the factor 1 / rows (itself rounded)
        bound = 13 * 2.0 ** -24 * chunks(size).sum(1) / rows
        got = lm[0, l, h].double()
        assert torch.all(got >= (mean - bound).to(torch.bfloat16).double()) and torch.all(got <= (mean + bound).to(torch.bfloat16).double())
        cos = (x * mean[:, None]).sum(2) / (x.norm(dim=2) * mean.norm(dim=1)[:, None]).clamp_min(1e-300)
        cos[-1, int(rows[-1]):] = 2.0
        # sums of 16 terms per lane in eight steps, three or two folds; both factors rounded; two norms, two roots, a quotient
        assert (mc[l, 0, h].double() - cos.min(1)[0]).abs().max() <= 32 * 2.0 ** -24
