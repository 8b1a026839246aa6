"""Precision of the attention logits: one selected row per problem, rebuilt exactly (one-hot token bases), so that the log-sum
handed back is the row's logit, against fp64."""
import math

import pytest
import torch

from paper_2503_18893_b200 import xkv

pytestmark = pytest.mark.gpu
G, T, R, K = 4, 16384, 64, 128


@pytest.mark.parametrize("bits", [16, 4])
@pytest.mark.parametrize("rows", ["in order", "out of order", "not rotated"])
@pytest.mark.parametrize("d_h,H_kv,n_rep,batch", [
    (128, 8, 1, 1), (128, 8, 4, 1), (128, 4, 7, 4), (128, 4, 16, 2), (64, 8, 4, 1), (64, 8, 8, 2),
    (128, 8, 4, 16), (64, 8, 3, 16),            # two tiles and more per CTA
])
def test_logits_of_single_rows(d_h, H_kv, n_rep, batch, rows, bits):
    g = torch.Generator(device="cuda").manual_seed(4400 + d_h + n_rep)
    H_q, half = H_kv * n_rep, d_h // 2
    rn = lambda *shape: torch.randn(shape, generator=g, device="cuda").to(torch.bfloat16)
    t = torch.arange(T, device="cuda")
    A = torch.zeros((batch, T, R), dtype=torch.bfloat16, device="cuda")
    A[:, t, t // 8 % R] = 1.0
    B, q = rn(batch, G, R, H_kv * d_h), rn(G, batch, H_q, d_h)
    rope_base = 0.0 if rows == "not rotated" else 10000.0
    grp = xkv.create_from_tensors(A, A, B, B, None, H_kv=H_kv, H_q=H_q, k_max=K, rope_base=rope_base)
    if bits != 16:
        codes, meta = xkv.xkv_quantize_rtn(A, bits)
        assert torch.equal(xkv.xkv_dequantize_rtn(codes, meta, bits), A)
        xkv.xkv_group_set_quantized_bases(grp, codes, meta, codes, meta, bits)
    out = torch.empty_like(q)
    lse = torch.empty((G, batch, H_q), dtype=torch.float32, device="cuda")
    theta = 10000.0 ** (-torch.arange(half, device="cuda").double() / half)
    err = []
    for _ in range(8):
        row = torch.randint(0, T // 8, (G, batch, H_kv, 1), generator=g, device="cuda", dtype=torch.int32) * 8
        row += 3 if rows == "out of order" else 0          # position 0 of a tile is not position 0 of a chunk then
        idx = torch.full((G, batch, H_kv, K), -1, dtype=torch.int32, device="cuda")
        idx[..., :1] = row
        xkv.xkv_sr_reconstruct_attend(grp, 0, G, q, idx, torch.ones((G, batch, H_kv), dtype=torch.int32, device="cuda"), K, out, lse)
        p = row.long()
        keys = B.view(batch, G, R, H_kv, d_h).permute(1, 0, 3, 2, 4)                        # G, batch, H_kv, R, d_h
        x = keys.gather(3, (p // 8 % R)[..., None].expand(-1, -1, -1, 1, d_h))[..., 0, :].double()
        p = p if rope_base > 0.0 else 0 * p
        cs, sn = (p.double() * theta).cos(), (p.double() * theta).sin()
        k = torch.cat([x[..., :half] * cs - x[..., half:] * sn, x[..., half:] * cs + x[..., :half] * sn], -1)
        terms = q.view(G, batch, H_kv, n_rep, d_h).double() * k[..., None, :] / math.sqrt(d_h)
        err.append(((lse.view(G, batch, H_kv, n_rep).double() - terms.sum(-1)) / terms.abs().sum(-1)).flatten())
    assert xkv.xkv_group_status(grp) == (0, 0)
    xkv.xkv_group_destroy(grp)
    err = torch.cat(err) * 2.0 ** 24
    # A term carries about ten roundings of 2^-24 (angles of two table entries, rotation, product), independent of the other
    # terms': 10 / sqrt(3) / sqrt(d_h) = 0.5 to 0.7 of 2^-24 sum |q k| if each were as large as it may be; the final sums and the
    # conversion of the log-sum add less than one rounding.  A sum cut off at every one of its steps is off by 1.2 and more, keys
    # of 11 bits by hundreds.
    assert err.square().mean().sqrt() <= 0.7
    assert err.abs().max() <= 7.0
