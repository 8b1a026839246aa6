"""Rows of whole landmark chunks in another order than ascending, or repeated, cost about what they cost in order: their rotary
rows are staged in shared memory all the same."""
import pytest
import torch

from paper_2503_18893_b200 import xkv

pytestmark = pytest.mark.gpu


def _time(f):
    ts = []
    for _ in range(15):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record()
        for _ in range(8):
            f()
        b.record()
        torch.cuda.synchronize()
        ts.append(a.elapsed_time(b))
    return sorted(ts)[7]


@pytest.mark.parametrize("d_h,H_kv,n_rep,T,r,batch,k", [(128, 8, 4, 65536, 512, 1, 4096), (128, 4, 7, 32768, 256, 4, 2048),
                                                      (128, 2, 16, 32768, 512, 4, 4096), (64, 8, 4, 32768, 256, 4, 4096)])
def test_rows_out_of_order_take_about_the_same_time(d_h, H_kv, n_rep, T, r, batch, k):
    G, H_q = 4, H_kv * n_rep
    g = torch.Generator(device="cuda").manual_seed(4500)
    rn = lambda *shape: torch.randn(shape, generator=g, device="cuda").to(torch.bfloat16)
    A, B, q = rn(batch, T, r), rn(batch, G, r, H_kv * d_h) * 0.05, rn(G, batch, H_q, d_h)
    grp = xkv.create_from_tensors(A, A, B, B, None, H_kv=H_kv, H_q=H_q, k_max=k)
    P = G * batch * H_kv
    chunks = torch.rand((P, T // 8), generator=g, device="cuda").topk(k // 8, dim=1).indices.sort(1).values
    rows = chunks[:, :, None] * 8 + torch.arange(8, device="cuda")
    mixed = rows.gather(2, torch.rand(rows.shape, generator=g, device="cuda").argsort(2))
    cnt = torch.full((G, batch, H_kv), k, dtype=torch.int32, device="cuda")
    out = torch.empty_like(q)
    times = []
    for lst in (rows, mixed, rows[:, :, :1].expand(rows.shape)):
        idx = lst.reshape(G, batch, H_kv, k).int().contiguous()
        times.append(_time(lambda: xkv.xkv_sr_reconstruct_attend(grp, 0, G, q, idx, cnt, k, out, None)))
    assert xkv.xkv_group_status(grp) == (0, 0)
    xkv.xkv_group_destroy(grp)
    assert max(times[1:]) <= 1.25 * times[0], times
