"""Decode steps one behind the other, as a model runs them: each appends a row to the tail, lengthens it and replaces the
queries in place, and nothing waits for the device in between.  The tail's kernel starts ahead of its turn; its results have
to be those of the same steps with a synchronisation after every operation, bit for bit."""
import pytest
import torch

from paper_2503_18893_b200 import synth
from tests import _cases as C

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d_h,by_layer", [(128, False), (128, True), (64, False), (64, True)])
def test_steps_in_a_row_equal_steps_one_at_a_time(d_h, by_layer):
    from paper_2503_18893_b200 import xkv
    s = synth.config(1, T=1024, k=128, d_h=d_h, r_k=64, r_v=64, batch=2)
    g = C.GpuCase(s, C.case_from_factors(s))
    steps, first, cap = 24, 120, 160                          # the tail grows from one split into a second
    gen = torch.Generator(device="cuda").manual_seed(d_h)
    rand = lambda *shape: torch.randn(shape, generator=gen, device="cuda").to(torch.bfloat16)
    all_q, all_k, all_v = rand(steps, s.G, s.batch, s.H_q, d_h), rand(s.G, s.batch, s.H_kv, cap, d_h), rand(s.G, s.batch, s.H_kv, cap, d_h)

    def run(sync):
        wait = torch.cuda.synchronize if sync else (lambda: None)
        q = torch.empty_like(all_q[0])
        tk, tv = torch.full_like(all_k, float("nan")), torch.full_like(all_v, float("nan"))
        tk[..., :first, :], tv[..., :first, :] = all_k[..., :first, :], all_v[..., :first, :]
        length = torch.tensor([first, first - 7], dtype=torch.int32, device="cuda")
        k_cap = -(-s.k // s.c) * s.c
        idx = torch.empty((s.G, s.batch, s.H_kv, k_cap), dtype=torch.int32, device="cuda")
        cnt = torch.empty((s.G, s.batch, s.H_kv), dtype=torch.int32, device="cuda")
        out = torch.empty((s.G, s.batch, s.H_q, d_h), dtype=torch.bfloat16, device="cuda")
        lse = torch.empty((s.G, s.batch, s.H_q), dtype=torch.float32, device="cuda")
        ws = torch.empty(xkv.xkv_tail_workspace_bytes(g.grp, cap), dtype=torch.uint8, device="cuda")
        got = []
        wait()
        for t in range(steps):
            q.copy_(all_q[t]); wait()
            tk[..., first + t, :] = all_k[..., first + t, :]; wait()
            tv[..., first + t, :] = all_v[..., first + t, :]; wait()
            length.add_(1); wait()
            for lo, hi in ([(l, l + 1) for l in range(s.G)] if by_layer else [(0, s.G)]):
                xkv.xkv_sr_select(g.grp, lo, hi, q, s.k, idx, cnt); wait()
                xkv.xkv_sr_reconstruct_attend_tail(g.grp, lo, hi, q, idx, cnt, k_cap, tk, tv, length, cap, ws, out, lse); wait()
            got.append((out.clone(), lse.clone())); wait()
        torch.cuda.synchronize()
        return got

    want, got = run(True), run(False)
    assert g.status() == (0, 0)
    for t in range(steps):
        assert torch.isfinite(got[t][1]).all()
        assert torch.equal(got[t][0].view(torch.int16), want[t][0].view(torch.int16)) and torch.equal(got[t][1], want[t][1]), t
    g.close()
