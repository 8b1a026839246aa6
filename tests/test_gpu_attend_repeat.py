"""Rows gathered by asynchronous copies reach the tensor core whole: two handles of the same shape and other bases take turns, so
that what a ring slot held before belongs to the other one, and every call returns the bits of the first.  (An order that is
missing shows here by chance at most; the order itself is the fence behind the wait for a slot pair.)"""
import numpy as np
import pytest
import torch

from paper_2503_18893_b200 import synth
from tests import _cases as C

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("over", [
    dict(T=4096, k=4096, G=4, H_kv=8, H_q=32, d_h=128, r_k=512, r_v=512),     # several tiles per CTA
    dict(T=2048, k=1024, G=2, H_kv=2, H_q=8, d_h=64, r_k=64, r_v=64),         # one tile per CTA, one slab and padding
    dict(T=3001, k=3001, G=1, H_kv=4, H_q=28, d_h=128, r_k=328, r_v=200),     # ragged slabs and rows
], ids=["many", "few", "ragged"])
def test_every_call_returns_the_same_bits(over):
    cases = []
    for seed in (3, 4):
        s = synth.config(1, seed=seed, **over)
        inp = C.case_from_factors(s)
        g = C.GpuCase(s, inp)
        idx, cnt = g.select(0)
        out, _ = g.attend(idx, cnt, 0)
        _, _, oout, _ = C.oracle_step(s, inp, 0, sel_idx=idx, sel_cnt=cnt, problems=[(0, 0, 0)])
        assert C.rel_err(out[0, 0, :s.n_rep], oout[0, 0, :s.n_rep]) <= 2e-2
        cases.append((g, torch.as_tensor(idx).cuda(), torch.as_tensor(cnt).cuda(), torch.as_tensor(out)))
    got = [torch.empty((50, *out.shape), dtype=torch.bfloat16, device="cuda") for *_, out in cases]
    for i in range(50):
        for (g, idx, cnt, _), o in zip(cases, got):
            g.xkv.xkv_sr_reconstruct_attend(g.grp, 0, g.shape.G, g.inp.q[0], idx, cnt, idx.shape[-1], o[i], None)
    torch.cuda.synchronize()
    for (g, _, _, out), o in zip(cases, got):
        assert np.array_equal(C.f32(o), np.broadcast_to(out.numpy(), o.shape))
        assert g.status() == (0, 0)
        g.close()
