"""The landmark scan that scores on the tensor core gives up (its loads are not issued, on the host's demand): the call
returns, the time-out is reported, indices and counts are in range whatever the scores were left as, for budgets up to all but
one chunk and with queries that make the error bound infinite, and the handle works again afterwards."""
import numpy as np
import pytest
import torch

from paper_2503_18893_b200 import synth, workload
from tests import _cases as C

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d_h,n_rep,T,k", [(128, 7, 65536, 2048), (128, 7, 65536, 65536 - 8), (64, 16, 40009, 40009 - 8),
                                           (128, 5, 262144, 262144 - 8)])
def test_scan_with_a_bound_gives_up_and_the_handle_recovers(d_h, n_rep, T, k):
    G, B, H_kv, n_c = 2, 2, 4, -(-T // 8)
    s = synth.config(1, T=T, k=k, G=G, H_kv=H_kv, H_q=H_kv * n_rep, d_h=d_h, batch=B, c=8, r_k=8, r_v=8, seed=8200)
    lm = synth.normal(synth.stream_key(8200, 91), (B, G, H_kv, n_c, d_h)).to(torch.bfloat16)
    q = synth.normal(synth.stream_key(8200, 92), (1, G, B, H_kv * n_rep, d_h)).to(torch.bfloat16)
    A = torch.zeros((B, T, 8), dtype=torch.bfloat16)
    Bm = torch.zeros((B, G, 8, H_kv * d_h), dtype=torch.bfloat16)
    g = C.GpuCase(s, workload.GroupInputs(A, A.clone(), Bm, Bm.clone(), lm, q))
    x, q = g.xkv, g.inp.q[0]
    wild = q.clone()
    wild[..., 5] = float("inf")
    k_ch, k_cap = -(-k // 8), -(-k // 8) * 8
    idx = torch.full((G, B, H_kv, k_cap), -7, dtype=torch.int32, device="cuda")
    cnt = torch.full((G, B, H_kv), -7, dtype=torch.int32, device="cuda")
    good, good_cnt = idx.clone(), cnt.clone()
    ragged = n_c * 8 - T
    for queries in (wild, q):                              # first on a handle that never scored anything, then on old scores
        x.xkv_debug_set_fault_injection(g.grp, x.XKV_INJECT_SCAN_NO_LOAD)
        x.xkv_sr_select(g.grp, 0, G, queries, k, idx, cnt)
        st, flags = g.status()
        assert st == x.XKV_ERR_TIMEOUT and flags & x.XKV_FLAG_TIMEOUT
        gi, gc = idx.cpu().numpy(), cnt.cpu().numpy()
        assert np.all((gc == k_ch * 8) | (gc == k_ch * 8 - ragged))
        for rows, n in zip(gi.reshape(-1, k_cap), gc.reshape(-1)):
            assert rows[0] >= 0 and np.all(np.diff(rows[:n]) > 0) and rows[n - 1] < T and np.all(rows[n:] == -1)
        x.xkv_debug_set_fault_injection(g.grp, 0)
        x.xkv_sr_select(g.grp, 0, G, q, k, idx, cnt)
        x.xkv_sr_select_static(G=G, batch=B, T=T, H_kv=H_kv, H_q=H_kv * n_rep, d_h=d_h, landmarks=g.inp.landmarks, layer_begin=0,
                               layer_end=G, q=q, k=k, sel_idx=good, sel_cnt=good_cnt)
        assert g.status() == (0, 0)
        assert torch.equal(idx, good) and torch.equal(cnt, good_cnt)
    g.close()
