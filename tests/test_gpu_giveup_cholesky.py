"""The give-up path of the Cholesky kernels of the factorisation (the injection is on the host, see test_gpu_giveup.py): one
CTA of the first launch skips its arrival at the first grid barrier, the others run out of polls and raise the time-out flag
and the abort word; the launches behind it, which count on arrivals that never came, end at once; the next call is right."""
import pytest
import torch

from paper_2503_18893_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r,q", [(64, 1), (8, 0), (200, 2)])          # 4, 2 and 8 blocks of 32; 4, 3 and 5 launches
def test_cholesky_barrier_wait_runs_out_and_the_next_factorisation_is_fine(r, q):
    from paper_2503_18893_b200 import xkv
    s = synth.config(1, T=2048)
    K, _ = synth.make_kv(s)
    X = torch.cat([K[l] for l in range(s.G)], dim=1).cuda().contiguous()          # (T, G d)
    cfg = xkv.make_clf_config(T=s.T, G=s.G, d=s.d, r=r, oversample=32, power_iters=q)
    l = xkv.xkv_clf_rank_l(cfg)
    omega = synth.normal(synth.stream_key(5, 31), (s.G * s.d, l)).to(torch.bfloat16).cuda()
    ws = torch.empty(xkv.xkv_clf_workspace_bytes(cfg), dtype=torch.uint8, device="cuda")
    A = torch.empty((s.T, r), dtype=torch.bfloat16, device="cuda")
    B = torch.empty((s.G, r, s.d), dtype=torch.bfloat16, device="cuda")
    sig = torch.empty(r, dtype=torch.float32, device="cuda")
    xkv.xkv_debug_set_clf_fault_injection(xkv.XKV_INJECT_CLF_CHOLESKY)
    try:
        xkv.xkv_clf_factorize(cfg, X, omega, ws, A, B, sig)                        # returns: every wait is bounded
        st, flags = xkv.xkv_clf_status(ws)
        assert st == xkv.XKV_ERR_TIMEOUT and flags & xkv.XKV_FLAG_TIMEOUT
    finally:
        xkv.xkv_debug_set_clf_fault_injection(0)
    xkv.xkv_clf_factorize(cfg, X, omega, ws, A, B, sig)
    assert xkv.xkv_clf_status(ws) == (0, 0)
    Xf = X.double()
    V = torch.cat([B[g] for g in range(s.G)], dim=1).double()                      # (r, G d)
    assert (V @ V.T - torch.eye(r, device="cuda")).abs().max() <= 2e-2
    res = float(((Xf - A.double() @ V) ** 2).sum())
    sv = torch.linalg.svdvals(Xf)
    assert res <= 1.25 * float((sv[r:] ** 2).sum())
