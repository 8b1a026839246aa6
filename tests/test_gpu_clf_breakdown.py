"""Caches on which the Cholesky factorisation breaks down: a NaN, an infinity, nothing but zeros.  The call returns, the flag word
says so (the status is not an error: every kernel ran), no entry of a cache of zeros' factors is other than zero, and the
next call with the same workspace is right."""
import pytest
import torch

from paper_2503_18893_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,N,r,q", [(2048, 256, 64, 2), (300, 192, 24, 0), (5000, 512, 264, 1)])
@pytest.mark.parametrize("what", ["nan", "inf", "zeros"])
def test_breakdown_is_reported_and_the_next_call_is_right(what, T, N, r, q):
    from paper_2503_18893_b200 import xkv
    g = torch.Generator(device="cuda").manual_seed(T)
    rho = r // 2
    X = (torch.randn(T, rho, generator=g, device="cuda") @ torch.randn(rho, N, generator=g, device="cuda") / rho ** 0.5
         + 0.05 * torch.randn(T, N, generator=g, device="cuda")).to(torch.bfloat16)
    bad = X.clone()
    if what == "zeros":
        bad.zero_()
    else:
        bad[T // 3, N // 2] = float(what)
    cfg = xkv.make_clf_config(T=T, G=2, d=N // 2, r=r, oversample=32, power_iters=q)
    l = xkv.xkv_clf_rank_l(cfg)
    omega = synth.normal(synth.stream_key(5, 31), (N, l)).to(torch.bfloat16).cuda()
    ws = torch.empty(xkv.xkv_clf_workspace_bytes(cfg), dtype=torch.uint8, device="cuda")
    A = torch.empty((T, r), dtype=torch.bfloat16, device="cuda")
    B = torch.empty((2, r, N // 2), dtype=torch.bfloat16, device="cuda")
    sig = torch.empty(r, dtype=torch.float32, device="cuda")
    xkv.xkv_clf_factorize(cfg, bad, omega, ws, A, B, sig)
    assert xkv.xkv_clf_status(ws) == (xkv.XKV_OK, xkv.XKV_FLAG_CLF_BREAKDOWN)
    if what == "zeros":
        assert not A.any() and not B.any() and not sig.any()
    xkv.xkv_clf_factorize(cfg, X, omega, ws, A, B, sig)
    assert xkv.xkv_clf_status(ws) == (xkv.XKV_OK, 0)
    Xd, V = X.double(), torch.cat([B[0], B[1]], dim=1).double()
    assert (V @ V.T - torch.eye(r, device="cuda")).abs().max() <= 2e-2
    res = float(((Xd - A.double() @ V) ** 2).sum())
    best = float((torch.linalg.svdvals(Xd)[r:] ** 2).sum())
    assert res <= 1.25 * best + 2e-5 * float((Xd ** 2).sum())       # (the second term: factors in bf16)
