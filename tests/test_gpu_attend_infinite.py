"""Rebuilt keys beyond the range of fp32: a row whose logits are minus infinity for every head takes no part in the softmax,
whichever way the key epilogue multiplies (one tile per CTA and several, four query heads and more)."""
import numpy as np
import pytest
import torch

from paper_2503_18893_b200 import synth
from tests import _cases as C

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d_h,n_rep,batch", [(128, 1, 1), (128, 4, 1), (128, 4, 16), (128, 7, 1), (128, 16, 1), (64, 4, 1), (64, 8, 1)])
def test_a_row_whose_logits_are_minus_infinity_drops_out(d_h, n_rep, batch):
    s = synth.config(1, T=1200, k=256, G=2, H_kv=2, H_q=2 * n_rep, d_h=d_h, batch=batch, r_k=96, r_v=72, seed=4300 + n_rep + d_h)
    if batch > 1:                       # two tiles and more per CTA
        s = synth.config(1, T=1200, k=256, G=4, H_kv=8, H_q=8 * n_rep, d_h=d_h, batch=batch, r_k=96, r_v=72, seed=4300)
    inp = C.case_from_factors(s)
    rows = np.sort(np.random.default_rng(4300).choice(s.T // 8, 24, replace=False))[:, None] * 8 + np.arange(8)
    rows = rows.reshape(-1)
    bad = int(rows[77])
    # dimension 0 of row `bad` overflows: rotated it is (x cos, x sin) in dimensions 0 and d_h / 2
    inp.A_k[:, :, 0] = 0.0
    inp.A_k[:, bad, 0] = 3e38
    inp.B_k[:, :, 0] = 0.0
    inp.B_k[:, :, 0, ::d_h] = 2.0
    inp.q[..., 0] = -np.sign(np.cos(bad))
    inp.q[..., d_h // 2] = -np.sign(np.sin(bad))
    P = (s.G, s.batch, s.H_kv)
    idx = np.broadcast_to(rows.astype(np.int32), P + rows.shape).copy()
    cnt = np.full(P, len(rows), dtype=np.int32)
    keep = np.broadcast_to(rows[rows != bad].astype(np.int32), P + (len(rows) - 1,)).copy()
    problems = [(0, 0, 0), (s.G - 1, s.batch - 1, s.H_kv - 1)]
    g = C.GpuCase(s, inp)
    out, lse = g.attend(idx, cnt, 0)
    less_out, less_lse = g.attend(keep, cnt - 1, 0)
    assert g.status() == (0, 0)
    g.close()
    assert np.isfinite(out).all() and np.isfinite(lse).all()
    # the same rows in other tile positions: bf16 weights and outputs
    assert C.rel_err(out, less_out) <= 2e-2
    np.testing.assert_allclose(lse, less_lse, atol=2.0 ** -8)
    _, _, oout, olse = C.oracle_step(s, inp, 0, sel_idx=keep, sel_cnt=cnt - 1, problems=problems)
    for l, b, h in problems:
        hs = slice(h * n_rep, (h + 1) * n_rep)
        assert C.rel_err(out[l, b, hs], oout[l, b, hs]) <= 2e-2
        np.testing.assert_allclose(lse[l, b, hs], olse[l, b, hs], atol=2.0 ** -8)
    assert torch.isfinite(inp.A_k).all()
