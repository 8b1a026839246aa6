"""Reconstruct+attend with several tiles per CTA at small ranks: one to four slabs of the reconstruction matrix per tile, so
that the ring of those slabs wraps in every way, against the oracle."""
import numpy as np
import pytest

from paper_2503_18893_b200 import synth
from tests import _cases as C

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r_k", [8, 64, 72, 128, 136, 256])
@pytest.mark.parametrize("over", [dict(H_kv=8, H_q=16, d_h=64), dict(H_kv=4, H_q=28, d_h=128)], ids=["d64", "rep7"])
def test_ring_of_slabs_wraps(r_k, over):
    s = synth.config(1, T=12288, k=12288, G=2, r_k=r_k, r_v=64, **over)     # 96 tiles per problem: 5 to 10 per CTA
    inp = C.case_from_factors(s)
    g = C.GpuCase(s, inp)
    idx, cnt = g.select(0)
    out, lse = g.attend(idx, cnt, 0)
    assert g.status() == (0, 0)
    problems = [(0, 0, 0), (1, 0, s.H_kv - 1)]
    _, _, oout, olse = C.oracle_step(s, inp, 0, sel_idx=idx, sel_cnt=cnt, problems=problems)
    n = s.n_rep
    for l, b, h in problems:
        heads = slice(h * n, (h + 1) * n)
        assert C.rel_err(out[l, b, heads], oout[l, b, heads]) <= 2e-2
        np.testing.assert_allclose(lse[l, b, heads], olse[l, b, heads], atol=2e-2)
    g.close()
