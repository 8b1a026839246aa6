"""The short-list top-k at the edges of its thread counts and items, with no tie, with a few tied keys at the threshold, and
with more tied keys than are ranked directly, against the oracle bit for bit."""
import numpy as np
import pytest
import torch

from oracle import xkv_oracle as O
from paper_2503_18893_b200 import synth, workload
from tests import _cases as C

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_c", [1, 5, 31, 2047, 2048, 2052, 4097, 8192, 16384, 16388, 32767, 32768])
@pytest.mark.parametrize("ties", ["none", "few", "many"])
def test_selection_at_the_edges(n_c, ties):
    d_h, T = 64, n_c * 8 - 3                                     # a ragged last chunk
    g = torch.Generator().manual_seed(n_c)
    lm = torch.zeros((1, 1, 1, n_c, d_h))
    v = torch.randn(n_c, generator=g)
    if ties == "few":
        v = (v * 64).round() / 64
    elif ties == "many":
        v = (v > 1.0).float() - (v < -1.0).float()
    lm[..., 0] = v
    q = torch.zeros((1, 1, 1, 1, d_h))
    q[..., 0] = 1.0
    lm, q = lm.to(torch.bfloat16), q.to(torch.bfloat16)
    ks = sorted({1, 8, n_c, 4 * n_c, max(1, n_c // 32) * 8, T - 1 if T > 1 else 1, n_c * 8})
    s = synth.config(1, T=T, k=max(ks), G=1, H_kv=1, H_q=1, d_h=d_h, r_k=8, r_v=8)
    A, B = torch.zeros((1, T, 8), dtype=torch.bfloat16), torch.zeros((1, 1, 8, d_h), dtype=torch.bfloat16)
    case = C.GpuCase(s, workload.GroupInputs(A, A.clone(), B, B.clone(), lm, q))
    for k in ks:
        idx, cnt = case.select(0, k=k)
        rows = O.sr_select(C.f32(q[0, 0, 0]), C.f32(lm[0, 0, 0]), k, 8, T, None)
        assert cnt[0, 0, 0] == len(rows), k
        np.testing.assert_array_equal(idx[0, 0, 0, :len(rows)], rows)
        assert np.all(idx[0, 0, 0, len(rows):] == -1)
    assert case.status() == (0, 0)
    case.close()
