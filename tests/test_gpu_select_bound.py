"""Selection from tensor-core scores with an error bound (more than four query heads per KV head, large calls): the index
sets are those of the canonical fp32 scores, bit for bit -- where almost every score ties, where an infinity or a NaN makes
the bound useless, at ragged tile edges, with and without the top-k's filter, for every number of keys and threads."""
import numpy as np
import pytest
import torch

from oracle import xkv_oracle as O
from paper_2503_18893_b200 import synth, workload
from tests import _cases as C

pytestmark = pytest.mark.gpu

#        d_h  H_kv n_rep G  B  T       k      (problems * ceil(T / 8) * n_rep >= 5 * 2^17, or just below it)
SHAPES = [(128, 4, 5, 4, 1, 65536, 2048),      # n_c = 8192: 512 threads, filter of one group a thread
          (128, 2, 7, 2, 2, 131072, 4096),     # n_c = 16384
          (64, 2, 8, 2, 1, 262144, 8000),      # n_c = 32768: keys read twice
          (128, 1, 16, 2, 2, 100003, 12000),   # two groups of heads; ragged last chunk, last tile; two groups a thread
          (64, 4, 9, 2, 2, 40009, 19000),      # no multiple of four chunks; no filter
          (128, 8, 6, 4, 4, 8 * 65, 24),       # a tile of one row per problem; (below the line: the canonical scan)
          (128, 8, 7, 4, 8, 8 * 513, 333)]     # 256 problems, nine tiles, the last of one row


def _inputs(shape, mode, seed):
    d_h, H_kv, n_rep, G, B, T, k = shape
    n_c = -(-T // 8)
    lm = synth.normal(synth.stream_key(seed, 91), (B, G, H_kv, n_c, d_h))
    q = synth.normal(synth.stream_key(seed, 92), (1, G, B, H_kv * n_rep, d_h))
    if mode == "ties":                         # a handful of distinct scores: thousands of chunks at the cut
        gen = torch.Generator().manual_seed(seed)
        lm, q = torch.sign(lm), torch.sign(q) * (torch.rand(q.shape, generator=gen) < 0.1)
    if mode == "grid":                         # half-integers: many exact ties, spread out
        lm, q = torch.round(lm * 2) / 2, torch.round(q)
    if mode == "spike":                        # one element a thousand times the others: a wide band
        lm[..., 3, 5] = 3000.0
    lm, q = lm.to(torch.bfloat16), q.to(torch.bfloat16)
    if mode == "inf":
        lm[..., 11, 0] = float("inf")
    if mode == "nan":
        lm[..., 11, 1] = float("nan")
        q[..., 2, 3] = float("nan")
    return lm, q


@pytest.mark.parametrize("mode", ["normal", "ties", "grid", "spike", "inf", "nan"])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "-".join(map(str, s)))
def test_index_sets_are_those_of_the_canonical_scores(shape, mode):
    d_h, H_kv, n_rep, G, B, T, k = shape
    n_c, seed = -(-T // 8), 8100
    lm, q = _inputs(shape, mode, seed)
    s = synth.config(1, T=T, k=k, G=G, H_kv=H_kv, H_q=H_kv * n_rep, d_h=d_h, batch=B, c=8, r_k=8, r_v=8, seed=seed)
    A = torch.zeros((B, T, 8), dtype=torch.bfloat16)
    Bm = torch.zeros((B, G, 8, H_kv * d_h), dtype=torch.bfloat16)
    g = C.GpuCase(s, workload.GroupInputs(A, A.clone(), Bm, Bm.clone(), lm, q))
    k_cap = -(-k // 8) * 8
    idx = torch.full((G, B, H_kv, k_cap), -7, dtype=torch.int32, device="cuda")
    cnt = torch.full((G, B, H_kv), -7, dtype=torch.int32, device="cuda")
    idx2, cnt2 = idx.clone(), cnt.clone()
    g.xkv.xkv_sr_select(g.grp, 0, G, g.inp.q[0], k, idx, cnt)
    # the call without a handle keeps the canonical scan
    g.xkv.xkv_sr_select_static(G=G, batch=B, T=T, H_kv=H_kv, H_q=H_kv * n_rep, d_h=d_h, landmarks=g.inp.landmarks, layer_begin=0,
                               layer_end=G, q=g.inp.q[0], k=k, sel_idx=idx2, sel_cnt=cnt2)
    torch.cuda.synchronize()
    assert g.status() == (0, 0)
    assert torch.equal(cnt, cnt2) and torch.equal(idx, idx2)
    if mode in ("normal", "ties"):
        gi, gc, qf, lf = idx.cpu().numpy(), cnt.cpu().numpy(), C.f32(q[0]), C.f32(lm)
        for l, b, h in ((0, 0, 0), (G - 1, B - 1, H_kv - 1)):
            rows = O.sr_select(qf[l, b, h * n_rep:(h + 1) * n_rep], lf[b, l, h], k, 8, T, None)
            assert gc[l, b, h] == len(rows)
            np.testing.assert_array_equal(gi[l, b, h, :len(rows)], rows)
    g.close()
