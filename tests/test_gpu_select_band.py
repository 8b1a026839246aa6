"""Selection from tensor-core scores with an error bound where the band around the cut could grow: elements and channels far
above the rest, zeros, equal scores, sums that cancel, a neighbouring problem that is not finite.  Index sets are those of the
call without a handle (canonical scores), for whole windows and for one layer of several, with and without outlier chunks."""
import numpy as np
import pytest
import torch

from paper_2503_18893_b200 import synth, workload
from tests import _cases as C

pytestmark = pytest.mark.gpu

#        d_h  H_kv n_rep G  B  n_c    k_ch   (problems * n_c * n_rep >= 5 * 2^17, for one layer too)
SHAPES = [(128, 4, 7, 3, 6, 4097, 256),        # the last tile of a problem holds one row, the others are the next problem's
          (128, 4, 16, 2, 3, 4000, 3990),      # no filter, nearly everything taken
          (64, 4, 9, 2, 2, 16385, 300),        # keys read twice
          (64, 8, 5, 2, 3, 6000, 700)]


def _fill(mode, lm, q, k_ch=256):
    if mode == "cluster":                      # two hundred scores around the cut that differ in their last bits only
        G, B = q.shape[1:3]
        H_kv, n_c, d_h = lm.shape[2:]
        g = torch.Generator().manual_seed(5)
        q[..., :16] = 2.0 ** -10 * torch.sign(q[..., :16])
        first = q[0].view(G, B, H_kv, -1, d_h)[:, :, :, :1].transpose(0, 1).to(torch.bfloat16).float()     # head 0 of every group
        lm *= 0.1
        above, below = k_ch - 100, min(k_ch + 100, n_c)
        lm[..., :above, :] = first
        lm[..., above:below, :] = 0.5 * first
        # one unit in the last place of the first sixteen elements, which weigh 2^-10
        lm[..., above:below, :16] += 2.0 ** -7 * torch.randint(-1, 2, lm[..., above:below, :16].shape, generator=g)
        lm[...] = lm[..., torch.randperm(n_c, generator=g), :].clone()
    elif mode == "element":
        lm[..., 3, 5] = 3000.0
    elif mode == "channel":
        lm[..., 7] = 100.0 + lm[..., 7]
        q[..., 7] = 1.0
    elif mode == "rows":                       # one row in a hundred a hundred times as long
        lm[..., ::100, :] *= 100.0
    elif mode == "zero queries":
        q.zero_()
    elif mode == "zero landmarks":             # all but the first hundred: the cut lies among zeros
        lm[..., 100:, :] = 0.0
    elif mode == "equal":                      # one score for all chunks, but for a few
        lm[...] = lm[..., :1, :].clone()
        lm[..., 17, :] *= -1.0
    elif mode == "tiny":                       # products around and below the smallest fp32 numbers
        lm *= 2.0 ** -126
        q *= 2.0 ** -20
    elif mode == "cancel":                     # scores are what is left of terms a thousand times as large
        half = lm.shape[-1] // 2
        lm[..., half:] = 30.0 * torch.sign(lm[..., half:])
        lm[..., half + 1::2] = -lm[..., half::2]
        q[..., half:] = 30.0
    elif mode == "neighbour":                  # the second layer's first head lies behind the first layer's last one
        lm[:, 1] = float("nan")


@pytest.mark.parametrize("mode", ["cluster", "element", "channel", "rows", "zero queries", "zero landmarks", "equal", "tiny", "cancel",
                                  "neighbour"])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "-".join(map(str, s)))
def test_index_sets_are_those_of_the_canonical_scores(shape, mode):
    d_h, H_kv, n_rep, G, B, n_c, k_ch = shape
    T, k = n_c * 8 - 3, k_ch * 8
    lm = synth.normal(synth.stream_key(8300, 91), (B, G, H_kv, n_c, d_h))
    q = synth.normal(synth.stream_key(8300, 92), (1, G, B, H_kv * n_rep, d_h))
    _fill(mode, lm, q, k_ch)
    lm, q = lm.to(torch.bfloat16), q.to(torch.bfloat16)
    s = synth.config(1, T=T, k=k, G=G, H_kv=H_kv, H_q=H_kv * n_rep, d_h=d_h, batch=B, c=8, r_k=8, r_v=8, seed=8300)
    A = torch.zeros((B, T, 8), dtype=torch.bfloat16)
    Bm = torch.zeros((B, G, 8, H_kv * d_h), dtype=torch.bfloat16)
    g = C.GpuCase(s, workload.GroupInputs(A, A.clone(), Bm, Bm.clone(), lm, q))
    x, q = g.xkv, g.inp.q[0]
    want = torch.full((G, B, H_kv, k), -7, dtype=torch.int32, device="cuda")
    want_cnt = torch.full((G, B, H_kv), -7, dtype=torch.int32, device="cuda")
    for l in range(G):                         # (its scratch is fixed: a layer at a time)
        x.xkv_sr_select_static(G=G, batch=B, T=T, H_kv=H_kv, H_q=H_kv * n_rep, d_h=d_h, landmarks=g.inp.landmarks,
                               layer_begin=l, layer_end=l + 1, q=q, k=k, sel_idx=want, sel_cnt=want_cnt)
    idx, cnt = torch.full_like(want, -9), torch.full_like(want_cnt, -9)
    x.xkv_sr_select(g.grp, 0, G, q, k, idx, cnt)
    assert torch.equal(idx, want) and torch.equal(cnt, want_cnt)
    idx.fill_(-9), cnt.fill_(-9)
    x.xkv_sr_select(g.grp, 1, 2, q, k, idx, cnt)
    assert torch.equal(idx[1], want[1]) and torch.equal(cnt[1], want_cnt[1])
    others = [l for l in range(G) if l != 1]
    assert (idx[others] == -9).all() and (cnt[others] == -9).all()
    # outlier chunks, in reach and out of it, join the sets
    n_out = 5
    out = torch.randint(-2, n_c + 2, (G, B, H_kv, n_out), generator=torch.Generator().manual_seed(1), dtype=torch.int32).cuda()
    x.xkv_group_set_outliers(g.grp, out, n_out)
    idx = torch.full((G, B, H_kv, k + 8 * n_out), -9, dtype=torch.int32, device="cuda")
    x.xkv_sr_select(g.grp, G - 1, G, q, k, idx, cnt)
    assert g.status() == (0, 0)
    sets, wn, cn, on = idx.cpu().numpy(), want.cpu().numpy(), cnt.cpu().numpy(), out.cpu().numpy()
    for b in range(B):
        for h in range(H_kv):
            more = [j for j in on[G - 1, b, h] if 0 <= j < n_c]
            rows = np.concatenate([wn[G - 1, b, h], np.array([j * 8 + i for j in more for i in range(8)], dtype=np.int32)])
            rows = np.unique(rows[(rows >= 0) & (rows < T)])
            assert cn[G - 1, b, h] == len(rows)
            np.testing.assert_array_equal(sets[G - 1, b, h, :len(rows)], rows)
    g.close()


def _time(x, grp, layers, q, k, idx, cnt):
    ts = []
    for _ in range(15):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record()
        for _ in range(8):
            x.xkv_sr_select(grp, 0, layers, q, k, idx, cnt)
        b.record()
        torch.cuda.synchronize()
        ts.append(a.elapsed_time(b))
    return sorted(ts)[7]


@pytest.mark.parametrize("mode", ["element", "channel", "rows", "zero queries", "zero landmarks", "neighbour"])
def test_the_band_does_not_decide_the_time(mode):
    """A selection over unusual landmarks takes about as long as one over Gaussian ones, as a scan of canonical scores does."""
    from paper_2503_18893_b200 import xkv as x
    G, B, H_kv, n_rep, d_h, n_c, k = 4, 8, 4, 7, 128, 8193, 2048
    g = torch.Generator().manual_seed(1)
    T = n_c * 8
    A = torch.zeros((B, T, 8), dtype=torch.bfloat16, device="cuda")
    Bm = torch.zeros((B, G, 8, H_kv * d_h), dtype=torch.bfloat16, device="cuda")
    base = torch.randn((B, G, H_kv, n_c, d_h), generator=g)
    q0 = torch.randn((G, B, H_kv * n_rep, d_h), generator=g)
    idx = torch.empty((G, B, H_kv, k), dtype=torch.int32, device="cuda")
    cnt = torch.empty((G, B, H_kv), dtype=torch.int32, device="cuda")
    times = []
    for m in ("normal", mode):
        lm, q = base.clone(), q0.clone()
        _fill(m, lm, q)
        grp = x.create_from_tensors(A, A, Bm, Bm, lm.to(torch.bfloat16).cuda(), H_kv=H_kv, H_q=H_kv * n_rep, k_max=k)
        times.append(_time(x, grp, 1 if mode == "neighbour" else G, q.to(torch.bfloat16).cuda(), k, idx, cnt))
        x.xkv_group_destroy(grp)
    assert times[1] <= 2.0 * times[0], times
