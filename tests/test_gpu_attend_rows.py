"""Reconstruct+attend where the rows of a tile are, and where they are not, the eight positions of whole landmark chunks in
their order (the key epilogue then shares a row among four lanes, or takes a row per lane), for one to sixteen query heads
per KV head and both head widths, against the oracle."""
import numpy as np
import pytest

from paper_2503_18893_b200 import synth
from tests import _cases as C

pytestmark = pytest.mark.gpu
T, ROWS = 1205, 301                     # a ragged last chunk; two tiles and a bit


def _rows(mode, rng):
    chunks = np.sort(rng.choice(T // 8, ROWS // 8, replace=False))
    whole = (chunks[:, None] * 8 + np.arange(8)).reshape(-1)
    if mode == "whole":                 # ... and the five rows of the last chunk
        return np.concatenate([whole, np.arange(T - 5, T)])
    if mode == "shifted":               # eight rows side by side that straddle two chunks
        return whole[:-8] + 3
    if mode == "shuffled":              # one coarse rotary row, positions out of order
        return np.concatenate([rng.permutation(c) for c in whole.reshape(-1, 8)])
    if mode == "repeated":
        return np.repeat(whole[::8], 8)
    mixed = whole.copy()                # only the second 32 rows are out of order
    mixed[32:64] = rng.permutation(mixed[32:64])
    return mixed


def _check(mode, d_h, n_rep, G, H_kv, batch):
    rng = np.random.default_rng(4100 + n_rep + d_h)
    s = synth.config(1, T=T, k=512, G=G, H_kv=H_kv, H_q=H_kv * n_rep, d_h=d_h, batch=batch, r_k=96, r_v=72, seed=4100 + n_rep)
    inp = C.case_from_factors(s)
    lists = [_rows(mode, rng) for _ in range(G * batch * H_kv)]
    idx = np.stack([np.pad(r, (0, ROWS - len(r)), constant_values=-1) for r in lists]).reshape(G, batch, H_kv, ROWS).astype(np.int32)
    cnt = np.array([len(r) for r in lists], dtype=np.int32).reshape(G, batch, H_kv)
    g = C.GpuCase(s, inp)
    gout, glse = g.attend(idx, cnt, 0)
    assert g.status() == (0, 0)
    _, _, oout, olse = C.oracle_step(s, inp, 0, sel_idx=idx, sel_cnt=cnt)
    assert C.rel_err(gout, oout) <= 2e-2
    # the weights are bf16 in the sum as in the product: 2^-9 of it at most, and as much again for the logits
    np.testing.assert_allclose(glse, olse, atol=2.0 ** -8)
    g.close()


@pytest.mark.parametrize("d_h,n_rep", [(128, 1), (128, 4), (128, 5), (128, 8), (128, 9), (128, 16), (64, 3), (64, 7), (64, 16)])
@pytest.mark.parametrize("mode", ["whole", "shifted", "shuffled", "repeated", "mixed"])
def test_rows_in_and_out_of_chunk_order(mode, d_h, n_rep):
    _check(mode, d_h, n_rep, G=2, H_kv=2, batch=1)


@pytest.mark.parametrize("d_h,n_rep", [(128, 2), (128, 4), (64, 1), (64, 4)])
@pytest.mark.parametrize("mode", ["whole", "mixed"])
def test_two_tiles_and_more_per_sm(mode, d_h, n_rep):
    _check(mode, d_h, n_rep, G=4, H_kv=8, batch=4)         # 384 tiles
