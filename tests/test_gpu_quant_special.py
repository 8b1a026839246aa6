"""The quantiser on scalars that are no numbers and on infinities: a NaN takes no part in its group's minimum and maximum
and gets code 0 (what clip(rint(q), 0, top) gives where the clip is fmin(fmax(q, 0), top)), the other scalars get the codes
they have without it; a group with an infinity has an infinite scale and only codes 0."""
import numpy as np
import pytest
import torch

from oracle import xkv_oracle as O
from paper_2503_18893_b200 import synth
from tests import _cases as C
from tests.test_gpu_quant import _meta, _unpack, _unpack3

pytestmark = pytest.mark.gpu


def _quantise(x, bits):
    from paper_2503_18893_b200 import xkv
    rows, cols = x.shape
    codes, meta = xkv.xkv_quantize_rtn(x.cuda(), bits)
    torch.cuda.synchronize()
    if bits == 4:
        return (_unpack(codes.cpu().numpy(), cols), *_meta(meta.cpu().numpy().reshape(rows, cols // 32)))
    return _unpack3(codes.cpu().numpy(), cols)


@pytest.mark.parametrize("bits", [4, 3])
@pytest.mark.parametrize("rows,cols", [(3, 32), (65, 160)])
def test_nan_scalars(rows, cols, bits):
    u = synth.normal(synth.stream_key(79, rows, cols, bits), (rows, cols))
    x = u.to(torch.bfloat16)
    holes = (u * 1000).round() % 5 == 0                      # about every fifth scalar
    holes.view(-1, 32)[0] = False
    holes.view(-1, 32)[0, 3::9] = True
    holes.view(-1, 32)[:, 7] = False                         # every group keeps a number
    x[holes] = float("nan")
    g = C.f32(x).reshape(-1, 32)
    filled = np.where(np.isnan(g), np.nanmin(g, axis=1, keepdims=True), g).reshape(rows, cols)
    oc, osc, oz = O.rtn_quantize(filled, bits)
    gc, gs, gz = _quantise(x, bits)
    np.testing.assert_array_equal(gs, osc.reshape(gs.shape))
    np.testing.assert_array_equal(gz, oz.reshape(gz.shape))
    np.testing.assert_array_equal(gc, oc.reshape(gc.shape))
    assert np.all(gc[holes.numpy()] == 0)


@pytest.mark.parametrize("bits", [4, 3])
def test_infinities_and_groups_of_nan(bits):
    x = synth.normal(synth.stream_key(80, bits), (5, 64)).to(torch.bfloat16)
    x[0, 5], x[1, 40], x[2, 0] = float("inf"), float("-inf"), float("inf")
    x[2, 9] = float("nan")
    x[3, 32:] = float("nan")
    plain = synth.normal(synth.stream_key(80, bits), (5, 64)).to(torch.bfloat16)
    oc, _, _ = O.rtn_quantize(C.f32(plain), bits)
    want = oc.reshape(10, 32).copy()
    for group in (0, 3, 4, 7):
        want[group] = 0
    gc, gs, gz = _quantise(x, bits)
    np.testing.assert_array_equal(gc.reshape(10, 32), want)
    assert np.all(np.isinf(gs.reshape(-1)[[0, 3, 4]])) and np.isneginf(gz.reshape(-1)[3])
