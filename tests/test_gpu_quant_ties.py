"""The quantiser where a quotient lies on or beside a half-integer, and at the ends of its pieces and ranges, against the
oracle bit for bit."""
import numpy as np
import pytest
import torch

from oracle import xkv_oracle as O
from paper_2503_18893_b200 import synth
from tests import _cases as C
from tests.test_gpu_quant import _meta, _unpack, _unpack3

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits", [4, 3])
@pytest.mark.parametrize("rows,cols", [(1, 32), (33, 96), (129, 256)])     # below, beside and beyond 1024 pieces of a block
@pytest.mark.parametrize("kind", ["ties", "wide", "tiny", "mixed"])
def test_codes_at_half_integers(rows, cols, bits, kind):
    from paper_2503_18893_b200 import xkv
    top = 2 ** bits - 1
    u = synth.normal(synth.stream_key(78, rows, cols, bits), (rows, cols))
    if kind == "ties":          # steps of a half on a grid of unit scale: every other quotient is a tie
        x = (u.abs() * 97).floor() % (2 * top + 1) * 0.5
        x.view(-1, 32)[:, 0] = 0.0
        x.view(-1, 32)[:, 1] = float(top)
    elif kind == "wide":        # exponents far apart: differences with all 24 bits
        x = u * torch.exp2((u * 1000).round() % 20 - 12)
    elif kind == "tiny":        # subnormal scales take the division
        x = u * 1e-38
    else:                       # constant groups, signed zeros
        x = (u * 4).round() * 0.25
        x.view(-1, 32)[::3] = -0.0
    x = x.to(torch.bfloat16)
    codes, meta = xkv.xkv_quantize_rtn(x.cuda(), bits)
    oc, osc, oz = O.rtn_quantize(C.f32(x), bits)
    torch.cuda.synchronize()
    if bits == 4:
        gc, (gs, gz) = _unpack(codes.cpu().numpy(), cols), _meta(meta.cpu().numpy().reshape(rows, cols // 32))
    else:
        gc, gs, gz = _unpack3(codes.cpu().numpy(), cols)
    np.testing.assert_array_equal(gs, osc.reshape(gs.shape))
    np.testing.assert_array_equal(gz, oz.reshape(gz.shape))
    np.testing.assert_array_equal(gc, oc.reshape(gc.shape))
    if kind == "tiny":          # the oracle's dequantiser rounds normal values only
        return
    back = xkv.xkv_dequantize_rtn(codes, meta, bits)
    want = O.rtn_dequantize(oc, osc, oz)
    np.testing.assert_array_equal(C.f32(back.cpu()), np.asarray(want, dtype=np.float32).reshape(rows, cols))
