"""The gather from codes at ranks of fewer groups than a slot pair has lanes for (a row of one to three groups), over whole
contexts: results only.  (What a lane beyond the rank fetches is never used, so a read past the row would not show here; that
every lane stays inside the row is checked in test_host_headers.py.)"""
import pytest

from tests.test_gpu_quant import test_decode_step_from_quantised_bases as check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits", [4, 3])
@pytest.mark.parametrize("name,over", [
    ("r32_whole", dict(T=520, k=520, d_h=128, r_k=32, r_v=32)),
    ("r32_r96", dict(T=777, k=777, d_h=64, r_k=32, r_v=96)),
    ("r64_r288", dict(T=1024, k=1024, d_h=128, r_k=64, r_v=288, batch=2)),
])
def test_few_groups(name, over, bits):
    check(name, over, bits)
