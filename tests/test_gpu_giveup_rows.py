"""The reconstruct+attend kernel gives up with copies of its own outstanding (the injection is on the host, see
test_gpu_giveup.py): the matrices are loaded, the rows that share their barriers never come.  The key stream makes up the
arrivals it owes, the loader stays for its bytes, the call returns, and the next one is right."""
import numpy as np
import pytest

from paper_2503_18893_b200 import synth
from tests import _cases as C

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r,T,k,bits", [
    (64, 1024, 128, 16),             # one slab and padding, one pair requested
    (512, 4096, 4096, 16),           # the loader waits for a release that does not come
    (512, 4096, 4096, 4),
])
def test_the_kernel_stays_for_its_copies_and_the_handle_recovers(r, T, k, bits):
    s = synth.config(1, T=T, k=k, G=2, H_kv=8, H_q=32, d_h=128, r_k=r, r_v=r)
    inp = C.case_from_factors(s)
    g = C.GpuCase(s, inp)
    x = g.xkv
    if bits != 16:
        ck, mk = x.xkv_quantize_rtn(g.inp.A_k, bits)
        cv, mv = x.xkv_quantize_rtn(g.inp.A_v, bits)
        x.xkv_group_set_quantized_bases(g.grp, ck, mk, cv, mv, bits)
    idx, cnt = g.select(0)
    want, want_lse = g.attend(idx, cnt, 0)
    x.xkv_debug_set_fault_injection(g.grp, x.XKV_INJECT_FUSED_NO_ROWS)
    g.attend(idx, cnt, 0)                                      # returns after the shortened limit; output unspecified
    st, flags = g.status()
    assert st == x.XKV_ERR_TIMEOUT and flags & x.XKV_FLAG_TIMEOUT
    x.xkv_debug_set_fault_injection(g.grp, 0)
    got, got_lse = g.attend(idx, cnt, 0)
    assert g.status() == (0, 0)
    assert np.array_equal(got, want) and np.array_equal(got_lse, want_lse)
    g.close()
