"""Landmarks of the default chunk at the edges of the kernel's split: one to 512 chunks side by side in a CTA, row groups
that take different layers, row blocks that end inside the context, a context shorter than one chunk."""
import pytest

from tests.test_gpu_landmarks import test_landmarks_min_cos_and_outliers as check

pytestmark = pytest.mark.gpu

CASES = [
    ("row_groups_over_layers", dict(T=1043, H_kv=1, H_q=4, d_h=64, batch=2), 5, 10000.0),
    ("more_groups_than_layers", dict(T=64, H_kv=2, H_q=4, d_h=64), 3, 10000.0),
    ("one_chunk_at_a_time", dict(T=201, H_kv=32, H_q=32, d_h=128), 4, 500000.0),
    ("four_chunks", dict(T=2500, H_kv=8, H_q=32, d_h=128, G=3), 7, 10000.0),
    ("no_rope", dict(T=777, H_kv=4, H_q=8, d_h=128), 2, 0.0),
    ("one_row", dict(T=1, H_kv=2, H_q=4, d_h=128), 1, 10000.0),
    ("one_chunk", dict(T=8, H_kv=2, H_q=4, d_h=64), 1, 10000.0),
]


@pytest.mark.parametrize("name,over,n_out,rope_base", CASES, ids=[c[0] for c in CASES])
def test_chunk8(name, over, n_out, rope_base):
    check(name, over, n_out, rope_base)
