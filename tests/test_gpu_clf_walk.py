"""The factorisation and its tensor-core product where a CTA walks several tiles: the operand ring runs on between them, the
accumulators are handed back before a tile is stored.  Whole and ragged tiles, widths of 128, 192 and 256 columns."""
import pytest

from tests.test_gpu_clf import test_tensor_core_product_against_fp64 as check_product
from tests.test_gpu_clf_shapes import test_factors_at_tile_edges as check_factors

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,G,d,r,p", [
    (80001, 1, 256, 96, 32),         # l = 128: 313 tiles of 256 x 128
    (40003, 2, 160, 128, 64),        # l = 192: 157 of 256 x 192
    (40003, 3, 128, 264, 40),        # l = 320: 314, every second one ragged
    (45000, 2, 128, 200, 40),        # l = 256: 176 of 256 x 256
])
def test_factors(T, G, d, r, p):
    check_factors(T, G, d, r, p)


@pytest.mark.parametrize("M,N,K", [(40104, 200, 136), (20000, 520, 64)])
def test_product(M, N, K):
    check_product(M, N, K)
