"""FP16 first pass at the sizes where its launches change: a chunk's block pairs
split into groups (fewer chunks than SMs, at least 32 blocks) and the update's
loads issued ahead (from 48 warps of 16 rows per SM), with the checks of
test_gpu_kernels."""
import pytest

from tests import test_gpu_kernels as K

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nb", [(1, 32), (1025, 33), (9000, 90), (40_000, 47), (155_648, 32), (155_647, 65)])
def test_gram_in_groups(n, nb):
    K.test_block_gram_f16_matches_fp64_product_of_the_fp16_basis(n, nb)


@pytest.mark.parametrize("n,nb,nnew", [(116_720, 7, 2), (116_736, 1, 2), (116_737, 6, 2), (116_737, 9, 0), (120_001, 12, 2)])
def test_update_with_loads_ahead(n, nb, nnew):
    K.test_block_update_f16old_matches_fp64_product(n, nb, nnew)
