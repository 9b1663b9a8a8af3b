"""Pair lists of grids one tile wide and more than 256 tiles high, whose keys have
no column digit, and of views whose columns and rows together exceed 31 bits,
against the plain numpy construction."""
import pytest

pytest.importorskip("torch")

from tests.test_gpu_binning import test_lists_equal_the_numpy_construction as _check  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P,sizes,tile,tight", [
    (1500, [(8, 2056)], 8, 1),                      # 257 rows
    (1500, [(8, 2056)], 8, 0),
    (3000, [(8, 4000)], 8, 1),
    (9000, [(5, 4000)], 8, 0),
    (2000, [(16, 4200)], 16, 0),
    (1200, [(1, 300)], 1, 0),
    (1200, [(8, 2300), (8, 2300), (7, 2600)], 8, 1),
    (900, [(8, 2056), (8, 64), (17, 40)], 8, 1),    # another view has columns
    (30, [(65536, 1), (64, 64), (1, 65536)], 1, 0),  # 32 bits of columns and rows
])
def test_narrow_grids(P, sizes, tile, tight):
    _check(P, sizes, tile, tight)
