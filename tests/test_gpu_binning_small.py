"""Pair lists at the edges of the rules that small calls take: grids around 256
tiles (one digit of linear keys), record counts around the one-record-per-thread
kernel's limit and pair capacities around the small pass tiles' limit, against the
plain numpy construction (which also bins with capacities on either side)."""
import pytest

pytest.importorskip("torch")

from tests.test_gpu_binning import test_lists_equal_the_numpy_construction as _check  # noqa: E402

pytestmark = pytest.mark.gpu

REC_LIMIT = 152 * 2 * 1024    # records: one per thread up to here; small depth tiles up to a quarter more


@pytest.mark.parametrize("P,sizes,tile,tight", [
    (3000, [(128, 128)], 8, 1),              # 256 tiles
    (3000, [(129, 128)], 8, 1),              # 272: two digits
    (3000, [(136, 120)], 8, 0),              # 255
    (2000, [(2048, 8)], 8, 1),               # one row of 256
    (2000, [(8, 2048)], 8, 1),               # one column of 256
    (5000, [(64, 64), (8, 8), (127, 90)], 8, 1),
    (256, [(100, 60)], 16, 0),
    (257, [(100, 60)], 16, 1),
    (REC_LIMIT, [(150, 100)], 16, 1),
    (REC_LIMIT * 5 // 16, [(150, 100), (30, 20), (90, 60), (50, 40)], 16, 1),  # at that limit
    (REC_LIMIT * 5 // 4 + 1, [(50, 40)], 16, 0),                               # one above
])
def test_small_grids_and_limits(P, sizes, tile, tight):
    _check(P, sizes, tile, tight)
