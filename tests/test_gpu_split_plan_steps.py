"""The one-block split plan at the tile counts where its threads take one, two, four
and eight consecutive tiles, compared as in test_gpu_split_plan."""
import pytest

pytest.importorskip("torch")

from tests.test_gpu_split_plan import test_plan_tile_counts as _check  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [8, 16, 32])
@pytest.mark.parametrize("more", [False, True])
def test_tiles_per_thread(rows, more):
    _check([(1024, 8 * rows)] + [(8, 8)] * more)  # 1024, 2048, 4096 tiles, or one more
