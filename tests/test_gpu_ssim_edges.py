"""The loss kernels at the edges of their strips (128 columns), rounds (2 rows)
and segments (16, 32 and 64 rows, by the size of the batch), against the oracle,
and with a workspace made for a larger image."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2503_18402_gb300 import capi  # noqa: E402
from tests.test_gpu_ssim import _check  # noqa: E402

pytestmark = pytest.mark.gpu


def _pair(rng, W, H):
    x = rng.random((3, H, W))
    return x, np.clip(x + 0.2 * rng.normal(size=x.shape), 0, 1)


@pytest.mark.parametrize("H", [3, 4, 16, 17, 33])
@pytest.mark.parametrize("W", [5, 123, 127, 128, 129, 133, 256, 257])
def test_strip_and_segment_edges(W, H):
    x, y = _pair(np.random.default_rng(W * 100 + H), W, H)
    _check([x], [y])


@pytest.mark.parametrize("V,W,H", [(16, 257, 130), (16, 513, 260), (3, 60, 40), (2, 129, 66)])
def test_longer_segments_and_view_counts(V, W, H):
    """16 views take 32-row and 64-row segments; two and three views share the
    summing block's warps differently."""
    rng = np.random.default_rng(V + W)
    pairs = [_pair(rng, W + v % 2, H - v % 3) for v in range(V)]
    _check([p[0] for p in pairs], [p[1] for p in pairs])


def test_workspace_of_a_larger_image_serves_smaller_ones():
    for big in [(1237, 822), (100, 32448), (4000, 64)]:
        need = capi.dg_ssim_workspace_size([big])
        for w in (big[0], max(1, big[0] - 1), big[0] // 2 + 1, 1):
            for h in (big[1], max(1, big[1] - 1), big[1] // 2 + 1, 1):
                assert capi.dg_ssim_workspace_size([(w, h)]) <= need
