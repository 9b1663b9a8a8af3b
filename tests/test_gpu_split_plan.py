"""The split plan at tile counts around its steps: one tile, a thread's eight
tiles and one more, the last count that one block plans and the first that the
scan kernels plan.  Lists cut at 5 entries (tiles with more chunks than a warp has
lanes) give the uncut lists' last / examined / blended and, to the rounding of the
chunk products, their image: each is within 1e-5 of the exact sum."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2503_18402_gb300 import capi, synth  # noqa: E402
from paper_2503_18402_gb300.raster import Rasterizer  # noqa: E402
from tests import _gpu as G  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [[(8, 8)], [(61, 7)], [(66, 8)], [(250, 130), (8, 8)], [(1024, 512)],
                                   [(1024, 512), (8, 8)]])
def test_plan_tile_counts(sizes):
    n = 3000
    g = synth.random_gaussians(n, 77)
    g[:, 0:2] *= 0.5
    g[:, 10] -= 2.0
    params = G.gpu_params(g)
    cams = [G.gpu_camera(synth.camera_cfg0(w, h, 4.0)) for w, h in sizes]
    out = []
    for split in (-1, 5):
        rz = Rasterizer("cuda", capi.raster_opts(tile=8, bg=(0.1, 0.2, 0.3), split_len=split))
        fr = rz.forward(params, n, cams, examined=True)
        torch.cuda.synchronize()
        m = G.np_(rz.ranges).view(np.uint32)
        out.append([np.concatenate([G.np_(v).ravel() for v in (x if isinstance(x, list) else [x])])
                    for x in (fr.img, fr.last, rz.examined, rz.blended)])
    tiles = sum(-(-w // 8) * -(-h // 8) for w, h in sizes)
    assert int((m[:tiles, 1] - m[:tiles, 0]).max()) > 160
    for a, b in zip(out[0][1:], out[1][1:]):
        np.testing.assert_array_equal(a, b)
    assert np.abs(out[0][0] - out[1][0]).max() <= 2e-5
