"""Colours that are not finite reach only the pixels that blend them, and through
those only the gradients of the entries these pixels blend, against the FP64
oracle fed the same records: where the oracle is finite the kernels are finite
and close, and where it is not they are not."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_2503_18402_gb300 import capi, synth  # noqa: E402
from paper_2503_18402_gb300.raster import Rasterizer  # noqa: E402
from tests import _gpu as G  # noqa: E402

pytestmark = pytest.mark.gpu


def _same(got, want, tol):
    """Finite in the same places, and there within tol(want)."""
    fin = np.isfinite(want)
    np.testing.assert_array_equal(np.isfinite(got), fin)
    assert (np.abs(got[fin] - want[fin]) <= tol(np.abs(want[fin]))).all()
    return fin


@pytest.mark.parametrize("tile,ppt", [(8, 1), (8, 2), (16, None)])
@pytest.mark.parametrize("split", [-1, 5, 32])
@pytest.mark.parametrize("n", [3, 40, 161])
def test_nonfinite_colours_stay_with_their_pixels(n, split, tile, ppt):
    W, H, bg = 29, 21, (0.2, 0.4, 0.1)
    g = synth.random_gaussians(n, 700 + n)
    rng = np.random.default_rng(n)
    g[:, 0:2] *= 0.6
    g[:, 3:6] = rng.normal(-2.0, 0.4, size=(n, 3))
    for i, (ch, val) in enumerate([(0, np.nan), (1, np.inf), (2, -np.inf)]):  # channels of three Gaussians
        g[(i * n) // 3, 11 + ch] = val
    cam = synth.camera_cfg0(W, H, 4.0)
    k = oracle.consts()
    rz = Rasterizer("cuda", capi.raster_opts(tile=tile, bg=bg, split_len=split), ppt_fwd=ppt, ppt_bwd=ppt)
    params = G.gpu_params(g)
    fr = rz.forward(params, n, G.gpu_camera(cam), examined=True)
    feat = G.np_(rz.feat[:n]).astype(np.float64)[:, :9]
    assert (~np.isfinite(feat[:, 6:9])).any(1).sum() >= 2
    gid = G.np_(rz.gid[: fr.M]).view(np.uint32)
    n_tiles = -(-W // tile) * -(-H // tile)
    ranges = G.np_(rz.ranges[:n_tiles]).view(np.uint32).reshape(-1)
    orf = oracle.render_fwd(feat, W, H, tile, gid, ranges, G.f32(bg), k)
    fin = _same(G.np_(fr.img), orf["img"], lambda a: 1e-5)
    if n > 3:
        assert fin.any() and not fin.all()
    np.testing.assert_array_equal(G.np_(fr.last), orf["last"])
    np.testing.assert_array_equal(G.np_(rz.examined), orf["examined"])
    np.testing.assert_array_equal(G.np_(rz.blended), orf["blended"])
    dL = (rng.normal(size=(3, H, W)) / (3 * H * W)).astype(np.float32)
    rz.backward_render(fr, torch.from_numpy(dL).cuda())
    og2 = oracle.render_bwd(feat, W, H, tile, gid, ranges, G.f32(bg), k, dL.astype(np.float64))
    fin = _same(G.np_(rz.grad2d[:n])[:, :9], og2, lambda a: 1e-4 * a + 1e-6)
    if n > 3:
        assert fin[:, :6].all(1).any() and not fin.all()


@pytest.mark.parametrize("split", [-1, 2])
def test_infinite_opacity_does_not_restart_a_stopped_pixel(split):
    """Records of infinite opacity blend at the clamp.  Behind a wide, a small and a
    second wide entry the pixels under the small one stop at the first of them, the
    others a step later; the stopped ones examine nothing more."""
    W, H, n = 13, 11, 6
    g = synth.random_gaussians(n, 41)
    g[:, 0:2] *= 0.1
    g[:, 3:6] = 0.5
    cam = synth.camera_cfg0(W, H, 4.0)
    gcam = G.gpu_camera(cam)
    k = oracle.consts()
    rz = Rasterizer("cuda", capi.raster_opts(tile=8, split_len=split, tight_bins=0), ppt_fwd=1, ppt_bwd=1)
    fr = rz.forward(G.gpu_params(g), n, gcam)
    order = [int(i) for i in rz.gid[:n]]  # of the first tile, and of all: every record is wide
    for i, o in zip(order, (0.9, 0.98, 0.3) + (float("inf"),) * 3):
        rz.feat[i, :6] = torch.tensor([6.1, 5.2, 1e-4, 0.0, 1e-4, o])
    rz.feat[order[1], :5] = torch.tensor([3.2, 2.7, 1.0, 0.0, 1.0])
    img, T = torch.empty_like(fr.img), torch.empty_like(fr.T)
    last, ex, bl = (torch.empty_like(fr.last) for _ in range(3))
    capi.dg_render_fwd(rz.feat, rz.gid, rz.ranges, gcam, 1, rz.opts_fwd, img, T, last, ex, bl, rz.rws, rz.rws.numel())
    feat = G.np_(rz.feat[:n]).astype(np.float64)[:, :9]
    orf = oracle.render_fwd(feat, W, H, 8, G.np_(rz.gid[: fr.M]).view(np.uint32),
                            G.np_(rz.ranges[:4]).view(np.uint32).reshape(-1), np.zeros(3), k)
    assert set(np.unique(orf["examined"])) == {4, 5}
    np.testing.assert_array_equal(G.np_(last), orf["last"])
    np.testing.assert_array_equal(G.np_(ex), orf["examined"])
    np.testing.assert_array_equal(G.np_(bl), orf["blended"])
    assert np.abs(G.np_(img) - orf["img"]).max() <= 1e-5
