"""The tile-8 render passes at list lengths around their steps (entry pairs,
batches of 32, groups of 16, the ring of 48 staged entries) with pixels that stop
at the first or the second entry of a pair, whole and in chunks, against the
FP64 oracle fed the same records."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_2503_18402_gb300 import capi, synth  # noqa: E402
from paper_2503_18402_gb300.raster import Rasterizer  # noqa: E402
from tests import _gpu as G  # noqa: E402

pytestmark = pytest.mark.gpu


def _scene(n, opaque, seed):
    g = synth.random_gaussians(n, seed)
    g[:, 0:2] *= 0.3
    g[:, 3:6] = np.random.default_rng(seed).normal(-1.4, 0.4, size=(n, 3))
    g[:, 10] += 2.5 if opaque else -3.0
    return g


@pytest.mark.parametrize("opaque", [False, True])
@pytest.mark.parametrize("split", [-1, 5, 32])
@pytest.mark.parametrize("n", [1, 2, 15, 16, 17, 31, 32, 33, 47, 48, 49, 64, 65, 97, 161])
def test_list_lengths(n, split, opaque):
    W, H, bg = 13, 11, (0.2, 0.4, 0.1)
    g = _scene(n, opaque, 900 + n)
    cam = synth.camera_cfg0(W, H, 4.0)
    k = oracle.consts()
    rz = Rasterizer("cuda", capi.raster_opts(tile=8, bg=bg, split_len=split), ppt_fwd=1, ppt_bwd=1)
    buf = torch.zeros((59, n + 3), device="cuda")
    buf[:, :n] = G.gpu_params(g)
    params = buf[:, :n]
    fr = rz.forward(params, n, G.gpu_camera(cam), examined=True)
    torch.cuda.synchronize()
    feat = G.np_(rz.feat[:n]).astype(np.float64)[:, :9]
    gid = G.np_(rz.gid[: fr.M]).view(np.uint32)
    ranges = G.np_(rz.ranges[:4]).view(np.uint32)
    orf = oracle.render_fwd(feat, W, H, 8, gid, ranges, G.f32(bg), k)
    assert np.abs(G.np_(fr.img) - orf["img"]).max() <= 1e-5
    np.testing.assert_array_equal(G.np_(fr.last), orf["last"])
    np.testing.assert_array_equal(G.np_(rz.examined), orf["examined"])
    np.testing.assert_array_equal(G.np_(rz.blended), orf["blended"])
    dL = (np.random.default_rng(n).normal(size=(3, H, W)) / (3 * H * W)).astype(np.float32)
    grads = torch.zeros_like(buf)[:, :n]
    rz.backward(params, fr, torch.from_numpy(dL).cuda(), grads)
    og2 = oracle.render_bwd(feat, W, H, 8, gid, ranges, G.f32(bg), k, dL.astype(np.float64))
    ok, worst, nbad = G.grad_close(G.np_(rz.grad2d[:n])[:, :9], og2)
    assert ok, (worst, nbad)
