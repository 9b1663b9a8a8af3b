"""Lists of a binning that reports an error are empty, so that passes launched
behind it read nothing."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2503_18402_gb300 import capi, synth  # noqa: E402
from paper_2503_18402_gb300.raster import Rasterizer, make_camera  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H", [(200, 120), (2100, 300)])
def test_a_mask_outside_the_grid_leaves_no_lists(W, H):
    """A record whose mask has as many tiles as were counted, but below the last
    tile row: the pair counts agree, the keys do not fit the grid."""
    P, B = 3000, 8
    g = synth.random_gaussians(P, 5)
    g[:, 3:6] -= 1.5
    cam = make_camera(np.asarray(synth.look_at(np.array([0.0, -4.0, 0.0])), np.float32).reshape(-1),
                      synth.intrinsics(W, H, 45.0), W, H)
    prm = torch.from_numpy(np.ascontiguousarray(g.T.astype(np.float32))).cuda()
    rz = Rasterizer("cuda", capi.raster_opts(tile=B, tight_bins=1))
    fr = rz.forward(prm, P, cam)
    feat, rad, tiles = (x.cpu().numpy() for x in (rz.feat[:P], rz.radius[:P], rz.tiles[:P]))
    y0 = np.clip((np.floor(feat[:, 1]).astype(np.int64) - rad) // B, 0, None)
    masked = feat[:, 9:11].copy().view(np.uint32).any(1)
    pick = np.nonzero(masked & (tiles > 0) & (tiles <= 8) & (y0 + 7 >= -(-H // B)))[0]
    assert len(pick)
    i = int(pick[0])
    bad = rz.feat.clone()
    hi = np.array([0, ((1 << int(tiles[i])) - 1) << 24], np.uint32)  # bits of the mask's eighth row
    bad[i, 9:11] = torch.from_numpy(hi.view(np.float32).copy()).cuda()
    capi.dg_bin_count(rz.depth, rz.tiles, P, 1, rz.ws, rz.ws.numel(), rz.M_cap, rz.M_dev)
    capi.dg_bin_sort(bad, rz.radius, P, cam, 1, B, rz.ws, rz.ws.numel(), rz.M_cap, rz.gid, rz.ranges, rz.status)
    assert int(rz.status.item()) == capi.DG_ERR_CUDA
    assert int(rz.ranges.abs().sum()) == 0 and fr.M > 0
    # the next call with matching records is whole again
    capi.dg_bin_count(rz.depth, rz.tiles, P, 1, rz.ws, rz.ws.numel(), rz.M_cap, rz.M_dev)
    capi.dg_bin_sort(rz.feat, rz.radius, P, cam, 1, B, rz.ws, rz.ws.numel(), rz.M_cap, rz.gid, rz.ranges, rz.status)
    r = rz.ranges.cpu().numpy().view(np.uint32).astype(np.int64)
    assert int(rz.status.item()) == 0 and int((r[:, 1] - r[:, 0]).sum()) == fr.M


def test_the_rasterizer_raises_for_a_failed_binning():
    """A status word that a failed binning left is raised by the next frame and by
    check(); a capacity overflow is not, and a frame that binned clears it."""
    P, W, H = 500, 64, 48
    cam = make_camera(np.asarray(synth.look_at(np.array([0.0, -4.0, 0.0])), np.float32).reshape(-1),
                      synth.intrinsics(W, H, 45.0), W, H)
    prm = torch.from_numpy(np.ascontiguousarray(synth.random_gaussians(P, 5).T.astype(np.float32))).cuda()
    rz = Rasterizer("cuda", capi.raster_opts(tile=8))
    rz.check()
    want = rz.forward(prm, P, cam).img.clone()
    rz.check()
    for code in (capi.DG_ERR_TIMEOUT, capi.DG_ERR_CUDA):
        rz.status.fill_(code)
        with pytest.raises(capi.DashGSError) as e:
            rz.check()
        assert e.value.status == code
        with pytest.raises(capi.DashGSError) as e:
            rz.forward(prm, P, cam)
        assert e.value.status == code
        assert torch.equal(rz.forward(prm, P, cam).img, want)  # the frame before this one binned
    rz.status.fill_(capi.DG_ERR_CAPACITY)
    rz.check()
    assert torch.equal(rz.forward(prm, P, cam).img, want)
    rz.status.fill_(capi.DG_ERR_CUDA)
    big = torch.cat([prm, prm], 1)
    with pytest.raises(capi.DashGSError):  # also when the record buffers grow
        rz.forward(big, 2 * P, cam)
