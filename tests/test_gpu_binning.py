"""Pair lists of the binning against a plain numpy construction, at the sizes
where the segmented radix passes can go wrong: grids whose tile key fits one
digit, grids with several column digits (more than 256 tiles per row), one row
or column of tiles, views of different sizes with culled records and views that
see nothing, tied depths, and both tile sizes of the passes (few and many
items).  Everything is a whole number, so lists and ranges must be equal."""
import numpy as np
import pytest

import torch

from paper_2503_18402_gb300 import capi, synth
from paper_2503_18402_gb300.raster import Rasterizer, make_camera

pytestmark = pytest.mark.gpu


def expected(feat, depth, radius, tiles, P, sizes, B):
    """gid and ranges: per view, the pairs (tile, depth bits, record) in lexicographic order."""
    gid, ranges = [], []
    start = 0
    for v, (W, H) in enumerate(sizes):
        r = slice(v * P, (v + 1) * P)
        TX, TY = -(-W // B), -(-H // B)
        f, rad, tl = feat[r], radius[r].astype(np.int64), tiles[r]
        vis = np.nonzero(tl > 0)[0]
        u, w = np.floor(f[vis, 0]).astype(np.int64), np.floor(f[vis, 1]).astype(np.int64)
        x0, x1 = np.clip((u - rad[vis]) // B, 0, TX), np.clip((u + rad[vis]) // B + 1, 0, TX)
        y0, y1 = np.clip((w - rad[vis]) // B, 0, TY), np.clip((w + rad[vis]) // B + 1, 0, TY)
        mask = f[vis, 9:11].copy().view(np.uint32).astype(np.uint64)
        mask = mask[:, 0] | (mask[:, 1] << np.uint64(32))
        tile, rec = [], []
        for dy in range(int((y1 - y0).max(initial=0))):
            for dx in range(int((x1 - x0).max(initial=0))):
                inside = (y0 + dy < y1) & (x0 + dx < x1)
                if dy < 8 and dx < 8:
                    bit = (mask >> np.uint64(8 * dy + dx)) & np.uint64(1)
                    inside &= (mask == 0) | (bit == 1)
                else:
                    inside &= mask == 0
                k = np.nonzero(inside)[0]
                tile.append((y0[k] + dy) * TX + x0[k] + dx)
                rec.append(vis[k])
        tile = np.concatenate(tile) if tile else np.zeros(0, np.int64)
        rec = np.concatenate(rec) if rec else np.zeros(0, np.int64)
        assert len(tile) == int(tl[vis].sum())
        key = depth[r].view(np.uint32)[rec]
        o = np.lexsort((rec, key, tile))
        gid.append(rec[o] + v * P)
        cnt = np.bincount(tile, minlength=TX * TY)
        end = np.cumsum(cnt)
        rg = np.stack([end - cnt, end], 1) + start
        rg[cnt == 0] = 0
        ranges.append(rg)
        start += len(tile)
    return np.concatenate(gid), np.concatenate(ranges)


CASES = [
    # P, sizes, tile, tight, distance of the cameras (0: the last view looks away)
    (1, [(64, 64)], 16, 0),
    (33, [(8, 8)], 8, 1),                       # one tile
    (700, [(500, 8)], 8, 1),                    # one row of tiles
    (700, [(8, 500)], 8, 0),                    # one column
    (900, [(300, 260)], 1, 0),                  # 300 tiles per row: two column digits, two row digits
    (4097, [(2100, 300)], 8, 1),                # 263 tiles per row
    (5000, [(103, 68)], 8, 1),                  # key of one digit
    (20000, [(309, 205), (64, 64), (155, 103)], 8, 1),
    (30001, [(120, 80)] * 5, 16, 0),
    (311297, [(400, 300)], 8, 1),               # just above the small passes' item count
    (150000, [(618, 411), (97, 33), (309, 205)], 8, 1),
]


@pytest.mark.parametrize("P,sizes,tile,tight", CASES)
def test_lists_equal_the_numpy_construction(P, sizes, tile, tight):
    g = synth.random_gaussians(P, 77 + P)
    g[:, 3:6] -= 1.5 if P > 1000 else 0.0
    g[:, 0:3] = np.round(g[:, 0:3] * 64.0) / 64.0   # tied depths
    rng = np.random.default_rng(P)
    cams = []
    for v, (W, H) in enumerate(sizes):
        d = 3.0 + 0.5 * v
        eye = np.array([0.0, -d, 0.0])
        target = (0.0, 0.0, 0.0)
        if len(sizes) > 1 and v == 1:
            target = (0.0, -2.0 * d, 0.0)           # this view sees nothing
        vm = synth.look_at(eye, target)
        cams.append(make_camera(np.asarray(vm, np.float32).reshape(-1), synth.intrinsics(W, H, 45.0), W, H))
    prm = torch.from_numpy(np.ascontiguousarray(g.T.astype(np.float32))).cuda()
    V = len(sizes)
    rz = Rasterizer("cuda", capi.raster_opts(tile=tile, tight_bins=tight))
    rz._ensure_records(V * P)
    capi.dg_project(prm, P, P, cams, V, rz.opts, rz.feat, rz.depth, rz.radius, rz.tiles, rz.clamp)
    M = int(rz.tiles[: V * P].sum())
    n_tiles = sum(-(-W // tile) * -(-H // tile) for W, H in sizes)
    feat, depth = rz.feat.cpu().numpy(), rz.depth.cpu().numpy()
    want_gid, want_ranges = expected(feat, depth, rz.radius.cpu().numpy(), rz.tiles.cpu().numpy(), P, sizes, tile)
    assert len(want_gid) == M
    # exact capacity, then a capacity that takes the passes' other tile size
    for cap in sorted({max(M, 1), M + int(rng.integers(1, 5000)), max(M, 400000)}):
        ws = torch.randint(0, 255, (capi.dg_bin_workspace_size(P, V, cap),), dtype=torch.uint8, device="cuda")
        gid = torch.full((cap + 7,), -5, dtype=torch.int32, device="cuda")
        ranges = torch.full((n_tiles, 2), -1, dtype=torch.int32, device="cuda")
        status = torch.full((1,), 9, dtype=torch.int32, device="cuda")
        Md = torch.full((1,), -1, dtype=torch.int64, device="cuda")
        capi.dg_bin_count(rz.depth, rz.tiles, P, V, ws, ws.numel(), cap, Md)
        capi.dg_bin_sort(rz.feat, rz.radius, P, cams, V, tile, ws, ws.numel(), cap, gid, ranges, status)
        assert int(Md.item()) == M and int(status.item()) == 0
        got = gid.cpu().numpy()
        np.testing.assert_array_equal(got[:M], want_gid)
        assert (got[M:] == -5).all()
        np.testing.assert_array_equal(ranges.cpu().numpy(), want_ranges)


def test_records_that_do_not_match_the_counted_tiles_are_refused():
    """Phase 2 with the radii of another projection: the pairs do not add up to
    phase 1's count, so nothing is emitted and the status says so."""
    P, W, H = 3000, 200, 120
    g = synth.random_gaussians(P, 5)
    vm = synth.look_at(np.array([0.0, -4.0, 0.0]))
    cam = make_camera(np.asarray(vm, np.float32).reshape(-1), synth.intrinsics(W, H, 45.0), W, H)
    prm = torch.from_numpy(np.ascontiguousarray(g.T.astype(np.float32))).cuda()
    rz = Rasterizer("cuda", capi.raster_opts(tile=8))
    fr = rz.forward(prm, P, cam)
    other = torch.clamp(rz.radius - 1, min=0)
    capi.dg_bin_count(rz.depth, rz.tiles, P, 1, rz.ws, rz.ws.numel(), rz.M_cap, rz.M_dev)
    capi.dg_bin_sort(rz.feat, other, P, cam, 1, 8, rz.ws, rz.ws.numel(), rz.M_cap, rz.gid, rz.ranges, rz.status)
    assert int(rz.status.item()) == capi.DG_ERR_CUDA
    assert int(rz.ranges.abs().sum()) == 0 and fr.M > 0
