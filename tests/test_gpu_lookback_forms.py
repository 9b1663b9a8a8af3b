"""Every form of the bounded look-back wait (64-bit and 32-bit words by one thread,
64-bit words by a whole warp): exact sums at lengths around the warp form's 32
words, an inclusive word ends the walk, and an unpublished word with a small poll
limit gives up with DG_ERR_TIMEOUT and the words walked before it.  And the
passes over 64-bit words, which a large capacity selects, give the same lists."""
from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2503_18402_gb300 import capi, synth  # noqa: E402
from paper_2503_18402_gb300.raster import Rasterizer, make_camera  # noqa: E402

pytestmark = pytest.mark.gpu

FORMS = [(0, 4, 1), (1, 4, 1), (2, 1, 0)]  # form, stride, column


def _probe(words, form, stride, digit, max_polls):
    """words: (state, count) of each tile."""
    dt, shift = (np.uint32, 30) if form == 1 else (np.uint64, 62)
    w = np.full((len(words) + 1, stride), 0x7777, dtype=dt)
    for t, (st, c) in enumerate(words):
        w[t, digit] = dt((st << shift) | c)
    look = torch.from_numpy(w.view(np.int32 if form == 1 else np.int64)).cuda()
    out = torch.full((1,), -1, dtype=torch.int64, device="cuda")
    err = torch.full((1,), 123, dtype=torch.int32, device="cuda")
    capi.dg_lookback_probe_form(look, len(words), stride, digit, max_polls, form, out, err)
    torch.cuda.synchronize()
    return int(out.item()), int(err.item())


@pytest.mark.parametrize("form,stride,digit", FORMS)
@pytest.mark.parametrize("n", [0, 1, 3, 4, 5, 31, 32, 33, 63, 64, 65, 100])
def test_sums_inclusive_words_and_give_up(n, form, stride, digit):
    rng = np.random.default_rng(n)
    top = (1 << 23) if form == 1 else (1 << 55)
    c = [int(x) for x in rng.integers(0, top, n)]
    agg = [(1, x) for x in c]
    first_inc = [(2, c[0])] + agg[1:] if n else []
    assert _probe(first_inc, form, stride, digit, 0) == (sum(c), 0)
    assert _probe(agg, form, stride, digit, 0) == (sum(c), 0)  # (every word is there, none inclusive)
    for at in sorted({0, n // 2, n - 1} & set(range(n))):
        # an inclusive word stops the walk, whatever lies before it
        words = [(0, 0)] * at + [(2, c[at])] + agg[at + 1:]
        assert _probe(words, form, stride, digit, 0) == (sum(c[at:]), 0)
        # a word that is never published
        words = first_inc[:at] + [(0, 0)] + agg[at + 1:]
        for polls in (0, 1, 50):
            assert _probe(words, form, stride, digit, polls) == (sum(c[at + 1:]), capi.DG_ERR_TIMEOUT)


def test_form_arguments():
    t = torch.zeros(8, dtype=torch.int64, device="cuda")
    e = torch.zeros(1, dtype=torch.int32, device="cuda")
    for args in ((t, 1, 4, 0, 0, 3), (t, 1, 4, 0, 0, -1), (t, 1, 4, 0, 0, 2), (t, -1, 1, 0, 0, 2),
                 (t, 1, 4, 0, (1 << 20) + 1, 1)):
        with pytest.raises(capi.DashGSError) as ex:
            capi.dg_lookback_probe_form(*args, t, e)
        assert ex.value.status == capi.DG_ERR_ARG


def test_a_capacity_of_2_30_pairs_takes_64_bit_words():
    P, W, H, B, cap = 20000, 700, 400, 8, 1 << 30
    cam = make_camera(np.asarray(synth.look_at(np.array([0.0, -3.0, 0.0])), np.float32).reshape(-1),
                      synth.intrinsics(W, H, 45.0), W, H)
    g = synth.random_gaussians(P, 3)
    g[:, 3:6] -= 1.5
    prm = torch.from_numpy(np.ascontiguousarray(g.T.astype(np.float32))).cuda()
    rz = Rasterizer("cuda", capi.raster_opts(tile=B))
    fr = rz.forward(prm, P, cam)
    want, ranges = rz.gid[: fr.M].clone(), rz.ranges.clone()
    need = capi.dg_bin_workspace_size(P, 1, cap)
    if torch.cuda.mem_get_info()[0] < need + 4 * cap + (8 << 30):
        pytest.skip("needs about 30 GB of device memory")
    ws = torch.empty(need, dtype=torch.uint8, device="cuda")
    gid = torch.empty(cap, dtype=torch.int32, device="cuda")
    capi.dg_bin_count(rz.depth, rz.tiles, P, 1, ws, need, cap, rz.M_dev)
    capi.dg_bin_sort(rz.feat, rz.radius, P, cam, 1, B, ws, need, cap, gid, rz.ranges, rz.status)
    assert int(rz.status.item()) == 0 and int(rz.M_dev.item()) == fr.M > 20000
    assert torch.equal(gid[: fr.M], want) and torch.equal(rz.ranges, ranges)
    del ws, gid
    torch.cuda.empty_cache()
