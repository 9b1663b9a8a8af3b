"""The projection adjoint of several views in one call against the sum of one-view
calls, at the view counts, degrees and sizes where the kernel's form changes: 2D
gradients loaded one view ahead or in place, stored gradients and the fused Adam
update (against dg_adam_step on the stored ones)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2503_18402_gb300 import capi, synth  # noqa: E402
from paper_2503_18402_gb300.raster import make_camera  # noqa: E402

pytestmark = pytest.mark.gpu

LR = [1e-3] * 59


def _setup(P, V, degree):
    W, H = 96, 64
    cams = [make_camera(np.asarray(c["viewmat"], np.float32).reshape(-1), c["intr"], W, H)
            for c in synth.ring_cameras(V, W, H, 4.0, 5)]
    gen = torch.Generator("cuda")
    gen.manual_seed(P + V)
    prm = torch.from_numpy(np.ascontiguousarray(synth.random_gaussians(min(P, 20000), 9).T.astype(np.float32))).cuda()
    prm = prm.repeat(1, -(-P // prm.shape[1]))[:, :P].contiguous()
    prm += 0.01 * torch.randn(prm.shape, generator=gen, device="cuda")
    opts = capi.raster_opts(tile=8, sh_degree=degree)
    feat = torch.empty((V * P, capi.FEAT_FLOATS), device="cuda")
    depth = torch.empty(V * P, device="cuda")
    radius, tiles = (torch.empty(V * P, dtype=torch.int32, device="cuda") for _ in range(2))
    clamp = torch.empty(V * P, dtype=torch.uint8, device="cuda")
    capi.dg_project(prm, P, P, cams, V, opts, feat, depth, radius, tiles, clamp)
    g2 = torch.randn((V * P, capi.FEAT_FLOATS), generator=gen, device="cuda")
    return prm, cams, opts, radius, clamp, g2


@pytest.mark.parametrize("degree", [0, 1, 2, 3])
@pytest.mark.parametrize("P,V", [(701, 2), (701, 5), (701, 6), (701, 8), (701, 12), (701, 16), (100001, 2), (100001, 5),
                                 (312501, 8)])
def test_views_in_one_call(P, V, degree):
    prm, cams, opts, radius, clamp, g2 = _setup(P, V, degree)
    total = torch.empty_like(prm)
    capi.dg_project_bwd(prm, P, P, cams, V, opts, radius, clamp, g2, total)
    want, mag = torch.zeros_like(prm, dtype=torch.float64), torch.zeros_like(prm, dtype=torch.float64)
    one = torch.empty_like(prm)
    for v in range(V):
        s = slice(v * P, (v + 1) * P)
        capi.dg_project_bwd(prm, P, P, cams[v], 1, opts, radius[s], clamp[s].clone(), g2[s], one)
        want += one.double()
        mag += one.double().abs()
    # some hundred roundings of 6e-8, of the terms' size (the row's, where terms cancel)
    tol = 1e-4 * mag + 1e-5 * mag.amax(1, keepdim=True)
    assert ((total.double() - want).abs() <= tol).all()
    # fused: the stored gradient and dg_adam_step's update of it
    m, v = 1e-3 * torch.ones_like(prm), 1e-4 * torch.ones_like(prm)
    p1, m1, v1, p2, m2, v2 = prm.clone(), m.clone(), v.clone(), prm.clone(), m.clone(), v.clone()
    stored = torch.empty_like(prm)
    capi.dg_project_bwd_adam(p1, P, P, cams, V, opts, radius, clamp, g2, stored, m1, v1, LR, 0.9, 0.999, 1e-15, 7)
    assert ((stored.double() - want).abs() <= tol).all()
    capi.dg_adam_step(p2, stored, m2, v2, P, P, LR, 0.9, 0.999, 1e-15, 7)
    for a, b in ((p1, p2), (m1, m2), (v1, v2)):
        assert ((a - b).abs() <= 1e-6 * b.abs() + 1e-9).all()
