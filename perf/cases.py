"""What the framework's users have it do, as cases that can be timed and compared.

Training of 3D Gaussian splatting under a resolution and primitive schedule
spends its time in a handful of calls: projection, binning, the two render
passes, the photometric loss, the projection adjoint fused with Adam and, every
100 iterations, densification.  The cases are these calls at the sizes the
training runs have (one full-resolution view of a 2M-Gaussian scene; 16 views
per step of a 480k to 650k-Gaussian model, even or at uneven schedule
resolutions), three whole calls (a full-resolution training step, a replayed
16-view step early in the schedule, a novel view of a 6M-Gaussian scene) and the
smallest differentiable call (1,000 Gaussians, 64x64).

Scenes are textured surfaces plus a background shell, closed at the spacing of
their Gaussians (the layout of ``paper_2503_18402_gb300.synth.textured_scene``,
drawn on the GPU), seen from ring views; the model is a jittered copy of the
scene that its targets are rendered from.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2503_18402_gb300 import capi, synth
from paper_2503_18402_gb300.graphstep import StepGraph
from paper_2503_18402_gb300.raster import Rasterizer, make_camera, rasterize

DEV = "cuda"
LAMBDA = 0.2          # D-SSIM weight of the training loss
LR = [1.6e-5] * 3 + [0.005] * 3 + [0.001] * 4 + [0.025] + [0.0025] * 3 + [0.0025 / 20] * 45
BETA1, BETA2, EPS, STEP = 0.9, 0.999, 1e-15, 1000


def _case(name, kind, P, width, height, views=1, factors="1", record=0, tight=1, tile=8, sh=3):
    c = dict(kind=kind, P=P, width=width, height=height, views=views, factors=factors, record=record, tight=tight,
             tile=tile, sh=sh)
    return dict(name=name, **c) if name else c


def listed():
    full = dict(width=1237, height=822)
    return [
        # the smallest differentiable call: a unit scene under torch.autograd, default options (16x16 tiles)
        _case("raster_1k_64x64", "autograd", 1000, 64, 64, tight=0, tile=16),
        # the plain arm's training step: one full-resolution view, FP32 records, an odd Gaussian count
        _case("step_2m_1237x822", "step", 1999999, **full),
        # the scheduled arm early on: 16 low-resolution views, mixed records, replayed as a CUDA graph
        _case("graph_16v_100k_309x205", "graph", 100000, 309, 205, views=16, record=1),
        # a novel view of the largest scene (evaluation, viewer): forward only
        _case("view_6m_1600x1063", "view", 6000000, 1600, 1063),
        # projection and colour of a 16-view step late in the schedule
        _case("project_16v_480k", "project", 480000, views=16, record=1, **full),
        # pair lists of one full-resolution view of the 2M-Gaussian scene
        _case("bin_2m_1237x822", "bin", 2000000, **full),
        # pair lists of 16 views at uneven schedule resolutions (1237x822 down to 309x205)
        _case("bin_16v_653k_uneven", "bin", 653001, views=16, factors="1,2,3,4", record=1, **full),
        # compositing of the 16-view step, mixed records
        _case("fwd_16v_480k", "fwd", 480000, views=16, record=1, **full),
        # its adjoint
        _case("bwd_16v_480k", "bwd", 480000, views=16, record=1, **full),
        # L1 + D-SSIM of the 16-view step
        _case("loss_16v_1237x822", "loss", 0, views=16, **full),
        # projection adjoint and Adam of the 16-view step
        _case("update_16v_480k", "update", 480000, views=16, record=1, **full),
        # prune, select, clone and split with the Adam moments, every 100 iterations
        _case("densify_480k", "densify", 480000, **full),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["autograd", "step", "graph", "view", "project", "bin", "bin", "fwd", "bwd", "loss", "update",
                       "densify"])
    width = log_int(51, 1600)
    height = max(34, int(width * rng.uniform(0.5, 0.8)))
    views = 1 if kind in ("autograd", "step", "view", "densify") else rng.choice([1, 2, 3, 5, 8, 16])
    views = max(1, min(views, 16000000 // (width * height)))
    P = log_int(1000, min(2000000, 7500000 // views))
    factors = rng.choice(["1", "1", "1,2", "1,2,3,4"]) if views > 1 and width >= 200 else "1"
    record, tight, tile, sh = rng.choice([0, 1]), rng.choice([0, 1, 1]), rng.choice([8, 8, 8, 16]), rng.choice([3, 3, 3, 2, 1, 0])
    if kind == "autograd":
        width, height, P = log_int(32, 160), log_int(32, 160), log_int(500, 20000)
        record, tight = 0, 0
    if kind == "loss":
        P = 0
    if kind == "graph":
        tile = 8
    return _case(None, kind, P, width, height, views, factors, record, tight, tile, sh)


# ------------------------------------------------------------------ inputs
def _sizes(case):
    f = [int(x) for x in case["factors"].split(",")]
    return [(case["width"] // f[v % len(f)], case["height"] // f[v % len(f)]) for v in range(case["views"])]


def _opts(case):
    return capi.raster_opts(tile=case["tile"], sh_degree=case["sh"], record=case["record"], tight_bins=case["tight"])


def _gen(seed):
    g = torch.Generator(DEV)
    g.manual_seed(int(seed))
    return g


def _randn(gen, *shape):
    return torch.randn(shape, generator=gen, device=DEV)


def _rand(gen, *shape):
    return torch.rand(shape, generator=gen, device=DEV)


def _scene(n, seed):
    """[59][n] float32 Gaussians on textured planes and spheres plus a shell."""
    rng, gen = np.random.default_rng(seed), _gen(seed)
    S, lo, hi, n_shell = 400, 0.04, 0.9, n // 10
    u = rng.uniform(size=S)
    size = 1.0 / np.sqrt(1.0 / lo ** 2 - u * (1.0 / lo ** 2 - 1.0 / hi ** 2))
    plane = np.arange(S) % 2 == 0
    area = np.where(plane, (2.0 * size) ** 2, 4.0 * math.pi * size ** 2)
    counts = np.floor((n - n_shell) * area / area.sum()).astype(np.int64)
    counts[np.argsort(-area)[: n - n_shell - counts.sum()]] += 1
    a = rng.normal(size=(S, 3))
    a /= np.linalg.norm(a, axis=1, keepdims=True)
    b = np.cross(a, rng.normal(size=(S, 3)))
    b /= np.linalg.norm(b, axis=1, keepdims=True)
    waves = 12
    f = np.exp(rng.uniform(math.log(0.5), math.log(40.0), size=(S, waves, 3)))
    th = rng.uniform(0, 2 * math.pi, size=(S, waves, 3))
    k = 2 * math.pi * f[:, :, None, :] * np.stack([np.cos(th), np.sin(th)], axis=2)
    amp = (1.0 / f) * 0.25 / np.sqrt(0.5 * ((1.0 / f) ** 2).sum(axis=1, keepdims=True))

    def dev(x):
        return torch.from_numpy(np.ascontiguousarray(x, dtype=np.float32)).to(DEV)

    sid = torch.repeat_interleave(torch.arange(S, device=DEV), torch.from_numpy(counts).to(DEV))
    m = n - n_shell
    size_t, centre = dev(size)[sid][:, None], dev(rng.uniform(-1.8, 1.8, size=(S, 3)))[sid]
    uv = 2 * _rand(gen, m, 2) - 1
    on_plane = uv[:, :1] * dev(a)[sid] + uv[:, 1:] * dev(b)[sid]
    t, p = torch.acos(uv[:, 0]), math.pi * uv[:, 1]
    on_sphere = torch.stack([t.sin() * p.cos(), t.sin() * p.sin(), t.cos()], 1)
    mean = centre + size_t * torch.where(dev(plane)[sid][:, None] > 0, on_plane, on_sphere)
    col = dev(rng.uniform(0.1, 0.9, size=(S, 3)))[sid]
    kd, ad, ph, st = dev(k), dev(amp), dev(rng.uniform(0, 2 * math.pi, size=(S, waves, 3))), uv * size_t / 0.65
    for w in range(waves):
        kw = kd[:, w][sid]
        col = col + ad[:, w][sid] * torch.sin(st[:, :1] * kw[:, 0] + st[:, 1:] * kw[:, 1] + ph[:, w][sid])
    sigma = dev(np.log(np.sqrt(area / np.maximum(counts, 1))))[sid]
    d = _randn(gen, n_shell, 3)
    d = d / d.norm(dim=1, keepdim=True)
    out = torch.empty((59, n), device=DEV)
    out[0:3] = torch.cat([mean, 12.0 * d]).T
    shell = math.log(math.sqrt(4.0 * math.pi * 144.0 / max(n_shell, 1)))
    out[3:6] = torch.cat([sigma, torch.full((n_shell,), shell, device=DEV)]) + 0.3 * _randn(gen, 3, n)
    q = _randn(gen, 4, n)
    out[6:10] = q / q.norm(dim=0, keepdim=True)
    out[10] = _randn(gen, n)
    out[11:59] = 0.2 * _randn(gen, 48, n)
    sky = 0.5 + 0.25 * torch.sin(d @ _randn(gen, 3, 3) * 6.0)
    out[11:14] = ((torch.cat([col, sky]).clamp(0, 1) - 0.5) / synth.SH_DC_NORM).T
    return out


def _unit_scene(n, seed):
    """[59][n] Gaussians in the unit cube (the 1,000-Gaussian scene's recipe)."""
    return torch.from_numpy(np.ascontiguousarray(synth.random_gaussians(n, seed).T.astype(np.float32))).to(DEV)


def _jitter(g, seed):
    gen, n, out = _gen(seed + 77), g.shape[1], g.clone()
    out[0:3] += 0.003 * _randn(gen, 3, n)
    out[3:6] += 0.1 * _randn(gen, 3, n)
    out[6:10] += 0.05 * _randn(gen, 4, n)
    out[10] += 0.2 * _randn(gen, n)
    out[11:59] += 0.05 * _randn(gen, 48, n)
    return out


def _views(case, seed):
    sizes = _sizes(case)
    ring = synth.ring_cameras(16, case["width"], case["height"], 5.0, seed + 1000)
    cams = []
    for v, (w, h) in enumerate(sizes):
        r = ring[(v * 16) // case["views"]]
        full = make_camera(np.asarray(r["viewmat"], np.float32).reshape(-1), r["intr"], case["width"], case["height"])
        cams.append(capi.dg_camera_scale(full, w, h))
    return cams, sizes


def _images(sizes, seed):
    """Image pairs in [0, 1] with structure at several scales: a target and a render close to it."""
    gen, xs, ys = _gen(seed), [], []
    for w, h in sizes:
        y = torch.zeros((3, h, w), device=DEV)
        for s in (4, 16, 64):
            n = _rand(gen, 1, 3, max(2, h // s), max(2, w // s))
            y += torch.nn.functional.interpolate(n, size=(h, w), mode="bilinear", align_corners=False)[0] / 3
        y = (y + 0.05 * _randn(gen, 3, h, w)).clamp(0, 1)
        xs.append((y + 0.03 * _randn(gen, 3, h, w)).clamp(0, 1).reshape(-1))
        ys.append(y.reshape(-1))
    return torch.cat(xs), torch.cat(ys)


def _moments(n, stride, seed):
    """Adam moments of a run under way: second moments around the gradients' size, first moments below them."""
    gen = _gen(seed + 5)
    m, v = torch.zeros((59, stride), device=DEV), torch.zeros((59, stride), device=DEV)
    s = 3e-7 * torch.exp(0.5 * _randn(gen, 59, n))
    v[:, :n] = s * s
    m[:, :n] = 0.3 * s * _randn(gen, 59, n)
    return m, v


class _Scene:
    """A model, its cameras, the targets and the rasterizer of a training program."""

    def __init__(self, case, seed, targets=True):
        self.case, self.P, self.V = case, case["P"], case["views"]
        self.cams, self.sizes = _views(case, seed)
        scene = _scene(self.P, seed)
        self.rz = Rasterizer(DEV, _opts(case), ppt_fwd=1 if case["tile"] == 8 else None,
                             ppt_bwd=1 if case["tile"] == 8 else None)
        self.npix = sum(w * h for w, h in self.sizes)
        if targets:
            fr = self.rz.forward(scene, self.P, self.cams)
            self.target = fr.flat_img.clone()
        self.stride = (self.P + 1024 + 3) // 4 * 4  # the trainer's buffers: room to grow, 16-byte rows
        self.params = torch.zeros((59, self.stride), device=DEV)
        self.params[:, : self.P] = _jitter(scene, seed)
        self.dL = torch.empty(3 * self.npix, device=DEV)
        self.loss = torch.zeros(self.V + 1, device=DEV)
        self.sws = torch.empty(capi.dg_ssim_workspace_size(self.sizes), dtype=torch.uint8, device=DEV)

    def forward(self):
        return self.rz.forward(self.params[:, : self.P], self.P, self.cams)

    def loss_and_gradient(self, fr):
        capi.dg_loss_l1_dssim(fr.flat_img, self.target, self.sizes, LAMBDA, self.dL, self.loss, self.sws,
                              self.sws.numel(), torch.cuda.current_stream())


def prepare(case, seed):
    kind = case["kind"]
    if kind == "autograd":
        st = _Bag(case=case, rz=Rasterizer(DEV, _opts(case)))
        cam = synth.camera_cfg0(case["width"], case["height"], 4.0)
        st.cam = make_camera(np.asarray(cam["viewmat"], np.float32).reshape(-1), cam["intr"], case["width"],
                             case["height"])
        st.params = _unit_scene(case["P"], seed).requires_grad_(True)
        st.target = _rand(_gen(seed), 3, case["height"], case["width"])
        n = st.target.numel()
        st.dL, st.loss = torch.empty_like(st.target), torch.zeros(1, device=DEV)
        st.ws = torch.empty(capi.dg_loss_workspace_size(n), dtype=torch.uint8, device=DEV)
        return st
    if kind == "loss":
        st = _Bag(case=case, sizes=_sizes(case))
        st.img, st.target = _images(st.sizes, seed)
        st.dL, st.loss = torch.empty_like(st.img), torch.zeros(case["views"] + 1, device=DEV)
        st.sws = torch.empty(capi.dg_ssim_workspace_size(st.sizes), dtype=torch.uint8, device=DEV)
        return st
    if kind == "densify":
        return _prepare_densify(case, seed)
    st = _Scene(case, seed, targets=kind in ("step", "graph", "bwd", "update"))
    if kind in ("step", "graph", "update"):
        st.m, st.v = _moments(st.P, st.stride, seed)
    if kind == "graph":
        fr = st.forward()
        st.hp = capi.dg_adam_hparams_fill(LR, BETA1, BETA2, EPS, STEP)
        st.targets, o = [], 0
        for w, h in st.sizes:
            st.targets.append(st.target[o: o + 3 * w * h].view(3, h, w))
            o += 3 * w * h
        keep = [x.clone() for x in (st.params, st.m, st.v)]  # capture() also runs a step
        st.graph = StepGraph(DEV, _opts(case), 1, 1, st.params, st.m, st.v, None, st.stride, st.P, st.cams,
                             int(fr.M * 1.5) + 4096, LAMBDA)
        st.graph.capture(st.cams, st.hp, st.targets)
        for x, k in zip((st.params, st.m, st.v), keep):
            x.copy_(k)
    if kind in ("bin", "fwd", "bwd", "update"):
        st.fr = st.forward()
    if kind == "bin":  # room for half as many pairs again as such a scene usually has
        cap = max(st.fr.M, int(1.5 * _pairs(case)[1]))
        st.rz.gid, st.rz.M_cap, st.rz.ws = torch.zeros(cap, dtype=torch.int32, device=DEV), cap, None
        st.rz._ensure_ws(st.P, st.V, cap)
    if kind in ("bwd", "update"):
        st.loss_and_gradient(st.fr)
    if kind == "update":
        st.rz.backward_render(st.fr, st.dL)
    if kind == "fwd":
        st.img, st.T = torch.empty(3 * st.npix, device=DEV), torch.empty(st.npix, device=DEV)
        st.last = torch.empty(st.npix, dtype=torch.int32, device=DEV)
    return st


class _Bag:
    def __init__(self, **kw):
        self.__dict__.update(kw)


def _prepare_densify(case, seed):
    P = case["P"]
    gen = _gen(seed + 9)
    st = _Bag(case=case, P=P, cap=(2 * P + 1024 + 3) // 4 * 4)
    st.params = torch.zeros((59, st.cap), device=DEV)
    st.params[:, :P] = _scene(P, seed)
    st.params[10, :P] -= 2.0  # after an opacity reset: some fall below the pruning bound
    st.m, st.v = _moments(P, st.cap, seed)
    st.den = torch.floor(_rand(gen, P) * 40.0)  # views that saw each Gaussian since the last time
    st.acc = st.den * 1e-4 * torch.exp(0.7 * _randn(gen, P))
    st.maxr = torch.floor(_rand(gen, P) * 30.0)
    st.opts = capi.densify_opts(2e-4, 0.005, 0.01, 5.5)
    st.budget = P // 12
    st.noise = _randn(gen, st.budget, 2, 3)
    st.counts = torch.zeros(2, dtype=torch.int64, device=DEV)
    st.P_out = torch.zeros(1, dtype=torch.int64, device=DEV)
    st.dst = [torch.zeros((59, st.cap), device=DEV) for _ in range(3)]
    st.ws = torch.empty(capi.dg_densify_workspace_size(P), dtype=torch.uint8, device=DEV)
    return st


# ------------------------------------------------------------------ one pass
def run(st):
    kind = st.case["kind"]
    stream = torch.cuda.current_stream()
    if kind == "autograd":
        st.params.grad = None
        img = rasterize(st.params, st.rz, st.cam)
        capi.dg_loss_l1(img.detach(), st.target, st.target.numel(), st.dL, st.loss, st.ws, st.ws.numel(), stream)
        img.backward(st.dL)
        return dict(img=img.detach(), loss=st.loss, grad=st.params.grad)
    if kind == "loss":
        capi.dg_loss_l1_dssim(st.img, st.target, st.sizes, LAMBDA, st.dL, st.loss, st.sws, st.sws.numel(), stream)
        return dict(loss=st.loss, dL=st.dL)
    if kind == "densify":
        capi.dg_densify_mark(st.params, st.cap, st.P, st.acc, st.den, st.maxr, st.opts, st.ws, st.ws.numel(),
                             st.counts, stream)
        _, n_cand = (int(x) for x in st.counts.cpu())  # the trainer reads the counts for the Eq. 5 budget
        capi.dg_densify_apply(st.params, st.m, st.v, st.cap, st.P, n_cand, st.budget, st.noise, st.ws, st.ws.numel(),
                              *st.dst, st.cap, st.P_out, stream)
        return dict(counts=st.counts, P=st.P_out, params=st.dst[0], m=st.dst[1], v=st.dst[2])
    rz, P, V, cams = st.rz, st.P, st.V, st.cams
    if kind == "step":
        fr = st.forward()
        st.loss_and_gradient(fr)
        rz.backward_render(fr, st.dL)
        rz.project_bwd_adam(st.params, st.stride, fr, st.m, st.v, LR, STEP, BETA1, BETA2, EPS)
        return dict(img=fr.flat_img, loss=st.loss, params=st.params, m=st.m, v=st.v)
    if kind == "graph":
        st.graph.replay(st.cams, st.hp, st.targets)
        return dict(loss=st.graph.loss, params=st.params, m=st.m, v=st.v)
    if kind == "view":
        fr = st.forward()
        return dict(img=fr.flat_img, T=fr.flat_T, last=fr.flat_last)
    if kind == "project":
        rz._ensure_records(V * P)
        capi.dg_project(st.params, st.stride, P, cams, V, rz.opts, rz.feat, rz.depth, rz.radius, rz.tiles, rz.clamp,
                        stream)
        return dict(feat=rz.feat[:, :9], mask=rz.feat[:, 9:11].view(torch.int32), depth=rz.depth, radius=rz.radius,
                    tiles=rz.tiles, clamp=rz.clamp)
    if kind == "bin":
        capi.dg_bin_count(rz.depth, rz.tiles, P, V, rz.ws, rz.ws.numel(), rz.M_cap, rz.M_dev, stream)
        capi.dg_bin_sort(rz.feat, rz.radius, P, cams, V, rz.opts.tile, rz.ws, rz.ws.numel(), rz.M_cap, rz.gid,
                         rz.ranges, rz.status, stream)
        return dict(M=rz.M_dev, status=rz.status, ranges=rz.ranges, gid=rz.gid)
    if kind == "fwd":
        capi.dg_render_fwd(rz.rfeat, rz.gid, rz.ranges, cams, V, rz.opts_fwd, st.img, st.T, st.last, None, None,
                           rz.rws, rz.rws.numel(), stream)
        return dict(img=st.img, T=st.T, last=st.last)
    if kind == "bwd":
        rz.backward_render(st.fr, st.dL)
        return dict(grad2d=rz.grad2d)
    if kind == "update":
        rz.project_bwd_adam(st.params, st.stride, st.fr, st.m, st.v, LR, STEP, BETA1, BETA2, EPS)
        return dict(params=st.params, m=st.m, v=st.v)
    raise ValueError(kind)


# ------------------------------------------------------------------ the work of a pass
def _pairs(case):
    """(records in view, tile pairs) that such a scene has, within a fifth or so: surfaces
    are closed at the Gaussians' spacing, so a record's footprint grows with the pixels per record."""
    rec = case["P"] * case["views"]
    vis = rec if case["kind"] == "autograd" else 0.83 * rec
    x = sum(w * h for w, h in _sizes(case)) / max(rec, 1)
    per = 1.65 + 3.8 * x if case["tile"] == 8 else 1.3 + 1.05 * x
    return vis, vis * per * (1.0 if case["tight"] else 1.4)


def work(case):
    kind, P, V = case["kind"], case["P"], case["views"]
    npix = sum(w * h for w, h in _sizes(case))
    rec = P * V
    feat = 24 if case["record"] else 48
    if kind == "loss":  # both images read, the gradient written; two 11-tap passes over four and three statistics
        return dict(bytes=3 * npix * 12, flops=3 * npix * 2 * 22 * 7)
    if kind == "densify":  # parameters and moments read and written once (moments of new Gaussians are zeros)
        return dict(bytes=int(P * 59 * 4 * 3 * 2.1), flops=60 * P)
    vis, pairs = _pairs(case)
    blends = 45.0 * npix                                     # blended (pixel, entry) evaluations
    n_par = 11 + 3 * (case["sh"] + 1) ** 2
    parts = dict(
        project=(P * n_par * 4 + rec * 61, rec * 300),
        bin=(rec * 8 + vis * 24 + pairs * 4, pairs),
        fwd=(vis * feat + pairs * 4 + npix * 20, blends * 19),
        loss=(3 * npix * 12, 3 * npix * 308),
        bwd=(vis * feat + pairs * 4 + npix * 20 + rec * 48, blends * 50),
        update=(vis * 48 + rec * 5 + P * 59 * 4 * 6, rec * 600),
        grads=(vis * 48 + rec * 5 + P * 59 * 4 * 2, rec * 600))
    chains = dict(autograd=("project", "bin", "fwd", "bwd", "grads"), view=("project", "bin", "fwd"),
                  step=("project", "bin", "fwd", "loss", "bwd", "update"))
    chains["graph"] = chains["step"]
    use = chains.get(kind, (kind,))
    return dict(bytes=int(sum(parts[k][0] for k in use)), flops=int(sum(parts[k][1] for k in use)))


# ------------------------------------------------------------------ the same in 64 bits
def _sh_basis(d):
    x, y, z = d
    xx, yy, zz = x * x, y * y, z * z
    pi = math.pi
    return [torch.full_like(x, 0.5 / math.sqrt(pi)),
            math.sqrt(3 / (4 * pi)) * y, math.sqrt(3 / (4 * pi)) * z, math.sqrt(3 / (4 * pi)) * x,
            math.sqrt(15 / pi) / 2 * x * y, math.sqrt(15 / pi) / 2 * y * z, math.sqrt(5 / pi) / 4 * (3 * zz - 1),
            math.sqrt(15 / pi) / 2 * x * z, math.sqrt(15 / pi) / 4 * (xx - yy),
            math.sqrt(35 / (2 * pi)) / 4 * y * (3 * xx - yy), math.sqrt(105 / pi) / 2 * x * y * z,
            math.sqrt(21 / (2 * pi)) / 4 * y * (5 * zz - 1), math.sqrt(7 / pi) / 4 * z * (5 * zz - 3),
            math.sqrt(21 / (2 * pi)) / 4 * x * (5 * zz - 1), math.sqrt(105 / pi) / 4 * z * (xx - yy),
            math.sqrt(35 / (2 * pi)) / 4 * x * (xx - 3 * yy)]


def _project64(p, cam, opts):
    """Projected records of the [59][P] float64 parameters: (u, v, A, B, C, o), colour before its clamp, depth, radius."""
    vm = torch.tensor(list(cam.viewmat), dtype=torch.float64, device=DEV).view(3, 4)
    R, t0 = vm[:, :3], vm[:, 3:]
    t = R @ p[0:3] + t0
    tx, ty, tz = t
    q = p[6:10] / p[6:10].norm(dim=0, keepdim=True)
    w, x, y, z = q
    rot = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                       2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                       2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)]).view(3, 3, -1)
    M = rot * torch.exp(p[3:6])[None]
    limx, limy = 1.3 * 0.5 * cam.width / cam.fx, 1.3 * 0.5 * cam.height / cam.fy
    gx, gy = (tx / tz).clamp(-limx, limx), (ty / tz).clamp(-limy, limy)
    zero = torch.zeros_like(tz)
    J = torch.stack([torch.stack([cam.fx / tz, zero, -cam.fx * gx / tz]),
                     torch.stack([zero, cam.fy / tz, -cam.fy * gy / tz])])
    K = torch.einsum("ijn,jk,kln->iln", J, R, M)  # 2 x 3 square root of the 2D covariance
    a = (K[0] * K[0]).sum(0) + opts.eps2d
    b = (K[0] * K[1]).sum(0)
    c = (K[1] * K[1]).sum(0) + opts.eps2d
    det = a * c - b * b
    lam = 0.5 * (a + c) + torch.sqrt(0.25 * (a - c) ** 2 + b * b)
    centre = -(R.T @ t0)
    d = p[0:3] - centre
    d = d / d.norm(dim=0, keepdim=True)
    Y = _sh_basis(d)
    col = torch.stack([sum(Y[k] * p[11 + 3 * k + ch] for k in range((opts.sh_degree + 1) ** 2)) for ch in range(3)]) + 0.5
    geo = torch.stack([cam.fx * tx / tz + cam.cx, cam.fy * ty / tz + cam.cy, c / det, -b / det, a / det,
                       torch.sigmoid(p[10])])
    return geo, col, tz, torch.ceil(3 * torch.sqrt(lam.detach()))


def _rect64(geo, radius, cam, B):
    """Tile rect [x0, x1) x [y0, y1) of each record."""
    fu, fv = torch.floor(geo[0].detach()), torch.floor(geo[1].detach())
    TX, TY = -(-cam.width // B), -(-cam.height // B)
    return (torch.floor((fu - radius) / B).clamp(0, TX), torch.floor((fu + radius) / B).add(1).clamp(0, TX),
            torch.floor((fv - radius) / B).clamp(0, TY), torch.floor((fv + radius) / B).add(1).clamp(0, TY))


def _exact_autograd(case, seed):
    st = prepare(case, seed)
    opts, cam, B = _opts(case), st.cam, case["tile"]
    p = st.params.detach().double().requires_grad_(True)
    geo, col, tz, radius = _project64(p, cam, opts)
    x0, x1, y0, y1 = _rect64(geo, radius, cam, B)
    vis = (tz > opts.near_plane) & (x0 < x1) & (y0 < y1)
    order = torch.argsort(torch.where(vis, tz.detach(), torch.inf), stable=True)[: int(vis.sum())]
    u, v, A, Bc, C, o = geo[:, order]
    ys, xs = torch.meshgrid(torch.arange(cam.height, device=DEV), torch.arange(cam.width, device=DEV), indexing="ij")
    px, py = xs.reshape(1, -1), ys.reshape(1, -1)
    member = ((px // B >= x0[order][:, None]) & (px // B < x1[order][:, None]) &
              (py // B >= y0[order][:, None]) & (py // B < y1[order][:, None]))
    dx, dy = u[:, None] - (px + 0.5), v[:, None] - (py + 0.5)
    power = -0.5 * (A[:, None] * dx * dx + C[:, None] * dy * dy) - Bc[:, None] * dx * dy
    alpha = (o[:, None] * torch.exp(power)).clamp(max=float(np.float32(0.99)))
    alpha = torch.where(member & (alpha.detach() >= float(np.float32(1) / np.float32(255))), alpha, 0.0)
    after = torch.cumprod(1 - alpha.detach(), 0)
    alpha = torch.where(after >= float(np.float32(1e-4)), alpha, 0.0)
    T = torch.cumprod(1 - alpha, 0)
    before = torch.cat([torch.ones_like(T[:1]), T[:-1]])
    img = torch.einsum("np,cn->cp", alpha * before, col[:, order].clamp(min=0)).view(3, cam.height, cam.width)
    diff = img - st.target.double()
    n = diff.numel()
    img.backward(torch.sign(diff.detach()) / n)
    return dict(img=img.detach(), loss=diff.detach().abs().mean().view(1), grad=p.grad)


def _exact_loss(case, seed):
    st = prepare(case, seed)
    k = torch.arange(-5, 6, device=DEV, dtype=torch.float64)
    win = torch.exp(-k * k / (2 * 1.5 * 1.5))
    win = win / win.sum()

    def blur(a):
        a = a[:, None]
        a = torch.nn.functional.conv2d(a, win.view(1, 1, 1, 11), padding=(0, 5))
        return torch.nn.functional.conv2d(a, win.view(1, 1, 11, 1), padding=(5, 0))[:, 0]

    losses, grads, o = [], [], 0
    for w, h in st.sizes:
        x = st.img[o: o + 3 * w * h].view(3, h, w).double().requires_grad_(True)
        y = st.target[o: o + 3 * w * h].view(3, h, w).double()
        o += 3 * w * h
        mx, my = blur(x), blur(y)
        sx, sy, sxy = blur(x * x) - mx * mx, blur(y * y) - my * my, blur(x * y) - mx * my
        c1, c2 = 0.01 ** 2, 0.03 ** 2
        S = (2 * mx * my + c1) * (2 * sxy + c2) / ((mx * mx + my * my + c1) * (sx + sy + c2))
        L = (1 - LAMBDA) * (x - y).abs().mean() + LAMBDA * (1 - S.mean())
        (L / len(st.sizes)).backward()
        losses.append(L.detach())
        grads.append(x.grad.reshape(-1))
    losses.append(sum(losses) / len(losses))
    return dict(loss=torch.stack(losses), dL=torch.cat(grads))


def _exact_project(case, seed):
    st = prepare(case, seed)
    opts = _opts(case)
    p = st.params[:, : st.P].double()
    feats, depths = [], []
    for cam in st.cams:
        geo, col, tz, radius = _project64(p, cam, opts)
        x0, x1, y0, y1 = _rect64(geo, radius, cam, case["tile"])
        vis = (tz > opts.near_plane) & (x0 < x1) & (y0 < y1)
        feats.append((torch.cat([geo, col.clamp(min=0)]) * vis).nan_to_num(0.0, 0.0, 0.0).T)
        depths.append(tz)
    return dict(feat=torch.cat(feats), mask=None, depth=torch.cat(depths), radius=None, tiles=None, clamp=None)


def _exact_update(case, seed):
    st = prepare(case, seed)
    opts, P, rz = _opts(case), st.P, st.rz
    p = st.params[:, :P].double().requires_grad_(True)
    total = torch.zeros_like(p)
    for i, cam in enumerate(st.cams):
        r = slice(i * P, (i + 1) * P)
        seen = torch.nonzero(rz.radius[r] > 0)[:, 0]
        if not len(seen):
            continue
        sub = p.detach()[:, seen].requires_grad_(True)
        geo, col, _, _ = _project64(sub, cam, opts)
        g2, cl = rz.grad2d[r][seen].double().T, rz.clamp[r][seen]
        gcol = torch.stack([torch.where((cl >> ch) & 1 > 0, 0.0, g2[6 + ch]) for ch in range(3)])
        torch.autograd.backward([geo, col], [g2[:6], gcol])
        total[:, seen] += sub.grad
    out = {k: x.double().clone() for k, x in (("params", st.params), ("m", st.m), ("v", st.v))}
    b1, b2 = float(np.float32(BETA1)), float(np.float32(BETA2))
    out["m"][:, :P] = b1 * out["m"][:, :P] + (1 - b1) * total
    out["v"][:, :P] = b2 * out["v"][:, :P] + (1 - b2) * total * total
    lr = torch.tensor(LR, dtype=torch.float64, device=DEV)[:, None]
    mh, vh = out["m"][:, :P] / (1 - b1 ** STEP), out["v"][:, :P] / (1 - b2 ** STEP)
    out["params"][:, :P] -= lr * mh / (vh.sqrt() + EPS)
    return out


def _exact_densify(case, seed):
    st = prepare(case, seed)
    P, prm = st.P, st.params[:, : st.P]
    keep = ~(prm[10] < float(np.float32(math.log(float(np.float32(0.005)) / (1 - float(np.float32(0.005)))))))
    score = torch.where(st.den > 0, st.acc / st.den.clamp(min=1), 0.0)
    cand = keep & (st.den > 0) & (score >= float(np.float32(2e-4)))
    split = prm[3:6].amax(0) > float(np.float32(math.log(float(np.float32(0.01)) * 5.5)))
    idx = torch.nonzero(cand)[:, 0]
    n_sel = min(len(idx), st.budget)
    best = torch.argsort(score[idx], descending=True, stable=True)[:n_sel]
    sel_idx = torch.sort(idx[best])[0]
    sel = torch.zeros(P, dtype=torch.bool, device=DEV)
    sel[sel_idx] = True
    left = torch.nonzero(keep & ~(sel & split))[:, 0]
    n_keep = len(left)
    outs = [torch.zeros((59, st.cap), dtype=torch.float64, device=DEV) for _ in range(3)]
    for o, s in zip(outs, (st.params, st.m, st.v)):
        o[:, :n_keep] = s[:, left].double()
    src, sp = prm[:, sel_idx].double(), split[sel_idx]
    pos = n_keep + torch.cumsum(torch.where(sp, 2, 1), 0) - torch.where(sp, 2, 1)
    outs[0][:, pos[~sp]] = src[:, ~sp]
    if bool(sp.any()):
        s, eps = src[:, sp], st.noise[:n_sel][sp].double()
        w, x, y, z = s[6:10] / s[6:10].norm(dim=0, keepdim=True)
        rot = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                           2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                           2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)]).view(3, 3, -1)
        for k in range(2):
            new = s.clone()
            new[0:3] += torch.einsum("ijn,jn->in", rot, torch.exp(s[3:6]) * eps[:, k].T)
            new[3:6] -= math.log(1.6)
            outs[0][:, pos[sp] + k] = new
    return dict(counts=None, P=None, params=outs[0], m=outs[1], v=outs[2])


def exact(case, seed):
    kind = case["kind"]
    if kind == "autograd" and case["P"] * case["width"] * case["height"] <= 60_000_000:
        return _exact_autograd(case, seed)
    if kind in ("loss", "project", "update", "densify"):
        return dict(loss=_exact_loss, project=_exact_project, update=_exact_update, densify=_exact_densify)[kind](case, seed)
    # binning gives whole numbers; whole steps and full-size compositing would take
    # minutes in 64 bits
    return None
