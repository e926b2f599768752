"""Performance cases of the sparse-voxel rasterizer and the steps around it.

Each case is one call, or one training iteration, that a program makes through
the package's public entry points (``raster``, ``litevoxel``):

  render     forward pass, for viewing or evaluation
  grad       differentiable forward + backward through ``rasterize`` with the
             per-voxel statistics of an accumulation window
  train      one training iteration: LF weights, forward, backward with the
             LF-weighted loss fused in, transmittance loss, Adam with TV
  prune      depth-quantile pruning with all of its guards
  subdivide  priority subdivision into new arrays, optimizer moments carried
  loss       LF-weighted loss of a set of views
  vertex     shared grid-vertex index, gather and scatter

``listed()`` gives the standing cases, ``draw(rng)`` one more of the same
ranges; ``prepare``, ``run``, ``work`` and ``exact`` make the inputs, run one
pass, state its least work and give its result in 64 bits.  Scenes are the
synthetic octrees of ``synth`` (spheres over a ground plane inside a background
shell), built on the GPU with a chosen voxel count.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2511_02510_gb300 import litevoxel as L
from paper_2511_02510_gb300 import synth
from paper_2511_02510_gb300.raster import CapturedStep, RasterContext, Scene, rasterize

DEV = "cuda"


# ---------------------------------------------------------------------------- the cases
def _raster(kind, name, **kw):
    c = {"name": name, "kind": kind, "voxels": 4000, "width": 128, "height": 128, "views": 1, "tile": 16,
         "persistent": False, "segment": False, "half": False, "degree": 3, "opaque": True, "graph": False}
    c.update(kw)
    return c


def listed():
    return [
        # the smallest calls: a thumbnail of the 4k-voxel unit-cube scene, where launches are all
        _raster("render", "render_tiny"),
        # evaluation of a trained 2M-voxel scene at the Mip-NeRF 360 view size, default options
        _raster("render", "render_360", voxels=1976376, width=1237, height=822),
        # a batch of evaluation views in one launch, FP16 corners and BF16 SH, tuned schedule
        _raster("render", "render_8_mixed", voxels=6000000, width=980, height=545, views=8, tile=32,
                persistent=True, half=True),
        # gradients while a scene is still small: odd image, two views, SH degree 1
        _raster("grad", "grad_odd", voxels=200001, width=641, height=479, views=2, tile=8, degree=1),
        # gradients of the trained scene through autograd, default options
        _raster("grad", "grad_360", voxels=1976376, width=1237, height=822),
        # semi-transparent matter: long sample lists, exact segment integration
        _raster("grad", "grad_fog", voxels=300000, width=979, height=545, segment=True, opaque=False),
        # the first iterations of a training run, launched call by call
        _raster("train", "train_start", voxels=50000, width=640, height=480, degree=0),
        # the iteration of a long run: captured in a CUDA graph, tuned schedule
        _raster("train", "train_360", voxels=1976376, width=1237, height=822, tile=32, persistent=True, graph=True),
        # adaptation of the trained scene: pruning with every guard on
        {"name": "prune_360", "kind": "prune", "voxels": 1976376, "bins": 16},
        # growth of a large scene: FP16 corners and BF16 SH, FP32 moments carried along
        {"name": "subdivide_tt", "kind": "subdivide", "voxels": 6000000, "half": True, "top_ppm": 50000},
        # the loss of sixteen uneven views
        {"name": "loss_16", "kind": "loss", "views": 16, "width": 640, "height": 480, "width1": 1600,
         "height1": 1060},
        # vertex numbering after a topology change of the shared-vertex variant
        {"name": "vertex_300k", "kind": "vertex", "voxels": 300000},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["render", "render", "grad", "grad", "grad", "train", "train", "prune", "subdivide", "loss",
                       "vertex"])
    if kind == "prune":
        return {"kind": kind, "voxels": _log(rng, 4000, 4000000), "bins": rng.choice([7, 16, 16, 31])}
    if kind == "subdivide":
        return {"kind": kind, "voxels": _log(rng, 4000, 4000000), "half": rng.random() < 0.5,
                "top_ppm": rng.choice([10000, 50000, 100000])}
    if kind == "loss":
        w, h = _log(rng, 60, 1200), _log(rng, 60, 800)
        return {"kind": kind, "views": rng.randint(1, 12), "width": w, "height": h,
                "width1": w + rng.randint(0, 400), "height1": h + rng.randint(0, 200)}
    if kind == "vertex":
        return {"kind": kind, "voxels": _log(rng, 4000, 300000)}
    views = rng.choice([1, 1, 1, 2, 4])
    c = _raster(kind, "", voxels=_log(rng, 4000, 4000000 // views), width=_log(rng, 100, 1300),
                height=_log(rng, 80, 900), views=views, tile=rng.choice([8, 16, 16, 32]),
                persistent=rng.random() < 0.5, segment=rng.random() < 0.2, half=rng.random() < 0.25,
                degree=rng.choice([0, 1, 2, 3, 3, 3]), opaque=rng.random() < 0.8)
    if not c["opaque"]:                     # long sample lists
        c["voxels"], c["views"] = min(c["voxels"], 300000), 1
        c["width"], c["height"] = min(c["width"], 979), min(c["height"], 545)
    if kind == "train":
        c["graph"], c["half"] = rng.random() < 0.5, False
    del c["name"]
    return c


# ---------------------------------------------------------------------------- scenes and images on the GPU
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _sdf_factory(spec):
    centers, radii = synth._shapes(spec.seed)
    fc = torch.tensor(spec.fg_center, dtype=torch.float64, device=DEV)
    cen = torch.tensor(centers, dtype=torch.float64, device=DEV)

    def sdf(p):
        q = (p - fc) / spec.fg_scale + 0.5
        d = q[..., 1] - 0.15
        for c, r in zip(cen, radii):
            d = torch.minimum(d, (q - c).norm(dim=-1) - float(r))
        box = (q - 0.5).abs().amax(-1) - spec.fg_box_half
        d = torch.maximum(d, box) * spec.fg_scale
        if spec.shell is not None:
            d = torch.minimum(d, spec.shell[0] - (p - fc).norm(dim=-1))
        return d

    return sdf


def _octree(spec, sdf, l_fg):
    """Leaves of the octree refined to level l_fg: (cells, levels, |sdf| / edge)."""
    rmin = torch.tensor(spec.root_min, dtype=torch.float64, device=DEV)
    fc = torch.tensor(spec.fg_center, dtype=torch.float64, device=DEV)
    g = torch.arange(1 << spec.l_min, device=DEV)
    cells = torch.stack(torch.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)
    offs = torch.tensor([[i & 1, (i >> 1) & 1, (i >> 2) & 1] for i in range(8)], device=DEV)
    reach = spec.fg_scale * (spec.fg_box_half + 0.1)
    out = []
    for level in range(spec.l_min, l_fg + 1):
        edge = spec.root_edge / (1 << level)
        cen = rmin + (cells + 0.5) * edge
        d = sdf(cen).abs()
        l_bg = min(spec.l_max_bg, l_fg)
        fine = (cen - fc).abs().amax(-1) < reach
        cap = torch.where(fine, l_fg, l_bg)
        straddle = d < 0.87 * edge
        inside = (cen - fc).norm(dim=-1) < spec.shell[1] if spec.shell is not None else torch.ones_like(fine)
        straddle &= inside
        refine = straddle & (level < cap)
        keep = inside & (((level >= cap) & (d < 2.6 * edge)) |
                         ((level < cap) & ~straddle & (d < (0.87 + spec.halo) * edge)))
        out.append((cells[keep], torch.full((int(keep.sum()),), level, dtype=torch.uint8, device=DEV),
                    d[keep] / edge))
        par = cells[refine]
        if not par.shape[0]:
            break
        cells = (2 * par[:, None, :] + offs).reshape(-1, 3)
    return [torch.cat(x) for x in zip(*out)]


def _spec(n, seed):
    if n <= 30000:                          # the unit cube's scene
        return synth.SceneSpec(seed=seed, l_min=4, l_max_bg=5, halo=0.2)
    return synth._spec_360(seed, 2.0, 1.0)  # the 360-degree scene


def _scene(n, seed, opaque=True, density_dtype=torch.float32, sh_dtype=torch.float32, degree=3):
    """A scene of n voxels: the octree's leaves nearest to the surface, in octree order."""
    spec = _spec(n, seed)
    sdf = _sdf_factory(spec)
    l_fg = spec.l_min + 1
    while True:
        cells, level, near = _octree(spec, sdf, l_fg)
        if cells.shape[0] >= n:
            break
        l_fg += 1
    spec.l_max_fg = l_fg
    keep = near.argsort(stable=True)[:n].sort().values
    cells, level = cells[keep], level[keep]
    edge = spec.root_edge / torch.exp2(level.double())
    rmin = torch.tensor(spec.root_min, dtype=torch.float64, device=DEV)
    cen = rmin + (cells + 0.5) * edge[:, None]
    geom = torch.cat([cen, 0.5 * edge[:, None]], 1).float().contiguous()
    g = _gen(seed)
    sign = torch.tensor([[(i & 1) * 2 - 1, ((i >> 1) & 1) * 2 - 1, ((i >> 2) & 1) * 2 - 1] for i in range(8)],
                        dtype=torch.float64, device=DEV)
    big = spec.root_edge > 1.0
    peak = 2.5 * (1 << l_fg) / spec.root_edge if opaque and big else spec.density_peak
    dens = torch.empty((n, 8), dtype=density_dtype, device=DEV)
    for s in range(0, n, 1 << 20):
        e = min(n, s + (1 << 20))
        p = geom[s:e, None, :3].double() + sign * geom[s:e, None, 3:].double()
        v = peak * torch.sigmoid(-sdf(p) / spec.sigmoid_scale)
        dens[s:e] = (v.float() + spec.density_noise * torch.randn(v.shape, device=DEV, generator=g)).to(density_dtype)
    sh = torch.empty((n, 48), dtype=sh_dtype, device=DEV)
    for s in range(0, n, 1 << 20):
        e = min(n, s + (1 << 20))
        sh[s:e, 3:] = (spec.sh_noise * torch.randn((e - s, 45), device=DEV, generator=g)).to(sh_dtype)
        sh[s:e, :3] = torch.rand((e - s, 3), device=DEV, generator=g).to(sh_dtype)
    return Scene(geom, level.contiguous(), dens, sh, degree)


def _cameras(case, seed):
    rng = np.random.default_rng(seed + 100)
    unit = case["voxels"] <= 30000
    return [synth.orbit_camera(case["width"], case["height"], 60.0, 1.6 if unit else 3.0, rng.uniform(0, 360),
                               rng.uniform(5, 30), (0.5, 0.4, 0.5) if unit else (0.0, 0.0, 0.0))
            for _ in range(case["views"])]


def _image(w, h, seed, blobs=12):
    """Piecewise-smooth target image [h * w, 3]: flat regions separated by edges, a little noise."""
    rng = np.random.default_rng(seed)
    ys = torch.arange(h, device=DEV, dtype=torch.float32)[:, None]
    xs = torch.arange(w, device=DEV, dtype=torch.float32)[None, :]
    img = torch.empty((h, w, 3), device=DEV)
    img[:] = torch.tensor(rng.uniform(0.2, 0.8, 3), device=DEV, dtype=torch.float32)
    for _ in range(blobs):
        cx, cy, r = rng.uniform(0, w), rng.uniform(0, h), rng.uniform(0.05, 0.3) * min(w, h)
        m = ((xs - cx) ** 2 + (ys - cy) ** 2 < r * r)[..., None]
        img = torch.where(m, torch.tensor(rng.uniform(0, 1, 3), device=DEV, dtype=torch.float32), img)
    img = img + 0.01 * torch.randn(img.shape, device=DEV, generator=_gen(seed))
    return (img + 0.05 * (xs / max(1, w - 1))[..., None]).clamp(0, 1).reshape(-1, 3).contiguous()


def _lf_params():
    p = L.lv_lf_params()
    p.eps, p.gamma_max, p.t0, p.t1, p.pctl_ppm = 1e-3, 0.6, 300.0, 600.0, 990000
    return p


# ---------------------------------------------------------------------------- prepare
def _inputs_raster(case, seed):
    half = case["half"]
    s = SimpleNamespace(case=case)
    s.scene = _scene(case["voxels"], seed, case["opaque"], torch.float16 if half else torch.float32,
                     torch.bfloat16 if half else torch.float32, case["degree"])
    s.cams = _cameras(case, seed)
    s.n_pix = sum(c["width"] * c["height"] for c in s.cams)
    return s


def _prepare_raster(case, seed):
    s = _inputs_raster(case, seed)
    s.ctx = RasterContext(s.cams, s.scene.n, tile=case["tile"], exact_segment=case["segment"],
                          persistent=case["persistent"])
    s.vox = s.scene.voxels()
    s.ctx.fit_capacity(s.vox)
    return s


def _image_grads(s, seed):
    """Loss gradients of the three images, as a photometric, a depth and a transmittance term leave them
    (with a loss scale where the parameters, and so their gradients, are kept in 16 bits)."""
    g = _gen(seed + 1)
    k = (65536.0 if s.case["half"] else 1.0) / s.n_pix
    return [k * torch.randn((s.n_pix, 3), device=DEV, generator=g), 0.1 * k * torch.randn(s.n_pix, device=DEV, generator=g),
            0.1 * k * torch.randn(s.n_pix, device=DEV, generator=g)]


def _prepare_render(case, seed):
    return _prepare_raster(case, seed)


def _prepare_grad(case, seed):
    s = _prepare_raster(case, seed)
    s.density = s.scene.density.requires_grad_()
    s.sh = s.scene.sh.requires_grad_()
    s.grads = _image_grads(s, seed)
    s.w_max = torch.empty(s.scene.n, device=DEV)
    return s


def _moments(n, seed):
    """Adam moments of a run under way: (m, v) of corners and SH."""
    g = _gen(seed + 2)
    out = []
    for width, scale in ((8, 1e-7), (48, 1e-6)):
        out.append(scale * torch.randn((n, width), device=DEV, generator=g))
        out.append((scale * (1.0 + torch.rand((n, width), device=DEV, generator=g))) ** 2)
    return out


def _adam():
    p = L.lv_adam_params()
    p.lr_density, p.lr_sh, p.beta1, p.beta2, p.eps, p.step, p.tv_weight = 1e-3, 1e-5, 0.9, 0.999, 1e-8, 4000, 1e-6
    return p


LF_T, TC_WEIGHT = 450.0, 1e-2


def _prepare_train(case, seed):
    s = _prepare_raster(case, seed)
    n = s.scene.n
    s.widths, s.heights = [c["width"] for c in s.cams], [c["height"] for c in s.cams]
    s.gt = torch.cat([_image(w, h, seed + 31 * i) for i, (w, h) in enumerate(zip(s.widths, s.heights))])
    s.lfp = _lf_params()
    s.lf_ws = torch.empty(L.lv_lf_workspace_size(s.widths, s.heights), dtype=torch.uint8, device=DEV)
    s.tr_ws = torch.empty(max(256, L.lv_train_workspace_size()), dtype=torch.uint8, device=DEV)
    s.loss, s.tc_loss = torch.zeros(case["views"], device=DEV), torch.zeros(1, device=DEV)
    s.dL_dT = torch.empty(s.n_pix, device=DEV)
    s.d_density, s.d_sh = torch.empty((n, 8), device=DEV), torch.empty((n, 48), device=DEV)
    s.w_max = torch.empty(n, device=DEV)
    s.moments = _moments(n, seed)
    s.adam = _adam()
    s.step = lambda: _iteration(s)
    if case["graph"]:
        state = [s.scene.density, s.scene.sh] + s.moments
        kept = [t.clone() for t in state]
        s.step = CapturedStep(s.step)
        for t, k in zip(state, kept):       # the capture's warm-up pass was an iteration too
            t.copy_(k)
    return s


def _prepare_prune(case, seed):
    n, g = case["voxels"], _gen(seed)

    def rand():
        return torch.rand(n, device=DEV, generator=g)

    s = SimpleNamespace(case=case)
    s.seen = (rand() < 0.6).to(torch.uint8)
    s.z = torch.where(rand() < 0.9, 1.7 + 2.6 * rand(), 9.0 + 10.0 * rand())   # object, background shell
    s.w_max = torch.where(rand() < 0.4, rand() ** 4, 0.0)                      # the others were never hit
    s.delta = s.z / 1071.3
    s.edge = rand() ** 3
    h = torch.exp2(-torch.randint(2, 9, (n,), device=DEV, generator=g).float())
    s.geom = torch.cat([4.0 * torch.randn((n, 3), device=DEV, generator=g), h[:, None]], 1).contiguous()
    s.ema, s.state = 0.25 + 0.75 * rand(), (rand() < 0.8).to(torch.uint8)
    s.pct = torch.tensor([1.8, 9.0], device=DEV)
    p = L.lv_prune_params()
    p.n_bins, p.q_ppm, p.ema_alpha, p.m_low, p.m_high = case["bins"], 50000, 0.1, 0.3, 0.7
    p.cap_ppm, p.lo_ppm, p.hi_ppm = 10000, 50000, 950000
    p.anneal, p.anneal_ppm, p.relax_ppm = 1, 820000, 250000
    p.halo_small, p.halo_w, p.halo_edge = 0.75, 0.5, 0.5
    p.geom, p.delta, p.edge = s.geom.data_ptr(), s.delta.data_ptr(), s.edge.data_ptr()
    p.pct_ema, p.pct_state = 0.1, s.pct.data_ptr()
    s.params = p
    s.mask = torch.empty(n, dtype=torch.uint8, device=DEV)
    s.count = torch.zeros(1, dtype=torch.int64, device=DEV)
    s.ws = torch.empty(L.lv_prune_workspace_size(n, p), dtype=torch.uint8, device=DEV)
    return s


def _inputs_subdivide(case, seed):
    n = case["voxels"]
    s = SimpleNamespace(case=case)
    half = case["half"]
    s.scene = _scene(n, seed, True, torch.float16 if half else torch.float32,
                     torch.bfloat16 if half else torch.float32)
    g = _gen(seed + 3)
    cam = np.array(synth.orbit_camera(1237, 822, 60.0, 3.0, 37.0, 15.0)["w2c"], np.float32).reshape(3, 4)
    s.z = (s.scene.geom[:, :3] @ torch.tensor(cam[2, :3], device=DEV) + float(cam[2, 3])).clamp_min(0.05)
    s.delta = s.z / 1071.3
    s.seen = (torch.rand(n, device=DEV, generator=g) < 0.6).to(torch.uint8)
    s.useful = torch.where(torch.rand(n, device=DEV, generator=g) < 0.5, torch.rand(n, device=DEV, generator=g) ** 4, 0.0)
    s.pruned = (torch.rand(n, device=DEV, generator=g) < 0.01).to(torch.uint8)
    s.moments = _moments(n, seed)
    return s


def _prepare_subdivide(case, seed):
    s = _inputs_subdivide(case, seed)
    n = case["voxels"]
    cap = n + 7 * (n * case["top_ppm"] // 1000000) + 16
    src = (s.scene.geom, s.scene.level, s.scene.density, s.scene.sh)
    s.out = [torch.zeros((cap,) + tuple(t.shape[1:]), dtype=t.dtype, device=DEV) for t in src]
    s.out_moments = [torch.zeros((cap, t.shape[1]), device=DEV) for t in s.moments]
    s.aux = []
    for a, b in zip(s.moments, s.out_moments):
        x = L.lv_aux_array()
        x.in_, x.out, x.width, x.elem_bytes, x.fill = a.data_ptr(), b.data_ptr(), a.shape[1], 4, 0
        s.aux.append(x)
    p = L.lv_subdiv_params()
    p.kappa, p.beta, p.top_ppm, p.l_max, p.budget, p.lo_ppm, p.hi_ppm = 1.0, 0.2, case["top_ppm"], 16, 1 << 40, 50000, 950000
    s.params = p
    s.vox = s.scene.voxels()
    s.vox_out = L.make_voxels(s.out[0], s.out[2], s.out[3], s.out[1])
    s.selected = torch.empty(n, dtype=torch.uint8, device=DEV)
    s.count = torch.zeros(1, dtype=torch.int64, device=DEV)
    s.status = torch.zeros(1, dtype=torch.int32, device=DEV)
    s.ws = torch.empty(L.lv_subdivide_workspace_size(n, p), dtype=torch.uint8, device=DEV)
    return s


def _sizes(case):
    k = max(1, case["views"] - 1)
    return ([case["width"] + (case["width1"] - case["width"]) * i // k for i in range(case["views"])],
            [case["height"] + (case["height1"] - case["height"]) * i // k for i in range(case["views"])])


def _prepare_loss(case, seed):
    s = SimpleNamespace(case=case)
    s.widths, s.heights = _sizes(case)
    s.gt = torch.cat([_image(w, h, seed + 31 * i) for i, (w, h) in enumerate(zip(s.widths, s.heights))])
    s.rgb = (s.gt + 0.1 * torch.randn(s.gt.shape, device=DEV, generator=_gen(seed + 4))).contiguous()
    s.lfp = _lf_params()
    s.ws = torch.empty(L.lv_lf_workspace_size(s.widths, s.heights), dtype=torch.uint8, device=DEV)
    s.loss, s.dL = torch.empty(case["views"], device=DEV), torch.empty_like(s.rgb)
    return s


def _prepare_vertex(case, seed):
    s = SimpleNamespace(case=case)
    s.scene = _scene(case["voxels"], seed)
    n = s.scene.n
    s.unit = float(s.scene.geom[:, 3].min())
    s.vidx = torch.empty((n, 8), dtype=torch.int32, device=DEV)
    s.count = torch.zeros(1, dtype=torch.int64, device=DEV)
    s.status = torch.zeros(1, dtype=torch.int32, device=DEV)
    s.sum, s.share = torch.empty(8 * n, device=DEV), torch.empty(8 * n, device=DEV)
    s.corners = torch.empty((n, 8), device=DEV)
    return s


def prepare(case, seed):
    return globals()["_prepare_" + case["kind"]](case, int(seed))


# ---------------------------------------------------------------------------- run
def _run_render(s):
    rgb, depth, T = s.ctx.forward(s.vox, stats=False)
    return {"rgb": rgb, "depth": depth, "T": T}


def _run_grad(s):
    s.ctx.reset_stats()
    out = rasterize(s.density, s.sh, s.scene, s.ctx)
    d_density, d_sh = torch.autograd.grad(out, (s.density, s.sh), s.grads)
    L.lv_unpack_wmax(s.ctx.wmax_packed, s.w_max)
    return {"rgb": out[0].detach(), "depth": out[1].detach(), "T": out[2].detach(), "d_density": d_density,
            "d_sh": d_sh, "w_max": s.w_max, "z_min": s.ctx.z_min, "delta_min": s.ctx.delta_min, "seen": s.ctx.seen}


def _iteration(s):
    ctx = s.ctx
    L.lv_lf_weights(s.gt, s.widths, s.heights, LF_T, s.lfp, s.lf_ws)
    ctx.reset_stats()
    ctx.forward(s.vox)
    L.lv_transmittance_loss(ctx.T, TC_WEIGHT, s.tc_loss, s.dL_dT, s.tr_ws)
    ctx.backward(s.vox, None, dL_dT=s.dL_dT, d_density=s.d_density, d_sh=s.d_sh, lf=(s.gt, s.lf_ws, None))
    L.lv_lf_loss_finish(s.widths, s.heights, s.loss, s.lf_ws)
    m = s.moments
    L.lv_adam_voxels(s.scene.density, s.scene.sh, s.d_density, s.d_sh, m[0], m[1], m[2], m[3], s.adam, s.tr_ws)


def _run_train(s):
    s.step()
    L.lv_unpack_wmax(s.ctx.wmax_packed, s.w_max)
    m = s.moments
    return {"loss": s.loss, "tc_loss": s.tc_loss, "rgb": s.ctx.rgb, "T": s.ctx.T, "w_max": s.w_max,
            "seen": s.ctx.seen, "d_density": s.d_density, "d_sh": s.d_sh, "density": s.scene.density,
            "sh": s.scene.sh, "m_density": m[0], "v_density": m[1], "m_sh": m[2], "v_sh": m[3]}


def _run_prune(s):
    L.lv_prune_depth_quantile(s.w_max, s.seen, s.z, s.ema, s.state, s.params, s.mask, s.count, s.ws)
    return {"mask": s.mask, "count": s.count, "ema": s.ema, "state": s.state, "pct": s.pct}


def _run_subdivide(s):
    L.lv_subdivide_priority(s.vox, s.delta, s.z, s.useful, s.seen, s.pruned, s.params, s.aux, s.vox_out, s.selected,
                            s.count, s.ws, s.status)
    return {"geom": s.out[0], "level": s.out[1], "density": s.out[2], "sh": s.out[3], "moments": s.out_moments,
            "selected": s.selected, "count": s.count, "status": s.status}


def _run_loss(s):
    L.lv_lf_weighted_loss(s.rgb, s.gt, s.widths, s.heights, LF_T, s.lfp, s.loss, s.dL, s.ws)
    return {"loss": s.loss, "dL": s.dL}


def _run_vertex(s):
    L.lv_build_vertex_index(s.scene.geom, s.unit, s.vidx, s.count, s.status)
    s.sum.zero_()
    s.share.zero_()
    L.lv_vertex_scatter_add(s.vidx, s.scene.density, s.sum, s.share)
    L.lv_vertex_gather(s.vidx, s.sum, s.corners)
    return {"vidx": s.vidx, "count": s.count, "sum": s.sum, "share": s.share, "corners": s.corners}


def run(state):
    return globals()["_run_" + state.case["kind"]](state)


# ---------------------------------------------------------------------------- least work
def work(case):
    """Each input read once and each output written once; FP32 operations of the arithmetic that every
    result needs (a dozen samples a pixel on opaque scenes, about sixty on semi-transparent ones)."""
    kind = case["kind"]
    if kind == "prune":
        n = case["voxels"]
        return {"bytes": n * (4 + 1 + 4 + 4 + 4 + 16 + 2 * (4 + 1) + 1), "flops": 20 * n}
    if kind == "subdivide":
        n, half = case["voxels"], case["half"]
        row = 16 + 1 + 8 * (2 if half else 4) + 48 * (2 if half else 4) + 4 * 112
        new = n + 7 * (n * case["top_ppm"] // 1000000)
        return {"bytes": n * (row + 14) + new * row, "flops": 20 * n}
    if kind == "loss":
        p = sum(w * h for w, h in zip(*_sizes(case)))
        return {"bytes": 36 * p, "flops": 80 * p}
    if kind == "vertex":
        n = case["voxels"]
        return {"bytes": n * (16 + 32 + 32 + 32 + 64), "flops": 40 * n}
    n, v = case["voxels"], case["views"]
    p = v * case["width"] * case["height"]
    row = 16 + 8 * (2 if case["half"] else 4) + 3 * (case["degree"] + 1) ** 2 * (2 if case["half"] else 4)
    samples = p * (12 if case["opaque"] else 60)
    b, f = n * row + 20 * p, 70 * samples + 100 * n * v
    if kind in ("grad", "train"):
        b += n * ((16 + 96) if case["half"] else (32 + 192)) + 20 * p + 21 * n
        f += 110 * samples
    if kind == "train":
        b += 2 * n * 56 * 4 + 4 * n * 56 * 4 - n * 224 + 24 * p   # parameters and moments updated
        f += 56 * 12 * n
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------- 64-bit results
def _sh_basis(d):
    x, y, z = d.unbind(-1)
    q = math.sqrt
    pi = math.pi
    return torch.stack([
        torch.full_like(x, 0.5 / q(pi)), q(3 / (4 * pi)) * y, q(3 / (4 * pi)) * z, q(3 / (4 * pi)) * x,
        q(15 / (4 * pi)) * x * y, q(15 / (4 * pi)) * y * z, q(5 / (16 * pi)) * (3 * z * z - 1),
        q(15 / (4 * pi)) * x * z, q(15 / (16 * pi)) * (x * x - y * y),
        q(35 / (32 * pi)) * y * (3 * x * x - y * y), q(105 / (4 * pi)) * x * y * z,
        q(21 / (32 * pi)) * y * (5 * z * z - 1), q(7 / (16 * pi)) * z * (5 * z * z - 3),
        q(21 / (32 * pi)) * x * (5 * z * z - 1), q(105 / (16 * pi)) * z * (x * x - y * y),
        q(35 / (32 * pi)) * x * (x * x - 3 * y * y)], -1)


_SIGNS = [[(i >> a & 1) * 2 - 1 for a in range(3)] for i in range(8)]


class _View64:
    """One view in 64 bits: every (pixel, voxel) crossing, in the pixels' front-to-back order."""

    def __init__(self, scene, cam, segment, t_stop=1e-4):
        geom = scene.geom.double()
        W, H = cam["width"], cam["height"]
        self.n_pix, self.n = W * H, scene.n
        m = torch.tensor(np.float32(cam["w2c"]).astype(np.float64), device=DEV).reshape(3, 4)
        R, t = m[:, :3], m[:, 3]
        fx, fy, cx, cy, zn = (float(np.float32(cam[k])) for k in ("fx", "fy", "cx", "cy", "z_near"))
        o = -(R.T @ t)
        cen, h = geom[:, :3], geom[:, 3]
        pc = cen @ R.T + t
        # depth order: the FP32 camera depth, one rounding per operation
        g32, m32 = scene.geom, m.float()
        z32 = g32[:, 0] * m32[2, 0] + g32[:, 1] * m32[2, 1]
        z32 = (z32 + g32[:, 2] * m32[2, 2]) + m32[2, 3]
        bits = z32.view(torch.int32).long()
        key = torch.where(bits < 0, -(bits & 0x7fffffff), bits) + (1 << 31)
        # candidate pixels of each voxel
        r = h * math.sqrt(3.0) * 1.001 + 1e-5
        vis = pc[:, 2] + r > zn
        for a, f, lo, hi in ((0, fx, -cx, W - cx), (1, fy, -cy, H - cy)):
            u = f * pc[:, a]
            vis &= u - lo * pc[:, 2] > -r * math.hypot(f, lo)
            vis &= u - hi * pc[:, 2] < r * math.hypot(f, hi)
        ids = vis.nonzero().flatten()
        corners = cen[ids, None, :] + h[ids, None, None] * torch.tensor(_SIGNS, dtype=torch.float64, device=DEV)
        q = corners @ R.T + t
        front = (q[..., 2] > zn).all(1)
        zc = q[..., 2].clamp_min(zn)
        u, v = fx * q[..., 0] / zc + cx, fy * q[..., 1] / zc + cy
        box = [torch.where(front, (u.amin(1) - 0.51).ceil().clamp(0, W), 0.0),
               torch.where(front, (u.amax(1) + 0.51).floor().clamp(0, W), float(W)),
               torch.where(front, (v.amin(1) - 0.51).ceil().clamp(0, H), 0.0),
               torch.where(front, (v.amax(1) + 0.51).floor().clamp(0, H), float(H))]
        x0, x1, y0, y1 = (b.long() for b in box)
        nx, ny = (x1 - x0).clamp_min(0), (y1 - y0).clamp_min(0)
        area = nx * ny
        pix, vox, tin, tout = [], [], [], []
        ends = area.cumsum(0)
        start, total = 0, int(ends[-1]) if ids.numel() else 0
        step = 1 << 23
        self.o, self.R, self.cam = o, R, (W, fx, fy, cx, cy, zn)
        for c0 in range(0, total, step):
            e = torch.arange(c0, min(total, c0 + step), device=DEV)
            j = torch.searchsorted(ends, e, right=True)
            k = e - (ends[j] - area[j])
            p = (y0[j] + k // nx[j]) * W + x0[j] + k % nx[j]
            i = ids[j]
            a, b, _ = self._chord(p, cen[i], h[i])
            hit = b > a
            pix.append(p[hit]); vox.append(i[hit]); tin.append(a[hit]); tout.append(b[hit])
        empty = torch.zeros(0, dtype=torch.int64, device=DEV)
        pix, vox = torch.cat(pix or [empty]), torch.cat(vox or [empty])
        tin, tout = torch.cat(tin or [empty.double()]), torch.cat(tout or [empty.double()])
        order = vox.sort(stable=True).indices
        order = order[((pix << 32) | key[vox])[order].sort(stable=True).indices]
        self.pix, self.vox = pix[order], vox[order]
        tin, tout = tin[order], tout[order]
        self.len, self.mid = tout - tin, 0.5 * (tin + tout)
        # density of each crossing: trilinear at the midpoint, or Simpson over the chord
        self.points = [(self.mid, 1.0)] if not segment else [(self.mid, 4 / 6), (tin, 1 / 6), (tout, 1 / 6)]
        self.cen, self.h = cen, h
        dens = scene.density.detach().double()
        raw = torch.zeros_like(self.mid)
        for tt, wt in self.points:
            raw += wt * sum(w * dens[self.vox, i] for i, w in enumerate(self._corner_weights(tt)))
        self.raw = raw
        self.x = raw.clamp_min(0) * self.len
        d = cen - o
        nn = d.norm(dim=1, keepdim=True)
        d = torch.where(nn > 0, d / nn.clamp_min(1e-300), torch.tensor([0.0, 0.0, 1.0], dtype=torch.float64, device=DEV))
        nb = (scene.sh_degree + 1) ** 2
        self.Y = _sh_basis(d)[:, :nb]
        self.c_raw = 0.5 + torch.einsum("njc,nj->nc", scene.sh.detach().double().reshape(-1, 16, 3)[:, :nb], self.Y)
        self.col = self.c_raw.clamp_min(0)
        # front to back, one crossing of every pixel at a time
        count = torch.bincount(self.pix, minlength=self.n_pix)
        first = count.cumsum(0) - count
        self.T = torch.ones(self.n_pix, dtype=torch.float64, device=DEV)
        self.used = torch.zeros_like(self.pix, dtype=torch.bool)
        self.Tk, before = torch.zeros_like(self.x), torch.zeros_like(self.x)
        alive, k = count.nonzero().flatten(), 0
        while alive.numel():
            e = first[alive] + k
            self.used[e] = True
            before[e] = self.T[alive]
            T = before[e] * torch.exp(-self.x[e])
            self.T[alive] = T
            self.Tk[e] = T
            k += 1
            alive = alive[(T >= t_stop) & (count[alive] > k)]
        self.w = -before * torch.expm1(-self.x)
        self.first, self.count = first, count
        self.rgb = torch.zeros((self.n_pix, 3), dtype=torch.float64, device=DEV).index_add_(
            0, self.pix, self.w[:, None] * self.col[self.vox])
        self.depth = torch.zeros(self.n_pix, dtype=torch.float64, device=DEV).index_add_(0, self.pix, self.w * self.mid)

    def _ray(self, p):
        W, fx, fy, cx, cy, zn = self.cam
        dc = torch.stack([((p % W).double() + 0.5 - cx) / fx, ((p // W).double() + 0.5 - cy) / fy,
                          torch.ones_like(p, dtype=torch.float64)], 1)
        d = dc @ self.R
        nn = d.norm(dim=1, keepdim=True)
        return d / nn, zn * nn[:, 0]

    def _chord(self, p, cen, h):
        d, near = self._ray(p)
        a, b = (cen - h[:, None] - self.o) / d, (cen + h[:, None] - self.o) / d
        return torch.maximum(torch.minimum(a, b).amax(1), near), torch.maximum(a, b).amin(1), d

    def _corner_weights(self, t):
        d, _ = self._ray(self.pix)
        u = ((self.o + t[:, None] * d - self.cen[self.vox]) / (2 * self.h[self.vox][:, None]) + 0.5).clamp(0, 1)
        for i in range(8):
            yield (u[:, 0] if i & 1 else 1 - u[:, 0]) * (u[:, 1] if i & 2 else 1 - u[:, 1]) * \
                (u[:, 2] if i & 4 else 1 - u[:, 2])

    def backward(self, g_rgb, g_depth, g_T, d_density, d_sh):
        a = (g_rgb[self.pix] * self.col[self.vox]).sum(1) + (0 if g_depth is None else g_depth[self.pix] * self.mid)
        q = self.w * a
        cum = torch.cat([q.new_zeros(1), q.cumsum(0)])
        after = cum[(self.first + self.count)[self.pix]] - cum[1:]
        ds = self.len * (self.Tk * a - after - (0 if g_T is None else (self.T * g_T)[self.pix]))
        ds = torch.where(self.used & (self.raw > 0), ds, 0.0)
        for tt, wt in self.points:
            for i, w in enumerate(self._corner_weights(tt)):
                d_density[:, i].index_add_(0, self.vox, wt * w * ds)
        dc = torch.zeros((self.n, 3), dtype=torch.float64, device=DEV).index_add_(
            0, self.vox, self.w[:, None] * g_rgb[self.pix])
        dc = torch.where(self.c_raw > 0, dc, 0.0)
        nb = self.Y.shape[1]
        d_sh.view(-1, 16, 3)[:, :nb] += self.Y[:, :, None] * dc[:, None, :]


def _too_long(case):
    """Crossings grow with the pixels, the views and the depth of the scene."""
    p = case["views"] * case["width"] * case["height"]
    return p * max(1.0, case["voxels"] / 2e5) ** 0.5 * (1.0 if case["opaque"] else 1.5) > 1.2e7


def _w_max(views, n):
    w = torch.zeros(n, dtype=torch.float64, device=DEV)
    for v in views:
        w.scatter_reduce_(0, v.vox, v.w, "amax")
    return w


def _exact_render(case, seed):
    s = _inputs_raster(case, seed)
    v = [_View64(s.scene, c, case["segment"]) for c in s.cams]
    return {k: torch.cat([getattr(x, k) for x in v]) for k in ("rgb", "depth", "T")}


def _grads64(s, views, g):
    d_density = torch.zeros((s.scene.n, 8), dtype=torch.float64, device=DEV)
    d_sh = torch.zeros((s.scene.n, 48), dtype=torch.float64, device=DEV)
    off = 0
    for v in views:
        e = off + v.n_pix
        v.backward(*[None if x is None else x[off:e].double() for x in g], d_density, d_sh)
        off = e
    return d_density, d_sh


def _exact_grad(case, seed):
    s = _inputs_raster(case, seed)
    v = [_View64(s.scene, c, case["segment"]) for c in s.cams]
    d_density, d_sh = _grads64(s, v, _image_grads(s, seed))
    out = {k: torch.cat([getattr(x, k) for x in v]) for k in ("rgb", "depth", "T")}
    return {**out, "d_density": d_density, "d_sh": d_sh, "w_max": _w_max(v, s.scene.n), "z_min": None,
            "delta_min": None, "seen": None}


def _lf64(rgb, gt, widths, heights):
    """Per-view LF-weighted loss and its gradient."""
    p = _lf_params()
    gamma = p.gamma_max * (LF_T - p.t0) / (p.t1 - p.t0)
    loss, dL, off = [], [], 0
    for w, h in zip(widths, heights):
        n = w * h
        a, b = rgb[off:off + n], gt[off:off + n].double()
        y = torch.nn.functional.pad(b.mean(1).reshape(1, 1, h, w), (1, 1, 1, 1), mode="replicate")[0, 0]
        l, r, u, d = y[:, :-2], y[:, 2:], y[:-2], y[2:]
        gx = (r[:-2] + 2 * r[1:-1] + r[2:]) - (l[:-2] + 2 * l[1:-1] + l[2:])
        gy = (d[:, :-2] + 2 * d[:, 1:-1] + d[:, 2:]) - (u[:, :-2] + 2 * u[:, 1:-1] + u[:, 2:])
        m = (gx * gx + gy * gy).sqrt().flatten()
        k = min(n, max(1, -(-p.pctl_ppm * n // 1000000)))
        top = m.sort().values[k - 1]
        sn = (m / top).clamp(0, 1) if top > 0 else torch.zeros_like(m)
        wt = (p.eps + 1 - sn) ** gamma
        wt = (wt / wt.mean())[:, None]
        loss.append((wt * (a - b) ** 2).sum() / (3 * n))
        dL.append(2.0 / (3 * n) * wt * (a - b))
        off += n
    return torch.stack(loss), torch.cat(dL)


def _exact_loss(case, seed):
    s = _prepare_loss(case, seed)
    loss, dL = _lf64(s.rgb.double(), s.gt, s.widths, s.heights)
    return {"loss": loss, "dL": dL}


def _exact_train(case, seed):
    s = _inputs_raster(case, seed)
    views = [_View64(s.scene, c, case["segment"]) for c in s.cams]
    rgb, T = torch.cat([v.rgb for v in views]), torch.cat([v.T for v in views])
    widths, heights = [c["width"] for c in s.cams], [c["height"] for c in s.cams]
    gt = torch.cat([_image(w, h, seed + 31 * i) for i, (w, h) in enumerate(zip(widths, heights))])
    loss, dL = _lf64(rgb, gt, widths, heights)
    out = {"loss": loss, "tc_loss": (TC_WEIGHT * (T * (1 - T)).mean())[None], "rgb": rgb, "T": T,
           "w_max": _w_max(views, s.scene.n), "seen": None}
    g = _grads64(s, views, (dL, None, TC_WEIGHT * (1 - 2 * T) / s.n_pix))
    del views
    out["d_density"], out["d_sh"] = g
    p, m = _adam(), _moments(s.scene.n, seed)
    b1, b2, eps = (float(np.float32(x)) for x in (p.beta1, p.beta2, p.eps))
    d = s.scene.density.double()
    tv = torch.zeros_like(d)
    for i in range(8):
        for bit in (1, 2, 4):
            tv[:, i] += d[:, i] - d[:, i ^ bit]
    for name, x, grad, mm, vv, lr in (("density", d, g[0] + 2 * p.tv_weight / s.scene.n * tv, m[0], m[1], p.lr_density),
                                      ("sh", s.scene.sh.double(), g[1], m[2], m[3], p.lr_sh)):
        mn = b1 * mm.double() + (1 - b1) * grad
        vn = b2 * vv.double() + (1 - b2) * grad * grad
        out["m_" + name], out["v_" + name] = mn, vn
        out[name] = x - lr * (mn / (1 - b1 ** p.step)) / ((vn / (1 - b2 ** p.step)).sqrt() + eps)
    return out


def _rank(ppm, m):
    return max(1, -(-ppm * m // 1000000))


def _exact_prune(case, seed):
    s = _prepare_prune(case, seed)
    p, nb = s.params, case["bins"]
    seen = s.seen.bool()
    zs = s.z[seen].sort().values
    f = torch.float32
    r = torch.tensor(p.pct_ema, dtype=f, device=DEV)
    pct = (1 - r) * s.pct + r * torch.stack([zs[_rank(q, zs.numel()) - 1] for q in (p.lo_ppm, p.hi_ppm)])
    bins = (nb * ((s.z - pct[0]) / (pct[1] - pct[0])).clamp(0, 1)).floor().clamp_max(nb - 1).long()
    x = torch.ones(case["voxels"], dtype=torch.float64, device=DEV)
    for b in range(nb):
        at = (seen & (bins == b)).nonzero().flatten()
        qa = p.q_ppm * p.anneal_ppm // 1000000
        qb = qa * (1000000 * nb - p.relax_ppm * abs(2 * b + 1 - nb)) // (1000000 * nb)
        if qb > 0 and at.numel():
            w = s.w_max[at]
            x[at] = (w > w.sort().values[_rank(qb, at.numel()) - 1]).double()
    a = float(np.float32(p.ema_alpha))
    ema = torch.where(seen, (1 - a) * s.ema.double() + a * x, s.ema.double())
    rd = float(r)
    step = torch.stack([zs[_rank(q, zs.numel()) - 1] for q in (p.lo_ppm, p.hi_ppm)]).double()
    return {"mask": None, "count": None, "ema": ema, "state": None, "pct": (1 - rd) * s.pct.double() + rd * step}


def _exact_subdivide(case, seed):
    s = _inputs_subdivide(case, seed)
    n, p = case["voxels"], SimpleNamespace(beta=np.float32(0.2), lo=50000, hi=950000)
    alive = s.pruned == 0
    ok = alive & (s.seen != 0)
    zs = s.z[ok].sort().values
    lo, hi = (zs[_rank(q, zs.numel()) - 1] for q in (p.lo, p.hi))
    zt = ((s.z - lo) / (hi - lo)).clamp(0, 1)
    prio = s.useful * (1 + torch.tensor(p.beta, device=DEV) * zt)
    eligible = ok & (s.scene.level < 16) & (s.scene.geom[:, 3] > s.delta)
    k = min(case["top_ppm"] * int(alive.sum()) // 1000000, int(eligible.sum()))
    order = torch.where(eligible, prio, -1.0).sort(descending=True, stable=True).indices[:k]
    split = torch.zeros(n, dtype=torch.bool, device=DEV)
    split[order] = True
    par, rest = split.nonzero().flatten(), (alive & ~split).nonzero().flatten()
    dens = s.scene.density.double()
    kids = []
    for c in range(8):                      # the parent's trilinear field at child c's corners
        for i in range(8):
            u = [0.5 * ((c >> a & 1) + (i >> a & 1)) for a in range(3)]
            kids.append(sum(dens[par, j] * math.prod(u[a] if j >> a & 1 else 1 - u[a] for a in range(3))
                            for j in range(8)))
    cap = n + 7 * (n * case["top_ppm"] // 1000000) + 16
    out = torch.zeros((cap, 8), dtype=torch.float64, device=DEV)
    out[:rest.numel()] = dens[rest]
    out[rest.numel():rest.numel() + 8 * k] = torch.stack(kids, 1).reshape(-1, 8)
    return {"geom": None, "level": None, "density": out, "sh": None, "moments": [None] * 4, "selected": None,
            "count": None, "status": None}


def _exact_vertex(case, seed):
    s = _prepare_vertex(case, seed)
    geom = s.scene.geom.double()
    sign = torch.tensor(_SIGNS, dtype=torch.float64, device=DEV)
    q = ((geom[:, None, :3] + geom[:, None, 3:] * sign) / s.unit).round().long() + (1 << 20)
    _, idx = ((q[..., 2] << 42) | (q[..., 1] << 21) | q[..., 0]).flatten().unique(return_inverse=True)
    total = torch.zeros(8 * s.scene.n, dtype=torch.float64, device=DEV)
    share = torch.zeros_like(total)
    total.index_add_(0, idx, s.scene.density.double().flatten())
    share.index_add_(0, idx, torch.ones_like(idx, dtype=torch.float64))
    return {"vidx": None, "count": None, "sum": total, "share": share, "corners": total[idx].reshape(-1, 8)}


def exact(case, seed):
    if case["kind"] in ("render", "grad", "train") and _too_long(case):
        return None
    with torch.no_grad():
        return globals()["_exact_" + case["kind"]](case, int(seed))
