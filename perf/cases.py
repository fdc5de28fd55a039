"""The work that this framework is used for, as a list of measurable cases.

Each case is a plain dict.  ``prepare`` makes what a program has in hand before the
call (a scene resident on the GPU, its occupancy structures, cameras, rays, targets,
gradient buffers), ``run`` is one pass through the package's public entry points,
and ``exact`` states what that pass returns in 64-bit arithmetic: it renders the same
inputs with plain torch from the method's definitions, without the package's kernels.

Kinds of cases:

* ``frame``      one call of ``Renderer.render``: a view (or several) of a scene.
* ``fast``       ``proposal.FastRenderer``: 16-bit tables, tensor-core MLP, learned
                 interval per ray and the fallback pass.
* ``train``      the render part of a training step as ``fit.fit`` runs it: rays in
                 tile order, Huber loss, reverse pass in the drawn order.
* ``autograd``   the same through ``RenderFunction`` and ``torch.autograd``.
* ``distortion`` the distortion regulariser of a training step and its reverse pass.
* ``proposal``   one gradient of the proposal network on a minibatch.
* ``occupancy``  the render-time occupancy pipeline after (or during) a fit.
* ``grid``       pyramid and distance grid from an occupancy grid.

Scenes: ``small`` (bounded, 4 levels), ``mid`` (8 levels to 512, 64^3 occupancy: the
reduced scene that the tests fit), ``hd`` (16 levels to 4096, 128^3 occupancy, the
benchmark's model), ``paper`` (hashed levels from 1024 up, 512^3 coarse grid and
occupancy, G at 256^3).
"""
import math
from dataclasses import replace

import numpy as np
import torch

from paper_2407_10482_gb300 import fit as F
from paper_2407_10482_gb300 import hdfit as HF
from paper_2407_10482_gb300 import ngprt as ng
from paper_2407_10482_gb300 import proposal as P
from paper_2407_10482_gb300 import scenes as S

DTYPES = {"f32": (ng.F32, torch.float32), "f16": (ng.F16, torch.float16), "bf16": (ng.BF16, torch.bfloat16)}


def listed():
    return [
        # a preview or probe view of the small bounded scene: the smallest call in use,
        # bound by latency and launches
        {"name": "small_view_f32", "kind": "frame", "scene": "small", "dtype": "f32", "views": 1, "W": 64, "H": 64},
        # the benchmark's plain renderer: one full-HD frame, FP32 tables and MLP
        {"name": "hd_frame_f32", "kind": "frame", "scene": "hd", "dtype": "f32", "views": 1, "W": 1920, "H": 1080},
        # the deployed precision form: FP16 tables, MLP on tensor cores
        {"name": "hd_frame_f16", "kind": "frame", "scene": "hd", "dtype": "f16", "views": 1, "W": 1920, "H": 1080},
        # BF16 tables in a window of odd size, with the per-ray counts a viewer's
        # statistics overlay reads
        {"name": "hd_window_bf16", "kind": "frame", "scene": "hd", "dtype": "bf16", "views": 1, "W": 1283, "H": 721},
        # the fastest form: learned interval, fallback, FP16
        {"name": "hd_fast_f16", "kind": "fast", "scene": "hd", "dtype": "f16", "views": 1, "W": 1920, "H": 1080},
        # the paper's render-time shape with the baked block-sparse coarse grid
        {"name": "paper_frame_f16", "kind": "frame", "scene": "paper", "dtype": "f16", "views": 1, "W": 1920,
         "H": 1080, "L": 2, "sparse": True},
        # the training batch of a fit: 2^18 rays of 8 views
        {"name": "hd_train_rays", "kind": "train", "scene": "hd", "dtype": "f32", "views": 8, "W": 1920, "H": 1080,
         "rays": 1 << 18},
        # a small model trained through torch.autograd on an odd number of free rays
        {"name": "mid_autograd", "kind": "autograd", "scene": "mid", "dtype": "f32", "rays": 50001},
        # the regulariser of the same fit, at its batch
        {"name": "hd_distortion", "kind": "distortion", "scene": "hd", "dtype": "f32", "views": 8, "W": 960, "H": 540,
         "rays": 1 << 18},
        # one minibatch of the proposal's training
        {"name": "proposal_batch", "kind": "proposal", "views": 64, "W": 1920, "H": 1080, "rays": 1 << 15},
        # occupancy refreshed from the model and its training views
        {"name": "hd_occupancy", "kind": "occupancy", "scene": "hd", "dtype": "f32", "views": 4, "W": 960, "H": 540},
        # the paper's 512^3 occupancy: pyramid and distance grid
        {"name": "paper_grid", "kind": "grid", "R": 512, "levels": 5, "dist_level": 1},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["frame", "frame", "frame", "fast", "train", "autograd", "distortion", "proposal", "occupancy",
                       "grid"])
    # an image of 2^12 to 1920x1080 pixels, odd sizes among them
    px = _log(rng, 4096, 1920 * 1080)
    W = max(33, min(1920, int(round(math.sqrt(px * rng.uniform(1.0, 1.9))))))
    H = max(31, min(1080, px // W))
    if kind == "frame":
        scene = rng.choice(["small", "mid", "hd", "hd", "paper"])
        c = {"kind": kind, "scene": scene, "dtype": rng.choice(["f32", "f16", "bf16"]),
             "views": rng.choice([1, 1, 2, 3]), "W": W, "H": H}
        if c["views"] > 1:
            c["W"], c["H"] = min(W, 960), min(H, 540)
        if scene == "paper":
            c["L"] = rng.choice([2, 3])
            c["sparse"] = rng.random() < 0.5
        return c
    if kind == "fast":
        return {"kind": kind, "scene": rng.choice(["mid", "hd"]), "dtype": "f16", "views": 1, "W": W, "H": H}
    if kind == "grid":
        R = rng.choice([32, 64, 128, 256])
        return {"kind": kind, "R": R, "levels": rng.choice([3, 4, 5]), "dist_level": rng.choice([0, 1])}
    if kind == "proposal":
        return {"kind": kind, "views": rng.choice([8, 64]), "W": W, "H": H, "rays": _log(rng, 1000, 1 << 16)}
    if kind == "autograd":
        return {"kind": kind, "scene": rng.choice(["small", "mid"]), "dtype": "f32", "rays": _log(rng, 1000, 1 << 17)}
    scene = rng.choice(["mid", "hd"])
    if kind == "occupancy":
        return {"kind": kind, "scene": scene, "dtype": "f32", "views": rng.choice([1, 3]), "W": min(W, 960),
                "H": min(H, 540)}
    return {"kind": kind, "scene": scene, "dtype": "f32", "views": rng.choice([3, 8]), "W": W, "H": H,
            "rays": _log(rng, 4096, 1 << 18)}


# ---------------------------------------------------------------------- inputs

def _cfg(case, seed):
    scene = case["scene"]
    kw = dict(seed=1000 + seed)
    if "W" in case:
        kw.update(W=case["W"], H=case["H"])
    if scene == "small":
        return S.small_config(blob_std=(0.05, 0.15), **kw)
    if scene == "mid":
        return S.hd_config(L=8, N=S.level_resolutions(16, 512, 8), T_log2=16, R_O=64, n_occ_levels=4, **kw)
    if scene == "paper":
        return S.paper_config(L=case["L"], **kw)
    return S.hd_config(**kw)


def _scene(case, seed):
    """The scene arrays of the case: tables, coarse grid, MLP weights, occupancy grid."""
    cfg = _cfg(case, seed)
    sc = S.make_scene(cfg) if cfg.bounded else S.make_scene_torch(cfg)
    return cfg, sc


def _mlp(case):
    return "f32" if case["dtype"] == "f32" else "f16"


def _cams(case, cfg, seed):
    return S.orbit_cameras(cfg, case["views"], azimuth0=7.0 + 31.0 * (seed % 11), step_deg=360.0 / case["views"])


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(77 + seed)
    return g


def _pixels(case, seed):
    n = case["views"] * case["W"] * case["H"]
    return torch.randint(0, n, (case["rays"],), device="cuda", generator=_gen(seed)).to(torch.int32)


def _free_rays(case, cfg, seed):
    o, d = S.random_rays(case["rays"], 5 + seed, cfg.bounded)
    return torch.as_tensor(o).cuda(), torch.as_tensor(d).cuda()


def _proposal_weights(seed):
    """Weights of a proposal network that predicts intervals around a scene on an orbit of
    radius 3: t_near near 2, t_far near 8, opacity near 1, each varying from ray to ray."""
    w = P.init_weights(seed, "cuda").clone()
    w[-99:] *= 0.3
    w[-3:] = torch.tensor([-1.9, 0.0, 4.0], device="cuda")
    return w


def _occupied(R, seed):
    """A blob-shaped occupancy grid of R^3 voxels, about a tenth of them occupied."""
    g = _gen(seed)
    c = torch.rand(24, 3, device="cuda", generator=g) * 0.6 + 0.2
    rad = torch.rand(24, device="cuda", generator=g) * 0.07 + 0.03
    x = (torch.arange(R, device="cuda") + 0.5) / R
    occ = torch.zeros(R, R, R, dtype=torch.bool, device="cuda")
    for k in range(24):
        dx, dy, dz = ((x - c[k, a]) ** 2 for a in range(3))
        occ |= dz[:, None, None] + dy[None, :, None] + dx[None, None, :] < rad[k] ** 2
    return occ.to(torch.uint8).reshape(-1)


def _device_scene(case, cfg, sc):
    return ng.DeviceScene(cfg, sc.tables, sc.coarse, sc.mlp_w, table_dtype=DTYPES[case["dtype"]][0],
                          mlp_dtype=DTYPES[_mlp(case)][0])


def prepare(case, seed):
    k = case["kind"]
    st = {"case": case, "kind": k}
    if k == "grid":
        st["occ"] = _occupied(case["R"], seed)
        return st
    if k == "proposal":
        cfg = S.hd_config(W=case["W"], H=case["H"])
        cams, n_cams = ng.cameras_struct(_cams(case, cfg, seed), case["W"], case["H"])
        n = case["rays"]
        r = torch.rand(n, 3, device="cuda", generator=_gen(seed + 1))
        # interval targets of opaque and half-transparent rays, some of them empty
        t0 = 1.6 + 1.8 * r[:, 0]
        A = torch.where(r[:, 2] < 0.1, torch.zeros_like(t0), 0.5 + 0.5 * r[:, 2])
        tg = torch.stack([t0 * (A > 0), (t0 + 0.1 + 6.0 * r[:, 1] ** 3) * (A > 0), A], 1).contiguous()
        w = _proposal_weights(seed)
        st.update(cams=cams, n_cams=n_cams, pix=_pixels(case, seed), targets=tg, w=w, g=torch.zeros_like(w),
                  loss=torch.zeros(1, device="cuda"))
        return st
    cfg, sc = _scene(case, seed)
    ds = _device_scene(case, cfg, sc)
    docc = ng.DeviceOcc(sc.occ, cfg.R_O, cfg.n_occ_levels, dist_level=cfg.dist_level)
    if case.get("sparse"):
        ds.sparsify_coarse(docc)
    opts = S.default_options(cfg)
    st.update(cfg=cfg, ds=ds, occ=docc, opts=opts, rend=ng.Renderer(ds, docc))
    if k != "autograd":
        st["cams"] = _cams(case, cfg, seed)
    if k == "fast":
        n = case["views"] * cfg.W * cfg.H
        st.update(fast=P.FastRenderer(ds, docc, _proposal_weights(seed)), rgb=torch.empty(n, 3, device="cuda"),
                  depth=torch.empty(n, device="cuda"), opacity=torch.empty(n, device="cuda"))
    elif k == "train":
        st.update(pix=_pixels(case, seed), targets=torch.rand(case["rays"], 3, device="cuda", generator=_gen(seed + 1)),
                  grads=[torch.zeros_like(t) for t in (ds.tables, ds.coarse, ds.mlp_w)],
                  loss=torch.zeros(1, device="cuda"), d_rgb=torch.empty(case["rays"], 3, device="cuda"))
    elif k == "autograd":
        o, d = _free_rays(case, cfg, seed)
        st.update(rays=dict(rays_o=o, rays_d=d),
                  targets=torch.rand(case["rays"], 3, device="cuda", generator=_gen(seed + 1)))
        for t in (ds.tables, ds.coarse, ds.mlp_w):
            t.requires_grad_(True)
    elif k == "distortion":
        cams, n_cams = ng.cameras_struct(st["cams"], cfg.W, cfg.H)
        st.update(pix=_pixels(case, seed), cam_arr=cams, n_cams=n_cams, ro=ng.render_opts(opts),
                  grads=[torch.zeros_like(t) for t in (ds.tables, ds.coarse)], loss=torch.zeros(1, device="cuda"),
                  dist_state=torch.empty(case["rays"], 4, device="cuda"))
    return st


# ------------------------------------------------------------------------ runs

def run(st):
    return globals()["_run_" + st["kind"]](st)


def _run_frame(st):
    c = st["cfg"]
    return st["rend"].render(st["opts"], cams=st["cams"], W=c.W, H=c.H, stats=st["case"]["dtype"] == "bf16")


def _run_fast(st):
    c = st["cfg"]
    st["fast"].render(st["opts"], st["cams"], c.W, c.H, st["rgb"], st["depth"], st["opacity"])
    return {"rgb": st["rgb"], "depth": st["depth"], "opacity": st["opacity"]}


def _run_train(st):
    c, pix, n = st["cfg"], st["pix"], st["pix"].numel()
    perm, back = F.tile_order(pix, c.W, c.H)
    out = st["rend"].render(st["opts"], cams=st["cams"], W=c.W, H=c.H, pixel_ids=pix[perm].contiguous(), state=True)
    st["loss"].zero_()
    ng.ngprt_huber_loss(out["rgb"], st["targets"][perm].contiguous(), 3 * n, 0.1, 1.0 / (3 * n), st["loss"],
                        st["d_rgb"])
    for g in st["grads"]:
        g.zero_()
    st["rend"].backward(st["opts"], out["state"][back].contiguous(), st["d_rgb"][back].contiguous(), None, None,
                        *st["grads"], cams=st["cams"], W=c.W, H=c.H, pixel_ids=pix)
    return {"loss": st["loss"], "rgb": out["rgb"], "tables": st["grads"][0], "coarse": st["grads"][1],
            "mlp_w": st["grads"][2]}


def _run_autograd(st):
    ds = st["ds"]
    p = (ds.tables, ds.coarse, ds.mlp_w)
    rgb, depth, opacity = ng.RenderFunction.apply(*p, st["rend"], st["opts"], st["rays"])
    loss = ((rgb - st["targets"]) ** 2).mean() + 0.01 * depth.mean() + 0.1 * opacity.mean()
    g = torch.autograd.grad(loss, p)
    return {"loss": loss, "rgb": rgb, "depth": depth, "opacity": opacity, "tables": g[0], "coarse": g[1],
            "mlp_w": g[2]}


def _run_distortion(st):
    n, a = st["pix"].numel(), (st["ds"].struct, st["occ"].struct, st["cam_arr"], st["n_cams"], st["pix"], None, None)
    st["loss"].zero_()
    for g in st["grads"]:
        g.zero_()
    ng.ngprt_distortion_loss(*a, n, st["ro"], 0.01 / n, st["dist_state"], st["loss"])
    ng.ngprt_distortion_backward(*a, n, st["ro"], st["dist_state"], 0.01 / n, *st["grads"])
    return {"loss": st["loss"], "state": st["dist_state"], "tables": st["grads"][0], "coarse": st["grads"][1]}


def _run_proposal(st):
    st["g"].zero_()
    st["loss"].zero_()
    pc = P.ProposalConfig()
    ng.ngprt_propose_backward(st["w"], st["cams"], st["n_cams"], st["pix"], None, None, st["pix"].numel(),
                              pc.in_scale, pc.t_scale, st["targets"], st["g"], st["loss"])
    return {"loss": st["loss"], "w": st["g"]}


def _run_occupancy(st):
    c, ds = st["cfg"], st["ds"]
    R = c.R_O
    occ = torch.empty(R ** 3, dtype=torch.uint8, device="cuda")
    sigma = torch.empty(R ** 3, device="cuda")
    ng.ngprt_occupancy_from_density(ds.struct, ng.render_opts(st["opts"]), R, 20.0, occ, sigma)
    vis = HF.visibility_occupancy(ds, st["occ"], st["opts"], st["cams"], c.W, c.H, 1e-3, 1, occ)
    out = ng.DeviceOcc(vis, R, c.n_occ_levels)
    return {"density": occ, "sigma": sigma, "visible": vis, "bits": out.bits, "dist": out.dist}


def _run_grid(st):
    c = st["case"]
    out = ng.DeviceOcc(st["occ"], c["R"], c["levels"], dist_level=c["dist_level"])
    return {"bits": out.bits, "dist": out.dist}


# ------------------------------------------------------------------------ work

def work(case):
    """Bytes: every scene array, occupancy structure and ray input once, every output once.
    Flops: the multiply-adds of about 20 samples a ray (trilinear sums of the coarse
    channels and of each level's 8, the gates) and of the deferred MLP."""
    k = case["kind"]
    if k == "grid":
        n = case["R"] ** 3
        return {"bytes": n + n / 7 + n / 8 ** case["dist_level"], "flops": 0.0}
    if k == "proposal":
        return {"bytes": 16.0 * case["rays"] + 8 * 1315, "flops": 3.0 * 2 * 1312 * case["rays"]}
    cfg = _cfg(case, 0)
    size = 4 if case["dtype"] == "f32" else 2
    tables, ch = S.table_entries(cfg) * 8, S.coarse_channels(cfg)
    coarse = cfg.R_C ** 3 * ch
    if case.get("sparse"):
        coarse = coarse * 0.37
    scene = (tables + coarse) * size + cfg.R_O ** 3 / 7 + cfg.R_O ** 3 / 8 ** cfg.dist_level
    rays = case["rays"] if "rays" in case else case["views"] * cfg.W * cfg.H
    sample = 2.0 * 8 * (ch + 8 * cfg.L) + 16.0 * cfg.L
    mlp = 2.0 * S.mlp_param_count(cfg)
    per_ray, times, extra = 20.0, 1.0, rays * 20.0
    if k in ("train", "autograd"):
        times, extra = 3.0, rays * 40.0 + (tables + coarse) * 4
    elif k == "distortion":
        times, mlp, sample, extra = 3.0, 0.0, sample / 8, rays * 20.0 + (tables + coarse) * 4
    elif k == "occupancy":
        mlp, extra = 0.0, cfg.R_O ** 3 * 8.0
    return {"bytes": scene + extra, "flops": times * rays * (per_ray * sample + mlp)}


# ----------------------------------------------------------------- 64-bit values

class _Model:
    """The scene of a case in plain torch: grids as stored (16-bit forms rounded), and the
    occupancy pyramid and distance grid from the definitions."""

    def __init__(self, case, cfg, sc):
        td = DTYPES[case["dtype"]][1]
        dev = "cuda"
        self.cfg = cfg
        self.tables = torch.as_tensor(sc.tables, device=dev).to(td)
        self.coarse = torch.as_tensor(sc.coarse, device=dev).to(td)
        w = torch.as_tensor(sc.mlp_w, device=dev).to(DTYPES[_mlp(case)][1]).double()
        self.w, at = [], 0
        for o, i in S.mlp_shapes(cfg):
            self.w.append(w[at:at + o * i].reshape(o, i))
            at += o * i
        R = cfg.R_O
        occ = torch.as_tensor(sc.occ, device=dev).reshape(R, R, R) != 0
        self.levels = [occ]
        for _ in range(cfg.n_occ_levels - 1):
            r = self.levels[-1].shape[0] // 2
            self.levels.append(self.levels[-1].reshape(r, 2, r, 2, r, 2).any(5).any(3).any(1))
        self.G = _box_distance(self.levels[cfg.dist_level])
        T = 1 << cfg.T_log2
        self.kind = [(n, n ** 3 <= T) for n in cfg.N]
        self.off = np.cumsum([0] + [min(n ** 3, T) for n in cfg.N]).tolist()
        self.mask = T - 1

    def corners(self, u, n):
        p = u * (n - 1)
        b = p.floor().clamp(0, n - 2)
        w = p - b
        b = b.long()
        c = torch.arange(8, device=u.device)
        bit = torch.stack([c & 1, (c >> 1) & 1, (c >> 2) & 1], 1)
        v = b[:, None, :] + bit[None]
        cw = torch.where(bit[None] == 1, w[:, None, :], 1 - w[:, None, :]).prod(2)
        return v, cw

    def coarse_rows(self, u):
        R = self.cfg.R_C
        v, cw = self.corners(u, R)
        return v[..., 0] + R * (v[..., 1] + R * v[..., 2]), cw

    def level_rows(self, l, u):
        n, dense = self.kind[l]
        v, cw = self.corners(u, n)
        if dense:
            row = v[..., 0] + n * (v[..., 1] + n * v[..., 2])
        else:
            m = 0xFFFFFFFF
            row = (v[..., 0] ^ ((v[..., 1] * 2654435761) & m) ^ ((v[..., 2] * 805459861) & m)) & self.mask
        return row + self.off[l], cw

    def features(self, u, chunk=1 << 19):
        out = torch.empty(len(u), 8, dtype=torch.float64, device=u.device)
        for s in range(0, len(u), chunk):
            x = u[s:s + chunk]
            row, cw = self.coarse_rows(x)
            a = (self.coarse[row].double() * cw[..., None]).sum(1)
            f = a[:, :8].clone()
            gate = torch.sigmoid(a[:, 8:]).reshape(len(x), self.cfg.L, 2)
            for l in range(self.cfg.L):
                row, cw = self.level_rows(l, x)
                e = (self.tables[row].double() * cw[..., None]).sum(1)
                f[:, 0] += gate[:, l, 0] * e[:, 0]
                f[:, 1:] += gate[:, l, 1:2] * e[:, 1:]
            out[s:s + chunk] = f
        return out

    def feature_grads(self, u, gf, chunk=1 << 19):
        """Sums over samples of the gradients of features(): (tables, coarse)."""
        gt = torch.zeros(self.tables.shape, dtype=torch.float64, device=u.device)
        gc = torch.zeros(self.coarse.shape, dtype=torch.float64, device=u.device)
        for s in range(0, len(u), chunk):
            x, g = u[s:s + chunk], gf[s:s + chunk]
            row_c, cw_c = self.coarse_rows(x)
            a = (self.coarse[row_c].double() * cw_c[..., None]).sum(1)
            gate = torch.sigmoid(a[:, 8:]).reshape(len(x), self.cfg.L, 2)
            ga = torch.empty_like(a)
            ga[:, :8] = g
            for l in range(self.cfg.L):
                row, cw = self.level_rows(l, x)
                e = (self.tables[row].double() * cw[..., None]).sum(1)
                om, be = gate[:, l, 0], gate[:, l, 1]
                ga[:, 8 + 2 * l] = g[:, 0] * e[:, 0] * om * (1 - om)
                ga[:, 9 + 2 * l] = (g[:, 1:] * e[:, 1:]).sum(1) * be * (1 - be)
                ge = torch.cat([(om * g[:, 0])[:, None], be[:, None] * g[:, 1:]], 1)
                gt.index_add_(0, row.reshape(-1), (cw[..., None] * ge[:, None, :]).reshape(-1, 8))
            gc.index_add_(0, row_c.reshape(-1), (cw_c[..., None] * ga[:, None, :]).reshape(-1, ga.shape[1]))
        return gt, gc

    def shade(self, Cd, Fv, A, d, bg=0.0):
        x, y, z = d.unbind(1)
        xx, yy, zz = x * x, y * y, z * z
        s = math.sqrt
        pi = math.pi
        sh = [0.5 * s(1 / pi) + 0 * x, s(3 / (4 * pi)) * y, s(3 / (4 * pi)) * z, s(3 / (4 * pi)) * x,
              0.5 * s(15 / pi) * x * y, 0.5 * s(15 / pi) * y * z, 0.25 * s(5 / pi) * (3 * zz - 1),
              0.5 * s(15 / pi) * x * z, 0.25 * s(15 / pi) * (xx - yy), 0.25 * s(35 / (2 * pi)) * y * (3 * xx - yy),
              0.5 * s(105 / pi) * x * y * z, 0.25 * s(21 / (2 * pi)) * y * (5 * zz - 1),
              0.25 * s(7 / pi) * z * (5 * zz - 3), 0.25 * s(21 / (2 * pi)) * x * (5 * zz - 1),
              0.25 * s(105 / pi) * z * (xx - yy), 0.25 * s(35 / (2 * pi)) * x * (xx - 3 * yy)]
        h = torch.cat([Cd, Fv, torch.stack(sh, 1), torch.zeros(len(x), 9, dtype=Cd.dtype, device=Cd.device)], 1)
        for w in self.w[:-1]:
            h = torch.relu(h @ w.T)
        return A[:, None] * torch.sigmoid(Cd + h @ self.w[-1].T) + (1 - A[:, None]) * bg


def _box_distance(occ):
    """floor of the distance between voxel boxes to the nearest occupied voxel, at most 255."""
    big = 1 << 28
    D = torch.where(occ, 0, big).to(torch.int32)
    R = occ.shape[0]
    for axis in (2, 1, 0):
        best = D.clone()
        for s in range(1, min(R, 258)):
            gap = (s - 1) ** 2
            lo, hi = D.narrow(axis, 0, R - s) + gap, D.narrow(axis, s, R - s) + gap
            b = best.narrow(axis, s, R - s)
            torch.minimum(b, lo, out=b)
            b = best.narrow(axis, 0, R - s)
            torch.minimum(b, hi, out=b)
        D = best
    return D.double().sqrt().floor().clamp(max=255).to(torch.uint8)


def _camera_rays(cams, W, H, ids):
    c = torch.as_tensor(cams, device="cuda").double()[ids // (W * H)]
    rem = ids % (W * H)
    px = ((rem % W).double() + 0.5 - c[:, 14]) / c[:, 12]
    py = ((rem // W).double() + 0.5 - c[:, 15]) / c[:, 13]
    m = c[:, :12].reshape(-1, 3, 4)
    return m[:, :, 3], px[:, None] * m[:, :, 0] + py[:, None] * m[:, :, 1] + m[:, :, 2]


def _contract(x, bounded):
    r = x.norm(dim=1)
    if bounded:
        return x, r
    far = r > 1
    k = torch.where(far, (2 - 1 / r.clamp(min=1)) / r.clamp(min=1), torch.ones_like(r))
    return x * k[:, None], r


def _speed(x, d, r):
    """J(x) d of the contraction beyond the unit ball."""
    k = (2 - 1 / r) / r
    m = (x * d).sum(1) * 2 * (1 - r) / r ** 4
    return k[:, None] * d + m[:, None] * x


def _march(model, o, d, opts, t_lo=None, t_hi=None, on_sample=None):
    """Walks the rays; on_sample(rays, u, t, delta) -> rays to stop.  Returns (unit d, counts)."""
    cfg, bounded = model.cfg, model.cfg.bounded
    B = 1.0 if bounded else 2.0
    R = cfg.R_O
    d = d / d.norm(dim=1, keepdim=True)
    n = len(o)
    inf = float("inf")
    f32 = lambda v: float(np.float32(v))  # noqa: E731
    if bounded:
        t0, t1 = (-1 - o) / d, (1 - o) / d
        t, t_out = torch.minimum(t0, t1).amax(1), torch.maximum(t0, t1).amin(1)
    else:
        b = (o * d).sum(1)
        disc = b * b - (o * o).sum(1) + f32(opts.r_far) ** 2
        s = disc.clamp(min=0).sqrt()
        t, t_out = -b - s, torch.where(disc >= 0, -b + s, torch.full_like(b, -inf))
    t = t.clamp(min=f32(opts.t_min))
    if t_lo is not None:
        t, t_out = torch.maximum(t, t_lo), torch.minimum(t_out, t_hi)
    dt0 = f32(np.float32(opts.step_base) * np.float32(opts.step_gamma))
    counts = torch.zeros(n, 2, dtype=torch.int32, device=o.device)
    vg = 2 * B / model.G.shape[0]
    live = torch.nonzero(t < t_out).squeeze(1)
    while len(live):
        counts[live, 0] += 1
        tt, dd = t[live], d[live]
        x = o[live] + tt[:, None] * dd
        y, r = _contract(x, bounded)
        u = (y + B) / (2 * B)
        f = (u * R).floor().clamp(0, R - 1).long()
        empty = torch.full((len(live),), -1, device=o.device)
        for k in range(cfg.n_occ_levels):
            c = f >> k
            hit = model.levels[k][c[:, 2], c[:, 1], c[:, 0]]
            empty = torch.where(hit, empty, torch.full_like(empty, k))
        occ = empty < 0
        step = torch.zeros_like(tt)
        i = torch.nonzero(~occ).squeeze(1)
        if len(i):
            step[i] = _empty_step(model, x[i], y[i], dd[i], r[i], f[i], empty[i], B, R)
            j = i[empty[i] > cfg.dist_level]
            if len(j) and opts.use_dist:
                c = f[j] >> cfg.dist_level
                g = model.G[c[:, 2], c[:, 1], c[:, 0]].double() * vg
                s = g
                if not bounded:
                    far = r[j] > 1
                    b2 = torch.cross(x[j], dd[j], dim=1).square().sum(1)
                    rl = torch.maximum((r[j] + 1) / 2, b2.sqrt())
                    q = (2 * rl - 1) / rl
                    s = torch.where(far, torch.maximum(g, torch.minimum(g * rl ** 2 / (1 + q * q * b2).sqrt(),
                                                                        (r[j] - 1) / 2)), g)
                step[j] = torch.where(g > 0, torch.maximum(s, step[j]) if opts.dist_rule == 1 else s, step[j])
        i = torch.nonzero(occ).squeeze(1)
        stop = torch.zeros(len(live), dtype=torch.bool, device=o.device)
        if len(i):
            dt = torch.full_like(tt[i], dt0) if bounded else dt0 * r[i].clamp(min=1)
            counts[live[i], 1] += 1
            stop[i] = on_sample(live[i], u[i], tt[i], torch.minimum(dt, t_out[live[i]] - tt[i]))
            step[i] = dt
        t[live] = tt + step
        c = counts[live]
        go = ~stop & (t[live] < t_out[live]) & (c[:, 0] < opts.max_march) & (c[:, 1] < opts.max_samples)
        live = live[go]
    return d, counts


def _empty_step(model, x, y, d, r, f, k, B, R):
    """The step that carries the image 2% of a finest voxel past the exit face of the empty
    voxel of level k: along the image's direction, then one Newton step on the exit axis."""
    curved = (r > 1) & (not model.cfg.bounded)
    v = torch.where(curved[:, None], _speed(x, d, r.clamp(min=1)), d)
    side = 2 * B * (2.0 ** k.double()) / R
    guard = 0.02 * 2 * B / R
    lo = (f >> k[:, None]).double() * side[:, None] - B
    plane = torch.where(v > 0, lo + side[:, None] + guard, lo - guard)
    ta = torch.where(v != 0, (plane - y) / v, torch.full_like(v, float("inf")))
    s0, ax = ta.min(1)
    s0 = s0.clamp(min=0)
    pick = lambda a: a.gather(1, ax[:, None]).squeeze(1)  # noqa: E731
    x1 = x + s0[:, None] * d
    y1, r1 = _contract(x1, False)
    v1 = torch.where((r1 > 1)[:, None], _speed(x1, d, r1.clamp(min=1)), d)
    y1 = torch.where((r1 > 1)[:, None], y1, x1)
    c = (pick(plane) - pick(y1)) / pick(v1)
    h = 0.5 * s0
    s1 = s0 + torch.minimum(torch.maximum(c, -h), h)
    return torch.where(curved & (pick(v1) * pick(v) > 0), s1, s0)


def _render(model, o, d, opts, t_lo=None, t_hi=None):
    """Composite state per ray (C_d, F, A, depth) by the march, in 64 bits."""
    n = len(o)
    T = torch.ones(n, dtype=torch.float64, device=o.device)
    acc = torch.zeros(n, 9, dtype=torch.float64, device=o.device)
    t_term = float(np.float32(opts.t_term))

    def sample(i, u, t, delta):
        f = model.features(u)
        tr = torch.exp(-torch.exp(f[:, 0]) * delta)
        w = T[i] * (1 - tr)
        acc[i] += w[:, None] * torch.cat([f[:, 1:], torch.ones_like(t)[:, None], t[:, None]], 1)
        T[i] *= tr
        return T[i] < t_term

    dn, counts = _march(model, o, d, opts, t_lo, t_hi, sample)
    return acc[:, :3], acc[:, 3:7], acc[:, 7], acc[:, 8], dn, counts


def _samples(model, o, d, opts):
    """(u, t, delta) of the samples of every ray as [rays, most samples] arrays, a mask of
    those that exist, and the unit directions."""
    n = len(o)
    T = torch.ones(n, dtype=torch.float64, device=o.device)
    got = []
    t_term = float(np.float32(opts.t_term))

    def sample(i, u, t, delta):
        T[i] *= torch.exp(-torch.exp(model.features(u)[:, 0]) * delta)
        got.append((i, u, t, delta))
        return T[i] < t_term

    dn, counts = _march(model, o, d, opts, None, None, sample)
    at = torch.zeros(n, dtype=torch.long, device=o.device)
    most = max(1, int(counts[:, 1].max()))
    u = torch.zeros(n, most, 3, dtype=torch.float64, device=o.device)
    t, delta = (torch.zeros(n, most, dtype=torch.float64, device=o.device) for _ in range(2))
    for i, a, b, c in got:
        u[i, at[i]], t[i, at[i]], delta[i, at[i]] = a, b, c
        at[i] += 1
    mask = torch.arange(most, device=o.device)[None] < at[:, None]
    return u, t, delta, mask, dn


def _weights(f0, delta, mask):
    tr = torch.where(mask, torch.exp(-torch.exp(f0) * delta), torch.ones_like(f0))
    T = torch.cumprod(tr, 1)
    before = torch.cat([torch.ones_like(T[:, :1]), T[:, :-1]], 1)
    return before * (1 - tr)


def _grads(model, o, d, opts, loss_of, chunk=1 << 14):
    """(loss outputs, gradients of the tables, the coarse grid and the MLP weights) of the sum
    over ray chunks of loss_of(rays, rgb, depth, opacity, w, t, delta) in 64 bits."""
    outs, U, GF = [], [], []
    for w in model.w:
        w.requires_grad_(True)
    for s in range(0, len(o), chunk):
        r = slice(s, s + chunk)
        u, t, delta, mask, dn = _samples(model, o[r], d[r], opts)
        f = torch.zeros(*mask.shape, 8, dtype=torch.float64, device=o.device)
        f[mask] = model.features(u[mask])
        f.requires_grad_(True)
        w = _weights(f[..., 0], delta, mask)
        c = (w[..., None] * f[..., 1:]).sum(1)
        A, depth = w.sum(1), (w * t).sum(1)
        rgb = model.shade(c[:, :3], c[:, 3:], A, dn)
        loss, kept = loss_of(r, rgb, depth, A, w, t, delta)
        loss.backward()
        outs.append([x.detach() for x in [loss.reshape(1)] + kept])
        U.append(u[mask])
        GF.append(f.grad[mask])
    gt, gc = model.feature_grads(torch.cat(U), torch.cat(GF))
    gm = torch.cat([(torch.zeros_like(w) if w.grad is None else w.grad).reshape(-1) for w in model.w])
    cat = [torch.cat([q[k] for q in outs]) for k in range(len(outs[0]))]
    return cat[0].sum().reshape(1), cat[1:], gt, gc, gm


def exact(case, seed):
    k = case["kind"]
    if k == "grid":
        return None  # whole numbers
    if k == "proposal":
        return _exact_proposal(case, seed)
    cfg, sc = _scene(case, seed)
    model = _Model(case, cfg, sc)
    opts = S.default_options(cfg)
    n = case["rays"] if "rays" in case else case["views"] * cfg.W * cfg.H
    if k == "autograd":
        o, d = (v.double() for v in _free_rays(case, cfg, seed))
    else:
        ids = _pixels(case, seed).long() if "rays" in case else torch.arange(n, device="cuda")
        o, d = _camera_rays(_cams(case, cfg, seed), cfg.W, cfg.H, ids)
    if k == "occupancy":
        R = cfg.R_O
        i = torch.arange(R ** 3, device="cuda")
        u = (torch.stack([i % R, (i // R) % R, i // (R * R)], 1).double() + 0.5) / R
        return {"density": None, "sigma": torch.exp(model.features(u)[:, 0]), "visible": None, "bits": None,
                "dist": None}
    if k == "frame":
        Cd, Fv, A, depth, dn, _ = _render(model, o, d, opts)
        out = {"rgb": model.shade(Cd, Fv, A, dn), "depth": depth, "opacity": A}
        return dict(out, stats=None) if case["dtype"] == "bf16" else out
    if k == "fast":
        pc = P.ProposalConfig()
        z = _proposal_net(_proposal_weights(seed).half().double(), o, d, pc)
        tn, tf, ah = pc.t_scale * torch.sigmoid(z[:, 0]), pc.t_scale * torch.sigmoid(z[:, 1]), torch.sigmoid(z[:, 2])
        inf = torch.full_like(tn, float("inf"))
        lo = torch.where(tf > tn, tn - pc.margin_near, -inf)
        hi = torch.where(tf > tn, tf + pc.margin_far, inf)
        lo, hi = torch.where(ah < pc.a_min, inf, lo), torch.where(ah < pc.a_min, -inf, hi)
        Cd, Fv, A, depth, dn, _ = _render(model, o, d, opts, lo, hi)
        again = torch.nonzero((ah - A > pc.fallback) & ~((lo == -inf) & (hi == inf))).squeeze(1)
        if len(again):
            for x, y in zip((Cd, Fv, A, depth), _render(model, o[again], d[again], opts)):
                x[again] = y
        return {"rgb": model.shade(Cd, Fv, A, dn), "depth": depth, "opacity": A}
    if k == "train":
        tg = torch.rand(n, 3, device="cuda", generator=_gen(seed + 1)).double()
        h = float(np.float32(0.1))

        def huber(r, rgb, depth, A, w, t, delta):
            e = rgb - tg[r]
            a = e.abs()
            return torch.where(a <= h, 0.5 * e * e, h * (a - 0.5 * h)).sum() / (3 * n), [rgb]

        loss, (rgb,), gt, gc, gm = _grads(model, o, d, opts, huber)
        perm, _ = F.tile_order(_pixels(case, seed), cfg.W, cfg.H)
        return {"loss": loss, "rgb": rgb[perm], "tables": gt, "coarse": gc, "mlp_w": gm}
    if k == "autograd":
        tg = torch.rand(n, 3, device="cuda", generator=_gen(seed + 1)).double()

        def l2(r, rgb, depth, A, w, t, delta):
            return ((rgb - tg[r]).square().sum() / (3 * n) + 0.01 * depth.sum() / n + 0.1 * A.sum() / n,
                    [rgb, depth, A])

        loss, (rgb, depth, A), gt, gc, gm = _grads(model, o, d, opts, l2)
        return {"loss": loss.squeeze(0), "rgb": rgb, "depth": depth, "opacity": A, "tables": gt, "coarse": gc,
                "mlp_w": gm}

    def distortion(r, rgb, depth, A, w, t, delta):
        m = t + 0.5 * delta
        W, Sm = torch.cumsum(w, 1) - w, torch.cumsum(w * m, 1) - w * m
        L = (2 * w * (m * W - Sm)).sum(1) + (w * w * delta).sum(1) / 3
        return 0.01 / n * L.sum(), [torch.stack([L, w.sum(1), (w * m).sum(1), torch.zeros_like(L)], 1)]

    loss, (state,), gt, gc, _ = _grads(model, o, d, opts, distortion)
    return {"loss": loss, "state": state, "tables": gt, "coarse": gc}


def _proposal_net(w, o, d, pc):
    e = torch.cat([o / pc.in_scale, d / d.norm(dim=1, keepdim=True)], 1)
    for fan_in, fan_out, last in ((6, 32, False), (32, 32, False), (32, 3, True)):
        e = e @ w[:fan_out * fan_in].reshape(fan_out, fan_in).T + w[fan_out * fan_in:fan_out * fan_in + fan_out]
        e = e if last else torch.relu(e)
        w = w[fan_out * fan_in + fan_out:]
    return e


def _exact_proposal(case, seed):
    st = prepare(case, seed)
    pc = P.ProposalConfig()
    cfg = S.hd_config(W=case["W"], H=case["H"])
    o, d = _camera_rays(_cams(case, cfg, seed), case["W"], case["H"], st["pix"].long())
    w = st["w"].double().requires_grad_(True)
    tg = st["targets"].double()
    z = torch.sigmoid(_proposal_net(w, o, d, pc))
    beta = 0.01
    x = z[:, :2] - tg[:, :2] / pc.t_scale
    sl1 = torch.where(x.abs() < beta, 0.5 * x * x / beta, x.abs() - 0.5 * beta)
    a = torch.stack([torch.where(x[:, 0] > 0, 4.0, 1.0), torch.where(x[:, 1] < 0, 4.0, 1.0)], 1)
    loss = (tg[:, 2] * (a * sl1).sum(1) + (z[:, 2] - tg[:, 2]) ** 2).mean()
    loss.backward()
    return {"loss": loss.detach().reshape(1), "w": w.grad}
