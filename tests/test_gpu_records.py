"""The reverse passes by records against the one-kernel form, and the passes on the
density plane against those on the whole entries: every built L, every gate mode, camera
pixels (taken in pixel-tile order) and free rays, a ragged last run of rays, and rays
with more samples than the records hold (finished by the one-kernel form).

Both forms add the same FP32 terms in another order, so a gradient may differ by the
rounding of its sum: 1e-3 of itself plus 3e-5 of the largest, the bound of the parity with
the FP64 oracle.  The density path's sums keep their order: equal bit for bit."""
import ctypes as C

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2407_10482_gb300 import scenes as S

pytestmark = pytest.mark.gpu

LEVELS = {1: [64], 2: [24, 96], 3: [16, 40, 100], 4: [16, 32, 64, 128], 8: [16 + 12 * l for l in range(8)],
          16: S.level_resolutions(16, 1024, 16)}


def _setup(L, n, pixels, **kw):
    from paper_2407_10482_gb300 import ngprt as ng
    cfg = S.small_config(L=L, N=LEVELS[L], T_log2=18, blob_std=(0.05, 0.15), W=160, H=96)
    sc = S.make_scene(cfg)
    sc.coarse[:, 8:] *= 10.0
    ds = ng.DeviceScene(cfg, sc.tables, sc.coarse, sc.mlp_w)
    occ = ng.DeviceOcc(sc.occ, cfg.R_O, cfg.n_occ_levels)
    opts = S.default_options(cfg, **kw)
    if pixels:
        rays = dict(cams=S.orbit_cameras(cfg, 3, azimuth0=5.0), W=cfg.W, H=cfg.H,
                    pixel_ids=torch.as_tensor(S.random_pixels(n, 3, cfg.W, cfg.H, 2)).cuda())
        cams, n_cams = ng.cameras_struct(rays["cams"], cfg.W, cfg.H)
        src = (cams, n_cams, rays["pixel_ids"], None, None)
    else:
        o, d = S.random_rays(n, 3, cfg.bounded)
        rays = dict(rays_o=torch.as_tensor(o).cuda(), rays_d=torch.as_tensor(d).cuda())
        src = (None, 0, None, rays["rays_o"], rays["rays_d"])
    return ng, ds, occ, opts, rays, src


def _close(a, b):
    a, b = a.double(), b.double()
    scale = float(b.abs().max())
    assert scale > 0
    bad = (a - b).abs() > 1e-3 * b.abs() + 3e-5 * scale
    assert not bool(bad.any()), (int(bad.sum()), float((a - b).abs().max()), scale)


def _render_gradients(L, n, pixels, **kw):
    ng, ds, occ, opts, rays, src = _setup(L, n, pixels, **kw)
    rend = ng.Renderer(ds, occ)
    out = rend.render(opts, state=True, **rays)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1)
    cot = [torch.randn(n, 3, device="cuda", generator=gen), torch.randn(n, device="cuda", generator=gen) * 0.3,
           torch.randn(n, device="cuda", generator=gen)]
    ro = ng.render_opts(opts)
    got = []
    for need in (ng.ngprt_render_backward_scratch_bytes(ds.struct, ro, n),
                 ng.ngprt_render_backward_workspace_bytes(ds.struct, ro, n)):
        g = [torch.zeros_like(t) for t in (ds.tables, ds.coarse, ds.mlp_w)]
        ws = torch.empty(need, dtype=torch.uint8, device="cuda")
        ng.ngprt_render_backward(ds.struct, occ.struct, *src, n, ro, out["state"], *cot, *g, ws)
        got.append((need, g))
    assert got[0][0] > got[1][0]
    for a, b in zip(got[0][1], got[1][1]):
        _close(a, b)


@pytest.mark.parametrize("pixels", [True, False])
@pytest.mark.parametrize("attn_mode", [0, 1, 2])
@pytest.mark.parametrize("L", sorted(LEVELS))
def test_render_reverse_pass_by_records(L, attn_mode, pixels):
    _render_gradients(L, 4096 + 33, pixels, attn_mode=attn_mode, t_term=0.0)


def test_rays_longer_than_their_records():
    """About 400 samples a ray, 128 recorded: the rest is added by the one-kernel form."""
    step = 2.0 * 3 ** 0.5 / 128.0 / 16.0
    _render_gradients(4, 4096, True, step_base=step, max_samples=1024, max_march=4096, t_term=0.0)


def _distortion(L, n, pixels, **kw):
    ng, ds, occ, opts, rays, src = _setup(L, n, pixels, **kw)
    ro = ng.render_opts(opts)
    lib = ng.lib()
    p = lambda t: None if t is None else C.c_void_p(t.data_ptr())  # noqa: E731
    raw = (C.byref(ds.struct), C.byref(occ.struct), src[0], src[1], p(src[2]), p(src[3]), p(src[4]), n, C.byref(ro))
    st = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    state = [torch.full((n, 4), float("nan"), device="cuda") for _ in range(2)]
    assert ng.ngprt_density_scratch_bytes(ds.struct, n) > 0
    ng.ngprt_distortion_loss(ds.struct, occ.struct, *src, n, ro, 1.0, state[0])
    assert lib.ngprt_distortion_loss(*raw, C.c_float(1.0), p(state[1]), None, st) == 0
    torch.testing.assert_close(state[0], state[1], rtol=1e-5, atol=1e-6)
    grads = [[torch.zeros_like(t) for t in (ds.tables, ds.coarse)] for _ in range(2)]
    ng.ngprt_distortion_backward(ds.struct, occ.struct, *src, n, ro, state[1], 1.0 / n, *grads[0])
    assert lib.ngprt_distortion_backward(*raw, p(state[1]), C.c_float(1.0 / n), p(grads[1][0]), p(grads[1][1]), None,
                                         None, None, 0, st) == 0
    for a, b in zip(*grads):
        _close(a, b)


@pytest.mark.parametrize("pixels", [True, False])
@pytest.mark.parametrize("attn_mode", [0, 1])
@pytest.mark.parametrize("L", sorted(LEVELS))
def test_distortion_on_the_density_plane(L, attn_mode, pixels):
    _distortion(L, 4096 + 33, pixels, attn_mode=attn_mode)


def test_distortion_of_rays_longer_than_their_records():
    step = 2.0 * 3 ** 0.5 / 128.0 / 16.0
    _distortion(4, 4096, False, step_base=step, max_samples=1024, max_march=4096, t_term=0.0)


@pytest.mark.parametrize("attn_mode", [0, 1, 2])
@pytest.mark.parametrize("L", [1, 4, 16])
def test_occupancy_on_the_density_plane(L, attn_mode):
    ng, ds, occ, opts, rays, src = _setup(L, 5000, True, attn_mode=attn_mode)
    ro = ng.render_opts(opts)
    lib = ng.lib()
    p = lambda t: None if t is None else C.c_void_p(t.data_ptr())  # noqa: E731
    st = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    R = 32
    o = [torch.empty(R ** 3, dtype=torch.uint8, device="cuda") for _ in range(2)]
    sg = [torch.empty(R ** 3, device="cuda") for _ in range(2)]
    ng.ngprt_occupancy_from_density(ds.struct, ro, R, 1.0, o[0], sg[0])
    assert lib.ngprt_occupancy_from_density(C.byref(ds.struct), C.byref(ro), R, C.c_float(1.0), p(o[1]), p(sg[1]),
                                            st) == 0
    assert torch.equal(o[0], o[1]) and torch.equal(sg[0], sg[1])
    v = [torch.zeros(R ** 3, dtype=torch.uint8, device="cuda") for _ in range(2)]
    ng.ngprt_occupancy_visibility(ds.struct, occ.struct, *src, 5000, ro, 1e-3, R, v[0])
    assert lib.ngprt_occupancy_visibility(C.byref(ds.struct), C.byref(occ.struct), src[0], src[1], p(src[2]), None, None,
                                          5000, C.byref(ro), C.c_float(1e-3), R, p(v[1]), st) == 0
    assert torch.equal(v[0], v[1]) and int(v[0].sum()) > 0


@pytest.mark.parametrize("n", [1, 31, 1000, 20011])
@pytest.mark.parametrize("dtype", ["F32", "F16", "BF16"])
def test_lane_groups_render_the_one_lane_rays(n, dtype):
    """Small batches (2 to 32 lanes a ray) against the same rays in a batch that fills the
    GPU (one lane a ray): equal up to the contraction of w = T (1 - t) into its sum, one
    rounding a sample."""
    from paper_2407_10482_gb300 import ngprt as ng
    cfg = S.small_config(blob_std=(0.05, 0.15))
    sc = S.make_scene(cfg)
    ds = ng.DeviceScene(cfg, sc.tables, sc.coarse, sc.mlp_w, table_dtype=getattr(ng, dtype))
    rend = ng.Renderer(ds, ng.DeviceOcc(sc.occ, cfg.R_O, cfg.n_occ_levels))
    o, d = S.random_rays(300000, 4, cfg.bounded)
    o, d = torch.as_tensor(o).cuda(), torch.as_tensor(d).cuda()
    for kw in (dict(), dict(max_samples=5), dict(max_march=9), dict(t_term=0.5)):
        opts = S.default_options(cfg, **kw)
        full = rend.render(opts, rays_o=o, rays_d=d, stats=True, state=True)
        part = rend.render(opts, rays_o=o[:n].contiguous(), rays_d=d[:n].contiguous(), stats=True, state=True)
        assert torch.equal(part["stats"], full["stats"][:n])
        torch.testing.assert_close(part["state"], full["state"][:n], rtol=2e-6, atol=2e-6)
        torch.testing.assert_close(part["rgb"], full["rgb"][:n], rtol=0, atol=2e-6)


@pytest.mark.parametrize("lattice_snap", [False, True])
@pytest.mark.parametrize("n", [33, 40000, 75001, 140001])
@pytest.mark.parametrize("dtype", ["F32", "F16", "BF16"])
def test_medium_batches_render_the_rays_of_a_full_one(n, dtype, lattice_snap):
    """Batches below a full GPU (march kernel with more registers, or lane groups, and
    neither where the samples stay on a lattice at few rays) against the same rays in a
    batch that fills it, with the bounds of the lane groups above."""
    from paper_2407_10482_gb300 import ngprt as ng
    cfg = S.small_config(blob_std=(0.05, 0.15))
    sc = S.make_scene(cfg)
    ds = ng.DeviceScene(cfg, sc.tables, sc.coarse, sc.mlp_w, table_dtype=getattr(ng, dtype))
    rend = ng.Renderer(ds, ng.DeviceOcc(sc.occ, cfg.R_O, cfg.n_occ_levels))
    o, d = S.random_rays(300000, 4, cfg.bounded)
    o, d = torch.as_tensor(o).cuda(), torch.as_tensor(d).cuda()
    opts = S.default_options(cfg, lattice_snap=lattice_snap)
    full = rend.render(opts, rays_o=o, rays_d=d, stats=True, state=True)
    part = rend.render(opts, rays_o=o[:n].contiguous(), rays_d=d[:n].contiguous(), stats=True, state=True)
    assert torch.equal(part["stats"], full["stats"][:n])
    torch.testing.assert_close(part["state"], full["state"][:n], rtol=2e-6, atol=2e-6)
    torch.testing.assert_close(part["rgb"], full["rgb"][:n], rtol=0, atol=2e-6)
