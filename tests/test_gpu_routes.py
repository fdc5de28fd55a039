"""Calls that take the general route because of their alignment, size or scene, against
the form that serves every call."""
import ctypes as C

import pytest

torch = pytest.importorskip("torch")

from paper_2407_10482_gb300 import scenes as S
from test_gpu_records import _close, _render_gradients, _setup

pytestmark = pytest.mark.gpu


def _ptr(t):
    return None if t is None else C.c_void_p(t.data_ptr())


def _distortion_gradients(L, n, pixels, offset=0, **kw):
    """(gradients of the binding's call, of the C entry without scratch); g_coarse of the
    first starts `offset` floats into a flat buffer."""
    ng, ds, occ, opts, rays, src = _setup(L, n, pixels, **kw)
    ro = ng.render_opts(opts)
    state = torch.empty(n, 4, device="cuda")
    ng.ngprt_distortion_loss(ds.struct, occ.struct, *src, n, ro, 1.0, state)
    flat = torch.zeros(ds.coarse.numel() + offset, device="cuda")
    got = [torch.zeros_like(ds.tables), flat[offset:].view_as(ds.coarse)]
    ref = [torch.zeros_like(t) for t in (ds.tables, ds.coarse)]
    ng.ngprt_distortion_backward(ds.struct, occ.struct, *src, n, ro, state, 1.0 / n, *got)
    st = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert ng.lib().ngprt_distortion_backward(
        C.byref(ds.struct), C.byref(occ.struct), src[0], src[1], _ptr(src[2]), _ptr(src[3]), _ptr(src[4]), n, C.byref(ro),
        _ptr(state), C.c_float(1.0 / n), _ptr(ref[0]), _ptr(ref[1]), None, None, None, 0, st) == 0
    return got, ref


@pytest.mark.parametrize("offset", [0, 1, 2, 4])
@pytest.mark.parametrize("L", [2, 8, 16])
def test_distortion_gradient_in_a_flat_buffer(L, offset):
    """Bounds of the records' tests: the same FP32 terms in another order."""
    for a, b in zip(*_distortion_gradients(L, 4096 + 33, True, offset)):
        _close(a, b)


@pytest.mark.parametrize("sparse", [False, True])
@pytest.mark.parametrize("attn_mode", [0, 2])
@pytest.mark.parametrize("L,R", [(2, 128), (4, 128), (8, 64), (16, 64)])
def test_occupancy_on_the_density_plane_of_large_calls(L, R, attn_mode, sparse):
    """The density channel's sums keep their order: equal bit for bit, on the dense coarse
    grid and on its block-sparse form."""
    n = 40000
    ng, ds, occ, opts, rays, src = _setup(L, n, True, attn_mode=attn_mode)
    if sparse:
        ds.sparsify_coarse(occ)
    ro, lib = ng.render_opts(opts), ng.lib()
    st = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert ng.ngprt_occupancy_from_density_scratch_bytes(ds.struct, R) > 0
    assert ng.ngprt_density_scratch_bytes(ds.struct, n) > 0
    o = [torch.empty(R ** 3, dtype=torch.uint8, device="cuda") for _ in range(2)]
    sg = [torch.empty(R ** 3, device="cuda") for _ in range(2)]
    ng.ngprt_occupancy_from_density(ds.struct, ro, R, 1.0, o[0], sg[0])
    assert lib.ngprt_occupancy_from_density(C.byref(ds.struct), C.byref(ro), R, C.c_float(1.0), _ptr(o[1]), _ptr(sg[1]),
                                            st) == 0
    assert torch.equal(o[0], o[1]) and torch.equal(sg[0], sg[1])
    v = [torch.zeros(R ** 3, dtype=torch.uint8, device="cuda") for _ in range(2)]
    ng.ngprt_occupancy_visibility(ds.struct, occ.struct, *src, n, ro, 1e-3, R, v[0])
    assert lib.ngprt_occupancy_visibility(C.byref(ds.struct), C.byref(occ.struct), src[0], src[1], _ptr(src[2]), None,
                                          None, n, C.byref(ro), C.c_float(1e-3), R, _ptr(v[1]), st) == 0
    assert torch.equal(v[0], v[1]) and int(v[0].sum()) > 0


def _overflow(L, n, pixels):
    """More samples a ray than the records hold (128, or 44 for 2^18 rays of 16 levels):
    the rest comes from the one-kernel form, whose list is taken in scattered order."""
    step = 2.0 * 3 ** 0.5 / 128.0 / 8.0
    _render_gradients(L, n, pixels, step_base=step, max_samples=512, max_march=4096, t_term=0.0)


@pytest.mark.parametrize("L,n,pixels", [(1, 4097, True), (4, 4096, False), (8, 5001, True), (16, 1 << 18, True)])
def test_rays_beyond_the_records_room(L, n, pixels):
    _overflow(L, n, pixels)


def test_distortion_beyond_the_records_room():
    step = 2.0 * 3 ** 0.5 / 128.0 / 8.0
    for a, b in zip(*_distortion_gradients(8, 5001, True, step_base=step, max_samples=512, max_march=4096, t_term=0.0)):
        _close(a, b)


@pytest.mark.parametrize("L", [2, 4])
def test_pixel_lists_of_few_levels_by_records(L):
    """2 and 4 levels take pixel lists by records above 2^15 rays."""
    _render_gradients(L, (1 << 15) + 33, True)


@pytest.mark.parametrize("L", [1, 4, 8, 16])
def test_pixel_lists_in_tile_order(L):
    """Lists of at least 2^16 pixels are recorded in pixel-tile order."""
    _render_gradients(L, (1 << 16) + 33, True)


@pytest.mark.parametrize("pixels", [True, False])
def test_more_rays_than_one_pass_of_records(pixels):
    _render_gradients(1, (1 << 18) + 4129, pixels)


def _contracted(L, dtype):
    """A contracted scene of L levels with tables small enough to draw quickly."""
    from paper_2407_10482_gb300 import ngprt as ng
    cfg = S.hd_config(L=L, N=S.level_resolutions(16, 1024, L), T_log2=14, R_O=64, n_occ_levels=4, W=643, H=517)
    sc = S.make_scene(cfg)
    dt = getattr(ng, dtype)
    ds = ng.DeviceScene(cfg, sc.tables, sc.coarse, sc.mlp_w, table_dtype=dt, mlp_dtype=ng.F32 if dt == ng.F32 else ng.F16)
    docc = ng.DeviceOcc(sc.occ, cfg.R_O, cfg.n_occ_levels)
    return ng, cfg, ds, docc


@pytest.mark.parametrize("L", [2, 8, 16])
@pytest.mark.parametrize("dtype", ["F32", "F16", "BF16"])
def test_batches_of_every_size_render_the_rays_of_a_full_one(L, dtype):
    """Free rays in batches that take 32, 16, 8, 4, 2 and 1 lanes a ray and each block count
    of the march, against the same rays in a batch that fills the GPU.  Decisions are equal;
    the groups contract w = T (1 - t) into its sum, one rounding (2^-24) a sample, of at most
    100 samples here."""
    ng, cfg, ds, docc = _contracted(L, dtype)
    rend = ng.Renderer(ds, docc)
    o, d = (torch.as_tensor(x).cuda() for x in S.random_rays(330011, 4, False))
    opts = S.default_options(cfg)
    full = rend.render(opts, rays_o=o, rays_d=d, stats=True, state=True)
    assert int(full["stats"][:, 1].max()) <= 100
    for n in (1, 2000, 4097, 8191, 13001, 25000, 55001, 90000, 110003, 140001, 180000):
        part = rend.render(opts, rays_o=o[:n].contiguous(), rays_d=d[:n].contiguous(), stats=True, state=True)
        assert torch.equal(part["stats"], full["stats"][:n])
        torch.testing.assert_close(part["state"], full["state"][:n], rtol=6e-6, atol=6e-6)


@pytest.mark.parametrize("L", [2, 8, 16])
@pytest.mark.parametrize("dtype,rtol", [("F16", 0.05), ("BF16", 1e-3)])
def test_density_grid_of_16_bit_tables(L, dtype, rtol):
    """Against FP32 tables of the rounded values.  BF16 differs by the rounding of FP32 sums
    and of the fixed-point cells; FP16 by its half2 sums: 8 roundings of 2^-11 of a raw
    density of about 4, 0.016, and as much for the levels together, in the exponent."""
    ng, cfg, ds, docc = _contracted(L, dtype)
    ds32 = ng.DeviceScene(cfg, ds.tables.float(), ds.coarse.float(), ds.mlp_w.float())
    ro, R = ng.render_opts(S.default_options(cfg)), 32
    occ = torch.empty(R ** 3, dtype=torch.uint8, device="cuda")
    sigma = [torch.empty(R ** 3, device="cuda") for _ in range(2)]
    for scene, out in zip((ds, ds32), sigma):
        ng.ngprt_occupancy_from_density(scene.struct, ro, R, 20.0, occ, out)
    torch.testing.assert_close(sigma[0], sigma[1], rtol=rtol, atol=0)


def test_small_tables_in_tile_order():
    """Few table rows: the pixel-tile order from 2^15 rays on."""
    from paper_2407_10482_gb300 import ngprt as ng
    cfg = S.small_config(blob_std=(0.05, 0.15), W=160, H=96)
    sc = S.make_scene(cfg)
    ds = ng.DeviceScene(cfg, sc.tables, sc.coarse, sc.mlp_w)
    docc = ng.DeviceOcc(sc.occ, cfg.R_O, cfg.n_occ_levels)
    opts, n = S.default_options(cfg), (1 << 15) + 33
    rays = dict(cams=S.orbit_cameras(cfg, 3, azimuth0=5.0), W=cfg.W, H=cfg.H,
                pixel_ids=torch.as_tensor(S.random_pixels(n, 3, cfg.W, cfg.H, 2)).cuda())
    rend = ng.Renderer(ds, docc)
    out = rend.render(opts, state=True, **rays)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1)
    d_rgb = torch.randn(n, 3, device="cuda", generator=gen)
    cams, n_cams = ng.cameras_struct(rays["cams"], cfg.W, cfg.H)
    ro = ng.render_opts(opts)
    got = []
    for need in (ng.ngprt_render_backward_scratch_bytes(ds.struct, ro, n),
                 ng.ngprt_render_backward_workspace_bytes(ds.struct, ro, n)):
        g = [torch.zeros_like(t) for t in (ds.tables, ds.coarse, ds.mlp_w)]
        ws = torch.empty(need, dtype=torch.uint8, device="cuda")
        ng.ngprt_render_backward(ds.struct, docc.struct, cams, n_cams, rays["pixel_ids"], None, None, n, ro,
                                 out["state"], d_rgb, None, None, *g, ws)
        got.append(g)
    for a, b in zip(*got):
        _close(a, b)


@pytest.mark.parametrize("mode", ["tiles", "pixel_ids", "rays"])
@pytest.mark.parametrize("dtype", ["F32", "F16", "BF16"])
def test_run_time_tiles_of_batches_beyond_the_resident_warps(mode, dtype):
    """More tiles than the GPU holds warps, so that warps take several from the counter:
    bit for bit the static grid's states and counts."""
    ng, cfg, ds, docc = _contracted(16, dtype)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    ro = ng.render_opts(S.default_options(cfg))
    cams, n_cams = ng.cameras_struct(S.orbit_cameras(cfg, 3, azimuth0=7.0, step_deg=120.0), cfg.W, cfg.H)
    pix = o = d = None
    n = sms * 64 * 32 + 18011
    if mode == "tiles":
        n = n_cams * cfg.W * cfg.H
    elif mode == "pixel_ids":
        pix = torch.as_tensor(S.random_pixels(n, 3, cfg.W, cfg.H, 5)).cuda()
    else:
        o, d = (torch.as_tensor(x).cuda() for x in S.random_rays(n, 9, False))
        cams, n_cams = None, 0
    assert (n + 31) // 32 > sms * 64
    out = []
    for ws_bytes in (0, ng.ngprt_render_workspace_bytes(ds.struct, n)):
        state = torch.full((n, ng.STATE_FLOATS), float("nan"), device="cuda")
        stats = torch.full((n, 2), -1, dtype=torch.int32, device="cuda")
        ws = torch.empty(ws_bytes, dtype=torch.uint8, device="cuda") if ws_bytes else None
        for _ in range(2):
            ng.ngprt_render(ds.struct, docc.struct, cams, n_cams, pix, o, d, n, None, ro, None, ray_stats=stats,
                            ray_state=state, workspace=ws)
        out.append((state.view(torch.int32), stats))
    assert bool((out[0][1] >= 0).all())
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])


@pytest.mark.parametrize("attn_mode", [0, 1, 2])
@pytest.mark.parametrize("L", [1, 4, 8, 16])
def test_distortion_records_of_every_gate_mode(L, attn_mode):
    for pixels in (True, False):
        for a, b in zip(*_distortion_gradients(L, 4096 + 33, pixels, attn_mode=attn_mode)):
            _close(a, b)


def _whole_images(ng, ds, docc, cfg, views=2):
    cams = S.orbit_cameras(cfg, views, azimuth0=5.0)
    arr, n_cams = ng.cameras_struct(cams, cfg.W, cfg.H)
    return views * cfg.W * cfg.H, dict(cams=cams, W=cfg.W, H=cfg.H), (arr, n_cams, None, None, None)


@pytest.mark.parametrize("L", [1, 2, 8, 16])
def test_whole_images_by_records(L):
    """Camera images without a pixel list: render's and the regulariser's reverse passes."""
    ng, ds, occ, opts, _, _ = _setup(L, 1, True)
    n, rays, src = _whole_images(ng, ds, occ, ds.cfg)
    ro, rend = ng.render_opts(opts), ng.Renderer(ds, occ)
    out = rend.render(opts, state=True, **rays)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1)
    d_rgb = torch.randn(n, 3, device="cuda", generator=gen)
    got = []
    for need in (ng.ngprt_render_backward_scratch_bytes(ds.struct, ro, n),
                 ng.ngprt_render_backward_workspace_bytes(ds.struct, ro, n)):
        g = [torch.zeros_like(t) for t in (ds.tables, ds.coarse, ds.mlp_w)]
        ws = torch.empty(need, dtype=torch.uint8, device="cuda")
        ng.ngprt_render_backward(ds.struct, occ.struct, *src, n, ro, out["state"], d_rgb, None, None, *g, ws)
        got.append(g)
    for a, b in zip(*got):
        _close(a, b)
    state = torch.empty(n, 4, device="cuda")
    ng.ngprt_distortion_loss(ds.struct, occ.struct, *src, n, ro, 1.0, state)
    g = [[torch.zeros_like(t) for t in (ds.tables, ds.coarse)] for _ in range(2)]
    ng.ngprt_distortion_backward(ds.struct, occ.struct, *src, n, ro, state, 1.0 / n, *g[0])
    st = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert ng.lib().ngprt_distortion_backward(
        C.byref(ds.struct), C.byref(occ.struct), src[0], src[1], None, None, None, n, C.byref(ro), _ptr(state),
        C.c_float(1.0 / n), _ptr(g[1][0]), _ptr(g[1][1]), None, None, None, 0, st) == 0
    for a, b in zip(*g):
        _close(a, b)


def test_calls_under_capture():
    """A render of a small batch (kernels this process may not have used yet), its reverse
    pass, the regulariser and the marks, captured at first use and replayed, against the
    same calls outside."""
    n = 4129
    ng, ds, occ, opts, rays, src = _setup(3, n, True, t_term=0.01)
    ro, rend = ng.render_opts(opts), ng.Renderer(ds, occ)
    d_rgb = torch.ones(n, 3, device="cuda") / n
    rend.workspace(n)

    def calls():
        out = rend.render(opts, state=True, **rays)
        g = [torch.zeros_like(t) for t in (ds.tables, ds.coarse, ds.mlp_w)]
        rend.backward(opts, out["state"], d_rgb, None, None, *g, **rays)
        state = torch.empty(n, 4, device="cuda")
        ng.ngprt_distortion_loss(ds.struct, occ.struct, *src, n, ro, 1.0, state)
        gd = [torch.zeros_like(t) for t in (ds.tables, ds.coarse)]
        ng.ngprt_distortion_backward(ds.struct, occ.struct, *src, n, ro, state, 1.0 / n, *gd)
        vis = torch.zeros(32 ** 3, dtype=torch.uint8, device="cuda")
        ng.ngprt_occupancy_visibility(ds.struct, occ.struct, *src, n, ro, 1e-3, 32, vis)
        return [out["rgb"], out["state"], vis, state], g + gd

    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        same, close = calls()
    graph.replay()
    torch.cuda.synchronize()
    ref_same, ref_close = calls()
    for a, b in zip(same, ref_same):
        assert torch.equal(a, b)
    for a, b in zip(close, ref_close):
        _close(a, b)


def _fine_coarse(L, n, pixels):
    """A bounded scene whose coarse grid is about as fine as the steps, with n rays."""
    from paper_2407_10482_gb300 import ngprt as ng
    cfg = S.small_config(L=L, N=S.level_resolutions(64, 128, L), T_log2=16, R_C=64, blob_std=(0.05, 0.15), W=160, H=96)
    sc = S.make_scene(cfg)
    ds = ng.DeviceScene(cfg, sc.tables, sc.coarse, sc.mlp_w)
    occ = ng.DeviceOcc(sc.occ, cfg.R_O, cfg.n_occ_levels)
    if pixels:
        rays = dict(cams=S.orbit_cameras(cfg, 3, azimuth0=5.0), W=cfg.W, H=cfg.H,
                    pixel_ids=torch.as_tensor(S.random_pixels(n, 3, cfg.W, cfg.H, 2)).cuda())
        src = (*ng.cameras_struct(rays["cams"], cfg.W, cfg.H), rays["pixel_ids"], None, None)
    else:
        o, d = (torch.as_tensor(x).cuda() for x in S.random_rays(n, 3, True))
        rays, src = dict(rays_o=o, rays_d=d), (None, 0, None, o, d)
    return ng, ds, occ, S.default_options(cfg), rays, src


@pytest.mark.parametrize("L,n,pixels", [(2, 20000, False), (2, (1 << 17) + 33, True), (4, 20000, False),
                                        (4, (1 << 15) + 33, False), (16, 5001, True), (16, (1 << 15) + 33, True)])
def test_reverse_pass_on_a_fine_coarse_grid(L, n, pixels):
    """On both sides of the sizes from which records serve a coarse grid as fine as the
    steps."""
    ng, ds, occ, opts, rays, src = _fine_coarse(L, n, pixels)
    ro, rend = ng.render_opts(opts), ng.Renderer(ds, occ)
    out = rend.render(opts, state=True, **rays)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1)
    d_rgb = torch.randn(n, 3, device="cuda", generator=gen)
    got = []
    for need in (ng.ngprt_render_backward_scratch_bytes(ds.struct, ro, n),
                 ng.ngprt_render_backward_workspace_bytes(ds.struct, ro, n)):
        g = [torch.zeros_like(t) for t in (ds.tables, ds.coarse, ds.mlp_w)]
        ws = torch.empty(need, dtype=torch.uint8, device="cuda")
        ng.ngprt_render_backward(ds.struct, occ.struct, *src, n, ro, out["state"], d_rgb, None, None, *g, ws)
        got.append(g)
    for a, b in zip(*got):
        _close(a, b)


@pytest.mark.parametrize("pixels", [True, False])
def test_marks_of_two_large_levels(pixels):
    """2 levels of 2^20 rows: pixel lists take the density plane, free rays do not."""
    from paper_2407_10482_gb300 import ngprt as ng
    cfg = S.hd_config(L=2, N=[128, 1024], T_log2=19, R_O=64, n_occ_levels=4, W=320, H=200)
    sc = S.make_scene(cfg)
    ds = ng.DeviceScene(cfg, sc.tables, sc.coarse, sc.mlp_w)
    docc = ng.DeviceOcc(sc.occ, cfg.R_O, cfg.n_occ_levels)
    ro, n = ng.render_opts(S.default_options(cfg)), 40000
    assert ng.ngprt_density_scratch_bytes(ds.struct, n) > 0
    if pixels:
        src = (*ng.cameras_struct(S.orbit_cameras(cfg, 2, azimuth0=5.0), cfg.W, cfg.H),
               torch.as_tensor(S.random_pixels(n, 2, cfg.W, cfg.H, 2)).cuda(), None, None)
    else:
        o, d = (torch.as_tensor(x).cuda() for x in S.random_rays(n, 3, False))
        src = (None, 0, None, o, d)
    v = [torch.zeros(64 ** 3, dtype=torch.uint8, device="cuda") for _ in range(2)]
    ng.ngprt_occupancy_visibility(ds.struct, docc.struct, *src, n, ro, 1e-3, 64, v[0])
    st = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert ng.lib().ngprt_occupancy_visibility(
        C.byref(ds.struct), C.byref(docc.struct), src[0], src[1], _ptr(src[2]), _ptr(src[3]), _ptr(src[4]), n,
        C.byref(ro), C.c_float(1e-3), 64, _ptr(v[1]), st) == 0
    assert torch.equal(v[0], v[1]) and int(v[0].sum()) > 0
