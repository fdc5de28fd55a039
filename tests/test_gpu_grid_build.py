"""Occupancy pyramid and distance grid, bit for bit against the oracle, where the build
can go wrong: rows shorter than a word and of one, two and many words, gaps at and past
the saturation at 255, an empty and a full grid, a grid whose address allows no wide
loads, and values other than 1."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O

pytestmark = pytest.mark.gpu


def _grid(R, fill, seed):
    rng = np.random.default_rng(seed)
    occ = np.zeros(R ** 3, np.uint8)
    if fill == "full":
        occ[:] = 1
    elif fill == "corner":           # every distance up to the body diagonal
        occ[0] = 7
    elif fill == "edge":             # the last voxel of a row in the last word
        occ[R ** 3 - 1] = 255
    elif fill == "plane":
        occ.reshape(R, R, R)[:, :, R // 2] = 1
    elif fill == "few":
        occ[rng.integers(0, R ** 3, max(1, R // 4))] = rng.integers(1, 256, max(1, R // 4)).astype(np.uint8)
    elif fill == "many":
        occ[:] = rng.random(R ** 3) < 0.3
    return occ


@pytest.mark.parametrize("fill", ["empty", "full", "corner", "edge", "plane", "few", "many"])
@pytest.mark.parametrize("R,n_levels", [(2, 2), (4, 3), (16, 5), (32, 3), (64, 6), (128, 5)])
def test_pyramid_and_distance_grid(R, n_levels, fill):
    from paper_2407_10482_gb300 import ngprt as ng
    occ = _grid(R, fill, R)
    for k in {0, min(1, n_levels - 1)}:
        d = ng.DeviceOcc(occ, R, n_levels, dist_level=k)
        torch.cuda.synchronize()
        assert np.array_equal(d.bits.cpu().numpy().view(np.uint32), O.build_pyramid(occ, R, n_levels))
        assert np.array_equal(d.dist.cpu().numpy(), O.occ_dist(O.downsample_occ(occ, R, k), R >> k))


@pytest.mark.parametrize("fill", ["corner", "edge"])
@pytest.mark.parametrize("R,dist_level", [(256, 0), (512, 0), (512, 1)])
def test_one_voxel_in_a_large_grid(R, dist_level, fill):
    """G around one voxel is min(255, floor sqrt of the sum of (distance - 1)^2)."""
    from paper_2407_10482_gb300 import ngprt as ng
    d = ng.DeviceOcc(_grid(R, fill, R), R, 3, dist_level=dist_level)
    Rg = R >> dist_level
    x = torch.arange(Rg, device="cuda")
    g = ((x if fill == "corner" else Rg - 1 - x) - 1).clamp(min=0).double() ** 2
    ref = (g[:, None, None] + g[None, :, None] + g[None, None, :]).sqrt().floor().clamp(max=255).to(torch.uint8)
    assert torch.equal(d.dist.reshape(Rg, Rg, Rg), ref)


@pytest.mark.parametrize("shift", [1, 4, 8])
def test_unaligned_occupancy(shift):
    from paper_2407_10482_gb300 import ngprt as ng
    R, n_levels = 32, 3
    occ = _grid(R, "many", 3)
    buf = torch.zeros(R ** 3 + 16, dtype=torch.uint8, device="cuda")
    buf[shift:shift + R ** 3] = torch.as_tensor(occ).cuda()
    bits = torch.empty(ng.ngprt_occ_bits_words(R, n_levels), dtype=torch.int32, device="cuda")
    dist = torch.empty(R ** 3, dtype=torch.uint8, device="cuda")
    ws = torch.empty(ng.ngprt_build_occ_dist_workspace_bytes(R), dtype=torch.uint8, device="cuda")
    ng.ngprt_build_occ_dist(buf[shift:shift + R ** 3], R, n_levels, bits, dist, ws)
    torch.cuda.synchronize()
    assert np.array_equal(bits.cpu().numpy().view(np.uint32), O.build_pyramid(occ, R, n_levels))
    assert np.array_equal(dist.cpu().numpy(), O.occ_dist(occ, R))
