"""Rules that choose between the forms of a call by its size, from the native library's size
queries.  No GPU: the library is only asked."""
import pytest

from paper_2407_10482_gb300 import build as B
from paper_2407_10482_gb300 import scenes as S


@pytest.fixture(scope="module")
def ng():
    B.build()
    from paper_2407_10482_gb300 import ngprt
    ngprt.lib()
    return ngprt


def _scene(ng, **kw):
    cfg = S.hd_config(**kw)
    s = ng.ngprt_scene()
    s.L, s.T_log2, s.R_C = cfg.L, cfg.T_log2, cfg.R_C
    for i, n in enumerate(cfg.N):
        s.N[i] = n
    return s


def test_small_calls_do_not_copy_the_density_channel(ng):
    """The copy of the tables' density channel is taken only where the pass is long enough
    for it: not for a few rays or a coarse grid of voxels, the less so the larger the
    tables."""
    hd, big, two = _scene(ng), _scene(ng, T_log2=22), _scene(ng, L=2, N=[128, 1024])
    plane = 4 * S.table_entries(S.hd_config())
    for n in (-1, 0, 1, 100, 4095):
        assert ng.ngprt_density_scratch_bytes(hd, n) == 0
    assert plane < ng.ngprt_density_scratch_bytes(hd, 4096) < plane + (1 << 20)
    assert ng.ngprt_density_scratch_bytes(big, 6912) == 0 < ng.ngprt_density_scratch_bytes(big, 65536)
    assert ng.ngprt_density_scratch_bytes(two, 4096) == 0 < ng.ngprt_density_scratch_bytes(two, 65536)
    for s, first in ((hd, 64), (big, 128), (two, 128)):
        for R in (2, 8, 16, 32, 64, 128, 256):
            assert (ng.ngprt_occupancy_from_density_scratch_bytes(s, R) > 0) == (R >= first), R
    for R in (-1, 0, 1, 100, 2048):
        assert ng.ngprt_occupancy_from_density_scratch_bytes(hd, R) == 0
    hd.table_dtype = ng.F16
    assert ng.ngprt_density_scratch_bytes(hd, 65536) == 0
    assert ng.ngprt_occupancy_from_density_scratch_bytes(hd, 128) == 0
