"""Scratch of the binding's calls: what a call keeps, asks for again and does without.  The
native library and the allocator are stood in for; no GPU is touched."""
import pytest

torch = pytest.importorskip("torch")

from paper_2407_10482_gb300 import ngprt as ng

NEED, BEST = 100, 1000


class _Scene:
    struct = None
    tables = torch.zeros(1)


@pytest.fixture
def renderer(monkeypatch):
    """A Renderer whose reverse pass records the workspaces it was given."""
    r = ng.Renderer(_Scene(), _Scene(), device="cpu")
    r.given, r.asked, r.room = [], [], True

    def scratch(nbytes, like, stream=None):
        r.asked.append(nbytes)
        return torch.empty(nbytes, dtype=torch.uint8) if r.room else None

    monkeypatch.setattr(ng, "_scratch", scratch)
    monkeypatch.setattr(ng, "render_opts", lambda o: None)
    monkeypatch.setattr(ng, "ngprt_render_backward_workspace_bytes", lambda *a: NEED)
    monkeypatch.setattr(ng, "ngprt_render_backward_scratch_bytes", lambda *a: BEST)
    monkeypatch.setattr(ng, "ngprt_render_backward", lambda *a, **k: r.given.append(a[16].numel()))
    monkeypatch.setattr(torch.cuda, "is_current_stream_capturing", lambda: False)
    return r


def _backward(r):
    z = torch.zeros(4, 3)
    r.backward(None, z, z, None, None, z, z, z, rays_o=z, rays_d=z)


def test_the_renderer_gives_the_records_scratch_back(renderer):
    for _ in range(2):
        _backward(renderer)
    assert renderer.given == [BEST, BEST]
    assert renderer._bws is None or renderer._bws.numel() <= NEED


def test_a_scratch_that_could_not_be_had_is_asked_for_once(renderer):
    renderer.room = False
    _backward(renderer)
    kept = renderer._bws
    for _ in range(3):
        _backward(renderer)
    assert renderer.given == [NEED] * 4 and renderer.asked == [BEST]
    assert renderer._bws is kept


def test_a_capture_keeps_the_workspace(renderer, monkeypatch):
    """Under capture there is no scratch; the buffer at hand serves, and the scratch is
    asked for again after the capture."""
    renderer.room = False
    monkeypatch.setattr(torch.cuda, "is_current_stream_capturing", lambda: True)
    _backward(renderer)
    kept = renderer._bws
    _backward(renderer)
    assert renderer._bws is kept and renderer.given == [NEED, NEED]
    monkeypatch.setattr(torch.cuda, "is_current_stream_capturing", lambda: False)
    renderer.room = True
    _backward(renderer)
    assert renderer.given[-1] == BEST


class _Stream:
    """A stream of another library: a handle and nothing else."""
    cuda_stream = 7


@pytest.fixture
def entry(monkeypatch):
    """ngprt_occupancy_from_density on a stand-in library that wants scratch; returns the
    arguments of the native calls, and the devices of the allocations."""
    calls, devices = [], []

    class Lib:
        def ngprt_last_error(self):
            return b"occ_out is NULL"

        def __getattr__(self, name):
            def call(*a):
                calls.append(a)
                return 0 if a[4] else -1
            return call

    empty = torch.empty

    def alloc(n, dtype=None, device=None):
        devices.append(str(device))
        return empty(n, dtype=dtype)

    monkeypatch.setattr(ng, "lib", lambda: Lib())
    for name in ("ngprt_density_scratch_bytes", "ngprt_occupancy_from_density_scratch_bytes"):
        monkeypatch.setattr(ng, name, lambda *a: 64, raising=False)
    ptr = ng._ptr
    monkeypatch.setattr(ng, "_ptr", lambda t: t.data_ptr() if isinstance(t, torch.Tensor) else ptr(t))
    monkeypatch.setattr(torch, "empty", alloc)
    monkeypatch.setattr(torch.cuda, "is_current_stream_capturing", lambda: False)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda *a: _Stream)
    return calls, devices


def _density(out, **kw):
    ng.ngprt_occupancy_from_density(ng.ngprt_scene(), ng.ngprt_render_opts(), 64, 1.0, out, **kw)


def test_outputs_given_as_addresses(entry):
    calls, devices = entry
    _density(4096)
    assert devices == ["cuda"] and calls[0][4] == 4096


def test_a_missing_output_is_the_library_s_error(entry):
    with pytest.raises(ng.NgprtError, match="occ_out is NULL"):
        _density(None)


def test_streams_that_torch_cannot_allocate_on(entry):
    calls, devices = entry
    _density(4096, stream=_Stream)
    assert devices == [] and calls[0][-1] == 7
