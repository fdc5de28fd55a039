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
