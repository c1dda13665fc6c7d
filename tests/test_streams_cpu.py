"""Memory that the binding allocates for a call with ``stream=`` belongs to that stream: no GPU needed, the
library's launches and torch's streams and allocations are stood in for."""
import contextlib

import pytest
import torch

from paper_2605_15684_gb300 import api, build


class _Stream:
    def __init__(self, ptr):
        self.cuda_stream = ptr


class _Lib:
    """The library's host-only entry points as they are, its launches as successes."""

    def __init__(self, lib):
        self._lib = lib

    def __getattr__(self, name):
        if name in ("ssba_keep_count", "ssba_last_error") or name.endswith("_bytes"):
            return getattr(self._lib, name)
        return lambda *a: 0


@pytest.fixture
def world(monkeypatch):
    build.build()
    lib = api.load_library()
    main, stack, made, recorded = _Stream(1), [], [], []
    stack.append(main)

    @contextlib.contextmanager
    def on(stream):
        stack.append(stream)
        yield
        stack.pop()

    def maker(f):
        def make(shape, dtype=None, device=None):
            t = f(shape, dtype=dtype)
            made.append((t.data_ptr(), stack[-1]))
            return t
        return make

    monkeypatch.setattr(api, "load_library", lambda path=None: _Lib(lib))
    monkeypatch.setattr(api, "_check", lambda *a: None)
    monkeypatch.setattr(api, "_ws_args", lambda ws: (None, 0) if ws is None else (ws.data_ptr(), ws.numel()))
    monkeypatch.setattr(api, "_fwd_ws", {})
    monkeypatch.setattr(lib, "ssba_forward_workspace_bytes", lambda d: 1024)  # asks the device
    monkeypatch.setattr(torch, "empty", maker(torch.empty))
    monkeypatch.setattr(torch, "zeros", maker(torch.zeros))
    monkeypatch.setattr(torch.cuda, "stream", on)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda *a: stack[-1])
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 0)
    monkeypatch.setattr(torch.cuda, "is_current_stream_capturing", lambda: False)
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda d: stack[-1].cuda_stream, raising=False)
    monkeypatch.setattr(torch.Tensor, "record_stream", lambda t, s: recorded.append((t.data_ptr(), s)))
    return main, made, recorded


def _calls(stream):
    d = api.SsbaDesc(1, 2, 16, 16, rho=0.5)
    x = torch.randn(1, 2, 256, 64)
    m, idx, cnt, lse = torch.randn(1, 2, 4, 64), torch.ones(1), torch.ones(1), torch.ones(1)
    img, kw = torch.randn(1, 2, 8, 8), dict(stream=stream)
    return [
        lambda: api.build_mask(d, x, x, scores=True, **kw), lambda: api.build_mask_noalloc(d, x, x, **kw),
        lambda: api.select_mask(d, m, m, scores=True, **kw), lambda: api.pool_blocks(d, x, x, **kw),
        lambda: api.qkv_rope_pool(d, x, x, **kw), lambda: api.forward(d, x, x, x, idx, cnt, **kw),
        lambda: api.forward_joint(d, x, x, x, x, x, idx, cnt, **kw), lambda: api.forward_dense(d, x, x, x, **kw),
        lambda: api.forward_select(d, x, x, x, m, m, **kw), lambda: api.forward_fused(d, x, x, x, **kw),
        lambda: api.backward(d, x, x, x, x, lse, x, idx, cnt, **kw), lambda: api.haar_dwt(img, **kw),
        lambda: api.haar_iwt(img, 1, nb=2, **kw), lambda: api.haar_dwt_pyramid(img, 2, **kw),
        lambda: api.haar_iwt_pyramid([img], 1, nb=2, **kw),
    ]


@pytest.mark.parametrize("i", range(15))
def test_what_a_call_allocates_belongs_to_its_stream(world, i):
    main, made, recorded = world
    side = _Stream(2)
    out = _calls(side)[i]()
    assert made and all(s is side for _, s in made)
    outs = [t for t in (out if isinstance(out, (list, tuple)) else [out]) if t is not None]
    for t in outs:  # read and freed by the caller on the current stream
        assert (t.data_ptr(), main) in recorded
    del made[:], recorded[:]
    for same in (None, main):  # on the current stream nothing is recorded
        _calls(same)[i]()
        assert made and all(s is main for _, s in made) and not recorded


def test_a_workspace_made_in_a_capture_is_not_kept(world, monkeypatch):
    """Its fill runs when the graph does, so a call outside the graph must not find it; it is zero where a call
    reads it, and one that exists already is used."""
    d = api.SsbaDesc(1, 2, 16, 16, rho=0.5)
    monkeypatch.setattr(torch.cuda, "is_current_stream_capturing", lambda: True)
    ws = api.default_forward_workspace(d, "cuda:0")
    assert ws.numel() == 1024 and not ws[-256:].any() and not api._fwd_ws
    monkeypatch.setattr(torch.cuda, "is_current_stream_capturing", lambda: False)
    kept = api.default_forward_workspace(d, "cuda:0")
    assert not kept.any() and kept is api.default_forward_workspace(d, "cuda:0")
    monkeypatch.setattr(torch.cuda, "is_current_stream_capturing", lambda: True)
    assert kept is api.default_forward_workspace(d, "cuda:0")
