"""Calls on a stream of their own, with the buffers that the binding allocates."""
import pytest
import torch

from paper_2605_15684_gb300 import api, build, synthetic

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    api.load_library()


def test_side_stream_with_default_buffers():
    """The current stream busy, and taking memory as soon as a call has returned: a forward_fused, a mask of
    144 blocks a head (pooled into scratch) and a backward on another stream give what they give on the
    current one."""
    H = W = 96
    q, k, v = (t.cuda() for t in synthetic.qkv(1, 6, H * W, 64, torch.bfloat16, 71))
    go = synthetic.qkv(1, 6, H * W, 64, torch.bfloat16, 72)[0].cuda()
    desc = api.SsbaDesc(1, 6, H, W, shift_r=4, shift_c=4, rho=0.8)

    def calls(stream=None):
        fused = api.forward_fused(desc, q, k, v, stream=stream)
        idx, cnt = api.build_mask(desc, q, k, stream=stream)
        junk = [torch.full((1 << 20,), -1, dtype=torch.int32, device="cuda") for _ in range(8)]
        grads = api.backward(desc, q, k, v, fused[0], fused[1], go, idx, cnt, stream=stream)
        junk += [torch.full((1 << 20,), -1, dtype=torch.int32, device="cuda") for _ in range(8)]
        return (*fused, idx, cnt, *grads)

    want = calls()
    torch.cuda.synchronize()
    busy = torch.randn(8192, 8192, device="cuda").bfloat16()
    for _ in range(3):
        s = torch.cuda.Stream()
        s.wait_stream(torch.cuda.current_stream())
        for _ in range(10):
            busy @ busy
        got = calls(s)
        torch.cuda.current_stream().wait_stream(s)
        torch.cuda.synchronize()
        assert api.get_status() == api.SSBA_OK
        for a, b in zip(got, want):
            assert torch.equal(a, b)


def test_fused_call_captured_before_any_other_on_its_stream():
    """A graph whose fused calls are the first on their stream, then a call outside it before its first replay."""
    q, k, v = (t.cuda() for t in synthetic.qkv(1, 4, 1024, 64, torch.bfloat16, 73))
    desc = api.SsbaDesc(1, 4, 32, 32, shift_r=4, shift_c=4, rho=0.75)
    want = api.forward_fused(desc, q, k, v)
    torch.cuda.synchronize()
    api._fwd_ws.clear()
    s, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        in_graph = [api.forward_fused(desc, q, k, v) for _ in range(2)]
    s.wait_stream(torch.cuda.current_stream())
    outside = api.forward_fused(desc, q, k, v, stream=s)
    torch.cuda.current_stream().wait_stream(s)
    for _ in range(2):
        g.replay()
    torch.cuda.synchronize()
    assert api.get_status() == api.SSBA_OK
    for got in (*in_graph, outside):
        for a, b in zip(got, want):
            assert torch.equal(a, b)
