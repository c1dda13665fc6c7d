"""The gating (Top-k, drop the smallest) at the edges of its code paths: row lengths around the register
layouts (32, 64, 256, 512, 1024 labels) and rows a warp takes, keep counts at both ends, ties across
the cut and infinities, from block means given (ssba_select_mask). The lists must be the oracle's gate
of the exported scores bit for bit; build_mask's must agree with the means' own lists."""
import numpy as np
import pytest
import torch

import oracle
from paper_2605_15684_gb300 import api, build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    api.load_library()


def _check(desc, qb, kb):
    idx, cnt, S = api.select_mask(desc, qb, kb, scores=True)
    torch.cuda.synchronize()
    keep, Tb = api.keep_count(desc), desc.Tb
    S, idx = S.cpu().numpy().reshape(-1, Tb, Tb), idx.cpu().numpy().reshape(-1, Tb, keep)
    for s, i in zip(S, idx):
        assert np.array_equal(oracle.gate(s, Tb - keep), i)
    assert bool((cnt == keep).all())
    return S


@pytest.mark.parametrize("h,H,W,rho", [
    (1, 8, 8, 0.0), (3, 64, 64, 0.8416), (24, 64, 64, 0.5), (2, 88, 96, 0.9), (2, 128, 128, 0.84), (1, 128, 128, 0.998),
    (2, 136, 128, 0.001), (2, 136, 240, 0.75), (1, 184, 184, 0.9), (1, 256, 320, 0.97),
    (5, 40, 40, 0.6), (3, 32, 64, 0.97),                               # 25 and 32 blocks: one key a lane
    (3, 136, 240, 0.75), (6, 136, 240, 0.999), (3, 184, 184, 0.5), (8, 184, 184, 0.9),  # two and four rows a warp
    (2, 256, 512, 0.9),                                                # 2048 blocks, the longest
])
def test_selection_is_exact(h, H, W, rho):
    desc = api.SsbaDesc(1, h, H, W, rho=rho)
    g = torch.Generator(device="cuda").manual_seed(H + W)
    qb, kb = (torch.randn(1, h, desc.Tb, 64, generator=g, device="cuda") * 0.125 for _ in range(2))
    S = _check(desc, qb, kb)
    want = torch.einsum("hid,hjd->hij", qb[0].double(), kb[0].double()).cpu().numpy()
    assert np.abs(S - want).max() <= 64 * 2.0 ** -24 * np.abs(want).max() * 16


@pytest.mark.parametrize("H,W", [(24, 24), (32, 64), (64, 64), (128, 128), (136, 240)])
def test_ties_and_infinities(H, W):
    """Every score one of five values (exact in fp32), so that the cut falls inside a run of equal ones;
    then one key block infinite (scores of +inf and -inf)."""
    desc = api.SsbaDesc(1, 1, H, W, rho=0.8)
    g = torch.Generator(device="cuda").manual_seed(1)
    qb = torch.zeros(1, 1, desc.Tb, 64, device="cuda")
    kb = torch.zeros_like(qb)
    qb[..., 0] = torch.randint(0, 2, (desc.Tb,), generator=g, device="cuda") * 2.0 - 1.0
    kb[..., 0] = torch.randint(-2, 3, (desc.Tb,), generator=g, device="cuda").float()
    _check(desc, qb, kb)
    kb[0, 0, 7, 0] = float("inf")
    _check(desc, qb, kb)


@pytest.mark.parametrize("H,W", [(88, 96), (128, 128)])  # above the one-launch build's rows: two kernels
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_build_mask_of_long_rows_equals_its_means_lists(H, W, dtype):
    desc = api.SsbaDesc(1, 3, H, W, shift_r=4, shift_c=4, rho=0.84, dtype=dtype)
    g = torch.Generator(device="cuda").manual_seed(3)
    q, k = (torch.randn(1, 3, H * W, 64, generator=g, device="cuda").to(dtype) for _ in range(2))
    idx, cnt = api.build_mask(desc, q, k)
    idx2, cnt2 = api.select_mask(desc, *api.pool_blocks(desc, q, k))
    torch.cuda.synchronize()
    assert torch.equal(idx, idx2) and torch.equal(cnt, cnt2)


def test_fused_with_many_items_equals_two_calls():
    """More query blocks than the attention launch selects itself (16 an SM): the lists, means and outputs
    of the separate calls, bit for bit."""
    desc = api.SsbaDesc(2, 24, 64, 64, shift_r=4, shift_c=4, rho=0.9)
    g = torch.Generator(device="cuda").manual_seed(4)
    q, k, v = (torch.randn(2, 24, 4096, 64, generator=g, device="cuda").bfloat16() for _ in range(3))
    O, lse, idx, cnt, qb, kb = api.forward_fused(desc, q, k, v)
    qb2, kb2 = api.pool_blocks(desc, q, k)
    O3, lse3, idx3, cnt3, S3 = api.forward_select(desc, q, k, v, qb2, kb2, scores=True)
    idx2, cnt2 = api.build_mask(desc, q, k)
    O2, lse2 = api.forward(desc, q, k, v, idx2, cnt2)
    torch.cuda.synchronize()
    assert api.get_status() == api.SSBA_OK
    assert torch.equal(qb, qb2) and torch.equal(kb, kb2)
    for a, b, c in ((idx, idx2, idx3), (cnt, cnt2, cnt3), (O, O2, O3), (lse, lse2, lse3)):
        assert torch.equal(a, b) and torch.equal(a, c)
    assert bool(torch.isfinite(S3).all())


@pytest.mark.parametrize("h,H,W", [(3, 64, 64), (3, 8, 520), (24, 48, 88), (2, 64, 96), (2, 72, 88), (40, 48, 88)])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_one_launch_mask_by_blocks_a_cta(h, H, W, dtype):
    """64 blocks a head (eight a CTA), 65 and 66 (nine), 96 (twelve), 99 (thirteen), and 66 with more CTAs than two
    an SM (two kernels): the lists of the same means, pooled and selected apart."""
    desc = api.SsbaDesc(1, h, H, W, shift_r=4, shift_c=4, rho=0.84, dtype=dtype)
    g = torch.Generator(device="cuda").manual_seed(H * W)
    q, k = (torch.randn(1, h, H * W, 64, generator=g, device="cuda").to(dtype) for _ in range(2))
    idx, cnt = api.build_mask(desc, q, k)
    idx2, cnt2 = api.select_mask(desc, *api.pool_blocks(desc, q, k))
    torch.cuda.synchronize()
    assert torch.equal(idx, idx2) and torch.equal(cnt, cnt2)


def test_fused_with_more_heads_than_a_grid_dimension():
    """65600 (batch, head) pairs, more than a launch's y dimension holds: as two calls of half of them."""
    h, H, W = 65600, 8, 16
    g = torch.Generator(device="cuda").manual_seed(5)
    q, k, v = (torch.randn(1, h, H * W, 64, generator=g, device="cuda", dtype=torch.bfloat16) for _ in range(3))
    got = api.forward_fused(api.SsbaDesc(1, h, H, W, rho=0.5), q, k, v)
    desc = api.SsbaDesc(1, h // 2, H, W, rho=0.5)
    for part in (slice(0, h // 2), slice(h // 2, h)):
        want = api.forward_fused(desc, *(t[:, part] for t in (q, k, v)))
        for a, b in zip(got, want):
            assert torch.equal(a[:, part], b)
    assert api.get_status() == api.SSBA_OK
