"""The bf16 forward's pairing of query blocks (two items as the halves of M=128 products, a left-over
item split over both halves) at the sizes where it can go wrong, against the oracle at the bf16
tolerance of tests/parity.py: item counts around whole rounds of pairs, lists of one to a few blocks,
counts that differ within a pair (zero among them), scores that raise the reference maximum, and
values of one item that must not reach its partner."""
import numpy as np
import pytest
import torch

import oracle
from paper_2605_15684_gb300 import api, build, synthetic
from tests.parity import check_out

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    api.load_library()
    yield
    torch.cuda.synchronize()
    assert api.get_status() == api.SSBA_OK


def _inputs(h, H, W, seed):
    q, k, v = synthetic.qkv(1, h, H * W, 64, torch.bfloat16, seed)
    return (q, k, v), [t.cuda() for t in (q, k, v)]


@pytest.mark.parametrize("h,H,W,rho,shift", [
    (1, 16, 16, 0.75, (4, 4)),     # 4 items of 1 block: one item a pipeline, half B empty
    (1, 8, 8, 0.0, (0, 0)),        # one item of one block
    (1, 8, 24, 0.5, (0, 4)),       # 3 items of 2 blocks
    (3, 24, 40, 0.6, (4, -4)),     # 45 items of 6 blocks
    (10, 64, 64, 0.96, (4, 4)),    # 640 items of 3 blocks: one round of pairs, then single items for some
    (17, 64, 64, 0.93, (0, 0)),    # 1088 items of 5 blocks: a pair for some pipelines, one item for the rest
    (19, 64, 64, 0.9, (4, 4)),     # 1216 items: two whole rounds of pairs (304 pipelines)
])
def test_item_counts(h, H, W, rho, shift):
    (q, k, v), d = _inputs(h, H, W, 40)
    desc = api.SsbaDesc(1, h, H, W, shift_r=shift[0], shift_c=shift[1], rho=rho)
    idx_o, cnt_o = oracle.build_mask(q, k, H, W, 8, shift, rho)
    O, lse = api.forward(desc, *d, torch.from_numpy(idx_o).cuda(), torch.from_numpy(cnt_o).cuda())
    torch.cuda.synchronize()
    check_out(O.float().cpu().numpy(), lse.cpu().numpy(), *oracle.forward(q, k, v, idx_o, H, W, 8, shift), "bf16")


@pytest.mark.parametrize("h", [2, 10])
def test_ragged_and_empty_counts(h):
    """Counts 0, 1, 2, 5 and keep mixed within the pairs and among the split items; an empty list
    gives O = 0 and lse = -inf."""
    H = W = 64
    rho, shift = 0.9, (4, 4)
    (q, k, v), d = _inputs(h, H, W, 41)
    desc = api.SsbaDesc(1, h, H, W, shift_r=4, shift_c=4, rho=rho)
    idx_o, _ = oracle.build_mask(q, k, H, W, 8, shift, rho)
    keep, Tb = idx_o.shape[-1], 64
    choices = np.array([keep, 0, 1, 2, 5], dtype=np.int32)
    cnt = choices[(np.arange(h * Tb).reshape(1, h, Tb) * 7 // 3) % len(choices)]
    O, lse = api.forward(desc, *d, torch.from_numpy(idx_o).cuda(), torch.from_numpy(cnt).cuda())
    torch.cuda.synchronize()
    rows = cnt[:, :, oracle.partition(H, W, 8, shift)]
    O, lse = O.float().cpu().numpy(), lse.cpu().numpy()
    assert np.all(O[rows == 0] == 0) and np.all(np.isneginf(lse[rows == 0]))
    for c in choices[choices > 0]:
        O_c, l_c = oracle.forward(q, k, v, np.ascontiguousarray(idx_o[..., :c]), H, W, 8, shift)
        check_out(O[rows == c], lse[rows == c], O_c[rows == c], l_c[rows == c], "bf16")


@pytest.mark.parametrize("scale", [1.5, 6.0])
def test_reference_maximum_raised(scale):
    """A softmax scale that spreads the scores over tens and hundreds of units: later blocks exceed the
    first one's maximum by more than the 2^24 at which the reference is raised. Almost all of a row's
    weight is then on a few keys, so O is a few bf16 values of V."""
    H = W = 32
    (q, k, v), d = _inputs(6, H, W, 42)
    desc = api.SsbaDesc(1, 6, H, W, rho=0.3, softmax_scale=scale)
    idx_o, cnt_o = oracle.build_mask(q, k, H, W, 8, (0, 0), 0.3)
    O, lse = api.forward(desc, *d, torch.from_numpy(idx_o).cuda(), torch.from_numpy(cnt_o).cuda())
    torch.cuda.synchronize()
    lab = oracle.partition(H, W, 8, (0, 0))
    for h in range(6):  # plain fp64 softmax over the kept blocks
        s = (q[0, h].double() @ k[0, h].double().T).numpy() * np.float32(scale)
        kept = np.zeros((16, 16), dtype=bool)
        np.put_along_axis(kept, idx_o[0, h], True, axis=1)
        s = np.where(kept[lab][:, lab], s, -np.inf)
        m = s.max(axis=1, keepdims=True)
        e = np.exp(s - m)
        ref = (e / e.sum(axis=1, keepdims=True)) @ v[0, h].double().numpy()
        # P = exp2 of fp32 scores: |s| 2^-22 of absolute error in the exponent, then bf16 roundings
        tol = 2e-2 + 2.0 ** -20 * np.abs(m) * np.abs(v[0, h].double().numpy()).max()
        assert np.all(np.abs(O[0, h].float().cpu().numpy() - ref) <= tol)
        l_ref = (m + np.log(e.sum(axis=1, keepdims=True)))[:, 0]
        assert np.allclose(lse[0, h].cpu().numpy(), l_ref, rtol=1e-5, atol=1e-2)


def test_infinite_values_stay_in_their_items():
    """One block of V infinite: query blocks that do not keep it give what they give without it."""
    h, H, W, rho = 4, 32, 32, 0.75
    (_, _, _), (q, k, v) = _inputs(h, H, W, 43)
    desc = api.SsbaDesc(1, h, H, W, rho=rho)
    idx, cnt = api.build_mask(desc, q, k)
    O, lse = api.forward(desc, q, k, v, idx, cnt)
    lab = torch.from_numpy(np.asarray(oracle.partition(H, W, 8, (0, 0)))).long().cuda()
    bad = 5
    v2 = v.clone()
    v2[:, :, lab == bad] = float("inf")
    O2, lse2 = api.forward(desc, q, k, v2, idx, cnt)
    torch.cuda.synchronize()
    hit = (idx == bad).any(-1)[:, :, lab]  # [1, h, N]
    assert bool(hit.any()) and not bool(hit.all())
    assert torch.equal(O2[~hit], O[~hit]) and torch.equal(lse2, lse)
    assert not bool(torch.isfinite(O2[hit].float()).any())


@pytest.mark.parametrize("scale,ramp", [(1.5, 1.0), (6.0, 1.0), (1.0, 12.0)])
def test_dense_reference_maximum_raised(scale, ramp):
    """The dense kernel's reference maximum: scores that outgrow the first tile's by more than 2^24, in the
    first chunks of a tile (their P is formed again) and in the last one (the rest of P is rescaled)."""
    H = W = 32
    (q, k, v), _ = _inputs(3, H, W, 44)
    k = (k.float() * torch.linspace(0.1, ramp, H * W).view(1, 1, -1, 1)).bfloat16()
    if ramp > 1:  # every 128-key tile's largest scores in its last 32 keys
        k = torch.where((torch.arange(H * W) % 128 < 96).view(1, 1, -1, 1), k * 0.05, k)
    desc = api.SsbaDesc(1, 3, H, W, softmax_scale=scale)
    O, lse = api.forward_dense(desc, q.cuda(), k.cuda(), v.cuda())
    torch.cuda.synchronize()
    for h in range(3):
        s = (q[0, h].double() @ k[0, h].double().T).numpy() * np.float32(scale)
        m = s.max(axis=1, keepdims=True)
        e = np.exp(s - m)
        ref = (e / e.sum(axis=1, keepdims=True)) @ v[0, h].double().numpy()
        # as in test_reference_maximum_raised
        tol = 2e-2 + 2.0 ** -20 * np.abs(m) * np.abs(v[0, h].double().numpy()).max()
        assert np.all(np.abs(O[0, h].float().cpu().numpy() - ref) <= tol)
        assert np.allclose(lse[0, h].cpu().numpy(), (m + np.log(e.sum(axis=1, keepdims=True)))[:, 0], rtol=1e-5, atol=1e-2)


@pytest.mark.parametrize("low", [float("-inf"), -2.0 ** 37])
@pytest.mark.parametrize("far", [16.0, -16.0])
def test_dense_first_keys_masked_by_low_scores(low, far):
    """Every key but the last 32 of the second tile scores -inf, or -2^37: the reference maximum is that low
    until those 32 come, in a tile's last chunk. Their scaled scores lie around +-177, where exp2 against a
    reference of 0 is out of fp32's range. Softmax over those 32 keys in fp64 is what both must give."""
    H = W = 16
    (q, k, v), _ = _inputs(2, H, W, 45)
    k = k.clone()
    q, real = (q * 0.5).bfloat16(), torch.arange(H * W) >= 224
    q[..., 0], q[..., 1] = 1.0, 8.0
    k[..., 0], k[..., 1] = torch.where(real, 0.0, low).bfloat16(), torch.where(real, far * 8, 0.0).bfloat16()
    scale = np.float32(np.log(2.0) / 4)  # times log2(e) 0.25 exactly: the low scores have no rounding of their own
    assert np.float32(scale * np.float32(1.4426950408889634)) == np.float32(0.25)
    desc = api.SsbaDesc(1, 2, H, W, softmax_scale=float(scale))
    O, lse = api.forward_dense(desc, q.cuda(), k.cuda(), v.cuda())
    torch.cuda.synchronize()
    for h in range(2):
        s = (q[0, h].double() @ k[0, h, 224:].double().T).numpy() * float(scale)
        m = s.max(axis=1, keepdims=True)
        assert (np.abs(m) > 100).all()
        e = np.exp(s - m)
        ref = (e / e.sum(axis=1, keepdims=True)) @ v[0, h, 224:].double().numpy()
        # as in test_reference_maximum_raised
        tol = 2e-2 + 2.0 ** -20 * np.abs(m) * np.abs(v[0, h].double().numpy()).max()
        assert np.all(np.abs(O[0, h].float().cpu().numpy() - ref) <= tol)
        assert np.allclose(lse[0, h].cpu().numpy(), (m + np.log(e.sum(axis=1, keepdims=True)))[:, 0], rtol=1e-5, atol=1e-2)


@pytest.mark.parametrize("heads", [1, 20])  # 4 items: one a pipeline, its two blocks in the two halves; 1280: pairs too
@pytest.mark.parametrize("low", [0, 1])
def test_infinite_value_under_a_vanishing_weight(heads, low):
    """Lists of two blocks, the scores of one (the `low`-th) 400 below the other's, where exp gives 0, and a column of its
    V infinite: that column of O is no number (0 x inf), wherever the item runs, and the rest is the other block's."""
    H = W = 16 if heads == 1 else 64
    (_, _, _), (q, k, v) = _inputs(heads, H, W, 46)
    desc = api.SsbaDesc(1, heads, H, W, rho=0.5 if heads == 1 else 62 / 64)
    Tb = desc.Tb
    lab = torch.from_numpy(np.asarray(oracle.partition(H, W, 8, (0, 0)))).long().cuda()
    blocks = (0, 2)
    q[..., 0] = 16.0
    k[..., 0] = torch.where(lab == blocks[low], -200.0, 0.0).bfloat16()
    v[:, :, lab == blocks[low], 5] = float("inf")
    idx = torch.tensor(blocks, dtype=torch.int32, device="cuda").expand(1, heads, Tb, 2).contiguous()
    cnt = torch.full((1, heads, Tb), 2, dtype=torch.int32, device="cuda")
    O, lse = api.forward(desc, q, k, v, idx, cnt)
    torch.cuda.synchronize()
    assert not bool(torch.isfinite(O[..., 5]).any())
    kk, vv = (t[:, :, lab == blocks[1 - low]].float() for t in (k, v))
    s = q.float() @ kk.transpose(-1, -2) / 8
    want, rest = torch.softmax(s, -1) @ vv, torch.arange(64, device="cuda") != 5
    assert float((O.float() - want)[..., rest].abs().max()) <= 2e-2  # the bf16 bound of tests/parity.py
    assert float((lse - torch.logsumexp(s, -1)).abs().max()) <= 1e-2
