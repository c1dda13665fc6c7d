"""The backward's row kernel, through the workspace that it fills: D of every row, and the transposed lists."""
import numpy as np
import pytest
import torch

from paper_2605_15684_gb300 import api, synthetic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,h,H,W,rho", [
    (1, 1, 8, 8, 0.0),        # 64 rows: half a CTA; one block
    (1, 1, 8, 24, 0.0),       # 192 rows: a whole CTA and a half
    (2, 3, 24, 40, 0.5),      # 960 rows a head, 15 blocks
    (1, 2, 128, 128, 0.84),   # 256 blocks a head, 41 kept: the largest lists
])
def test_row_sums_and_transposed_lists(B, h, H, W, rho):
    q, k, v = (x.cuda() for x in synthetic.qkv(B, h, H * W, 64, torch.bfloat16, 61))
    go = synthetic.qkv(B, h, H * W, 64, torch.bfloat16, 62)[0].cuda()
    desc = api.SsbaDesc(B, h, H, W, shift_r=4, shift_c=4, rho=rho)
    idx, cnt = api.build_mask(desc, q, k)
    keep, Tb, BH, N = idx.shape[-1], desc.Tb, B * h, H * W
    cnt = torch.clamp(cnt - torch.arange(cnt.numel(), device="cuda").reshape(cnt.shape).to(torch.int32) % 3, min=1)
    O, lse = api.forward(desc, q, k, v, idx, cnt)
    ws = torch.full((api.backward_workspace_bytes(desc),), 0x55, dtype=torch.uint8, device="cuda")
    api.backward(desc, q, k, v, O, lse, go, idx, cnt, workspace=ws)
    torch.cuda.synchronize()
    assert api.get_status() == api.SSBA_OK
    w = ws.cpu().numpy()

    D = w[: BH * N * 4].view(np.float32)
    x, y = go.double().cpu().numpy().reshape(-1, 64), O.double().cpu().numpy().reshape(-1, 64)
    # 64 products of bf16 (exact in fp32), fewer than 64 roundings of sums
    assert (np.abs(D - (x * y).sum(1)) <= 64 * 2.0 ** -24 * np.abs(x * y).sum(1)).all()

    up = lambda n: (n + 255) // 256 * 256
    toff = up(BH * N * 4) + 256
    tcnt = toff + up(BH * Tb * 4)
    tlist = tcnt + up(BH * Tb * 4)
    off = w[toff: toff + BH * Tb * 4].view(np.int32).reshape(BH, Tb)
    num = w[tcnt: tcnt + BH * Tb * 4].view(np.int32).reshape(BH, Tb)
    lst = w[tlist: tlist + BH * Tb * keep * 4].view(np.int32)
    idx_n, cnt_n = idx.cpu().numpy().reshape(BH, Tb, keep), cnt.cpu().numpy().reshape(BH, Tb)
    kept = np.zeros((BH, Tb, Tb), dtype=bool)  # [head][query block][key block]
    for b in range(BH):
        for i in range(Tb):
            kept[b, i, idx_n[b, i, : cnt_n[b, i]]] = True
        for j in range(Tb):
            want = np.flatnonzero(kept[b, :, j])
            assert num[b, j] == len(want)
            assert (lst[off[b, j]: off[b, j] + len(want)] == want).all()
