"""The fp32 path (CUDA cores, register-tiled products) at the edges of its ranges: one block, a
non-square grid, shifts that are no multiple of 4, and more than 128 query blocks a head (the key
blocks' lists are gathered 128 query blocks at a time). Forward and gradients against the oracle, with
the tolerances of tests/test_parity_gpu.py (1e-4 of O; 1e-5 of the largest gradient, measured 1e-6)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2605_15684_gb300 import api, build, synthetic
from tests.parity import check_out

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,h,H,W,rho,shift", [
    (1, 1, 8, 8, 0.0, (0, 0)),
    (2, 2, 24, 40, 0.6, (3, -5)),
    (1, 2, 96, 96, 0.98, (1, 90)),   # 144 blocks: two gathers of a key block's list
])
def test_fp32_forward_and_gradients(B, h, H, W, rho, shift):
    build.build()
    api.load_library()
    q, k, v = synthetic.qkv(B, h, H * W, 64, torch.float32, 50)
    go = synthetic.qkv(B, h, H * W, 64, torch.float32, 51)[0]
    desc = api.SsbaDesc(B, h, H, W, shift_r=shift[0], shift_c=shift[1], rho=rho, dtype=torch.float32)
    idx_o, cnt_o = oracle.build_mask(q, k, H, W, 8, shift, rho)
    idx, cnt = torch.from_numpy(idx_o).cuda(), torch.from_numpy(cnt_o).cuda()
    qd, kd, vd = q.cuda(), k.cuda(), v.cuda()
    O, lse = api.forward(desc, qd, kd, vd, idx, cnt)
    grads = api.backward(desc, qd, kd, vd, O, lse, go.cuda(), idx, cnt)
    torch.cuda.synchronize()
    check_out(O.cpu().numpy(), lse.cpu().numpy(), *oracle.forward(q, k, v, idx_o, H, W, 8, shift), "fp32")
    for got, want in zip(grads, oracle.backward(q, k, v, go, idx_o, H, W, 8, shift)):
        got = got.cpu().double().numpy()
        assert np.all(np.isfinite(got))
        assert np.abs(got - want).max() <= 1e-5 * max(1.0, np.abs(want).max())
    assert api.get_status() == api.SSBA_OK
