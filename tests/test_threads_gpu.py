"""Host threads that launch the same kernel with different amounts of shared memory."""
import threading

import pytest
import torch

from paper_2605_15684_gb300 import api, build

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,sides", [(64, ((136, 240), (136, 152))), (64, ((128, 128), (96, 128))), (32, ((136, 240), (88, 88)))])
def test_selections_of_several_row_lengths_from_two_threads(d, sides):
    """Rows of 510 and 323 blocks, 256 and 192, and of another width: every call is accepted and gives the lists that
    it gives alone."""
    build.build()
    api.load_library()
    work = []
    for i, (H, W) in enumerate(sides):
        desc = api.SsbaDesc(1, 24 if d == 64 else 2, H, W, head_dim=d, rho=0.8)
        g = torch.Generator(device="cuda").manual_seed(i)
        qb, kb = (torch.randn(1, desc.heads, desc.Tb, d, generator=g, device="cuda") for _ in range(2))
        work.append((desc, qb, kb, *api.select_mask(desc, qb, kb)))
    torch.cuda.synchronize()
    bad, start = [], threading.Barrier(len(work))

    def run(desc, qb, kb, idx, cnt):
        try:
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                start.wait()
                for _ in range(1500):
                    got = api.select_mask(desc, qb, kb)
            s.synchronize()
            if not (torch.equal(got[0], idx) and torch.equal(got[1], cnt)):
                bad.append("lists differ")
        except Exception as e:  # a refused launch
            bad.append(str(e))

    threads = [threading.Thread(target=run, args=w) for w in work]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
