"""Replayed graphs of blocking calls over sizes, D, penalties and path counts: three
calls on the same buffers (kernel by kernel, making the graph, replaying it), the
images changed in between; bit-exact against the oracle (no tolerance)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H", [(1, 1), (2, 33), (17, 23), (64, 40), (77, 45), (200, 31), (31, 200), (301, 214)])
@pytest.mark.parametrize("D,P1,P2", [(32, 7, 84), (96, 7, 120), (128, 10, 85), (160, 50, 20), (256, 7, 200)])
def test_three_calls_on_the_same_buffers(W, H, D, P1, P2):
    import torch

    from paper_1610_04121_gb300 import sgm

    rng = np.random.default_rng(W * 7 + H + D)
    left, right, out = (torch.zeros((H, W), dtype=torch.uint8, device="cuda") for _ in range(3))
    out16 = torch.zeros((H, W), dtype=torch.int16, device="cuda")
    with sgm.Context(0) as c:
        for k in range(3):
            a, b = (rng.integers(0, 256, (H, W), dtype=np.uint8) for _ in range(2))
            left.copy_(torch.from_numpy(a))
            right.copy_(torch.from_numpy(b))
            for sched, n_paths in ((0, 4), (1, 4), (2, 4), (2, 2), (2, 8)):
                sgm.sgm_set_schedule(c.handle, sched)
                out.fill_(255)
                torch.cuda.synchronize()
                sgm.sgm_compute(c.handle, left, right, W, H, D, P1, P2, n_paths, out)
                assert (out.cpu().numpy() == oracle.sgm(a, b, D, P1, P2, n_paths)).all(), (k, sched, n_paths)
            out16.zero_()
            torch.cuda.synchronize()
            sgm.sgm_compute_ex(c.handle, left, right, W, H, D, P1, P2, 4, 7, out16)
            assert (out16.cpu().numpy().view(np.uint16) == oracle.sgm_ex(a, b, D, P1, P2, 4, 7)).all(), k
