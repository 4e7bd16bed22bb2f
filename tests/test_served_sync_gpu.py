"""Served batches beside a caller that synchronizes the whole device.

The first wave of every shape builds its graph on the scheduler's thread.  A
stream capture there would make cudaDeviceSynchronize on any other thread fail
with "operation not permitted when stream is capturing".
"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def test_device_synchronize_while_waves_are_built():
    import torch

    from paper_1610_04121_gb300 import sgm

    rng = np.random.default_rng(3)
    with sgm.Context(0) as c:
        for D in (32, 64, 96, 128, 160, 192, 224, 256):
            left, right = (rng.integers(0, 256, (40, 300), dtype=np.uint8) for _ in range(2))
            dl, dr = torch.from_numpy(left).cuda(), torch.from_numpy(right).cuda()
            outs = {n: torch.zeros((40, 300), dtype=torch.uint8, device="cuda") for n in (2, 4, 8)}
            torch.cuda.synchronize()
            tickets = [sgm.sgm_submit(c.handle, dl, dr, 300, 40, D, 7, 84, n, o) for n, o in outs.items()]
            for _ in range(2000):
                torch.cuda.synchronize()
            for t in tickets:
                assert sgm.sgm_poll(c.handle, t, -1) == sgm.SGM_OK
            for n, o in outs.items():
                assert (o.cpu().numpy() == oracle.sgm(left, right, D, 7, 84, n)).all(), (D, n)
