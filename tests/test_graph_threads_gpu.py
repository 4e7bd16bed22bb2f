"""Blocking calls, whose graphs are made on the second call with a set of
buffers, beside another thread that synchronizes the whole device.  A stream
capture would make that cudaDeviceSynchronize fail with "operation not permitted
when stream is capturing"; the graphs are built node by node.  Bit-exact against
the oracle.
"""
import threading

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("timed", [False, True])
def test_device_synchronize_while_graphs_are_made(timed):
    import torch

    from paper_1610_04121_gb300 import sgm

    W, H, D = 60, 40, 32
    rng = np.random.default_rng(9)
    stop, errors, syncs = threading.Event(), [], [0]

    def synchronize():
        while not stop.is_set() and not errors:
            try:
                torch.cuda.synchronize()
                syncs[0] += 1
            except Exception as e:  # noqa: BLE001
                errors.append(e)

    torch.cuda.init()
    t = threading.Thread(target=synchronize)
    with sgm.Context(0, flags=sgm.SGM_FLAG_STAGE_TIMING if timed else 0) as c:
        for n_paths in (2, 4, 8):
            c.compute(*(np.zeros((H, W), np.uint8) for _ in range(2)), D, 7, 84, n_paths)  # tuned
        t.start()
        try:
            for k in range(150):
                n_paths = (2, 4, 8)[k % 3]
                left, right = (rng.integers(0, 256, (H, W), dtype=np.uint8) for _ in range(2))
                out = np.zeros((H, W), np.uint8)
                for _ in range(3):
                    out[:] = 255
                    sgm.sgm_compute(c.handle, left, right, W, H, D, 7, 84, n_paths, out)
                    assert (out == oracle.sgm(left, right, D, 7, 84, n_paths)).all()
                if timed:
                    assert len(sgm.sgm_stage_times(c.handle)) == (7 if n_paths == 8 else 5)
        finally:
            stop.set()
            t.join()
    assert not errors, errors
    assert syncs[0] > 0
