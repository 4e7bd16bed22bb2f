"""Asynchronous calls that find their stream idle (a replayed graph, given the
call's buffers) or busy (kernel by kernel), mixed, on buffers that change from
call to call, and beside a capture of another thread; bit-exact against the
oracle (no tolerance).
"""
import threading
import time

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

W, H, D = 71, 38, 64


def _images(rng):
    return [rng.integers(0, 256, (H, W), dtype=np.uint8) for _ in range(2)]


# per-line sweeps: the schedule of 4 paths, or a memory cap that two passes' paired cubes would strain
@pytest.mark.parametrize("n_paths,post,per_line", [(2, None, False), (4, None, False), (8, None, False), (2, 7, False),
                                                   (4, 1, False), (8, 7, False), (4, None, True), (8, 7, True)])
def test_idle_and_busy_calls_on_changing_buffers(n_paths, post, per_line):
    import torch

    from paper_1610_04121_gb300 import sgm

    rng = np.random.default_rng(n_paths)
    kind = torch.uint8 if post is None else torch.int16
    with sgm.Context(0, mem_cap_bytes=64 << 20 if per_line else 0) as c:
        sgm.sgm_set_stream(c.handle, torch.cuda.Stream())
        if n_paths == 4:
            sgm.sgm_set_schedule(c.handle, sgm.SGM_SCHED_V_THEN_H if per_line else sgm.SGM_SCHED_PAIRS)

        def call(b):
            a = (c.handle, b[0], b[1], W, H, D, 7, 84, n_paths)
            if post is None:
                sgm.sgm_compute_async(*a, b[2])
            else:
                sgm.sgm_compute_ex_async(*a, post, b[2])

        def check(b):
            left, right = (b[i].cpu().numpy() for i in (0, 1))
            if post is None:
                assert (b[2].cpu().numpy() == oracle.sgm(left, right, D, 7, 84, n_paths)).all()
            else:
                assert (b[2].cpu().numpy().view(np.uint16) == oracle.sgm_ex(left, right, D, 7, 84, n_paths, post)).all()

        sets = [[*(torch.from_numpy(x).cuda() for x in _images(rng)), torch.zeros((H, W), dtype=kind, device="cuda")]
                for _ in range(4)]
        for order in ([0, 0, 0], [1, 2, 3, 1], [0, 3, 3, 2]):  # waited for, one by one
            for k in order:
                sets[k][2].zero_()
                torch.cuda.synchronize()
                call(sets[k])
                torch.cuda.synchronize()
                check(sets[k])
        for b in sets:  # an idle call and three behind it, without a wait
            b[2].zero_()
        torch.cuda.synchronize()
        for b in sets:
            call(b)
        torch.cuda.synchronize()
        for b in sets:
            check(b)


@pytest.mark.parametrize("legacy", [False, True])
def test_idle_calls_beside_a_capture_of_another_thread(legacy):
    import torch

    from paper_1610_04121_gb300 import sgm

    rng = np.random.default_rng(2)
    left, right = _images(rng)
    l, r = torch.from_numpy(left).cuda(), torch.from_numpy(right).cuda()
    outs = [torch.zeros((H, W), dtype=torch.uint8, device="cuda") for _ in range(12)]
    x = torch.zeros(1000, device="cuda")
    errors = []
    with sgm.Context(0) as c:
        st = torch.cuda.default_stream() if legacy else torch.cuda.Stream()
        sgm.sgm_set_stream(c.handle, st)
        sgm.sgm_compute_async(c.handle, l, r, W, H, D, 7, 84, 8, outs[0])
        torch.cuda.synchronize()

        def calls():
            try:
                for o in outs:
                    sgm.sgm_compute_async(c.handle, l, r, W, H, D, 7, 84, 8, o)
                    time.sleep(0.002)  # the stream has run dry by the next call
            except Exception as e:  # noqa: BLE001
                errors.append(e)

        t = threading.Thread(target=calls)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):  # capture mode "global"
            x.add_(1)
            t.start()
            t.join()
            x.add_(1)
        torch.cuda.synchronize()
        assert not errors, errors
        g.replay()
        torch.cuda.synchronize()
        assert (x == 2).all()
        ref = oracle.sgm(left, right, D, 7, 84, 8)
        for o in outs:
            assert (o.cpu().numpy() == ref).all()
