"""The asynchronous calls (kernels launched with programmatic serialization)
captured into the caller's own graph and replayed back to back on changing
images, and run by several threads with contexts and streams of their own;
bit-exact against the oracle (no tolerance).
"""
import threading

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def _pair(rng, W, H):
    return [rng.integers(0, 256, (H, W), dtype=np.uint8) for _ in range(2)]


@pytest.mark.parametrize("kind", ["plain", "post", "static"])
@pytest.mark.parametrize("W,H,D,n_paths", [(70, 34, 64, 2), (70, 34, 64, 4), (71, 35, 96, 8), (200, 120, 256, 8)])
def test_replays_of_a_captured_call(kind, W, H, D, n_paths):
    import torch

    from paper_1610_04121_gb300 import sgm

    if kind == "static" and D == 256:
        pytest.skip("past the static scratch")
    rng = np.random.default_rng(W + D)
    st = torch.cuda.Stream()
    with sgm.Context(0) as c:
        sgm.sgm_set_stream(c.handle, st)
        left, right = (torch.zeros((H, W), dtype=torch.uint8, device="cuda") for _ in range(2))
        out = torch.zeros((H, W), dtype=torch.int16 if kind == "post" else torch.uint8, device="cuda")

        def call():
            if kind == "plain":
                sgm.sgm_compute_async(c.handle, left, right, W, H, D, 7, 84, n_paths, out)
            elif kind == "post":
                sgm.sgm_compute_ex_async(c.handle, left, right, W, H, D, 7, 84, n_paths, 7, out)
            else:
                sgm.sgm_compute_static(left, right, W, H, D, 7, 84, n_paths, out, st)

        torch.cuda.synchronize()
        call()  # tunes the schedule, sizes the arena, sets up the static scratch
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=st):
            call()
        for _ in range(3):
            a, b = _pair(rng, W, H)
            left.copy_(torch.from_numpy(a))
            right.copy_(torch.from_numpy(b))
            out.zero_()
            torch.cuda.synchronize()
            for _ in range(3):
                graph.replay()
            torch.cuda.synchronize()
            if kind == "post":
                assert (out.cpu().numpy().view(np.uint16) == oracle.sgm_ex(a, b, D, 7, 84, n_paths, 7)).all()
            else:
                assert (out.cpu().numpy() == oracle.sgm(a, b, D, 7, 84, n_paths)).all()


def test_threads_with_contexts_and_streams_of_their_own():
    import torch

    from paper_1610_04121_gb300 import sgm

    wrong, done = [], []

    def work(seed):
        rng = np.random.default_rng(seed)
        st = torch.cuda.Stream()
        with sgm.Context(0) as c:
            sgm.sgm_set_stream(c.handle, st)
            for k in range(18):
                W, H, D, n = int(rng.integers(8, 200)), int(rng.integers(8, 120)), 32 * int(rng.integers(1, 9)), (2, 4, 8)[k % 3]
                a, b = _pair(rng, W, H)
                with torch.cuda.stream(st):
                    left, right = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()
                    out = torch.zeros_like(left)
                    for _ in range(3):
                        sgm.sgm_compute_async(c.handle, left, right, W, H, D, 7, 84, n, out)
                    st.synchronize()
                if not (out.cpu().numpy() == oracle.sgm(a, b, D, 7, 84, n)).all():
                    wrong.append((W, H, D, n))
                done.append(k)

    threads = [threading.Thread(target=work, args=(s,)) for s in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert len(done) == 72 and not wrong
