"""The walks of 8 paths over a cube larger than L2 (the three directions that go
down, or up, from a column pair in one block): plain, with both passes of the
left-right check and penalties per step, and as replayed graphs of the library
and of the caller; whole frames, bit-exact against the oracle (no tolerance).
"""
import numpy as np
import pytest

import oracle
import stereo_synth as synth

pytestmark = pytest.mark.gpu

# padded W * H * D above 96 MiB: even and odd sizes, a low and a high image (lines that wrap many times)
SHAPES = [(1500, 270, 256), (1501, 263, 256), (261, 1535, 256), (1243, 633, 128)]


@pytest.mark.parametrize("W,H,D", SHAPES)
def test_frames_with_a_cube_larger_than_l2(W, H, D):
    import torch

    from paper_1610_04121_gb300 import sgm

    assert (W + W % 2) * (H + H % 2) * D > 96 << 20
    p = synth.make_pair(synth.PairSpec(W, H, D, 8, 2, D - 8), W)
    left, right = (torch.from_numpy(x).cuda() for x in (p.left, p.right))
    out = torch.zeros((H, W), dtype=torch.uint8, device="cuda")
    out16 = torch.zeros((H, W), dtype=torch.int16, device="cuda")
    ref = oracle.sgm(p.left, p.right, D, 10, 120, 8)
    ref16 = oracle.sgm_ex(p.left, p.right, D, 10, 84, 8, 7)
    st = torch.cuda.Stream()
    with sgm.Context(0) as c:
        sgm.sgm_set_stream(c.handle, st)

        def plain():
            sgm.sgm_compute_async(c.handle, left, right, W, H, D, 10, 120, 8, out)

        def post():
            sgm.sgm_compute_ex_async(c.handle, left, right, W, H, D, 10, 84, 8, 7, out16)

        def check(run, o, want, reps=1):
            o.zero_()
            torch.cuda.synchronize()
            for _ in range(reps):
                run()
            torch.cuda.synchronize()
            assert (o.cpu().numpy().view(want.dtype) == want).all()

        for reps in (1, 1, 1, 4):  # kernel by kernel, making the graph, replaying it, one behind the other
            check(post, out16, ref16, reps)
            check(plain, out, ref, reps)
        for run, o, want in ((post, out16, ref16), (plain, out, ref)):
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=st):
                run()
            check(g.replay, o, want, 3)
