"""Pairs of a batch that run alone, one after the other, work in one region of the
arena; bit-exact against the oracle, with device, pinned and pageable buffers.
"""
import numpy as np
import pytest

import oracle
import stereo_synth as synth

pytestmark = pytest.mark.gpu

# 2^28 path steps make a pair run alone; the last two go through the lists
SHAPES = [(760, 560, 128, 8), (601, 450, 256, 4), (762, 558, 128, 8), (600, 452, 256, 4), (77, 45, 128, 8), (64, 40, 256, 4)]
CUBES = 760 * 560 * 128 * 7  # bytes of the largest pair's cubes


@pytest.fixture(scope="module")
def pairs():
    ps = [synth.make_pair(synth.PairSpec(W, H, D, 4, 2, 48), 40 + i) for i, (W, H, D, _) in enumerate(SHAPES)]
    refs = [oracle.sgm(p.left, p.right, D, 7, 84, n) for p, (_, _, D, n) in zip(ps, SHAPES)]
    return ps, refs


@pytest.mark.parametrize("kind", ["device", "pinned", "pageable"])
def test_pairs_that_run_alone_share_a_region(pairs, kind):
    import torch

    from paper_1610_04121_gb300 import sgm

    ps, refs = pairs
    place = {"device": lambda t: t.cuda(), "pinned": lambda t: t.pin_memory(), "pageable": lambda t: t}[kind]
    bufs = [[place(torch.from_numpy(x.copy())) for x in (p.left, p.right, np.full_like(p.left, 255))] for p in ps]
    with sgm.Context(0) as c:
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        for _ in range(2):
            for b in bufs:
                b[2].fill_(255)
            torch.cuda.synchronize()
            sgm.sgm_compute_batch(c.handle, [(*b, W, H, D, 7, 84, n) for b, (W, H, D, n) in zip(bufs, SHAPES)])
            for b, ref in zip(bufs, refs):
                assert (b[2].cpu().numpy() == ref).all()
        held = before - torch.cuda.mem_get_info()[0]
        assert held < 1.5 * CUBES, (held, CUBES)


def test_served_pairs_that_run_alone(pairs):
    from paper_1610_04121_gb300 import sgm

    ps, refs = pairs
    with sgm.Context(0) as c:
        jobs = []
        for _ in range(2):
            for p, (W, H, D, n) in zip(ps, SHAPES):
                out = np.full((H, W), 255, np.uint8)
                jobs.append((out, sgm.sgm_submit(c.handle, p.left, p.right, W, H, D, 7, 84, n, out)))
        for k, (out, t) in enumerate(jobs):
            assert sgm.sgm_poll(c.handle, t, -1) == sgm.SGM_OK
            assert (out == refs[k % len(refs)]).all()
