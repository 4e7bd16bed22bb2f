"""Batched and served pairs on the paired-line lists, bit-exact against the
oracle: groups large enough for them, pairs that run alone in front of the
lists, and caps that leave room for the per-line sweeps only."""
import numpy as np
import pytest

import oracle
import stereo_synth as synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sgm():
    from paper_1610_04121_gb300 import sgm as m

    return m


def _items(shapes, seed):
    out = []
    for i, (W, H, D, n_paths, P2) in enumerate(shapes):
        p = synth.make_pair(synth.PairSpec(W, H, D, 4, 2, min(48, D - 1)), seed + i)
        out.append((p, np.full((H, W), 255, np.uint8), W, H, D, P2, n_paths))
    return out


def _check(items):
    for p, o, W, H, D, P2, n_paths in items:
        assert (o == oracle.sgm(p.left, p.right, D, 7, P2, n_paths)).all(), (W, H, D, P2, n_paths)


# pairs alike together pass 2^18 pixels for 2 and 4 paths; odd sizes, one segment, every class of sums
SHAPES = ([(401, 333, 64, 4, 84), (400, 330, 64, 4, 84), (15, 700, 64, 4, 84), (330, 401, 64, 4, 84)]
          + [(399, 333, 96, 4, 120), (390, 360, 96, 4, 120)] + [(380, 360, 32, 2, 84), (381, 351, 32, 2, 200)]
          + [(390, 350, 32, 4, 200), (391, 351, 32, 4, 200)]
          + [(77, 45, 128, 8, 84), (65, 90, 128, 8, 84), (80, 31, 160, 8, 120), (33, 64, 256, 8, 200), (14, 20, 64, 8, 84)])


def test_paired_lists_match_the_oracle(sgm):
    items = _items(SHAPES, 7000)
    with sgm.Context(0) as c:
        for _ in range(2):  # tuned, then replayed
            for it in items:
                it[1].fill(255)
            sgm.sgm_compute_batch(c.handle, [(p.left, p.right, o, W, H, D, 7, P2, n) for p, o, W, H, D, P2, n in items])
            _check(items)


def test_pairs_that_run_alone_beside_lists(sgm):
    # 760x560 D=128 with 8 paths passes 2^28 path steps
    items = _items([(760, 560, 128, 8, 120), (90, 60, 128, 8, 120), (761, 561, 256, 4, 84), (60, 40, 32, 2, 84)], 7100)
    with sgm.Context(0) as c:
        sgm.sgm_compute_batch(c.handle, [(p.left, p.right, o, W, H, D, 7, P2, n) for p, o, W, H, D, P2, n in items])
        _check(items)
        only = items[:1]  # a wave without lists
        only[0][1].fill(255)
        sgm.sgm_compute_batch(c.handle, [(p.left, p.right, o, W, H, D, 7, P2, n) for p, o, W, H, D, P2, n in only])
        _check(only)


def test_served_pairs_with_and_without_room(sgm):
    items = _items([(200, 180, 64, 4, 84), (77, 45, 64, 8, 120), (210, 170, 64, 4, 84), (96, 64, 128, 8, 84)] * 3, 7200)
    for cap in (0, 14 << 20):  # the cap holds 200x180 D=64 in per-line records, not every pair's paired cubes
        with sgm.Context(0, mem_cap_bytes=cap) as c:
            ts = []
            for p, o, W, H, D, P2, n in items:
                o.fill(255)
                ts.append(sgm.sgm_submit(c.handle, p.left, p.right, W, H, D, 7, P2, n, o))
            for t in ts:
                assert sgm.sgm_poll(c.handle, t, -1) == sgm.SGM_OK
        _check(items)
