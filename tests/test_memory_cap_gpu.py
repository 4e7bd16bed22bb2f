"""Under a memory cap a call leaves as much room for served requests as the
per-line sweeps would: the paired lines, which hold up to twice as much, are
taken only where they need no more.  Results bit-exact against the oracle.
"""
import numpy as np
import pytest

import oracle
import stereo_synth as synth

pytestmark = pytest.mark.gpu

W, H, D = 160, 120, 64
WH, STATE = W * H, 3 * W * 64 * 4 * 4  # pixels, the per-line path states of 8 paths in bytes
SINGLE_EX = WH * (7 * D + 20) + STATE + 4096   # per-line arena of sgm_compute_ex with 8 paths
SINGLE = WH * (7 * D + 12) + STATE + 4096      # of sgm_compute
BATCHED = WH * (4 * D + 12) + STATE + 4096     # per-line region of a batched or served pair


def _served(sgm, c, p, n_paths):
    out = np.zeros((H, W), np.uint8)
    t = sgm.sgm_submit(c.handle, p.left, p.right, W, H, D, 10, 120, n_paths, out)
    assert sgm.sgm_poll(c.handle, t, -1) == sgm.SGM_OK
    assert (out == oracle.sgm(p.left, p.right, D, 10, 120, n_paths)).all()


# "ex": two passes' paired cubes (14 D bytes a pixel) fit the cap too, but not beside a served pair
@pytest.mark.parametrize("call,cap", [("ex", 20 << 20), ("plain", SINGLE + BATCHED), ("batch", 2 * BATCHED)])
def test_a_call_leaves_the_room_that_served_pairs_had(call, cap):
    from paper_1610_04121_gb300 import sgm

    p = synth.make_pair(synth.PairSpec(W, H, D, 4, 2, 40), 11)
    assert SINGLE_EX + BATCHED <= 20 << 20 < 14 * WH * D + BATCHED
    with sgm.Context(0, mem_cap_bytes=cap) as c:
        for _ in range(2):
            if call == "ex":
                got = c.compute_ex(p.left, p.right, D, 10, 120, 8, 2)
                assert (got == oracle.sgm_ex(p.left, p.right, D, 10, 120, 8, 2)).all()
            elif call == "plain":
                assert (c.compute(p.left, p.right, D, 10, 120, 8) == oracle.sgm(p.left, p.right, D, 10, 120, 8)).all()
            else:
                out = np.zeros((H, W), np.uint8)
                sgm.sgm_compute_batch(c.handle, [(p.left, p.right, out, W, H, D, 10, 120, 8)])
                assert (out == oracle.sgm(p.left, p.right, D, 10, 120, 8)).all()
        _served(sgm, c, p, 8)
        _served(sgm, c, p, 4)


@pytest.mark.parametrize("n_paths", [2, 4, 8])
def test_capped_results(n_paths):
    from paper_1610_04121_gb300 import sgm

    p = synth.make_pair(synth.PairSpec(W, H, D, 4, 2, 40), 12)
    for cap in (SINGLE_EX + (1 << 16), 4 * SINGLE_EX):
        with sgm.Context(0, mem_cap_bytes=cap) as c:
            assert (c.compute(p.left, p.right, D, 10, 120, n_paths)
                    == oracle.sgm(p.left, p.right, D, 10, 120, n_paths)).all()
            for post in (1, 7):
                assert (c.compute_ex(p.left, p.right, D, 10, 120, n_paths, post)
                        == oracle.sgm_ex(p.left, p.right, D, 10, 120, n_paths, post)).all()
