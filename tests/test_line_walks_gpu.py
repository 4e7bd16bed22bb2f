"""The paired-line walks of 2, 4 and 8 paths at the sizes where they can go
wrong, bit-exact against the oracle (integer arithmetic: no tolerance).

Widths around a segment (16 columns, 8 for D > 128) and far below the height
(a diagonal line wraps around the image many times and starts a path at every
wrap), odd sizes (padding row and column), one-quad rows, and the three ways
stored costs add in a byte (P2 up to 85, up to 127, above).
"""
import numpy as np
import pytest

import oracle
import stereo_synth as synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sgm():
    from paper_1610_04121_gb300 import sgm as m

    return m


@pytest.fixture(scope="module")
def ctx(sgm):
    with sgm.Context(0) as c:
        sgm.sgm_set_schedule(c.handle, sgm.SGM_SCHED_PAIRS)
        yield c


def _images(W, H):
    rng = np.random.default_rng(W * 1000 + H)
    return (rng.integers(0, 256, (H, W), dtype=np.uint8) for _ in range(2))


@pytest.mark.parametrize("W,H", [(2, 97), (3, 64), (5, 200), (15, 31), (16, 16), (17, 40), (18, 90), (33, 70), (48, 5),
                                 (98, 33), (130, 2)])
@pytest.mark.parametrize("D,P2", [(32, 84), (96, 120), (128, 85), (128, 127), (160, 84), (256, 120), (64, 200)])
def test_walks_match_the_oracle(ctx, W, H, D, P2):
    left, right = _images(W, H)
    for n_paths in (2, 4, 8):
        ref = oracle.sgm(left, right, D, 7, P2, n_paths, debug=True)
        got = ctx.debug(left, right, D, 7, P2, n_paths)
        assert (got["S"].astype(np.int32) == ref["S"]).all(), n_paths
        assert (got["raw"] == ref["raw"]).all() and (got["disp"] == ref["disp"]).all(), n_paths
        assert (ctx.compute(left, right, D, 7, P2, n_paths) == ref["disp"]).all(), n_paths


@pytest.mark.parametrize("W,H", [(5, 60), (17, 40), (40, 17), (67, 35)])
@pytest.mark.parametrize("D,P1,P2", [(64, 7, 84), (128, 10, 120), (160, 50, 20)])
def test_post_form_of_the_walks(ctx, W, H, D, P1, P2):
    left, right = _images(W, H)
    for n_paths in (2, 4, 8):
        for post in (1, 4, 7):
            assert (ctx.compute_ex(left, right, D, P1, P2, n_paths, post)
                    == oracle.sgm_ex(left, right, D, P1, P2, n_paths, post)).all(), (n_paths, post)


def test_per_line_sweeps_where_memory_is_short(sgm):
    # 8 paths hold 7 bytes per pixel and disparity in the paired schedule: a cap
    # below that and above the per-line sweeps' need gives the same result
    pair = synth.make_pair(synth.PairSpec(160, 120, 64, 4, 2, 40), 3)
    per_line = 160 * 120 * (7 * 64 + 13) + (1 << 20)
    for n_paths, cap in ((8, 0), (8, per_line), (2, 0)):
        with sgm.Context(0, mem_cap_bytes=cap) as c:
            out = c.compute(pair.left, pair.right, 64, 10, 120, n_paths)
            assert (out == oracle.sgm(pair.left, pair.right, 64, 10, 120, n_paths)).all()
    with sgm.Context(0, mem_cap_bytes=1 << 20) as c:
        with pytest.raises(sgm.SgmError) as e:
            c.compute(pair.left, pair.right, 64, 10, 120, 8)
        assert e.value.code == sgm.SGM_ENOMEM


def test_stage_timing_contexts_time_the_per_line_sweeps(sgm):
    import torch

    pair = synth.make_pair(synth.PairSpec(96, 64, 64, 4, 2, 40), 4)
    left, right = (torch.from_numpy(x).cuda() for x in (pair.left, pair.right))
    out = torch.empty_like(left)
    with sgm.Context(0, flags=sgm.SGM_FLAG_STAGE_TIMING) as c:
        for n_paths, stages in ((2, 5), (8, 7)):
            sgm.sgm_compute_async(c.handle, left, right, 96, 64, 64, 10, 120, n_paths, out)
            assert len(sgm.sgm_stage_times(c.handle)) == stages
            assert (out.cpu().numpy() == oracle.sgm(pair.left, pair.right, 64, 10, 120, n_paths)).all()
