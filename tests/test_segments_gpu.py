"""The paired lines with each length of a segment (2, 4 and 8 quads of columns;
2 and 4 for D > 128), which follows from the frame's size: frames on both sides
of the two bounds, last segments of every remainder, odd sizes, one segment per
row pair; bit-exact against the oracle (integer arithmetic: no tolerance).
"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def _quads(W, H, D):
    """Quads of a segment by the rule of the library."""
    q = 8 if D <= 128 else 4
    while q > 2 and -(-H // 2) * -(-(-(-W // 2)) // q) <= 1216:
        q //= 2
    return q


# W, H: 2432 rows make 1216 row pairs
SHAPES = [(8, 2432), (7, 2433), (16, 1216), (17, 1216), (15, 1217), (33, 203), (34, 487), (19, 609), (37, 700), (41, 601),
          (16, 2432), (17, 1217), (21, 1300), (33, 1000), (50, 701), (300, 129), (643, 67), (40, 100), (23, 99)]


def test_the_shapes_cover_every_length():
    for most, Ds in ((8, (32, 96, 128)), (4, (160, 256))):
        for D in Ds:
            assert {_quads(W, H, D) for W, H in SHAPES} == {2, 4, most}


@pytest.mark.parametrize("W,H", SHAPES)
@pytest.mark.parametrize("D", [32, 96, 128, 160])
def test_frames_around_the_bounds(W, H, D):
    from paper_1610_04121_gb300 import sgm

    rng = np.random.default_rng(W * 1000 + H + D)
    left, right = (rng.integers(0, 256, (H, W), dtype=np.uint8) for _ in range(2))
    with sgm.Context(0) as c:
        sgm.sgm_set_schedule(c.handle, sgm.SGM_SCHED_PAIRS)
        for n_paths, P2 in ((2, 84), (4, 84), (8, 120)):
            ref = oracle.sgm(left, right, D, 7, P2, n_paths)
            assert (c.compute(left, right, D, 7, P2, n_paths) == ref).all(), n_paths
        assert (c.compute_ex(left, right, D, 7, 84, 4, 7) == oracle.sgm_ex(left, right, D, 7, 84, 4, 7)).all()
