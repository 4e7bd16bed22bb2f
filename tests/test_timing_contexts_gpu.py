"""Contexts created with SGM_FLAG_STAGE_TIMING: the post form is never timed, so
it runs the same kernels there as in any other context.  Bit-exact against the
oracle.
"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_paths", [2, 4, 8])
def test_post_form_of_timing_contexts(n_paths):
    from paper_1610_04121_gb300 import sgm

    rng = np.random.default_rng(n_paths)
    left, right = (rng.integers(0, 256, (45, 77), dtype=np.uint8) for _ in range(2))
    launches = []
    for flags in (0, sgm.SGM_FLAG_STAGE_TIMING):
        with sgm.Context(0, flags=flags) as c:
            for _ in range(3):
                before = c.launches
                got = c.compute_ex(left, right, 64, 7, 84, n_paths, 7)
                launches.append(c.launches - before)
                assert (got == oracle.sgm_ex(left, right, 64, 7, 84, n_paths, 7)).all()
            assert (c.compute(left, right, 64, 7, 84, n_paths) == oracle.sgm(left, right, 64, 7, 84, n_paths)).all()
    assert len(set(launches)) == 1, launches
