"""The Census and the median kernels at the sizes and addresses where they can
go wrong, bit-exact against the oracle (integer arithmetic: no tolerance):
rows that are whole words or not, images and outputs off a word boundary, tile
edges, images of a few rows, and both tile heights of the Census.
"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sgm():
    from paper_1610_04121_gb300 import sgm as m

    return m


def _at(offset, host):
    """A device copy of `host` that starts `offset` bytes past an allocation."""
    import torch

    buf = torch.empty(host.size + offset, dtype=torch.uint8, device="cuda")
    view = buf[offset:].view(host.shape)
    view.copy_(torch.from_numpy(host))
    return view


@pytest.mark.parametrize("full", [False, True])
@pytest.mark.parametrize("W,H", [(2, 9), (9, 7), (60, 5), (64, 33), (66, 34), (67, 6), (68, 8), (128, 3), (132, 70),
                                 (641, 67), (1244, 66)])
def test_words_and_bytes_match_the_oracle(sgm, W, H, full):
    import torch

    rng = np.random.default_rng(W * 100 + H)
    left, right = (rng.integers(0, 256, (H, W), dtype=np.uint8) for _ in range(2))
    ref = {n: oracle.sgm(left, right, 32, 7, 84, n, census="ct62" if full else "csct") for n in (2, 4)}
    ref_ex = None if full else oracle.sgm_ex(left, right, 32, 7, 84, 4, 7)
    with sgm.Context(0, flags=sgm.SGM_FLAG_CENSUS_FULL if full else 0) as c:
        sgm.sgm_set_schedule(c.handle, sgm.SGM_SCHED_PAIRS)
        for li, ri, oi in ((0, 0, 0), (0, 1, 0), (4, 2, 2), (3, 0, 1)):
            dl, dr, out = _at(li, left), _at(ri, right), _at(oi, np.zeros_like(left))
            for n in (2, 4):
                out.zero_()
                sgm.sgm_compute_async(c.handle, dl, dr, W, H, 32, 7, 84, n, out)
                torch.cuda.synchronize()
                assert (out.cpu().numpy() == ref[n]).all(), (li, ri, oi, n)
            if ref_ex is not None:
                got = c.compute_ex(dl, dr, 32, 7, 84, 4, 7)
                assert (got.cpu().numpy().view(np.uint16) == ref_ex).all(), (li, ri)
