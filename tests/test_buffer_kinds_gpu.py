"""Blocking calls on host buffers that change their kind between calls: pageable
memory that the caller registers (page-locks), and the way back; bit-exact
against the oracle (no tolerance).  The graph made while a buffer was of one
kind must not serve it as the other.
"""
import mmap

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

W, H, D = 70, 34, 64


class Buffers:
    """left, right and out on pages of their own, pageable or registered."""

    def __init__(self, out_type):
        self.maps = [mmap.mmap(-1, 4 * mmap.PAGESIZE) for _ in range(3)]
        self.left, self.right, self.out = (np.frombuffer(m, t, W * H).reshape(H, W)
                                           for m, t in zip(self.maps, (np.uint8, np.uint8, out_type)))
        self.pinned = [False] * 3

    def pin(self, on):
        import torch

        rt = torch.cuda.cudart()
        for i, a in enumerate((self.left, self.right, self.out)):
            if self.pinned[i] != on[i]:
                rc = (rt.cudaHostRegister(a.ctypes.data, 4 * mmap.PAGESIZE, 0) if on[i]
                      else rt.cudaHostUnregister(a.ctypes.data))
                assert int(rc) == 0
                self.pinned[i] = on[i]


def _run(calls, post):
    from paper_1610_04121_gb300 import sgm

    rng = np.random.default_rng(5)
    b = Buffers(np.uint8 if post is None else np.uint16)
    with sgm.Context(0) as c:
        try:
            for k, on in enumerate(calls):
                b.pin(on)
                b.left[:], b.right[:] = (rng.integers(0, 256, (H, W), dtype=np.uint8) for _ in range(2))
                b.out[:] = 7
                if post is None:
                    sgm.sgm_compute(c.handle, b.left, b.right, W, H, D, 7, 84, 4, b.out)
                    ref = oracle.sgm(b.left, b.right, D, 7, 84, 4)
                else:
                    sgm.sgm_compute_ex(c.handle, b.left, b.right, W, H, D, 7, 84, 4, post, b.out)
                    ref = oracle.sgm_ex(b.left, b.right, D, 7, 84, 4, post)
                assert (b.out == ref).all(), (k, on)
        finally:
            b.pin([False] * 3)


ALL, NONE = (True,) * 3, (False,) * 3


@pytest.mark.parametrize("post", [None, 7])
@pytest.mark.parametrize("which", [ALL, (True, False, False), (False, True, False), (False, False, True)])
def test_pageable_buffers_registered_between_calls(which, post):
    _run([NONE] * 3 + [which] * 3, post)


@pytest.mark.parametrize("post", [None, 7])
def test_registered_buffers_unregistered_between_calls(post):
    _run([ALL] * 3 + [NONE] * 3 + [ALL] + [(False, True, False)] * 3, post)
