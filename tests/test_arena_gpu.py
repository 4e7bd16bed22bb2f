"""The context's work arena where the paired lines would need a larger one than
the per-line sweeps: a refusal by the device is met once, calls that the caller
captures allocate nothing, and graphs that the caller captured earlier keep the
arena they use.  Bit-exact against the oracle.

SGM_TEST_ALLOC_LIMIT stands for the device's refusal: host code answers with the
allocation error, nothing is allocated.
"""
import os

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

D = 64


class Call:
    """One asynchronous call on buffers of its own."""

    def __init__(self, c, W, H, post=None, n_paths=8):
        import torch

        self.c, self.W, self.H, self.post, self.n_paths = c, W, H, post, n_paths
        self.rng = np.random.default_rng(W)
        self.left, self.right = (torch.zeros((H, W), dtype=torch.uint8, device="cuda") for _ in range(2))
        self.out = torch.zeros((H, W), dtype=torch.uint8 if post is None else torch.int16, device="cuda")

    def run(self):
        from paper_1610_04121_gb300 import sgm

        a = (self.c.handle, self.left, self.right, self.W, self.H, D, 10, 120, self.n_paths)
        if self.post is None:
            sgm.sgm_compute_async(*a, self.out)
        else:
            sgm.sgm_compute_ex_async(*a, self.post, self.out)

    def check(self, run):
        """`run` on new images gives the oracle's result."""
        import torch

        a, b = (self.rng.integers(0, 256, (self.H, self.W), dtype=np.uint8) for _ in range(2))
        self.left.copy_(torch.from_numpy(a))
        self.right.copy_(torch.from_numpy(b))
        self.out.zero_()
        torch.cuda.synchronize()
        run()
        torch.cuda.synchronize()
        got = self.out.cpu().numpy()
        if self.post is None:
            assert (got == oracle.sgm(a, b, D, 10, 120, self.n_paths)).all()
        else:
            assert (got.view(np.uint16) == oracle.sgm_ex(a, b, D, 10, 120, self.n_paths, self.post)).all()

    def capture(self, stream):
        import torch

        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream):
            self.run()
        return g


@pytest.fixture()
def ctx_on_stream(monkeypatch):
    import torch

    from paper_1610_04121_gb300 import sgm

    made = []

    def make(alloc_limit=None):
        if alloc_limit:
            monkeypatch.setenv("SGM_TEST_ALLOC_LIMIT", str(alloc_limit))
        c, st = sgm.Context(0), torch.cuda.Stream()
        monkeypatch.delenv("SGM_TEST_ALLOC_LIMIT", raising=False)
        sgm.sgm_set_stream(c.handle, st)
        made.append(c)
        return c, st

    yield make
    for c in made:
        c.close()


# per-line arenas of 8 paths with the left-right check: 160x120 9.5 MB, paired 18 MB
def test_a_refusal_by_the_device_is_met_once(ctx_on_stream):
    c, st = ctx_on_stream(12 << 20)
    call = Call(c, 160, 120, post=2)
    call.check(call.run)
    g = call.capture(st)  # allocates and frees nothing
    for _ in range(2):
        call.check(call.run)
        call.check(g.replay)
    small = Call(c, 96, 64, post=7)  # the paired cubes fit the arena as it is
    small.check(small.run)
    call.check(g.replay)
    larger = Call(c, 170, 122, post=2)  # the arena has to grow, and the device refuses the paired cubes again
    larger.check(larger.run)
    gl = larger.capture(st)
    larger.check(gl.replay)


def test_no_allocation_for_the_paired_lines_under_capture(ctx_on_stream):
    c, st = ctx_on_stream()
    plain = Call(c, 200, 150)  # 14 MB
    plain.check(plain.run)
    ex = Call(c, 160, 120, post=2)  # the per-line arena fits, the paired cubes do not
    g = ex.capture(st)
    ex.check(g.replay)
    ex.check(ex.run)  # outside a capture the arena may grow
    ex.check(g.replay)


def test_graphs_of_the_caller_outlive_a_larger_arena(ctx_on_stream):
    c, st = ctx_on_stream()
    plain = Call(c, 200, 150)
    plain.check(plain.run)
    g = plain.capture(st)
    for W, H in ((160, 120), (176, 128), (192, 140)):
        ex = Call(c, W, H, post=2)
        ex.check(ex.run)
        plain.check(g.replay)
        plain.check(plain.run)


def test_an_arena_holds_what_the_per_line_sweeps_would(ctx_on_stream):
    c, st = ctx_on_stream()
    two = Call(c, 200, 150, n_paths=2)  # per-line sweeps 6.2 MB, paired lines 4.2 MB
    two.check(two.run)
    eight = Call(c, 100, 110)  # 5.2 MB
    g = eight.capture(st)
    eight.check(g.replay)
    two.check(two.run)
