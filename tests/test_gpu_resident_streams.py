"""Steps of several handles on several streams: resident launches that do not fit side by side take turns, so many small grids that step
at the same time are left to the other kernels, which share the GPU; results are the same either way."""
import numpy as np
import pytest
import torch

import jacobi_inputs as J
import oracle

pytestmark = pytest.mark.gpu

INIT = dict(bc="uniform", bc_seed=3, interior="uniform", interior_seed=4)
N = 4000  # iterations of a call: under way for some 10 ms, noted for twice that


class Handles:
    """Handles on streams of their own; step(q) tells whether the call was resident."""

    def __init__(self, *specs):
        import paper_2102_12416_gb300 as jg
        self.h = []
        for size, dtype, path in specs:
            s = jg.Jacobi3D((size,) * 3, ("shape", (32, 32, 32)), dtype, INIT, path=path, stream=torch.cuda.Stream())
            s.done, s.path = 0, path
            self.h.append(s)
        for s in self.h:  # loads the kernels of both kinds: loading one may wait for those that run
            for what in (-2, -1):  # resident launches refused, then taken
                jg.jacobi_debug_resident(s.h, what)
                s.set_path("fused")  # (forgets the refusal)
                s.set_path(s.path)
                s.step(100)
                s.done += 100
                s.sync()

    def step(self, q, n=N):
        s = self.h[q]
        before = s.info.resident_launches
        s.step(n)
        s.done += n
        return s.info.resident_launches > before

    def check(self):
        for s in self.h:
            s.sync()
            u = J.initial_grid(*s.grids[0], dtype=s.np_dtype, **INIT)
            if s.done * u.size < 2e9:
                assert np.array_equal(s.copy_out(), J.interior_of(oracle.jacobi(u, s.done)))
            s.close()


def test_two_small_grids_take_turns_and_more_share():
    w = Handles(*[(32, "f32", "graph")] * 6)
    taken = [w.step(q) for q in range(6)]
    assert taken[:2] == [True, True] and not any(taken[4:]), taken
    for s in w.h:
        s.sync()
    assert w.step(0)  # waited for: alone again
    w.check()


@pytest.mark.parametrize("wait", [lambda s: s.sync(), lambda s: s.residual(), lambda s: s.copy_out()])
def test_larger_grids_share_at_once(wait):
    w = Handles((64, "f64", "graph"), (64, "f64", "graph"))
    assert w.step(0) and not w.step(1)
    wait(w.h[0])
    wait(w.h[1])
    assert w.step(1)
    w.check()


def test_short_steps_beside_a_long_one_take_turns():
    w = Handles((64, "f64", "graph"), (64, "f64", "graph"))
    assert w.step(0, 5 * N) and w.step(1, N // 10) and w.step(1, N // 10)
    w.check()


def test_one_box_grids_run_side_by_side():
    w = Handles(*[(8, "f32", "graph")] * 8)
    assert all(w.step(q) for q in range(8))
    w.check()


def test_one_stream_and_closed_handles():
    """Steps of one stream follow each other: all resident; a closed handle has none under way."""
    import paper_2102_12416_gb300 as jg
    st = torch.cuda.Stream()
    hs = [jg.Jacobi3D((64, 64, 64), ("shape", (32, 32, 32)), "f64", INIT, path="graph", stream=st) for _ in range(4)]
    for s in hs:
        s.step(N)
    assert all(s.info.resident_launches > 0 for s in hs)
    for s in hs:
        s.close()
    w = Handles((64, "f64", "graph"))
    assert w.step(0)
    w.check()
