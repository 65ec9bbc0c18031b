"""Failures of the resident kernel: a wait that runs out (a box that sends nothing, made by the host) is reported by the next call that
waits for the handle, the handle works again afterwards, a refused launch falls back, and a late start is no failure."""
import numpy as np
import pytest

import jacobi_inputs as J
import oracle

pytestmark = pytest.mark.gpu

GRID, SPLIT = (45, 37, 29), ("shape", (16, 16, 16))
INIT = dict(bc="uniform", bc_seed=3, interior="uniform", interior_seed=4)

CALLS = {"sync": lambda s: s.sync(), "residual": lambda s: s.residual(), "copy_out": lambda s: s.copy_out(),
         "read_face": lambda s: s.read_face(0, 1), "step_timed": lambda s: s.step_timed(0), "solve": lambda s: s.solve(1e-3, 100, 50)}


@pytest.mark.parametrize("call", list(CALLS))
@pytest.mark.parametrize("path,dtype", [("graph", "f64"), ("persistent", "f32")])
def test_expired_wait_is_reported(path, dtype, call, monkeypatch):
    import paper_2102_12416_gb300 as jg
    monkeypatch.setenv("JACOBI_WAIT_MS", "100")
    u = J.initial_grid(*GRID, dtype=jg.NP_DTYPES[jg.DTYPES[dtype]], **INIT)
    with jg.Jacobi3D(GRID, SPLIT, dtype, INIT, path=path) as s:
        jg.jacobi_debug_resident(s.h, 5)
        s.step(20)
        assert s.info.resident_launches == 1
        with pytest.raises(jg.JacobiError) as e:
            CALLS[call](s)
        assert e.value.code == jg.JACOBI_ETIMEDOUT
        jg.jacobi_debug_resident(s.h, -1)
        s.sync()  # reported once
        for n in (20, 33):  # the same handle, from a new state
            s.set_state(u)
            s.step(n)
            assert np.array_equal(s.copy_out(), J.interior_of(oracle.jacobi(u, n)))
        assert s.info.resident_launches >= 3
        s.sync()


@pytest.mark.parametrize("path", ["graph", "persistent"])
def test_refused_launch_falls_back(path):
    import paper_2102_12416_gb300 as jg
    u = J.initial_grid(*GRID, **INIT)
    with jg.Jacobi3D(GRID, SPLIT, "f64", INIT, path=path) as s:
        jg.jacobi_debug_resident(s.h, -2)
        s.step(20)
        s.step(21)
        assert s.info.resident_launches == 0 and s.info.iteration == 41
        assert np.array_equal(s.copy_out(), J.interior_of(oracle.jacobi(u, 41)))
        s.sync()


def test_late_start_is_no_failure(monkeypatch):
    """Another stream's kernel holds an SM for longer than the wait limit while the launch, which wants all of them, is there."""
    import torch

    import paper_2102_12416_gb300 as jg
    monkeypatch.setenv("JACOBI_WAIT_MS", "20")
    grid, init = (128, 128, 128), dict(bc="uniform", bc_seed=3, interior="zero")
    u = J.initial_grid(*grid, dtype=np.float32, **init)
    other = torch.cuda.Stream()
    with jg.Jacobi3D(grid, ("shape", (32, 32, 32)), "f32", init, path="graph") as s:
        s.step(20)
        s.sync()
        with torch.cuda.stream(other):
            torch.cuda._sleep(300_000_000)  # cycles: about 150 ms
        s.step(20)
        s.sync()
        assert s.info.resident_launches == 2
        assert np.array_equal(s.copy_out(), J.interior_of(oracle.jacobi(u, 40)))
    torch.cuda.synchronize()
