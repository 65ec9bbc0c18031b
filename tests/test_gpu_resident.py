"""The resident kernel (small problems, 8 iterations or more on the GRAPH and PERSISTENT paths): iterates and receive slots equal the
oracle's and the other kernels', over box cuts and block splits of every kind, call lengths of both parities, batches, frozen grids."""
import numpy as np
import pytest

import jacobi_inputs as J
import oracle

pytestmark = pytest.mark.gpu

# one box; thin and one-point extents; ragged rows; cuts in every axis; more blocks than boxes; largest extents that fit
SHAPES = [((5, 4, 3), ("count", (1, 1, 1))), ((1, 1, 40), ("count", (1, 1, 4))), ((130, 1, 9), ("shape", (50, 1, 9))),
          ((33, 17, 29), ("count", (3, 2, 4))), ((64, 64, 64), ("count", (2, 2, 2))), ((61, 47, 50), ("shape", (7, 5, 6))),
          ((700, 6, 11), ("shape", (64, 64, 64))), ((96, 40, 77), ("shape", (32, 32, 32)))]


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("path", ["graph", "persistent"])
@pytest.mark.parametrize("grid,split", SHAPES)
def test_resident_iterates_and_slots(grid, split, path, dtype):
    import paper_2102_12416_gb300 as jg
    init = dict(bc="uniform", bc_seed=31, interior="uniform", interior_seed=32)
    u = J.initial_grid(*grid, dtype=jg.NP_DTYPES[jg.DTYPES[dtype]], **init)
    with jg.Jacobi3D(grid, split, dtype, init, path=path) as s, jg.Jacobi3D(grid, split, dtype, init, path="fused") as f:
        done = 0
        for n in (8, 9, 1, 33):  # resident launches from both parities, with other kernels between
            s.step(n)
            f.step(n)
            done += n
            s.sync()
            assert np.array_equal(s.copy_out(padded=True), f.copy_out(padded=True))
            for b in {0, s.info.n_blocks // 2, s.info.n_blocks - 1}:
                for face in range(6):
                    assert np.array_equal(s.read_face(b, face), f.read_face(b, face))
        assert np.array_equal(s.copy_out(), J.interior_of(oracle.jacobi(u, done)))
        assert s.residual() == f.residual()


def test_resident_negative_and_replaced_state():
    import paper_2102_12416_gb300 as jg
    grid = (40, 30, 20)
    u = J.initial_grid(*grid, bc="uniform", bc_seed=5, interior="uniform", interior_seed=6)
    with jg.Jacobi3D(grid, ("shape", (16, 16, 16)), "f64", path="graph") as s:
        for state in (u - 0.5, u):  # the first keeps the FP64 pipe
            s.set_state(state)
            s.step(17)
            assert np.array_equal(s.copy_out(), J.interior_of(oracle.jacobi(state, 17)))


@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_resident_batch_solve_freezes_grids(dtype, monkeypatch):
    """Grids of a batch converge one after another: the boxes are cut anew for those that run on; results are those of the per-step
    kernels."""
    import paper_2102_12416_gb300 as jg
    grids = [(12, 9, 10), (30, 21, 17), (8, 40, 6), (33, 32, 31)]
    splits = [("shape", (16, 16, 16))] * 4
    inits = [dict(bc="linear_noise", bc_seed=g, noise_amp=1e-3, interior="zero") for g in range(4)]
    got = []
    for on in ("1", "0"):
        monkeypatch.setenv("JACOBI_RESIDENT", on)
        with jg.Jacobi3D(grids, splits, dtype, inits, path="graph") as s:
            res = s.solve(1e-4, 5000, 25)
            s.step(12)
            got.append((res, [s.copy_out(g) for g in range(4)]))
    assert got[0][0] == got[1][0] and len(set(got[0][0][0])) > 1
    assert all(np.array_equal(a, b) for a, b in zip(got[0][1], got[1][1]))


def test_resident_on_two_streams_and_long_calls():
    """Two handles whose resident launches overlap on the GPU, each in more than one launch per call (16384 iterations at most)."""
    import torch

    import paper_2102_12416_gb300 as jg
    grid, n = (20, 17, 19), 20011
    u = [J.initial_grid(*grid, bc="uniform", bc_seed=q, interior="uniform", interior_seed=q + 9, dtype=np.float32) for q in (1, 2)]
    streams = [torch.cuda.Stream() for _ in u]
    hs = [jg.Jacobi3D(grid, ("shape", (8, 8, 8)), "f32", path="graph", stream=s) for s in streams]
    for h, x in zip(hs, u):
        h.set_state(x)
    for h in hs:
        h.step(n)
    for h, x in zip(hs, u):
        h.sync()
        assert np.array_equal(h.copy_out(), J.interior_of(oracle.jacobi(x, n)))
        h.close()
