"""State transfer kernels: install a padded array, read it back, |b| and the domain flag, over the block shapes where the row
walk can go wrong (one-point extents, rows narrower or wider than a warp, partial edge blocks, split blocks)."""
import numpy as np
import pytest

import jacobi_inputs as J
import oracle

pytestmark = pytest.mark.gpu

SHAPES = [((1, 1, 1), ("count", (1, 1, 1))), ((1, 5, 7), ("count", (1, 2, 1))), ((3, 2, 9), ("shape", (2, 2, 4))),
          ((31, 6, 5), ("count", (1, 1, 1))), ((33, 65, 34), ("shape", (32, 32, 32))), ((67, 9, 40), ("count", (2, 1, 3))),
          ((130, 4, 70), ("count", (1, 1, 1))), ((1040, 9, 3), ("count", (1, 1, 1)))]


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("grid,split", SHAPES)
@pytest.mark.parametrize("before", [0, 1])
def test_set_state_copy_out_residual(grid, split, dtype, before):
    import paper_2102_12416_gb300 as jg
    u = J.initial_grid(*grid, bc="uniform", bc_seed=11, interior="uniform", interior_seed=12, dtype=jg.NP_DTYPES[jg.DTYPES[dtype]])
    with jg.Jacobi3D([grid, (7, 6, 5)], [split, ("count", (1, 1, 1))], dtype, [dict(bc="linear"), dict(bc="uniform", bc_seed=3)]) as s:
        s.step(before)  # the state goes to the buffers of either parity
        other = s.copy_out(1, padded=True)
        s.set_state(u, 0)
        back = s.copy_out(0, padded=True)
        face = J.boundary_mask(*grid)
        two = np.zeros(u.shape, int)  # edges and corners lie on two or three boundary planes and come back as 0
        for ax in range(3):
            sl = [slice(None)] * 3
            for end in (0, -1):
                sl[ax] = end
                two[tuple(sl)] += 1
        assert np.array_equal(back, np.where(two > 1, 0, u)) and face.any()
        assert np.array_equal(s.copy_out(0), J.interior_of(u))
        assert np.array_equal(s.copy_out(1, padded=True), other)
        r, b, _ = oracle.residual(u)
        rel, res = s.residual()
        assert abs(res[0] - r) <= 1e-12 * r and abs(rel[0] - r / b) <= 1e-12 * (r / b)
        s.step(3)
        assert np.array_equal(s.copy_out(0), J.interior_of(oracle.jacobi(u, 3)))


@pytest.mark.parametrize("where", [(0, 4, 5), (3, 4, 0), (2, 5, 6), (4, 8, 3)])
def test_negative_value_keeps_the_fp64_pipe_until_replaced(where):
    """A value outside the integer adder's domain, in the interior or on any face, is seen wherever it stands; the next state clears
    the flag again (FP64 iterates stay the oracle's either way)."""
    import paper_2102_12416_gb300 as jg
    grid = (9, 7, 8)
    u = J.initial_grid(*grid, bc="uniform", bc_seed=5, interior="uniform", interior_seed=6)
    bad = u.copy()
    bad[where] = -2.5
    with jg.Jacobi3D(grid, ("shape", (4, 4, 4)), "f64") as s:
        for state in (bad, u, bad):
            s.set_state(state)
            s.step(5)
            assert np.array_equal(s.copy_out(), J.interior_of(oracle.jacobi(state, 5)))
