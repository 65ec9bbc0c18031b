"""FP64 states that mix zeros, subnormals below 2^-1042 and ordinary values in every neighbour position: sums whose operands are out of
the short integer adder's reach.  Resident iterates equal the FUSED path's and the oracle's bit for bit, the allocation-free residual
keeps the residual bar."""
import numpy as np
import pytest
import torch

import jacobi_inputs as J
import oracle
from test_gpu_residual_values import TOL, _norms

pytestmark = pytest.mark.gpu

HIGH = [1.0, 2.0 ** -15, 2.0 ** -20, 1e100]


def _state(grid, high, seed):
    r = np.random.RandomState(seed)
    u = r.choice([0.0, 0.0, 5e-324, 2.0 ** -1043, 2.1e-314, 2.0 ** -1022, high], size=tuple(n + 2 for n in grid[::-1]))
    return u * np.where(u == high, r.uniform(0.5, 1.0, u.shape), 1.0)


@pytest.mark.parametrize("high", HIGH)
@pytest.mark.parametrize("grid", [(40, 30, 20), (33, 7, 9)])
def test_resident_far_operands(grid, high):
    import paper_2102_12416_gb300 as jg
    split = ("shape", (16, 16, 16))
    for seed in (1, 2):
        u = _state(grid, high, seed)
        with jg.Jacobi3D(grid, split, "f64", path="graph") as s, jg.Jacobi3D(grid, split, "f64", path="fused") as f:
            for h in (s, f):
                h.set_state(u)
                h.step(8)
            got = s.copy_out()
            assert np.array_equal(got, f.copy_out())
        assert np.array_equal(got, J.interior_of(oracle.jacobi(u, 8)))


@pytest.mark.parametrize("high", HIGH)
@pytest.mark.parametrize("grid", [(1, 1, 1), (33, 17, 5), (64, 3, 40)])
def test_noalloc_far_operands(grid, high):
    import paper_2102_12416_gb300 as jg
    out = torch.zeros(3, dtype=torch.float64, device="cuda")
    for seed in (1, 2, 3):
        u = _state(grid, high, seed)
        u[1:-1, 1:-1, 1:-1] *= np.random.RandomState(seed).uniform(size=grid[::-1]) < 0.5  # neighbour sums that stand alone
        r, b = _norms(u)
        d = torch.from_numpy(u).cuda()
        jg.jacobi_residual_noalloc(d.data_ptr(), grid, "f64", out.data_ptr())
        got = out.cpu().numpy()
        assert abs(got[0] - r) <= TOL * r and abs(got[1] - b) <= TOL * b
