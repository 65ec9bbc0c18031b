"""FP64 states that mix zeros, subnormals below 2^-1042 and ordinary values in every neighbour position: sums whose operands are out of
the short integer adder's reach.  Resident iterates equal the FUSED path's and the oracle's bit for bit, the allocation-free residual
keeps the residual bar.  And FP32 states whose neighbours span or cancel too far for the split form of their FP64 residual: r of every
point is that of the FP64 sums."""
import numpy as np
import pytest
import torch

import jacobi_inputs as J
import oracle
from test_gpu_residual_values import TOL, _norms
from test_host_arith import _states32

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


def _point(row):
    """The padded state of a grid of one point: its neighbours xm xp ym yp zm zp and itself."""
    u = np.zeros((3, 3, 3), np.float32)
    u[1, 1, 0], u[1, 1, 2], u[1, 0, 1], u[1, 2, 1], u[0, 1, 1], u[2, 1, 1], u[1, 1, 1] = row
    return u


# r^2 and its root are each rounded once (FP64): 2^-53 / 2 + 2^-53, below 1e-15
ONE = 1e-15


@pytest.mark.parametrize("what", ["wide", "wide signed", "cancel", "exponents", "near", "zeros"])
def test_fp32_residual_of_single_points(what):
    import paper_2102_12416_gb300 as jg
    rows = next(v for k, v, _ in _states32(1024) if k == what)
    with np.errstate(over="ignore"):
        rows = rows.astype(np.float32)
    rows = rows[np.isfinite(rows).all(1)][:96]
    w = rows.astype(np.float64)
    r = np.abs((((w[:, 0] + w[:, 1]) + (w[:, 2] + w[:, 3])) + (w[:, 4] + w[:, 5])) - 6.0 * w[:, 6])
    with jg.Jacobi3D([(1, 1, 1)] * len(rows), [("count", (1, 1, 1))] * len(rows), "f32") as s:
        for g, row in enumerate(rows):
            s.set_state(_point(row), g)
        _, got = s.residual()
        assert np.all(np.abs(got - r) <= ONE * r)
    out = torch.zeros(3, dtype=torch.float64, device="cuda")
    for row, want in zip(rows, r):
        jg.jacobi_residual_noalloc(torch.from_numpy(_point(row)).cuda().data_ptr(), (1, 1, 1), "f32", out.data_ptr())
        assert abs(float(out[0]) - want) <= ONE * want


@pytest.mark.parametrize("grid,split", [((32, 32, 8), ("count", (1, 1, 1))), ((37, 9, 11), ("shape", (16, 8, 8))), ((1030, 5, 4), ("count", (1, 1, 1)))])
def test_fp32_residual_of_wide_signed_states(grid, split):
    """Streamed, ragged and tiled rows with points of every span side by side."""
    import paper_2102_12416_gb300 as jg
    rng = np.random.RandomState(8)
    shape = tuple(n + 2 for n in grid[::-1])
    u = (rng.choice([-1.0, 1.0], shape) * rng.uniform(0.5, 1.0, shape) * 2.0 ** rng.randint(-28, 1, shape)).astype(np.float32)
    r, b = _norms(u)
    with jg.Jacobi3D(grid, split, "f32") as s:
        s.set_state(u)
        rel, res = s.residual()
        assert abs(res[0] - r) <= TOL * r and abs(rel[0] - r / b) <= TOL * (r / b)
        _, rel, _ = s.solve(1e30, 1, 1)  # from the step-and-residual kernels
        assert abs(rel[0] - r / b) <= TOL * (r / b)
