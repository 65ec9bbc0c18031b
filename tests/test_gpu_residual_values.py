"""FP64 residual of FP32 states (rounding errors of the FP32 sums carried exactly) and the allocation-free residual, over values where
they can go wrong: wide and narrow spans, signs, subnormals, sums that overflow FP32, infinities and NaN.

Bar: with a span of up to 2^19 between the nonzero neighbours every term is exact; beyond it one point's r is off by at most 2^-46 of
its neighbour sum (1.5e-14), and r is of that sum's size at such points here, so the norms keep the residual bar of 1e-12."""
import numpy as np
import pytest
import torch

import jacobi_inputs as J

pytestmark = pytest.mark.gpu

TOL = 1e-12


def _norms(u):
    u = u.astype(np.float64)
    with np.errstate(all="ignore"):
        s = ((u[1:-1, 1:-1, :-2] + u[1:-1, 1:-1, 2:]) + (u[1:-1, :-2, 1:-1] + u[1:-1, 2:, 1:-1])) + (u[:-2, 1:-1, 1:-1] + u[2:, 1:-1, 1:-1])
        v = np.where(J.boundary_mask(*(n - 2 for n in u.shape[::-1])), u, 0.0)
        b = ((v[1:-1, 1:-1, :-2] + v[1:-1, 1:-1, 2:]) + (v[1:-1, :-2, 1:-1] + v[1:-1, 2:, 1:-1])) + (v[:-2, 1:-1, 1:-1] + v[2:, 1:-1, 1:-1])
        return float(np.sqrt(((s - 6.0 * u[1:-1, 1:-1, 1:-1]) ** 2).sum())), float(np.sqrt((b * b).sum()))


def _state(kind, grid, dtype):
    r = np.random.RandomState(3)
    shape = tuple(n + 2 for n in grid[::-1])
    u = r.uniform(0.5, 1.0, shape)
    if kind == "span":
        u = r.uniform(1.0, 2.0, shape) * 2.0 ** r.randint(-40, 1, shape)
    elif kind == "signed":
        u = r.standard_normal(shape)
    elif kind == "smooth":
        u = J.linear_function(*grid) + 1e-6 * u
    elif kind == "subnormal":
        u = u * 2.0 ** -140
    elif kind == "overflow":
        u[r.uniform(size=shape) < 0.1] = 3.0e38
    elif kind == "inf":
        u[2, 3, 4] = np.inf
    elif kind == "nan":
        u[2, 3, 4] = np.nan
    return np.ascontiguousarray(u.astype(dtype))


def _same(got, want):
    if np.isnan(want):
        return np.isnan(got)
    return got == want if np.isinf(want) else abs(got - want) <= TOL * want


KINDS = ["plain", "span", "signed", "smooth", "subnormal", "overflow", "inf", "nan"]


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("grid,split", [((32, 32, 8), ("count", (1, 1, 1))), ((37, 9, 11), ("shape", (16, 8, 8))), ((1030, 5, 4), ("count", (1, 1, 1)))])
def test_fp32_residual_values(kind, grid, split):
    import paper_2102_12416_gb300 as jg
    u = _state(kind, grid, np.float32)
    r, b = _norms(u)
    with jg.Jacobi3D(grid, split, "f32") as s:
        s.set_state(u)
        rel, res = s.residual()
        assert _same(res[0], r) and (not np.isfinite(r) or _same(rel[0], r / b))
        # the check of a solve takes it from the step-and-residual kernels
        it, rel2, _ = s.solve(0.0, 1, 1)
        assert it == [1]
        s.set_state(u)
        _, rel3, _ = s.solve(1e30, 1, 1)
        assert not np.isfinite(r) or _same(rel3[0], r / b)


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("grid", [(1, 1, 1), (33, 17, 5), (64, 3, 40), (7, 9, 1300)])
def test_noalloc_values(kind, grid, dtype):
    import paper_2102_12416_gb300 as jg
    if kind in ("inf", "nan") and min(n + 2 for n in grid) < 5:
        pytest.skip("the planted point lies outside")
    u = _state(kind, grid, jg.NP_DTYPES[jg.DTYPES[dtype]])
    r, b = _norms(u)
    d, out = torch.from_numpy(u).cuda(), torch.zeros(3, dtype=torch.float64, device="cuda")
    jg.jacobi_residual_noalloc(d.data_ptr(), grid, dtype, out.data_ptr())
    got = out.cpu().numpy()
    assert _same(got[0], r) and _same(got[1], b) and (not np.isfinite(r) or _same(got[2], r / b))
