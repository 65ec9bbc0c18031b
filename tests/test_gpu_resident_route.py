"""Which calls run the resident kernel (jacobi_info counts its launches), so that the tests of its results cannot pass on the other
kernels alone."""
import pytest

from test_gpu_resident import SHAPES

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("path", ["graph", "persistent", "fused", "explicit"])
@pytest.mark.parametrize("grid,split", SHAPES)
def test_small_grids_run_resident(grid, split, path, dtype):
    import paper_2102_12416_gb300 as jg
    with jg.Jacobi3D(grid, split, dtype, dict(bc="uniform", bc_seed=31, interior="uniform"), path=path) as s:
        taken = []
        for n in (1, 33, 8):
            before = s.info.resident_launches
            s.step(n)
            taken.append(s.info.resident_launches - before)
        s.sync()
    on = int(path in ("graph", "persistent"))
    assert taken[:2] == [0, on] and taken[2] in (0, on)


def test_batch_solve_and_long_calls_run_resident():
    import paper_2102_12416_gb300 as jg
    grids = [(12, 9, 10), (30, 21, 17), (8, 40, 6), (33, 32, 31)]
    inits = [dict(bc="linear_noise", bc_seed=g, noise_amp=1e-3, interior="zero") for g in range(4)]
    with jg.Jacobi3D(grids, [("shape", (16, 16, 16))] * 4, "f64", inits, path="graph") as s:
        iters, _, _ = s.solve(1e-4, 5000, 25)
        assert s.info.resident_launches >= max(iters) // 25  # one between any two checks
    with jg.Jacobi3D((20, 17, 19), ("shape", (8, 8, 8)), "f32", path="graph") as s:
        s.step(20011)
        assert s.info.resident_launches >= 2


@pytest.mark.parametrize("env", [{"JACOBI_RESIDENT": "0"}, {"JACOBI_PERSIST_WS": "1"}])
def test_switched_off(env, monkeypatch):
    import paper_2102_12416_gb300 as jg
    for k, v in env.items():
        monkeypatch.setenv(k, v)
    with jg.Jacobi3D((33, 17, 29), ("count", (3, 2, 4)), "f64", path="graph") as s:
        s.step(40)
        assert s.info.resident_launches == 0


def test_large_grids_do_not():
    import paper_2102_12416_gb300 as jg
    with jg.Jacobi3D((160, 160, 160), ("shape", (64, 64, 64)), "f64", path="graph") as s:
        s.step(40)
        assert s.info.resident_launches == 0
