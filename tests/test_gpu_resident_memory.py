"""The resident path's memory: a solve whose grids converge one after another cuts its boxes anew between the checks, and neither
allocates nor frees device memory for them, in a workspace of the library's or of the caller's."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

# 96 grids, a CTA each at first; those left are cut into ever more boxes with ever more surface
GRIDS = [(24, 24, 8 + q // 6) for q in range(96)]
SPLITS = [("shape", (16, 16, 16))] * len(GRIDS)
INITS = [dict(bc="uniform", bc_seed=q, interior="zero") for q in range(len(GRIDS))]


@pytest.mark.parametrize("own", [True, False])
@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_solve_allocates_nothing(dtype, own, monkeypatch):
    import paper_2102_12416_gb300 as jg

    def solve(watch):
        ws, kw = None, {}
        if not own:
            n = jg.jacobi_workspace_bytes_batch(GRIDS, SPLITS, dtype)
            ws = torch.empty(n, dtype=torch.uint8, device="cuda")
            kw = dict(workspace=ws.data_ptr(), ws_bytes=n)
        with jg.Jacobi3D(GRIDS, SPLITS, dtype, INITS, path="graph", **kw) as s:
            free = torch.cuda.mem_get_info()[0]
            res = s.solve(1e-5, 2000, 20)
            if watch:
                assert torch.cuda.mem_get_info()[0] == free
                # FP32: between any two checks, whatever was left running; FP64: once so few are left that it is the faster path
                assert s.info.resident_launches >= (max(res[0]) // 20 if dtype == "f32" else 1)
            return res, [s.copy_out(g) for g in range(0, len(GRIDS), 7)]

    first = solve(False)  # loads every kernel
    got = solve(True)
    monkeypatch.setenv("JACOBI_RESIDENT", "0")
    want = solve(False)
    assert len(set(want[0][0])) > 2
    assert got[0] == want[0] == first[0]
    assert all(np.array_equal(a, b) for a, b in zip(got[1], want[1]))
