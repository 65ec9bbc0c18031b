"""The autotuner on grids that the resident kernel takes: the choice keeps it, and the time that it reports is that of the calls that
follow."""
import pytest

pytestmark = pytest.mark.gpu

CASE = ((64, 64, 64), ("count", (2, 2, 2)))


@pytest.mark.parametrize("path", [None, "graph", "persistent"])
@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_tuned_handle_runs_what_was_timed(dtype, path, monkeypatch):
    import paper_2102_12416_gb300 as jg
    monkeypatch.delenv("JACOBI_TUNE_CACHE", raising=False)
    with jg.Jacobi3D(*CASE, dtype, dict(bc="linear", interior="uniform")) as s:
        r = s.autotune(100, path=path)
        assert r["path"] in ("graph", "persistent") and (path is None or r["path"] == path)
        before = s.info.resident_launches
        ms = min(s.step_timed(100)[0] for _ in range(20)) / 100
        assert s.info.resident_launches == before + 20
        # the launches per iteration take 1.5 times as long or more
        assert r["ms_per_iter"] / 1.25 < ms < r["ms_per_iter"] * 1.25


@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_short_trials_keep_the_resident_kernel(dtype, monkeypatch):
    import paper_2102_12416_gb300 as jg
    monkeypatch.delenv("JACOBI_TUNE_CACHE", raising=False)
    with jg.Jacobi3D(*CASE, dtype, dict(bc="linear", interior="uniform")) as s:
        assert s.autotune(1)["path"] != "fused"
        s.step(100)
        assert s.info.resident_launches == 1
        assert s.autotune(1, path="fused")["path"] == "fused"  # asked for by name


def test_switched_off_is_not_tuned(monkeypatch):
    import paper_2102_12416_gb300 as jg
    monkeypatch.delenv("JACOBI_TUNE_CACHE", raising=False)
    monkeypatch.setenv("JACOBI_RESIDENT", "0")
    with jg.Jacobi3D(*CASE, "f64", dict(bc="linear", interior="uniform")) as s:
        r = s.autotune(100)
        ms = min(s.step_timed(100)[0] for _ in range(20)) / 100
        assert s.info.resident_launches == 0 and r["ms_per_iter"] / 1.5 < ms < r["ms_per_iter"] * 1.5
