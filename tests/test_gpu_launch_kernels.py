"""The kernels of a launch per iteration, graph replays and persistent launches on small grids: the tests of those kernels once more with
the resident kernel off, which takes most of their calls otherwise (on the GRAPH and PERSISTENT paths, 4 to some tens of iterations)."""
import pytest

import paper_2102_12416_gb300 as jg
from test_gpu_fp64_adder import test_stencil_same_with_and_without_integer_adds  # noqa: F401
from test_gpu_parity import (  # noqa: F401
    test_autotune_keeps_results, test_autotune_path_keeps_path_and_results, test_config1_bit_exact, test_decomposition_invariance,
    test_fp32_64c_blocks_bit_exact, test_fp32_ragged_61x62x64_blocks, test_persistent_replays_continue, test_ragged_block_shapes,
    test_shapes_give_identical_iterates, test_solve_matches_oracle, test_tile_only_persistent_solve_matches_oracle,
    test_wide_rows_take_the_tile_kernel)

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _launches_only(monkeypatch):
    from paper_2102_12416_gb300 import _build
    _build.build()
    monkeypatch.setenv("JACOBI_RESIDENT", "0")
    destroyed = []
    close = jg.Jacobi3D.close

    def counted(self):
        if self.h:
            destroyed.append(self.info.resident_launches)
        close(self)

    monkeypatch.setattr(jg.Jacobi3D, "close", counted)
    yield
    assert destroyed and not any(destroyed)
