"""Steps of grids around the line (2,048 cells) up to which one cluster takes E and B in one launch:
three steps in one call, with particles, both solvers, deterministic or not, against the FP64 oracle.
The merged half steps, the cleared current (both words of a deterministic FP64 run), the second
differences of M4 across block borders and the FP32 shadows the next gather reads all enter.
Tolerance: three times the one-step tolerance of the form (test_gpu_parity), one per step."""
import pytest

import oracle
import plasma

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1909_09613_gb300 as pic  # noqa: E402
from test_gpu_parity import FP32_TOL, FP64_TOL, make_pair, rel, smooth_fields  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1909_09613_gb300 import _build
    _build.build()
    oracle.build()


@pytest.mark.parametrize("det", [False, True], ids=["atomic", "det"])
@pytest.mark.parametrize("solver", [pic.PIC_SOLVER_YEE, pic.PIC_SOLVER_M4], ids=["yee", "m4"])
@pytest.mark.parametrize("prec", [pic.PIC_FP64, pic.PIC_FP32_MIXED], ids=["fp64", "fp32"])
@pytest.mark.parametrize("grid", [(64, 32), (61, 35), (16, 16, 8), (13, 13, 13)])
def test_steps_match_oracle(grid, prec, solver, det):
    dim = len(grid)
    wl = plasma.pair_plasma(grid, (1.0,) * dim, 0.35, 2, 1, 5.0, 0.1, 4, omega_p=0.3, seed=11)
    f = smooth_fields((grid[2] if dim == 3 else 1, grid[1], grid[0]), 0.05, seed=3)
    run, orc = make_pair(wl, prec, f, solver=solver, deterministic=det)
    run.step(3)
    orc.step(3)
    tol = 3 * (FP64_TOL if prec == pic.PIC_FP64 else FP32_TOL)
    errs = [rel(run.field(c), orc.field(c)) for c in range(9)]
    assert max(errs) <= tol, errs
    assert run.diag()["error_flags"] == 0
    run.close()
    orc.close()
