"""The 2D particle pass with several CTAs per tile (a grid of few tiles is spread over the GPU):
one step against the FP64 oracle where the parts are ragged.  Tolerances as in test_gpu_parity."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1909_09613_gb300 as pic  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1909_09613_gb300 import _build
    _build.build()
    oracle.build()


# (grid, spline order, particles of each species): fewer particles than a warp, one more than a
# warp, an empty species and uneven species in both forms; and, FP64 form only (the FP32 form
# never splits a grid of several waves, and its FP32 sums over the 150,000 particles of one cell
# round by sqrt(150000) 2^-24 = 2e-5 of their size), parts that span several waves
SMALL = [((9, 7), 2, (1, 31)), ((64, 8), 3, (33, 0)), ((33, 17), 4, (257, 64)),
         ((70, 9), 1, (5000, 130))]
CASES = ([c + (pic.PIC_FP64, 1e-12) for c in SMALL + [((512, 128), 3, (300001, 299999))]]
         + [c + (pic.PIC_FP32_MIXED, 2e-6) for c in SMALL])


@pytest.mark.parametrize("grid,l,counts,prec,tol", CASES)
def test_split_tiles_match_oracle(grid, l, counts, prec, tol):
    rng = np.random.default_rng(sum(counts))
    n = (grid[0], grid[1], 1)
    run = pic.Run(n, (1.0, 1.0), 0.4, l, pic.PIC_SCHEME_WT, precision=prec,
                  capacity=[max(c, 1) for c in counts])
    orc = oracle.Sim(grid, (1.0, 1.0), 0.4, l, pic.PIC_SCHEME_WT)
    perms = []
    for s, c in enumerate(counts):
        # offsets in [0, 1) and momenta that FP32 holds exactly; half of the particles crowd one cell
        cell = rng.integers(0, [[grid[0]], [grid[1]]], size=(2, c))
        cell[:, : c // 2] = np.array([[grid[0] - 1], [0]])
        x = cell + rng.random((2, c), dtype=np.float32).astype(np.float64)
        u = rng.normal(0.0, 0.5, (3, c)).astype(np.float32).astype(np.float64)
        run.load(s, 1.0 - 2.0 * s, 1.0, 0.01, x, u)
        orc.add_species(1.0 - 2.0 * s, 1.0, 0.01, x, u)
        cells = np.floor(x[1]).astype(np.int64) * grid[0] + np.floor(x[0]).astype(np.int64)
        order = oracle.SLOT_MAJOR if run.slot_major else oracle.CELL_MAJOR
        perms.append(oracle.tile_sort(n, run.tile, cells, order)[0])
    for c in range(6):
        f = 0.1 * rng.standard_normal((1, grid[1], grid[0])).astype(np.float32).astype(np.float64)
        run.set_field(c, f)
        orc.set_field(c, f)
    run.step(1)
    orc.step(1)
    for c in range(9):
        a, b = run.field(c), orc.field(c)
        assert np.max(np.abs(a - b)) <= tol * np.max(np.abs(b)), c
    for s in range(2):
        _, u, _ = run.particles(s)
        uo = orc.particles(s)[1][:, perms[s]]
        assert counts[s] == 0 or np.max(np.abs(u - uo)) <= tol * np.max(np.abs(uo))
    assert run.diag()["error_flags"] == 0
