"""The 3D particle pass of the plain FP64 form (weights and currents in fixed point): one step
against the FP64 oracle at every order, with tiles split over several CTAs, ragged counts and a
crowded cell.  Tolerance: FP64 round-off of sums of this size, as in test_gpu_parity."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1909_09613_gb300 as pic  # noqa: E402

TOL = 1e-12


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1909_09613_gb300 import _build
    _build.build()
    oracle.build()


# (grid, spline order, scheme, time step, particles of each species)
CASES = [((5, 3, 2), 1, pic.PIC_SCHEME_WT, 0.2, (1, 31)),
         ((9, 7, 5), 1, pic.PIC_SCHEME_WT, 0.55, (33, 0)),
         ((16, 8, 8), 2, pic.PIC_SCHEME_WT, 0.4, (5000, 4097)),
         ((17, 9, 5), 2, pic.PIC_SCHEME_WT, 0.52, (130, 257)),
         ((17, 9, 5), 2, pic.PIC_SCHEME_MC, 0.3, (257, 64)),
         ((11, 6, 9), 3, pic.PIC_SCHEME_WT, 0.55, (600, 31)),
         ((8, 4, 4), 3, pic.PIC_SCHEME_MC, 0.3, (64, 300)),
         ((7, 13, 6), 4, pic.PIC_SCHEME_WT, 0.3, (400, 129)),
         ((12, 5, 7), 4, pic.PIC_SCHEME_WT, 0.55, (257, 64))]


@pytest.mark.parametrize("det", [0, 1])
@pytest.mark.parametrize("grid,l,scheme,dt,counts", CASES)
def test_fp64_3d_matches_oracle(grid, l, scheme, dt, counts, det):
    rng = np.random.default_rng(sum(counts) + l)
    run = pic.Run(grid, (1.0, 1.0, 1.0), dt, l, scheme, precision=pic.PIC_FP64,
                  capacity=[max(c, 1) for c in counts], deterministic=bool(det))
    orc = oracle.Sim(grid, (1.0, 1.0, 1.0), dt, l, scheme)
    perms = []
    for s, c in enumerate(counts):
        cell = rng.integers(0, [[grid[0]], [grid[1]], [grid[2]]], size=(3, c))
        cell[:, : c // 2] = np.array([[grid[0] - 1], [0], [grid[2] - 1]])
        x = cell + rng.random((3, c))
        u = rng.normal(0.0, 0.7, (3, c))
        run.load(s, 1.0 - 2.0 * s, 1.0, 0.01, x, u)
        orc.add_species(1.0 - 2.0 * s, 1.0, 0.01, x, u)
        k = np.floor(x).astype(np.int64)
        cells = (k[2] * grid[1] + k[1]) * grid[0] + k[0]
        perms.append(oracle.tile_sort(grid, run.tile, cells, oracle.SLOT_MAJOR)[0])
    for c in range(6):
        f = 0.1 * rng.standard_normal((grid[2], grid[1], grid[0]))
        run.set_field(c, f)
        orc.set_field(c, f)
    run.step(1)
    orc.step(1)
    for c in range(9):
        a, b = run.field(c), orc.field(c)
        assert np.max(np.abs(a - b)) <= TOL * np.max(np.abs(b)), c
    for s in range(2):
        if counts[s] == 0:
            continue
        _, u, _ = run.particles(s)
        uo = orc.particles(s)[1][:, perms[s]]
        assert np.max(np.abs(u - uo)) <= TOL * np.max(np.abs(uo))
    assert run.diag()["error_flags"] == 0
