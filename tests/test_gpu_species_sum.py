"""The species' currents of the 2D FP32 form are summed per tile in FP32 and added to each other in
FP64: two runs of one particle each, of weights 2^30 apart, and one run of both.  The particles do
not see each other in the step, so the currents of the two add up to the third's within one FP64
rounding per node (of two terms) -- single runs and members of a batch alike, in both tile orders
(a tile per species in the slot-major one, one tile flushed per species in the cell-major one)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1909_09613_gb300 as pic  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1909_09613_gb300 import _build
    _build.build()


@pytest.mark.parametrize("batch", [False, True], ids=["run", "batch"])
@pytest.mark.parametrize("order", [pic.PIC_ORDER_SLOT, pic.PIC_ORDER_CELL], ids=["slot", "cell"])
@pytest.mark.parametrize("l", [2, 3])
def test_species_are_added_in_fp64(l, order, batch):
    rng = np.random.default_rng(l)
    x = np.array([[9.0], [6.0]]) + rng.random((2, 1)).astype(np.float32)
    u = rng.normal(0.0, 1.0, (3, 1)).astype(np.float32).astype(np.float64)
    none = (np.empty((2, 0)), np.empty((3, 0)))
    runs = []
    for first, second in ((True, False), (False, True), (True, True)):
        run = pic.Run((24, 16, 1), (1.0, 1.0, 1.0), 0.4, l, pic.PIC_SCHEME_WT,
                      precision=pic.PIC_FP32_MIXED, capacity=(1, 1), tile_order=order)
        run.load(0, 1.0, 1.0, 1.0, *((x, u) if first else none))
        run.load(1, -1.0, 1.0, 2.0 ** -30, *((x, u) if second else none))
        runs.append(run)
    if batch:
        b = pic.Batch(runs)
        b.step(1)
        b.sync()
    else:
        for run in runs:
            run.step(1)
    for c in range(6, 9):
        one, two, both = [run.field(c) for run in runs]
        assert np.count_nonzero(two) > 0
        assert np.max(np.abs(both - (one + two)) / np.maximum(np.abs(one), 1e-300)) <= 2.0 ** -52


@pytest.mark.parametrize("order", [pic.PIC_ORDER_SLOT, pic.PIC_ORDER_CELL], ids=["slot", "cell"])
@pytest.mark.parametrize("l,counts", [(1, (300, 0, 500)), (2, (1, 700, 0, 400)), (3, (400, 33, 1, 900)),
                                      (4, (0, 250, 31, 700))])
def test_several_species_match_oracle(l, counts, order):
    """Three and four species, some without particles: tiles of their own (three, slot-major), one tile
    flushed per species (four, or cell-major).  Tolerance as in test_gpu_parity."""
    import oracle
    oracle.build()
    rng = np.random.default_rng(l)
    grid = (40, 21)
    run = pic.Run(grid + (1,), (1.0, 1.0, 1.0), 0.4, l, pic.PIC_SCHEME_WT,
                  precision=pic.PIC_FP32_MIXED, capacity=[max(c, 1) for c in counts], tile_order=order)
    orc = oracle.Sim(grid, (1.0, 1.0), 0.4, l, pic.PIC_SCHEME_WT)
    for s, c in enumerate(counts):
        x = np.floor(rng.random((2, c)) * np.array(grid)[:, None]) + rng.random((2, c), dtype=np.float32)
        u = rng.normal(0.0, 0.5, (3, c)).astype(np.float32).astype(np.float64)
        run.load(s, (1.0, -1.0, 2.0, -0.5)[s], 1.0 + s, 0.01, x, u)
        orc.add_species((1.0, -1.0, 2.0, -0.5)[s], 1.0 + s, 0.01, x, u)
    for c in range(6):
        f = 0.1 * rng.standard_normal((1, grid[1], grid[0])).astype(np.float32).astype(np.float64)
        run.set_field(c, f)
        orc.set_field(c, f)
    run.step(1)
    orc.step(1)
    for c in range(9):
        a, b = run.field(c), orc.field(c)
        assert np.max(np.abs(a - b)) <= 2e-6 * np.max(np.abs(b)), c
    assert run.diag()["error_flags"] == 0
    run.close()
    orc.close()
