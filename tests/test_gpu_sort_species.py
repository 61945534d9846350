"""All species sorted by the same launches: the stable order of every species, bit for bit, with
uneven and empty species, on grids of few and of many keys (two sets of stages)."""
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


@pytest.mark.parametrize("prec", [pic.PIC_FP64, pic.PIC_FP32_MIXED], ids=["fp64", "fp32"])
@pytest.mark.parametrize("grid,tile,counts", [
    ((9, 7, 1), None, (300, 0, 1)),              # one tile
    ((45, 27, 1), (1, 1, 1), (1000, 33, 257)),   # tiles of one cell: a block of one warp each
    ((256, 240, 1), None, (5000, 70001, 31)),    # few keys (61,440)
    ((300, 257, 1), None, (5000, 70001, 31)),    # many keys
    ((12, 10, 8), None, (3000, 64, 0))])
def test_sort_of_all_species_is_stable(grid, tile, counts, prec):
    rng = np.random.default_rng(sum(counts))
    dim = 3 if grid[2] > 1 else 2
    run = pic.Run(grid, (1.0,) * dim, 0.3, 2, pic.PIC_SCHEME_WT, precision=prec,
                  capacity=[max(c, 1) for c in counts], tile=tile, sort_interval=4)
    for s, c in enumerate(counts):
        x = rng.random((dim, c)) * np.array(grid[:dim])[:, None]
        u = rng.normal(0.0, 0.5, (3, c))
        u[2] = np.arange(c) * 2.0**-20  # a tag that FP32 holds (no force acts: q = 0, B = 0)
        run.load(s, 0.0, 1.0, 1.0, x, u)
    run.step(3)
    before = [run.particles(s) for s in range(3)]
    run.sort()
    order = oracle.SLOT_MAJOR if run.slot_major else oracle.CELL_MAJOR
    for s in range(3):
        xb, ub, cb = before[s]
        xa, ua, ca = run.particles(s)
        perm, ts = oracle.tile_sort(grid, run.tile, cb, order)
        assert np.array_equal(run.tile_offsets(s), ts)
        assert np.array_equal(ua, ub[:, perm])
        assert np.array_equal(xa, xb[:, perm])
        assert np.array_equal(ca, cb[perm])
    run.close()
