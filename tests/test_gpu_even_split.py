"""The FP32 2D particle pass with the grid's tiles divided evenly over the CTAs (shares that cross
tile borders), and the charge density with blocks that take shares of a tile, against the oracle.
Tolerances as in test_gpu_parity and test_gpu_diag_det."""
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


def load(run, orc, grid, counts, rng, u_th):
    dim = len(grid)
    for s, c in enumerate(counts):
        # offsets and momenta that FP32 holds exactly
        cell = rng.integers(0, [[g] for g in grid], size=(dim, c))
        x = cell + rng.random((dim, c), dtype=np.float32).astype(np.float64)
        u = rng.normal(0.0, u_th, (3, c)).astype(np.float32).astype(np.float64)
        run.load(s, 1.0 - 2.0 * s, 1.0, 0.01, x, u)
        if orc is not None:
            orc.add_species(1.0 - 2.0 * s, 1.0, 0.01, x, u)


# about 1,100 to 2,000 particles of the fuller species per CTA on 304 slots; 64, 128 and 375 tiles
@pytest.mark.parametrize("grid,l,counts", [((250, 126), 3, (333333, 1000)),
                                           ((512, 125), 2, (400001, 399999)),
                                           ((260, 600), 4, (700000, 650001))])
def test_even_split_matches_oracle(grid, l, counts):
    rng = np.random.default_rng(7)
    run = pic.Run(grid + (1,), (1.0, 1.0), 0.4, l, pic.PIC_SCHEME_WT,
                  precision=pic.PIC_FP32_MIXED, capacity=counts)
    orc = oracle.Sim(grid, (1.0, 1.0), 0.4, l, pic.PIC_SCHEME_WT)
    load(run, orc, grid, counts, rng, 0.5)
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


# particles that drift past the window (FP64 3D: up to 4 cells between sorts), a tile wider than
# any window, dense and sparse cells, both orders of the store
@pytest.mark.parametrize("prec", [pic.PIC_FP64, pic.PIC_FP32_MIXED], ids=["fp64", "fp32"])
@pytest.mark.parametrize("grid,tile,l,dt,counts,steps", [
    ((9, 7), None, 1, 0.4, (1, 0), 1), ((33, 17), None, 2, 0.4, (9000, 8999), 3),
    ((70, 9), None, 3, 0.6, (300, 40000), 2), ((37, 21), (1, 3, 1), 4, 0.3, (5000, 1), 3),
    ((14, 10, 9), None, 2, 0.55, (4000, 4001), 7), ((12, 5, 7), None, 4, 0.3, (300, 31), 3),
    ((200, 5, 4), (200, 5, 1), 3, 0.3, (9000, 2), 2)])
def test_charge_density_matches_oracle(grid, tile, l, dt, counts, steps, prec):
    dim = len(grid)
    if dim == 3 and tile and prec == pic.PIC_FP32_MIXED:
        tile = None  # (its stage would not fit)
    rng = np.random.default_rng(3)
    run = pic.Run(grid + (1,) * (3 - dim), (1.0,) * dim, dt, l, pic.PIC_SCHEME_WT, precision=prec,
                  capacity=[max(c, 1) for c in counts], tile=tile)
    load(run, None, grid, counts, rng, 2.0)
    run.step(steps)
    d = run.diag()
    orc = oracle.Sim(grid, (1.0,) * dim, dt, l, pic.PIC_SCHEME_WT)
    for s in range(2):
        x, u, _ = run.particles(s)
        orc.add_species(1.0 - 2.0 * s, 1.0, 0.01, x, u)
    rho = orc.rho()
    E = [run.field(c) for c in range(3)]
    div = sum(E[a] - np.roll(E[a], 1, axis=2 - a) for a in range(dim))
    want = np.max(np.abs(div.reshape(-1) - rho.reshape(-1)))
    assert abs(d["max_gauss_residual"] - want) <= 1e-10 * np.max(np.abs(rho))
    assert d["error_flags"] == 0
