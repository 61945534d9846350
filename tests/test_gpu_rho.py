"""Charge density of the diagnostics, seen through max |D.E - rho|."""
from fractions import Fraction

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


@pytest.mark.parametrize("trial", range(6))
def test_rounding_in_a_crowded_tile(trial):
    """Linear splines, E = 0: 4,000 charges of either sign on one node cancel exactly and leave one
    charge elsewhere in the tile, whose largest weight comes back with one rounding at 2^-53 of
    a weight of one (the tile's fixed-point unit) beside those of its product (2^-59)."""
    rng = np.random.default_rng(trial)
    off = rng.random(2)
    crowd = np.repeat([[3.0], [2.0]], 4000, axis=1)
    run = pic.Run((32, 8, 1), (1.0, 1.0, 1.0), 0.3, 1, pic.PIC_SCHEME_WT, precision=pic.PIC_FP64,
                  capacity=(4001, 4001))
    run.load(0, 1.0, 1.0, 1.0, np.hstack([crowd, [[14.0 + off[0]], [5.0 + off[1]]]]),
             np.zeros((3, 4001)))
    run.load(1, -1.0, 1.0, 1.0, crowd, np.zeros((3, 4000)))
    got = run.diag()["max_gauss_residual"]
    run.close()
    d = [Fraction(14.0 + off[0]) - 14, Fraction(5.0 + off[1]) - 5]
    want = max(a * b for a in (d[0], 1 - d[0]) for b in (d[1], 1 - d[1]))
    assert abs(Fraction(got) - want) <= Fraction(1, 2 ** 53) + Fraction(1, 2 ** 58)


@pytest.mark.parametrize("prec", [pic.PIC_FP64, pic.PIC_FP32_MIXED], ids=["fp64", "fp32"])
@pytest.mark.parametrize("share", [1.0, 0.1, 0.002], ids=["even", "tenth", "clump"])
@pytest.mark.parametrize("grid,l,counts", [((96, 40), 1, (60000, 59990)), ((61, 35), 3, (30000, 1)),
                                           ((128, 8), 2, (20000, 0)), ((33, 17, 9), 2, (60000, 777)),
                                           ((16, 16, 16), 3, (9000, 9000))])
def test_uneven_plasma_matches_oracle(grid, l, counts, share, prec):
    """Half of the particles in a part of the box, the others spread over it, so that blocks hold whole
    tiles, parts of one, and many tiles of a few particles: every node, as max |D.E - rho| of
    fields that cancel the oracle's density."""
    dim, rng = len(grid), np.random.default_rng(sum(counts))
    g = tuple(grid) + (1,) * (3 - dim)
    run = pic.Run(g, (1.0,) * 3, 0.3, l, pic.PIC_SCHEME_WT, precision=prec,
                  capacity=[max(c, 1) for c in counts])
    orc = oracle.Sim(grid, (1.0,) * dim, 0.3, l, pic.PIC_SCHEME_WT)
    ext = np.array(grid, dtype=np.float64)[:, None]
    for s, c in enumerate(counts):
        cell = np.floor(rng.random((dim, c)) * ext)
        cell[:, : c // 2] = np.floor(rng.random((dim, c // 2)) * ext * share ** (1.0 / dim) + 3.0) % ext
        x = cell + rng.random((dim, c), dtype=np.float32)
        run.load(s, 1.0 - 2.0 * s, 1.0, 1.0, x, np.zeros((3, c)))
        orc.add_species(1.0 - 2.0 * s, 1.0, 1.0, x, np.zeros((3, c)))
    rho = np.asarray(orc.rho()).reshape(g[2], g[1], g[0])
    size = np.max(np.abs(rho))
    rest, left = rho - rho.mean(), rho.mean()
    # E with D.E = rho - <rho>: along x up to the rows' means, along y up to the planes', along z
    for a, axis in enumerate((2, 1, 0)[:dim]):
        mean = rest.mean(axis=axis, keepdims=True)
        run.set_field(a, np.cumsum(np.broadcast_to(rest - mean, rho.shape), axis=axis))
        rest = np.broadcast_to(mean, rho.shape)
    got = run.diag()["max_gauss_residual"]
    # FP64 rounding of the cumulated field, up to 128 nodes of one size, and of up to 60,000 charges
    assert abs(got - abs(left)) <= 1e-10 * size
    run.close()
    orc.close()


def test_largest_window():
    """Tiles of 1 x 17 x 25 cells and their reach are 8 x 24 x 32 = 6,144 nodes, 48 KB of words: the most
    shared memory a launch takes unasked, of which the kernel needs a little besides."""
    grid, n = (4, 17, 25), 40000
    rng = np.random.default_rng(4)
    run = pic.Run(grid, (1.0, 1.0, 1.0), 0.3, 1, pic.PIC_SCHEME_WT, precision=pic.PIC_FP64,
                  capacity=(n,), tile=(1, 17, 25))
    orc = oracle.Sim(grid, (1.0, 1.0, 1.0), 0.3, 1, pic.PIC_SCHEME_WT)
    x = rng.random((3, n)) * np.array(grid)[:, None]
    run.load(0, 1.0, 1.0, 1.0, x, np.zeros((3, n)))
    orc.add_species(1.0, 1.0, 1.0, x, np.zeros((3, n)))
    want = np.max(np.abs(orc.rho()))
    got = run.diag()
    assert got["status"] == pic.PIC_OK
    assert abs(got["max_gauss_residual"] - want) <= 1e-11 * want
    run.close()
    orc.close()
