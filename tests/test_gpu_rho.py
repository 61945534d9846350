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
