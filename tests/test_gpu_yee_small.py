"""Field updates of small grids, where one cluster takes E and B in one launch, and of the first grid
past that line: five steps of random fields without particles against the FP64 oracle (sums of a few
FP64 terms per step: 1e-12 of the largest field), in calls of one and of several steps."""
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
@pytest.mark.parametrize("grid", [(8, 4), (64, 32), (64, 64), (241, 17), (16, 16, 16), (17, 13, 19)])
def test_field_updates_match_oracle(grid, prec):
    dim = len(grid)
    rng = np.random.default_rng(5)
    run = pic.Run(grid + (1,) * (3 - dim), (1.0,) * dim, 0.4, 2, pic.PIC_SCHEME_WT, precision=prec,
                  capacity=(1, 1))
    orc = oracle.Sim(grid, (1.0,) * dim, 0.4, 2, pic.PIC_SCHEME_WT)
    for c in range(6):
        f = rng.standard_normal(tuple((grid + (1,) * (3 - dim))[::-1]))
        run.set_field(c, f)
        orc.set_field(c, f)
    for n in (1, 3, 1):
        run.step(n)
        orc.step(n)
        for c in range(6):
            a, b = run.field(c), orc.field(c)
            assert np.max(np.abs(a - b)) <= 1e-12 * np.max(np.abs(b)), (c, n)
