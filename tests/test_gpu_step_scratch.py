"""What pic_step keeps in memory that loads, reads and diagnostics use too (the copy of B, the further
species' sort scratch): a run that is read and diagnosed between its calls, and one that is not,
give the same bits (deterministic), and a load between calls changes nothing of the other species."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1909_09613_gb300 as pic  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1909_09613_gb300 import _build
    _build.build()


# one particle of capacity per cell and species and more: all in the staging buffer; fewer: apart
@pytest.mark.parametrize("grid,l,n", [((40, 24, 1), 4, 1000), ((40, 24, 1), 3, 5000), ((12, 10, 8), 2, 3000),
                                      ((64, 48, 1), 4, 100)])
def test_reads_between_calls_leave_a_run_alone(grid, l, n):
    rng = np.random.default_rng(n)
    dim = 3 if grid[2] > 1 else 2
    x = rng.random((2, dim, n)) * np.array(grid[:dim])[None, :, None]
    u = rng.normal(0.0, 0.5, (2, 3, n))
    f = 0.1 * rng.standard_normal((6,) + grid[::-1])
    runs = []
    for read in (False, True):
        run = pic.Run(grid, (1.0, 1.0, 1.0), 0.4, l, pic.PIC_SCHEME_WT, precision=pic.PIC_FP64,
                      capacity=(n, n), deterministic=True, stream=torch.cuda.Stream())
        for s in range(2):
            run.load(s, 1.0 - 2.0 * s, 1.0, 0.01, x[s], u[s])
        for c in range(6):
            run.set_field(c, f[c])
        for k in range(4):
            run.step(3)
            if read:
                run.diag()
                for s in range(2):
                    run.particles(s)
        runs.append([run.field(c) for c in range(9)] + [a for s in range(2) for a in run.particles(s)])
        run.close()
    for a, b in zip(*runs):
        assert np.array_equal(a, b)
