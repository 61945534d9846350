"""Reads of fields and particles on both sides of the size that passes through the page-locked stage
(256 kB), from one thread and from several at once: the bytes that were loaded come back."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1909_09613_gb300 as pic  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1909_09613_gb300 import _build
    _build.build()


def check(grid, n, seed):
    rng = np.random.default_rng(seed)
    run = pic.Run(grid, (1.0, 1.0), 0.3, 2, pic.PIC_SCHEME_WT, capacity=(max(n, 1), 1),
                  stream=torch.cuda.Stream())
    f = [rng.standard_normal((1, grid[1], grid[0])) for _ in range(6)]
    for c in range(6):
        run.set_field(c, f[c])
    x = rng.random((2, n)) * np.array(grid[:2])[:, None]
    u = rng.standard_normal((3, n))
    run.load(0, 1.0, 1.0, 1.0, x, u)
    for _ in range(3):
        for c in range(6):
            assert np.array_equal(run.field(c), f[c])
        xr, ur, cr = run.particles(0)
        order = np.argsort(ur[0])
        want = np.argsort(u[0])
        assert np.array_equal(ur[:, order], u[:, want])
        assert np.array_equal(xr[:, order], x[:, want])
        cells = np.floor(x[1]).astype(np.int64) * grid[0] + np.floor(x[0]).astype(np.int64)
        assert np.array_equal(cr[order], cells[want])
    run.close()


# 48 bytes per particle: 5461 are the most that pass through the stage
@pytest.mark.parametrize("grid,n", [((5, 3, 1), 0), ((256, 128, 1), 5461), ((257, 128, 1), 5462)])
def test_read_back_around_the_stage(grid, n):
    check(grid, n, 1)


def test_read_back_from_several_threads():
    failed = []

    def work(k):
        try:
            check((64, 33, 1), 4000 + k, k)
        except BaseException as e:  # noqa: BLE001 (reported below)
            failed.append(e)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(6)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed
