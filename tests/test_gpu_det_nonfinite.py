"""A non-finite momentum in a deterministic FP64 run, whose current is summed in integer words: the
error word reports it at the next syncing call, and the current holds what the finite particles
deposit (bit for bit: a particle that cannot move and has no velocity adds nothing)."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1909_09613_gb300 as pic  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1909_09613_gb300 import _build
    _build.build()


def _current(run):
    out = np.empty((3, run.ncell))
    for a in range(3):
        pic.load_library().pic_read_fields(run.ctx, 6 + a, out[a].ctypes.data_as(
            ctypes.POINTER(ctypes.c_double)), run.ncell)
    return out


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("grid", [(12, 10, 1), (8, 6, 5)], ids=["2d", "3d"])
def test_nonfinite_momentum_is_reported(grid, bad):
    dim, n = (3 if grid[2] > 1 else 2), 300
    rng = np.random.default_rng(2)
    x = rng.random((dim, n)) * np.array(grid[:dim])[:, None]
    u = rng.normal(0.0, 0.5, (3, n))
    current = []
    for k in (n, n - 1):  # with the particle of the bad momentum, and without it
        v = u[:, :k].copy()
        v[0, n - 1:] = bad
        run = pic.Run(grid, (1.0, 1.0, 1.0), 0.4, 2, pic.PIC_SCHEME_WT, precision=pic.PIC_FP64,
                      capacity=(n,), deterministic=True)
        run.load(0, -1.0, 1.0, 0.01, np.ascontiguousarray(x[:, :k]), v)
        run.step(1)
        if k == n:
            with pytest.raises(pic.PicError) as e:
                run.sync()
            assert e.value.status == pic.PIC_ENAN
        else:
            run.sync()
        current.append(_current(run))
        run.close()
    assert np.isfinite(current[0]).all()
    assert np.array_equal(current[0], current[1])
