"""Reads into device memory (the copy knows where a pointer points): the same bytes as into host memory,
for sizes that pass through the page-locked stage on their way to the host and for larger ones."""
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


def _ptr(t, kind=ctypes.c_double):
    return ctypes.cast(ctypes.c_void_p(t.data_ptr()), ctypes.POINTER(kind))


@pytest.mark.parametrize("grid,n", [((64, 32, 1), 300), ((256, 256, 1), 20000)])
def test_reads_into_device_memory(grid, n):
    rng = np.random.default_rng(n)
    run = pic.Run(grid, (1.0, 1.0, 1.0), 0.3, 2, pic.PIC_SCHEME_WT, capacity=(n,))
    f = rng.standard_normal((1, grid[1], grid[0]))
    run.set_field(2, f)
    run.load(0, 1.0, 1.0, 1.0, rng.random((2, n)) * np.array(grid[:2])[:, None],
             rng.standard_normal((3, n)))
    lib = pic.load_library()
    d = torch.zeros(run.ncell, dtype=torch.float64, device="cuda")
    assert lib.pic_read_fields(run.ctx, 2, _ptr(d), run.ncell) == 0
    assert np.array_equal(d.cpu().numpy(), f.reshape(-1))
    x = torch.zeros((2, n), dtype=torch.float64, device="cuda")
    u = torch.zeros((3, n), dtype=torch.float64, device="cuda")
    cell = torch.zeros(n, dtype=torch.int64, device="cuda")
    assert lib.pic_read_particles(run.ctx, 0, _ptr(x), _ptr(u), _ptr(cell, ctypes.c_int64), n) == 0
    for got, want in zip((x, u, cell), run.particles(0)):
        assert np.array_equal(got.cpu().numpy(), want)
    run.close()
