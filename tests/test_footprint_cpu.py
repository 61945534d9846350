"""Device memory of a run, against the bytes it took when the gather read B in place (before a call's steps
kept a copy of it): the copy lies in memory that is idle during a step, so no run of one particle of
capacity per cell or more takes more, and no FP64 run reserves memory that it does not use, but
for the cubic 2D form's published estimate."""
import pytest

import paper_1909_09613_gb300 as pic
from paper_1909_09613_gb300 import _build


@pytest.fixture(scope="module", autouse=True)
def _built():
    _build.build()
    pic.load_library()


@pytest.mark.parametrize("grid,l,prec,cap,det,before", [
    ((2048, 1024, 1), 3, pic.PIC_FP64, (67108864, 67108864), 0, 20820731392),
    ((64, 32, 1), 3, pic.PIC_FP64, (4096, 4096), 0, 1664512),
    ((255, 130, 1), 4, pic.PIC_FP64, (265200, 265200), 0, 62879488),
    ((255, 130, 1), 4, pic.PIC_FP64, (33150, 33150), 1, 11695616),
    ((96, 40, 36), 2, pic.PIC_FP64, (552960, 552960), 0, 160393472),
    ((128, 64, 64), 1, pic.PIC_FP64, (2097152, 2097152), 0, 608282112),
    ((64, 64, 1), 2, pic.PIC_FP64, (8192, 8192), 0, 3057152),
    ((512, 256, 1), 1, pic.PIC_FP64, (524288,), 0, 105920256),
    ((512, 256, 1), 3, pic.PIC_FP32_MIXED, (1 << 20, 1 << 20), 0, 184565248)])
def test_footprint_did_not_grow(grid, l, prec, cap, det, before):
    o = pic.pic_options()
    o.n_species, o.precision, o.deterministic = len(cap), prec, det
    for i, c in enumerate(cap):
        o.capacity[i] = c
    ctx = pic.pic_create(grid, (1.0, 1.0, 1.0), 0.3, l, pic.PIC_SCHEME_WT, o)
    try:
        got = pic.pic_footprint(ctx)
    finally:
        pic.pic_destroy(ctx)
    assert got <= before
    if prec == pic.PIC_FP64 and grid[2] == 1 and l < 3:  # 2 (l + 1) doubles a particle were reserved
        assert got <= before - 16 * (l + 1) * sum(cap)
