"""The gather of the 2D FP64 form, which sums a tile's fields in fixed point at one scale per
component, where the fields of a tile differ by more than that scale resolves: an exactly zero field
beside a large one, small fields beside a large one, fields too small for a scale, a non-finite
node.  Particles at rest feel the electric field alone: u = (q dt / m) E, E interpolated from at
most 36 nodes, so that FP64 gives it to some 36 roundings of the largest field in the stencil."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1909_09613_gb300 as pic  # noqa: E402

GRID, TOL = (32, 16), 36 * 2.0 ** -53


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1909_09613_gb300 import _build
    _build.build()
    oracle.build()


CASES = [(1, 0.3), (1, 0.55), (2, 0.3), (2, 0.55), (3, 0.3), (3, 0.55), (4, 0.3), (4, 0.55)]


def _step(l, dt, fields, x, det, want=True):
    """u after one step of particles at rest at x (sorted by the tile order), here and by the
    oracle."""
    n = x.shape[1]
    run = pic.Run(GRID + (1,), (1.0, 1.0, 1.0), dt, l, pic.PIC_SCHEME_WT, precision=pic.PIC_FP64,
                  capacity=(n,), deterministic=det)
    run.load(0, 1.0, 1.0, 1e-3, x, np.zeros((3, n)))
    for c in range(6):
        run.set_field(c, fields[c])
    run.step(1)
    u = run.particles(0)[1]
    cells = np.floor(x[1]).astype(np.int64) * GRID[0] + np.floor(x[0]).astype(np.int64)
    perm = oracle.tile_sort(GRID + (1,), run.tile, cells, oracle.SLOT_MAJOR)[0]
    run.close()
    if not want:
        return u, None, perm
    orc = oracle.Sim(GRID, (1.0, 1.0), dt, l, pic.PIC_SCHEME_WT)
    orc.add_species(1.0, 1.0, 1e-3, x, np.zeros((3, n)))
    for c in range(6):
        orc.set_field(c, fields[c])
    orc.step(1)
    uo = orc.particles(0)[1][:, perm]
    orc.close()
    return u, uo, perm


def _inputs(l, seed=0):
    """Large fields (about 1) in the columns x < 4, zero elsewhere; particles at 13 <= x < 19."""
    rng = np.random.default_rng(10 * l + seed)
    f = np.zeros((6, 1, GRID[1], GRID[0]))
    f[:, :, :, :4] = rng.standard_normal((6, 1, GRID[1], 4))
    x = rng.random((2, 64)) * np.array([[6.0], [16.0]]) + np.array([[13.0], [0.0]])
    return rng, f, x


@pytest.mark.parametrize("det", [False, True], ids=["atomic", "det"])
@pytest.mark.parametrize("l,dt", CASES + [(3, 1e-6)])
def test_zero_field_beside_a_large_one(l, dt, det):
    _, f, x = _inputs(l)
    u, _, _ = _step(l, dt, f, x, det, want=False)
    assert np.all(u == 0.0)


@pytest.mark.parametrize("small", [1e-3, 1e-8, 1e-14, 1e-40])
@pytest.mark.parametrize("l,dt", CASES)
def test_small_fields_beside_a_large_one(l, dt, small):
    rng, f, x = _inputs(l, 1)
    f[:3, :, :, 6:26] = small * rng.standard_normal((3, 1, GRID[1], 20))
    u, uo, _ = _step(l, dt, f, x, False)
    assert np.max(np.abs(u - uo)) <= TOL * np.max(np.abs(f[:3, :, :, 6:26])) * dt


@pytest.mark.parametrize("scale", [1e-280, 1e-295, 1e-302])
@pytest.mark.parametrize("l,dt", [(2, 0.3), (3, 0.55)])
def test_fields_below_any_scale(l, dt, scale):
    rng, f, x = _inputs(l, 2)
    f[:] = 0.0
    f[:3] = scale * rng.standard_normal((3, 1, GRID[1], GRID[0]))
    u, uo, _ = _step(l, dt, f, x, False)
    assert np.max(np.abs(u - uo)) <= TOL * np.max(np.abs(f[:3])) * dt
    assert np.count_nonzero(u) == u.size


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("l,dt", [(1, 0.3), (2, 0.55), (3, 0.3), (4, 0.55)])
def test_nonfinite_node_reaches_its_stencils_only(l, dt, bad):
    rng, f, x = _inputs(l, 3)
    f[:, :, :, 4:] = rng.standard_normal((6, 1, GRID[1], GRID[0] - 4))
    u, uo, _ = _step(l, dt, f, x, False)
    assert np.max(np.abs(u - uo)) <= 1e-12 * np.max(np.abs(uo))
    f[0, 0, 5, 1] = bad  # out of reach of x >= 13
    v, _, _ = _step(l, dt, f, x, False, want=False)
    assert np.max(np.abs(v - uo)) <= 1e-12 * np.max(np.abs(uo))


def test_stage_without_room_for_masks():
    """The largest stages leave no shared memory for the masks of small fields: the tiles are then
    gathered in FP64."""
    from test_gpu_parity import FP64_TOL, compare_state, make_pair, smooth_fields
    import plasma
    wl = plasma.pair_plasma((64, 64), (1.0, 1.0), 0.5, 2, 1, 5.0, 0.1, 4, omega_p=0.3, seed=7)
    f = smooth_fields((1, 64, 64), 0.05, seed=5)
    for ty in range(32, 20, -1):
        try:
            run, orc = make_pair(wl, pic.PIC_FP64, f, tile=(32, ty), sort_interval=33)
        except pic.PicError:
            continue  # more than 227 KB
        break
    assert 227 * 1024 - 4000 < pic.pic_smem_info(run.ctx)[0] <= 227 * 1024
    run.step(1)
    orc.step(1)
    compare_state(run, orc, 2, FP64_TOL)
    run.close()
    orc.close()
