"""The workloads this library is timed on: what they are, their inputs, one pass over each through
the public entry points, and what a plain FP64 evaluation of the method gives for the same inputs.

A case is one drifting e-/e+ pair plasma (or a batch of them) at a grid, spline order, time step,
density and precision form; a pass advances it by a few steps and reads the result back the way a
program that monitors a run does: the nine field components and the energies.  The FP32 form's
snapshots are taken in single precision, which is what that form carries.

Sizes are those of the benchmark configurations (64x32 quadratic at 4 particles per cell, 2048x1024
cubic at 64, the batch of uneven runs from 64x32 to 512x256 at 4..32 per cell, 3D boxes at 8 per
cell, and the quartic 256x128 runs of the paper's Table 1) and ragged sizes between them.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1909_09613_gb300 as pic

MC, WT = pic.PIC_SCHEME_MC, pic.PIC_SCHEME_WT


def _case(name, kind, precision, nx, ny, nz, l, ppc, steps, dt, gamma=20.0, u_th=0.01,
          scheme=WT, m4=False, runs=1):
    c = dict(kind=kind, precision=precision, nx=nx, ny=ny, nz=nz, l=l, ppc=ppc, steps=steps, dt=dt,
             gamma=gamma, u_th=u_th, scheme=scheme, m4=m4, runs=runs)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the parity and instability-scan run: a cold beam on the smallest grid, launch-bound;
        # the particles are read back too (a restart file)
        _case("fp64_64x32_l2_ppc4", "restart", "fp64", 64, 32, 1, 2, 4, 50, 0.35, u_th=0.0),
        # the smallest request of a scan service, precision form
        _case("fp32_64x32_l2_ppc4", "run", "fp32", 64, 32, 1, 2, 4, 50, 0.45, gamma=30.0),
        # a small scan run on a ragged grid
        _case("fp32_250x126_l3_ppc8", "run", "fp32", 250, 126, 1, 3, 8, 20, 0.3),
        # a run of Table 1: quartic splines, M4 solver, gamma 1000, hot, 64 per cell
        _case("fp32_256x128_l4_ppc64_m4", "run", "fp32", 256, 128, 1, 4, 64, 10, 0.35,
              gamma=1000.0, u_th=0.1, m4=True),
        # the densest scan run, quadratic
        _case("fp32_512x256_l2_ppc32", "run", "fp32", 512, 256, 1, 2, 32, 10, 0.4),
        # the large plasma in the precision form (134M particles)
        _case("fp32_2048x1024_l3_ppc64", "run", "fp32", 2048, 1024, 1, 3, 64, 10, 0.25,
              gamma=50.0),
        # the same plasma in the plain FP64 form
        _case("fp64_2048x1024_l3_ppc64", "run", "fp64", 2048, 1024, 1, 3, 64, 2, 0.25,
              gamma=50.0),
        # a quartic FP64 run with the momentum-conserving gather, ragged
        _case("fp64_255x130_l4_ppc16_mc", "run", "fp64", 255, 130, 1, 4, 16, 5, 0.3, scheme=MC),
        # the 3D service request, precision form
        _case("fp32_256x64x64_l2_ppc8", "run", "fp32", 256, 64, 64, 2, 8, 10, 0.4),
        # a small 3D run in the plain form
        _case("fp64_96x40x36_l2_ppc8", "run", "fp64", 96, 40, 36, 2, 8, 4, 0.4),
        # uneven runs advanced together (the scan's batch)
        _case("batch_48_runs", "batch", "fp32", 512, 256, 1, 3, 32, 10, 0.4, runs=48),
        # a whole call from pinned host arrays: load both species, ten steps, diagnostics
        _case("load_step_512x256_l3_ppc32", "load", "fp32", 512, 256, 1, 3, 32, 10, 0.25,
              gamma=50.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run2d", "run2d", "run2d", "run3d", "batch", "load", "restart"])
    gamma = 10.0 ** rng.uniform(1.0, 3.0 if rng.random() < 0.2 else 2.0)
    u_th = rng.choice([0.0, 0.01, 0.01, 0.03, 0.1])
    scheme = MC if rng.random() < 0.2 else WT
    m4 = rng.random() < 0.2
    precision = rng.choice(["fp32", "fp32", "fp64"])
    if kind == "run3d":
        cells = math.exp(rng.uniform(math.log(8e3), math.log(5e5)))
        ny, nz = _log_int(rng, 16, 64), _log_int(rng, 16, 64)
        nx = min(512, max(16, int(cells / (ny * nz))))
        return _case("", "run", precision, nx, ny, nz, rng.choice([1, 2, 2, 3]),
                     rng.choice([2, 4, 8, 16]), rng.randint(2, 6),
                     round(rng.uniform(0.1, 0.5), 3), gamma, u_th, scheme, m4)
    dt = round(rng.uniform(0.1, 0.7), 3)
    ppc = rng.choice([2, 4, 8, 12, 16, 32, 64])
    l = rng.choice([1, 2, 2, 3, 3, 3, 4])
    if kind == "batch":
        return _case("", "batch", "fp32", rng.choice([128, 256, 512]), 0, 1, 3, 32,
                     rng.randint(4, 12), dt, gamma, 0.01, WT, False, rng.randint(3, 40))
    if kind == "load":
        precision = "fp32"
    hi = 1536 if kind == "run2d" else 400
    nx, ny = _log_int(rng, 33, hi), _log_int(rng, 17, max(64, hi // 2))
    while nx * ny * ppc > 3e7:
        ppc //= 2
    steps = rng.randint(4, 30) if nx * ny * ppc < 1e6 else rng.randint(2, 8)
    if kind == "restart":
        precision = "fp64"
    return _case("", {"run2d": "run"}.get(kind, kind), precision, nx, ny, 1, l, max(2, ppc), steps,
                 dt, gamma, u_th, scheme, m4)


# ---- inputs -----------------------------------------------------------------------------------

def _members(case):
    """The runs of a case: one, or the uneven members of a batch (grid 64x32 up to the case's,
    4..32 per cell, quadratic or cubic, c dt/dx 0.1..0.7), which the case's numbers fix."""
    if case["kind"] != "batch":
        return [dict(case)]
    out = []
    h = 12345 + 7 * case["runs"] + case["nx"] + int(1000 * case["dt"])
    for r in range(case["runs"]):
        v = []
        for _ in range(5):
            h = (h * 1103515245 + 12345) % (1 << 31)
            v.append(h / (1 << 31))
        sizes = [n for n in (64, 128, 256, 512) if n <= case["nx"]]
        nx = sizes[min(int(v[0] * len(sizes)), len(sizes) - 1)]
        out.append(dict(case, nx=nx, ny=nx // 2, nz=1, ppc=(4, 8, 16, 32)[min(int(v[1] * 4), 3)],
                        l=2 if v[2] < 0.5 else 3, dt=0.1 + 0.6 * v[3], gamma=10.0 ** (1.0 + v[4])))
    return out


def _weight(m):
    # 16 cells per relativistic skin depth: n q^2 / (gamma m) = (1/16)^2, n = (ppc / 2) w
    return m["gamma"] / 256.0 / (m["ppc"] // 2)


def _dim(m):
    return 3 if m["nz"] > 1 else 2


def _ncell(m):
    return m["nx"] * m["ny"] * m["nz"]


def _species(m, seed, member, s):
    """x (dim, n) and u (3, n), FP64 on the device: ppc / 2 particles in every cell (cells x
    fastest) at uniform offsets, Gaussian momenta of spread u_th in the frame that drifts along x
    with gamma, the x component flipped for the volume transform.  Offsets and momenta are drawn
    as FP32 values, so that both forms store them exactly."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    g = torch.Generator(device=dev)
    g.manual_seed((int(seed) * 1000003 + member * 17 + s) % (1 << 62))
    per, n = m["ppc"] // 2, _ncell(m) * (m["ppc"] // 2)
    dim = _dim(m)
    x = torch.empty((dim, n), dtype=torch.float64, device=dev)
    u = torch.empty((3, n), dtype=torch.float64, device=dev)
    cell = torch.arange(n, device=dev, dtype=torch.int64).div_(per, rounding_mode="floor")
    ext = (m["nx"], m["ny"], m["nz"])
    for a in range(dim):
        off = torch.rand(n, generator=g, device=dev, dtype=torch.float32)
        x[a] = cell.remainder(ext[a]).to(torch.float64) + off
        cell = cell.div_(ext[a], rounding_mode="floor")
    beta = math.sqrt(1.0 - 1.0 / m["gamma"] ** 2)
    v = m["u_th"] * torch.randn((3, n), generator=g, device=dev, dtype=torch.float32)
    e = torch.sqrt(1.0 + (v * v).sum(0))
    flip = torch.rand(n, generator=g, device=dev) > 0.5 * (1.0 + beta * v[0] / e)
    v[0] = torch.where(flip, -v[0], v[0])
    u[0] = (m["gamma"] * (v[0] + beta * e)).to(torch.float32)
    u[1:] = v[1:]
    return x, u


def _new_run(m):
    n = _ncell(m) * (m["ppc"] // 2)
    return pic.Run((m["nx"], m["ny"], m["nz"]), (1.0, 1.0, 1.0), m["dt"], m["l"], m["scheme"],
                   precision=pic.PIC_FP32_MIXED if m["precision"] == "fp32" else pic.PIC_FP64,
                   capacity=(n, n), solver=pic.PIC_SOLVER_M4 if m["m4"] else pic.PIC_SOLVER_YEE)


def prepare(case, seed):
    members = _members(case)
    runs, host = [], []
    for k, m in enumerate(members):
        run = _new_run(m)
        for s, q in enumerate((-1.0, 1.0)):
            x, u = _species(m, seed, k, s)
            if case["kind"] == "load":
                host.append((x.cpu().pin_memory().numpy(), u.cpu().pin_memory().numpy()))
            else:
                run.load(s, q, 1.0, _weight(m), x, u)
        runs.append(run)
    torch.cuda.synchronize()
    return dict(case=case, members=members, runs=runs, host=host,
                batch=pic.Batch(runs) if case["kind"] == "batch" else None)


# ---- one pass ---------------------------------------------------------------------------------

def _snapshot(run, fp32):
    out = []
    for c in range(9):
        f = torch.from_numpy(run.field(c).reshape(-1))
        out.append(f.float() if fp32 else f)
    return out


def _energies(run, fp32):
    d = run.diag()
    v = [d["field_energy"], d["kinetic_energy"], d["total_charge"], d["max_gauss_residual"]]
    return np.array(v, dtype=np.float32 if fp32 else np.float64)


def run(state):
    case, runs = state["case"], state["runs"]
    fp32 = case["precision"] == "fp32"
    if case["kind"] == "batch":
        state["batch"].step(case["steps"])
        state["batch"].sync()
        snaps = [_snapshot(r, fp32) for r in runs]
        return {"fields": [torch.cat([s[c] for s in snaps]) for c in range(9)]}
    r = runs[0]
    if case["kind"] == "load":
        for s, q in enumerate((-1.0, 1.0)):
            r.load(s, q, 1.0, _weight(case), *state["host"][s])
        for c in range(6):
            r.set_field(c, np.zeros(r.ncell))
    r.step(case["steps"])
    out = {"energies": _energies(r, fp32), "fields": _snapshot(r, fp32)}
    if case["kind"] == "restart":
        out["particles"] = [list(r.particles(s)) for s in range(2)]
    return out


def work(case):
    """What a pass cannot do without: every step reads and writes each particle's state and the
    fields once (E, B read and written, J written and read, FP64; the FP32 form gathers from and
    writes FP32 shadows too) and evaluates the method's weights, gather, push and current."""
    nbytes = flops = 0.0
    for m in _members(case):
        dim, l, n, cells = _dim(m), m["l"], _ncell(m) * (m["ppc"] // 2) * 2, _ncell(m)
        k = l + 1
        fp32 = m["precision"] == "fp32"
        state = (4 + 4 * (dim + 3)) if fp32 else 8 * (dim + 3)
        gather = 12 * k ** dim + 6 * k ** (dim - 1)
        current = 6 * k ** (dim - 1) * (k + 1) + 12 * (k + 1)
        weights = dim * (2 * k * l + 4 * k + 2 * k)
        nbytes += case["steps"] * (2.0 * state * n + (150 if not fp32 else 174) * cells) + 72.0 * cells
        flops += case["steps"] * (n * (gather + current + weights + 90.0) + 60.0 * cells)
        if case["kind"] == "load":
            nbytes += n * (8 * (dim + 3) + state)
        if case["kind"] == "restart":
            nbytes += n * (state + 8 * (dim + 4))
    return {"bytes": nbytes, "flops": flops}


# ---- the method in plain FP64 -----------------------------------------------------------------

def _spline(k, t):
    """Cardinal B-spline of order k (support [0, k]) at the numpy points t."""
    if k == 1:
        return ((t >= 0.0) & (t < 1.0)).astype(np.float64)
    return (t * _spline(k - 1, t) + (k - t) * _spline(k - 1, t - 1.0)) / (k - 1)


def _w(l, x):
    return _spline(l + 1, x + 0.5 * (l + 1))


def _t(l, dtt, x):
    """The unit-area box of half-width dtt averaged over W_{l-1}; the integral of a cardinal
    B-spline up to t is the sum of the next order's shifts t, t - 1, ..."""
    def integral(y):
        t = y + 0.5 * l
        return sum(_spline(l + 1, t - j) for j in range(10))
    return (integral(x + dtt) - integral(x - dtt)) / (2.0 * dtt)


class _Axis:
    """A symmetric interpolation function along one axis as polynomials of the in-cell offset:
    the weight of node lo + i of a particle at offset d of its cell, exact on each of the pieces
    between the offsets where the function's knots fall."""

    def __init__(self, f, l, half, radius, knots, dev):
        lo, hi = math.ceil(-radius - half - 1e-9), math.floor(1.0 + radius - half + 1e-9)
        br = sorted({0.0, 1.0} | {round((k + half) % 1.0, 12) for k in knots})
        pieces, nodes = [], range(lo, hi + 1)
        for a, b in zip(br[:-1], br[1:]):
            t = 0.5 * (1.0 - np.cos(np.pi * (np.arange(l + 1) + 0.5) / (l + 1)))
            d = a + (b - a) * t
            v = np.vander(t, l + 1, increasing=True)
            pieces.append([np.linalg.solve(v, f(d - (n + half))) for n in nodes])
        keep = [i for i in range(len(nodes)) if any(np.abs(p[i]).max() > 1e-15 for p in pieces)]
        self.lo, self.n, self.l = lo + keep[0], keep[-1] - keep[0] + 1, l
        c = np.array([p[keep[0]:keep[-1] + 1] for p in pieces])
        self.c = torch.tensor(c, dtype=torch.float64, device=dev)  # (piece, node, power)
        self.br = torch.tensor(br, dtype=torch.float64, device=dev)

    def __call__(self, d):
        p = torch.bucketize(d, self.br[1:-1], right=True)
        a, b = self.br[p], self.br[p + 1]
        t = (d - a) / (b - a)
        out = []
        for i in range(self.n):
            r = self.c[p, i, self.l]
            for m in range(self.l - 1, -1, -1):
                r = r * t + self.c[p, i, m]
            out.append(r)
        return out


class _Plain:
    """One run in FP64 with plain tensor operations, particle chunk by particle chunk."""

    CHUNK = 1 << 22

    def __init__(self, m, dev):
        self.m, self.dev, self.dim = m, dev, _dim(m)
        self.n = (m["nx"], m["ny"], m["nz"])
        self.F = [torch.zeros(_ncell(m), dtype=torch.float64, device=dev) for _ in range(9)]
        l, dt = m["l"], m["dt"]
        kw = [j - 0.5 * (l + 1) for j in range(l + 2)]
        self.wh = _Axis(lambda x: _w(l, x), l, 0.5, 0.5 * (l + 1), kw, dev)
        self.wi = _Axis(lambda x: _w(l, x), l, 0.0, 0.5 * (l + 1), kw, dev)
        if m["scheme"] == WT:
            kt = [j - 0.5 * l + sg * dt for j in range(l + 1) for sg in (-1, 1)]
            self.ti = _Axis(lambda x: _t(l, dt, x), l, 0.0, 0.5 * l + dt, kt, dev)
        else:
            self.ti = self.wi
        self.sp = []

    def add(self, q, w, x, u):
        c = [torch.floor(v).to(torch.int64) for v in x]
        self.sp.append(dict(q=q, w=w, c=c, d=[v - k.to(torch.float64) for v, k in zip(x, c)],
                            u=list(u)))

    def _nodes(self, c, a, lo, count):
        """Linear index contributions of `count` wrapped nodes along axis a."""
        stride = (1, self.n[0], self.n[0] * self.n[1])[a]
        return [((c + (lo + i)).remainder_(self.n[a])).mul_(stride) for i in range(count)]

    def _gather(self, c, d):
        dim = self.dim
        tab = [[None, None] for _ in range(dim)]
        for a in range(dim):
            for h, ax in enumerate((self.ti, self.wh)):
                tab[a][h] = (ax(d[a]), self._nodes(c[a], a, ax.lo, ax.n))
        eb = []
        for comp in range(6):
            h = [(a == comp) if comp < 3 else (a != comp - 3) for a in range(3)]
            wx, ix = tab[0][int(h[0])]
            wy, iy = tab[1][int(h[1])]
            zs = [(None, None)] if dim == 2 else list(zip(*tab[2][int(h[2])]))
            acc = torch.zeros_like(d[0])
            for wz, iz in zs:
                plane = torch.zeros_like(acc)
                for vy, jy in zip(wy, iy):
                    base = jy if iz is None else jy + iz
                    row = torch.zeros_like(acc)
                    for vx, jx in zip(wx, ix):
                        row.addcmul_(vx, self.F[comp][base + jx])
                    plane.addcmul_(vy, row)
                acc.add_(plane) if wz is None else acc.addcmul_(wz, plane)
            eb.append(acc)
        return eb

    def _deposit(self, qw, c, d, sh, dn, vz):
        dim, dt = self.dim, self.m["dt"]
        S0, DS, idx = [], [], []
        for a in range(dim):
            w0, w1 = self.wi(d[a]), self.wi(dn[a])
            zero = torch.zeros_like(d[a])
            s0 = [zero] + w0 + [zero]
            s1 = []
            for i in range(len(s0)):  # node lo - 1 + i carries w1[i - 1 - sh]
                v = [w1[i - 1 - k] if 0 <= i - 1 - k < len(w1) else zero for k in (-1, 0, 1)]
                s1.append(torch.where(sh[a] == 0, v[1], torch.where(sh[a] < 0, v[0], v[2])))
            S0.append(s0)
            DS.append([p - q for p, q in zip(s1, s0)])
            idx.append(self._nodes(c[a], a, self.wi.lo - 1, len(s0)))
        if dim == 2:
            nx, ny = len(S0[0]), len(S0[1])
            for j in range(ny):
                f = (S0[1][j] + 0.5 * DS[1][j]) * (-qw / dt)
                acc = torch.zeros_like(f)
                for i in range(nx - 1):
                    acc = acc + DS[0][i]
                    self.F[6].index_add_(0, idx[0][i] + idx[1][j], acc * f)
            for i in range(nx):
                f = (S0[0][i] + 0.5 * DS[0][i]) * (-qw / dt)
                acc = torch.zeros_like(f)
                for j in range(ny - 1):
                    acc = acc + DS[1][j]
                    self.F[7].index_add_(0, idx[0][i] + idx[1][j], acc * f)
            for j in range(ny):
                f0 = (S0[1][j] + 0.5 * DS[1][j]) * (qw * vz)
                f1 = (0.5 * S0[1][j] + DS[1][j] / 3.0) * (qw * vz)
                for i in range(nx):
                    self.F[8].index_add_(0, idx[0][i] + idx[1][j], S0[0][i] * f0 + DS[0][i] * f1)
            return
        for a in range(3):
            b, e = (a + 1) % 3, (a + 2) % 3
            for kb in range(len(S0[b])):
                for ke in range(len(S0[e])):
                    f = (S0[b][kb] * (S0[e][ke] + 0.5 * DS[e][ke])
                         + DS[b][kb] * (0.5 * S0[e][ke] + DS[e][ke] / 3.0)) * (-qw / dt)
                    base = idx[b][kb] + idx[e][ke]
                    acc = torch.zeros_like(f)
                    for ka in range(len(S0[a]) - 1):
                        acc = acc + DS[a][ka]
                        self.F[6 + a].index_add_(0, base + idx[a][ka], acc * f)

    def _push(self):
        m, dt = self.m, self.m["dt"]
        for k in range(6, 9):
            self.F[k].zero_()
        for sp in self.sp:
            h = 0.5 * sp["q"] * dt
            for p in range(0, sp["d"][0].numel(), self.CHUNK):
                cut = slice(p, p + self.CHUNK)
                c = [v[cut] for v in sp["c"]]
                d = [v[cut] for v in sp["d"]]
                u = [v[cut] for v in sp["u"]]
                eb = self._gather(c, d)
                E, B = eb[:3], eb[3:]
                um = [u[a] + h * E[a] for a in range(3)]
                g = torch.sqrt(1.0 + um[0] ** 2 + um[1] ** 2 + um[2] ** 2)
                t = [h * B[a] / g for a in range(3)]
                s = 2.0 / (1.0 + t[0] ** 2 + t[1] ** 2 + t[2] ** 2)
                up = [um[a] + um[(a + 1) % 3] * t[(a + 2) % 3] - um[(a + 2) % 3] * t[(a + 1) % 3]
                      for a in range(3)]
                un = [um[a] + s * (up[(a + 1) % 3] * t[(a + 2) % 3]
                                   - up[(a + 2) % 3] * t[(a + 1) % 3]) + h * E[a] for a in range(3)]
                gi = 1.0 / torch.sqrt(1.0 + un[0] ** 2 + un[1] ** 2 + un[2] ** 2)
                sh, dn = [], []
                for a in range(self.dim):
                    y = d[a] + dt * un[a] * gi
                    f = torch.floor(y)
                    sh.append(f.to(torch.int64))
                    dn.append(y - f)
                self._deposit(sp["q"] * sp["w"], c, d, sh, dn, un[2] * gi)
                for a in range(3):
                    sp["u"][a][cut] = un[a]
                for a in range(self.dim):
                    sp["c"][a][cut] = (c[a] + sh[a]).remainder(self.n[a])
                    sp["d"][a][cut] = dn[a]

    def _diff(self, f, a, sign):
        """Forward (+1) or backward (-1) difference along axis a of a (nz, ny, nx) array."""
        if a >= self.dim:
            return torch.zeros_like(f)
        ax = 2 - a
        return torch.roll(f, -1, ax) - f if sign > 0 else f - torch.roll(f, 1, ax)

    def _faraday(self, f, a):
        d = self._diff(f, a, 1)
        if not self.m["m4"] or a >= self.dim:
            return d
        r, dt = d, self.m["dt"]
        for b in range(self.dim):
            ax = 2 - b
            coef = (dt * dt - 1.0) / 12.0 if b == a else dt * dt / 12.0
            r = r + coef * (torch.roll(d, -1, ax) - 2.0 * d + torch.roll(d, 1, ax))
        return r

    def _half_b(self):
        g = [v.view(self.n[2], self.n[1], self.n[0]) for v in self.F]
        D = self._faraday
        c = [D(g[2], 1) - D(g[1], 2), D(g[0], 2) - D(g[2], 0), D(g[1], 0) - D(g[0], 1)]
        for a in range(3):
            g[3 + a] -= 0.5 * self.m["dt"] * c[a]

    def step(self):
        self._push()
        self._half_b()
        g = [v.view(self.n[2], self.n[1], self.n[0]) for v in self.F]
        d = [[self._diff(g[3 + k], a, -1) for a in range(3)] for k in range(3)]
        c = [d[2][1] - d[1][2], d[0][2] - d[2][0], d[1][0] - d[0][1]]
        for a in range(3):
            g[a] += self.m["dt"] * (c[a] - g[6 + a])
        self._half_b()

    def energies(self):
        fe = 0.5 * sum(float((v * v).sum()) for v in self.F[:6])
        ke = qt = 0.0
        rho = torch.zeros_like(self.F[0])
        for sp in self.sp:
            u2 = sp["u"][0] ** 2 + sp["u"][1] ** 2 + sp["u"][2] ** 2
            ke += sp["w"] * float((u2 / (torch.sqrt(1.0 + u2) + 1.0)).sum())
            qt += sp["q"] * sp["w"] * u2.numel()
            for p in range(0, u2.numel(), self.CHUNK):
                cut = slice(p, p + self.CHUNK)
                ws = [self.wi(sp["d"][a][cut]) for a in range(self.dim)]
                ids = [self._nodes(sp["c"][a][cut], a, self.wi.lo, self.wi.n)
                       for a in range(self.dim)]
                zs = [(1.0, 0)] if self.dim == 2 else list(zip(ws[2], ids[2]))
                for wz, iz in zs:
                    for wy, iy in zip(ws[1], ids[1]):
                        f = wy * (wz * (sp["q"] * sp["w"]))
                        for wx, ix in zip(ws[0], ids[0]):
                            rho.index_add_(0, ix + iy + iz, wx * f)
        g = [v.view(self.n[2], self.n[1], self.n[0]) for v in self.F[:3]]
        div = sum(self._diff(g[a], a, -1) for a in range(self.dim))
        res = float((div.reshape(-1) - rho).abs().max())
        return np.array([fe, ke, qt, res])


def exact(case, seed):
    """What one pass over a new state gives in plain FP64; nothing for the restart file's
    particles (their order is the library's) and for cases that would take too long."""
    members = _members(case)
    total = sum(_ncell(m) * m["ppc"] * (m["nz"] > 1 and 8 or 1) for m in members)
    if total * case["steps"] > 1.5e9:
        return None
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    fields, energies = [], None
    for k, m in enumerate(members):
        sim = _Plain(m, dev)
        for s, q in enumerate((-1.0, 1.0)):
            x, u = _species(m, seed, k, s)
            sim.add(q, _weight(m), list(x), list(u))
        for _ in range(case["steps"]):
            sim.step()
        fields.append(sim.F)
        if case["kind"] != "batch":
            energies = sim.energies()
    out = {"fields": [torch.cat([f[c] for f in fields]) for c in range(9)]}
    if energies is not None:
        out["energies"] = energies
    if case["kind"] == "restart":
        out["particles"] = None
    return out
