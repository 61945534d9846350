// Grid kernels: periodic Yee FDTD updates (FP64), FP32 field shadows, particle packing and
// unpacking, and the FP64 diagnostics.
#include "pic_fixed.cuh"
#include "pic_grid_dev.cuh"
#include "pic_launch.h"

#include <cmath>

namespace pic {

namespace {

constexpr int kBlock = 256;

// Half steps B <- B - h curl E on the staggered grid (Sec. 1 Yee; App. C with A_i = 1), as the
// flags name them (yee_b_cell).
__global__ void __launch_bounds__(kBlock) k_yee_b(const __grid_constant__ RunDev rd, double h,
                                                  int flags)
{
    const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (c < rd.ncell) yee_b_cell(rd, c, h, flags);
}

// E <- E + dt curl B - dt J.
__global__ void __launch_bounds__(kBlock) k_yee_e(const __grid_constant__ RunDev rd, int shadow)
{
    const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (c < rd.ncell) yee_e_cell(rd, c, shadow);
}

// Both updates of a step of a small grid in one launch: one cluster of kYeeCtas blocks takes E, then
// (cluster barrier: B reads E of the neighbouring cells, other blocks' among them) B.  Two launches
// of a few blocks are 5 us each, nearly all of it launch and first loads (50 steps of 64x32 cells:
// 1960 -> 1843 us in the FP64 form, 1747 -> 1695 in the FP32 form).  Up to one cell per thread: a
// second one waits for the FP64 pipes of the eight SMs while two launches have more of them (50
// steps, two launches -> cluster, us: 2,048 cells Yee 2018 -> 1970, M4 2328 -> 2185, 3D M4 6442 ->
// 6290; 3,072 cells Yee 2328 -> 2384, M4 2635 -> 2810; 4,096 cells M4 2668 -> 2854, 3D 6485 -> 6879).
constexpr int kYeeCtas = 8;
constexpr int64_t kYeeOneCells = kYeeCtas * kBlock;

__global__ void __cluster_dims__(kYeeCtas, 1, 1) __launch_bounds__(kBlock)
k_yee_eb(const __grid_constant__ RunDev rd, double h, int shadow, int flags)
{
    const int c = blockIdx.x * kBlock + threadIdx.x;
    if (c < rd.ncell) yee_e_cell(rd, c, shadow);
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
    if (c < rd.ncell) yee_b_cell(rd, c, h, flags);
}

__global__ void __launch_bounds__(kBlock) k_shadow(const __grid_constant__ RunDev rd)
{
    const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (c >= rd.ncell) return;
#pragma unroll
    for (int f = 0; f < 6; ++f) rd.Fs[f][c] = (float)rd.F[f][c];
}

// FP64 physical (x, u) -> the context's particle form, for particles p0 .. p0 + m - 1.
// x[a * xs + i], u[a * us + i] hold particle p0 + i.  Positions are divided by dx (IEEE
// division, so the cell index floor(x/dx) matches a plain FP64 evaluation) and wrapped into
// [0, n).
__device__ __forceinline__ void pack_one(const RunDev &rd, const SpeciesDev &sp, int64_t p,
                                         const double *xp, const double *up)
{
    int cell[3] = {0, 0, 0};
    double off[3] = {0, 0, 0};
    for (int a = 0; a < rd.dim; ++a) {
        double xi = xp[a] / rd.dx[a];
        if (!isfinite(xi)) {  // a non-finite input position: flag it, keep the index in range
            set_err(rd.err, 2);  // PIC_ERR_NONFINITE
            xi = 0.0;
        }
        const double N = (double)rd.n[a];
        if (xi >= N) xi -= N;
        if (xi < 0.0) xi += N;
        if (xi >= N) xi = 0.0;  // -tiny + N rounded up to N
        const double f = floor(xi);
        cell[a] = (int)f;
        off[a] = xi - f;
    }
    if (rd.prec == 1) {
        int c[3] = {cell[0], cell[1], cell[2]};
        float o[3];
        for (int a = 0; a < rd.dim; ++a) {
            o[a] = (float)off[a];
            if (o[a] >= 1.0f) {  // offset rounded to 1: carry into the next cell
                o[a] = 0.0f;
                c[a] += 1;
                if (c[a] >= rd.n[a]) c[a] -= rd.n[a];
            }
            ((float *)sp.pos[a])[p] = o[a];
        }
        sp.cell[p] = (int32_t)gidx(rd, c[0], c[1], rd.dim == 3 ? c[2] : 0);
        for (int a = 0; a < 3; ++a) ((float *)sp.mom[a])[p] = (float)up[a];
    } else {
        for (int a = 0; a < rd.dim; ++a) ((double *)sp.pos[a])[p] = (double)cell[a] + off[a];
        for (int a = 0; a < 3; ++a) ((double *)sp.mom[a])[p] = up[a];
    }
}

__global__ void __launch_bounds__(kBlock) k_pack(const __grid_constant__ RunDev rd, int s,
                                                 const double *x, int64_t xs, const double *u,
                                                 int64_t us, int64_t m, int64_t p0)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= m) return;
    double xp[3] = {0, 0, 0}, up[3];
    for (int a = 0; a < rd.dim; ++a) xp[a] = x[a * xs + i];
    for (int a = 0; a < 3; ++a) up[a] = u[a * us + i];
    pack_one(rd, rd.sp[s], p0 + i, xp, up);
}

// ---- drifting plasma generated on the device (App. D) ------------------------------------
// SplitMix64 finaliser (Steele, Lea, Flood 2014) and U[0,1) from its 53 high bits.
__device__ __forceinline__ uint64_t sm64_mix(uint64_t z)
{
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

constexpr int kJuttnerAttempts = 128;

__device__ __forceinline__ double sm64_uniform(uint64_t key, uint64_t ctr)
{
    return (double)(sm64_mix(ctr * 0x9E3779B97F4A7C15ull + key) >> 11) * (1.0 / 9007199254740992.0);
}

__global__ void __launch_bounds__(kBlock) k_load_plasma(const __grid_constant__ RunDev rd, int s,
                                                        LoadKeys keys, int64_t per_cell,
                                                        double gamma, double u_th, double theta,
                                                        int64_t n)
{
    const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p >= n) return;
    const int64_t cell = p / per_cell;
    int64_t ci[3];
    ci[0] = cell % rd.n[0];
    ci[1] = (cell / rd.n[0]) % rd.n[1];
    ci[2] = cell / ((int64_t)rd.n[0] * rd.n[1]);
    double xp[3] = {0, 0, 0}, up[3] = {0, 0, 0};
    // every operation rounded on its own (no fused multiply-add), as a plain evaluation does
    for (int a = 0; a < rd.dim; ++a) {
        const double L = __dmul_rn((double)rd.n[a], rd.dx[a]);
        const double off = sm64_uniform(keys.pos[a], (uint64_t)p);
        double xa = __dmul_rn(__dadd_rn((double)ci[a], off), rd.dx[a]);
        if (xa >= L) xa = __dsub_rn(xa, L);
        xp[a] = xa;
    }
    const double beta = sqrt(__dsub_rn(1.0, __ddiv_rn(1.0, __dmul_rn(gamma, gamma))));
    if (theta > 0.0 || u_th > 0.0) {
        double v[3];
        if (theta > 0.0) {
            // Sobol's method: attempt a draws X1..X4 at counter p * kJuttnerAttempts + a;
            // u = -theta ln(X1 X2 X3), eta = -theta ln(X1 X2 X3 X4), accepted when
            // eta^2 - u^2 > 1.  The loop is bounded; a particle left without an accepted
            // attempt (about 1e-14 at theta = 0.3) is flagged and loaded at rest.
            double um = -1.0;
            for (int a = 0; a < kJuttnerAttempts && um < 0.0; ++a) {
                const uint64_t ctr = (uint64_t)p * kJuttnerAttempts + a;
                const double x1 = __dsub_rn(1.0, sm64_uniform(keys.jut[0], ctr));
                const double x2 = __dsub_rn(1.0, sm64_uniform(keys.jut[1], ctr));
                const double x3 = __dsub_rn(1.0, sm64_uniform(keys.jut[2], ctr));
                const double x4 = __dsub_rn(1.0, sm64_uniform(keys.jut[3], ctr));
                const double p3 = __dmul_rn(__dmul_rn(x1, x2), x3);
                const double u = __dmul_rn(-theta, log(p3));
                const double eta = __dmul_rn(-theta, log(__dmul_rn(p3, x4)));
                if (__dsub_rn(__dmul_rn(eta, eta), __dmul_rn(u, u)) > 1.0) um = u;
            }
            if (um < 0.0) {
                set_err(rd.err, 4);  // PIC_ERR_TIMEOUT: a bounded device loop gave up
                um = 0.0;
            }
            const double x5 = sm64_uniform(keys.dir[0], (uint64_t)p);
            const double x6 = sm64_uniform(keys.dir[1], (uint64_t)p);
            const double ct = __dsub_rn(__dmul_rn(2.0, x5), 1.0);
            const double st = __dmul_rn(2.0, sqrt(__dmul_rn(x5, __dsub_rn(1.0, x5))));
            const double ph = __dmul_rn(6.283185307179586, x6);
            v[0] = __dmul_rn(um, ct);
            v[1] = __dmul_rn(__dmul_rn(um, st), cos(ph));
            v[2] = __dmul_rn(__dmul_rn(um, st), sin(ph));
        } else
        for (int a = 0; a < 3; ++a) {
            const double u1 = __dsub_rn(1.0, sm64_uniform(keys.mom[2 * a], (uint64_t)p));  // (0, 1]
            const double u2 = sm64_uniform(keys.mom[2 * a + 1], (uint64_t)p);
            const double r = sqrt(__dmul_rn(-2.0, log(u1)));
            v[a] = __dmul_rn(u_th, __dmul_rn(r, cos(__dmul_rn(6.283185307179586, u2))));
        }
        const double s2 = __dadd_rn(__dadd_rn(__dmul_rn(v[0], v[0]), __dmul_rn(v[1], v[1])),
                                    __dmul_rn(v[2], v[2]));
        const double ep = sqrt(__dadd_rn(1.0, s2));
        const double x1 = sm64_uniform(keys.flip, (uint64_t)p);
        const double thr = __dmul_rn(0.5, __dadd_rn(1.0, __ddiv_rn(__dmul_rn(beta, v[0]), ep)));
        const double vx = (x1 > thr) ? -v[0] : v[0];
        up[0] = __dmul_rn(gamma, __dadd_rn(vx, __dmul_rn(beta, ep)));
        up[1] = v[1];
        up[2] = v[2];
    } else {
        up[0] = sqrt(__dsub_rn(__dmul_rn(gamma, gamma), 1.0));
    }
    pack_one(rd, rd.sp[s], p, xp, up);
}

// Particles p0 .. p0 + m - 1 -> FP64 physical x[a * m + i], u[a * m + i], cell[i].
__global__ void __launch_bounds__(kBlock) k_unpack(const __grid_constant__ RunDev rd, int s,
                                                   double *x, double *u, int64_t *cell,
                                                   int64_t m, int64_t p0)
{
    const SpeciesDev &sp = rd.sp[s];
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= m) return;
    const int64_t p = p0 + i;
    if (rd.prec == 1) {
        const int c = sp.cell[p];
        int ci[3];
        ci[0] = c % rd.n[0];
        ci[1] = (c / rd.n[0]) % rd.n[1];
        ci[2] = c / (rd.n[0] * rd.n[1]);
        for (int a = 0; a < rd.dim; ++a)
            x[a * m + i] = ((double)ci[a] + (double)((const float *)sp.pos[a])[p]) * rd.dx[a];
        for (int a = 0; a < 3; ++a) u[a * m + i] = (double)((const float *)sp.mom[a])[p];
        if (cell) cell[i] = c;
    } else {
        int ci[3] = {0, 0, 0};
        for (int a = 0; a < rd.dim; ++a) {
            const double xi = ((const double *)sp.pos[a])[p];
            ci[a] = (int)floor(xi);
            x[a * m + i] = xi * rd.dx[a];
        }
        for (int a = 0; a < 3; ++a) u[a * m + i] = ((const double *)sp.mom[a])[p];
        if (cell) cell[i] = gidx(rd, ci[0], ci[1], ci[2]);
    }
}

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ double warp_max(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

__device__ double block_sum(double v)
{
    __shared__ double red[32];
    v = warp_sum(v);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) red[w] = v;
    __syncthreads();
    const int nw = (blockDim.x + 31) >> 5;
    v = (threadIdx.x < nw) ? red[threadIdx.x] : 0.0;
    if (w == 0) v = warp_sum(v);
    __syncthreads();
    return v;
}

__device__ double block_max(double v)
{
    __shared__ double red[32];
    v = warp_max(v);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) red[w] = v;
    __syncthreads();
    const int nw = (blockDim.x + 31) >> 5;
    v = (threadIdx.x < nw) ? red[threadIdx.x] : 0.0;
    if (w == 0) v = warp_max(v);
    __syncthreads();
    return v;
}

__device__ __forceinline__ void atomic_max_nonneg(double *a, double v)
{
    atomicMax((unsigned long long *)a, (unsigned long long)__double_as_longlong(v));
}

// sum over nodes of E^2 + B^2 (FP64); non-finite values raise the error bit.
__global__ void __launch_bounds__(kBlock) k_field_energy(const __grid_constant__ RunDev rd,
                                                         double *out)
{
    double acc = 0.0;
    bool bad = false;
    for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < rd.ncell;
         c += (int64_t)gridDim.x * blockDim.x) {
        for (int f = 0; f < 6; ++f) {
            const double v = rd.F[f][c];
            if (!isfinite(v)) bad = true;
            acc += v * v;
        }
    }
    if (bad) set_err(rd.err, 2);
    acc = block_sum(acc);
    if (threadIdx.x == 0) atomicAdd(out, acc);
}

// The FP64 value of an FP32 one, by its bits: a conversion instruction runs at the rate of the
// FP64 pipe (2 per clock and SM), which bounds k_kinetic.
__device__ __forceinline__ double widen(float v)
{
    const uint32_t b = __float_as_uint(v), e = (b >> 23) & 0xff;
    if (e == 0 || e == 0xff) return (double)v;  // zero, subnormal, non-finite
    return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + (896u << 20))),
                            (int)(b << 29));
}

// sum over particles of w m (gamma - 1).  Bound by the FP64 pipe: the division of the form
// u^2 / (gamma + 1), free of cancellation for slow particles, is evaluated only by warps that
// hold a particle below gamma = 2; above it gamma - 1 loses at most one bit to the subtraction,
// no more than the quotient's roundings.  Together with k_rho's fixed point: pic_diag of 134M
// particles 24.1 -> 10.5 ms (FP32 form), 24.6 -> 11.7 ms (FP64 form).
__global__ void __launch_bounds__(kBlock) k_kinetic(const __grid_constant__ RunDev rd, int s,
                                                    double *out)
{
    const SpeciesDev &sp = rd.sp[s];
    double acc = 0.0;
    bool bad = false;
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < sp.n;
         p += (int64_t)gridDim.x * blockDim.x) {
        double u0, u1, u2;
        if (rd.prec == 1) {
            u0 = widen(((const float *)sp.mom[0])[p]);
            u1 = widen(((const float *)sp.mom[1])[p]);
            u2 = widen(((const float *)sp.mom[2])[p]);
        } else {
            u0 = ((const double *)sp.mom[0])[p];
            u1 = ((const double *)sp.mom[1])[p];
            u2 = ((const double *)sp.mom[2])[p];
        }
        const double u2s = u0 * u0 + u1 * u1 + u2 * u2;
        if ((__double2hiint(u2s) & 0x7ff00000) == 0x7ff00000) bad = true;
        const double g = sqrt(1.0 + u2s);
        acc += __double2hiint(g) >= 0x40000000 ? g - 1.0 : u2s / (g + 1.0);
    }
    if (bad) set_err(rd.err, 2);
    acc = block_sum(acc);
    if (threadIdx.x == 0) atomicAdd(out, acc * sp.w * sp.m);
}

// rho = sum q w W_l / V_c at integer nodes: the l + 1 non-zero B-spline weights per axis, the same
// S0 the Esirkepov deposit starts from, evaluated in 62-bit fixed point (pic_fixed.cuh); in FP64
// they bound the kernel (k_kinetic has the figures).  A block takes an equal share of the particles of
// species blockIdx.y, whatever the tiles hold, with its ends moved to a tile's where one is near
// (rho_edge), and sums every tile's part of it in shared memory, kRhoEpoch particles at a time: 64-bit words in units of 2^(k - 62), k = b - 2 for fewer than 2^b particles, so
// that no sum reaches 2^64 and each product is rounded at 2^(k - 63) <= 2^-53 of a weight of 1, the
// rounding of an FP64 sum there.  A word is two 32-bit atomics, the low one's carry going to the high
// one.  The window covers particles up to `drift` cells away from their tile; what lies outside, tiles of
// few particles, and everything when no window fits (nodes = 0), goes to the global density one
// reduction per node, which is what bounded the kernel when every particle did
// (pic_diag of 134M particles 10.6 -> 7.5 ms, FP32 form, and 11.7 -> 6.7 ms, FP64 form).  Equal
// shares instead of equal parts of every tile cost an even plasma 3% (2048x1024 quadratic, 8 of a
// species per cell: 2.11 -> 2.18 ms, the search for the ends) and spare a dense one the walk
// of its few full tiles by a few blocks (all particles in 1% of the cells 3.2 -> 2.2 ms, in 0.1% 11.8
// -> 2.2; FP32 form 6.8 -> 2.8 and 29.8 -> 2.9).
// The lanes of a warp take particles 2^sh apart: in the cell-major order neighbours in the store
// share a cell, and their atomics would collide, while particles about a cell's occupancy apart
// (at most 32) sit in neighbouring cells; in the slot-major order neighbours in the store already
// do (sh = 0).
constexpr int kRhoEpoch = 4095;

struct RhoWin {
    int drift[3], pre[3], w[3];
    int nodes;
    int64_t least;  // particles of a tile from which the window pays
};

// *(hi, lo) += v
__device__ __forceinline__ void shared_add64(uint32_t *lo, uint32_t *hi, uint64_t v)
{
    const uint32_t l = (uint32_t)v;
    const uint32_t old = atomicAdd(lo, l);
    atomicAdd(hi, (uint32_t)(v >> 32) + (old + l < old ? 1u : 0u));
}

template <int L, int DIM>
__device__ __forceinline__ void rho_particle(const RunDev &rd, const SpeciesDev &sp,
                                             const RhoWin &win, bool window, const int *org,
                                             int64_t p, int k, uint32_t *lo, uint32_t *hi, double qw,
                                             double *rho)
{
    int c[3] = {0, 0, 0};
    uint64_t f[DIM];
    if (rd.prec == 1) {
        const int cc = sp.cell[p];
        c[2] = DIM == 3 ? fast_div(cc, rd.div_n01.m, rd.div_n01.s) : 0;
        const int r = cc - c[2] * rd.n[0] * rd.n[1];
        c[1] = fast_div(r, rd.div_n0.m, rd.div_n0.s);
        c[0] = r - c[1] * rd.n[0];
#pragma unroll
        for (int a = 0; a < DIM; ++a)
            f[a] = offset_fixed(((const uint32_t *)sp.pos[a])[p]);
    } else {
#pragma unroll
        for (int a = 0; a < DIM; ++a)  // (a non-finite position stays in range)
            c[a] = min(decode_position(((const uint64_t *)sp.pos[a])[p], f[a]), rd.n[a] - 1);
    }
    Limbs w[DIM][L + 1];
    int b[DIM], at[DIM];
    bool in = window;
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        uint64_t psi, t[L + 1];
        b[a] = spline_base62<L>(f[a], false, psi);
        bspline62<L>(psi, t);
#pragma unroll
        for (int i = 0; i <= L; ++i) w[a][i] = limbs(t[i]);
        in = local_coord(c[a], org[a], rd.tile[a], win.drift[a], rd.n[a], at[a]) && in;
        at[a] += win.pre[a] + b[a];
    }
    if (in) {
        const uint64_t half = k > 0 ? (uint64_t)1 << (k - 1) : 0;
#pragma unroll
        for (int kk = 0; kk <= (DIM == 3 ? L : 0); ++kk) {
#pragma unroll
            for (int jj = 0; jj <= L; ++jj) {
                const Limbs wjk = DIM == 3 ? limbs(mul62(w[DIM - 1][kk], w[1][jj])) : w[1][jj];
                const int row = ((DIM == 3 ? (at[DIM - 1] + kk) * win.w[1] : 0) + at[1] + jj) * win.w[0]
                                + at[0];
#pragma unroll
                for (int ii = 0; ii <= L; ++ii)
                    shared_add64(lo + row + ii, hi + row + ii, (mul62(w[0][ii], wjk) + half) >> k);
            }
        }
    } else {
        const Scale62 q = scale62((uint64_t)__double_as_longlong(qw));
        const Limbs m = limbs(q.m);
#pragma unroll 1
        for (int kk = 0; kk <= (DIM == 3 ? L : 0); ++kk) {
            const int gk = DIM == 3 ? wrap_near(c[DIM - 1] + b[DIM - 1] + kk, rd.n[2]) : 0;
            Limbs wk = m;
            if (DIM == 3) {
#pragma unroll
                for (int i = 0; i <= L; ++i)
                    if (i == kk) wk = limbs(mul62(w[DIM - 1][i], m));
            }
#pragma unroll
            for (int jj = 0; jj <= L; ++jj) {
                double *row = rho + gidx(rd, 0, wrap_near(c[1] + b[1] + jj, rd.n[1]), gk);
                const Limbs wjk = limbs(mul62(w[1][jj], wk));
#pragma unroll
                for (int ii = 0; ii <= L; ++ii)
                    red_fixed(row + wrap_near(c[0] + b[0] + ii, rd.n[0]), mul62(w[0][ii], wjk), q.top);
            }
        }
    }
}

// The tile of store position p (start[0] = 0 <= p < start[nt]), found by a whole warp together.
__device__ __forceinline__ int64_t tile_of(const int64_t *start, int64_t nt, int64_t p)
{
    const int lane = threadIdx.x & 31;
    int64_t a = 0, b = nt;  // start[a] <= p < start[b]
    while (b - a > 1) {
        const int64_t step = (b - a + 31) / 32, at = a + (lane + 1) * step;
        a += __popc(__ballot_sync(0xffffffffu, at < b && start[at] <= p)) * step;
        b = min(b, a + step);
    }
    return a;
}

// First particle of block i of nb and its tile (-1: to be searched for): the equal share's, or a
// tile's first where one lies within half a share of it, so that a plasma of even density is divided
// into whole tiles.
__device__ __forceinline__ longlong2 rho_edge(const int64_t *start, int64_t nt, int64_t n, int64_t i,
                                              int64_t nb)
{
    const int64_t p = n * i / nb, near = n / (2 * nb);
    if (p >= n) return make_longlong2(n, -1);
    const int64_t t = tile_of(start, nt, p), below = p - start[t], above = start[t + 1] - p;
    if (below <= near && below <= above) return make_longlong2(p - below, t);
    if (above > near) return make_longlong2(p, t);
    // (tiles may be empty: the next particle's is not always t + 1)
    return make_longlong2(p + above, start[min(t + 2, nt)] > p + above ? t + 1 : -1);
}

template <int L, int DIM>
__global__ void __launch_bounds__(kBlock) k_rho(const __grid_constant__ RunDev rd,
                                                const __grid_constant__ RhoWin win, int sh,
                                                double *rho)
{
    extern __shared__ uint32_t words[];  // low words, then high words
    uint32_t *lo = words, *hi = words + win.nodes;
    const SpeciesDev &sp = rd.sp[blockIdx.y];
    const int64_t *start = sp.tile_start;
    const int64_t n = sp.n, nt = rd.ntiles, nb = gridDim.x, none = win.nodes == 0;
    if (n == 0) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __shared__ longlong2 edge[2];
    int64_t first = n * blockIdx.x / nb, last = n * (blockIdx.x + 1) / nb, tile = 0;
    if (!none) {
        if (warp < 2) {  // a search each, side by side
            const longlong2 e = rho_edge(start, nt, n, blockIdx.x + warp, nb);
            if (lane == 0) edge[warp] = e;
        }
        __syncthreads();
        first = edge[0].x;
        tile = edge[0].y;
        last = edge[1].x;
    }
    const double vc = rd.dx[0] * rd.dx[1] * (DIM == 3 ? rd.dx[2] : 1.0);
    const double qw = sp.q * sp.w / vc;
    for (int64_t p = first; p < last;) {  // block-uniform
        // what is summed together: the part of p's tile, or, with no window, all up to the next part
        // that takes one
        int64_t end = last;
        bool window = false;
        int org[3] = {0, 0, 0};
        if (!none) {
            int64_t t = p > first || tile < 0 ? tile_of(start, nt, p) : tile;
            org[0] = (int)(t % rd.ntile[0]) * rd.tile[0];
            org[1] = (int)(t / rd.ntile[0] % rd.ntile[1]) * rd.tile[1];
            org[2] = (int)(t / rd.ntile[0] / rd.ntile[1]) * rd.tile[2];
            end = max(min(last, start[t + 1]), p + 1);  // (start[t] <= p < start[t + 1])
            window = end - p >= win.least;
            while (!window && end < last) {  // 32 tiles at a time, the warp's lanes one each
                const int64_t u = t + 1 + lane;
                const int64_t s = u < nt ? min(start[u], last) : last;
                const unsigned stop = __ballot_sync(
                    0xffffffffu, s >= last || min(start[u + 1], last) - s >= win.least);
                if (stop) {
                    end = max(end, __shfl_sync(0xffffffffu, s, __ffs(stop) - 1));
                    break;
                }
                t += 32;
            }
        }
        const int64_t step = window ? kRhoEpoch : (int64_t)1 << 20;
        for (; p < end; p += step) {
            const int cnt = (int)min(end - p, step);
            const int k = max(30 - __clz(cnt), 0);  // cnt < 2^(k + 2)
            if (window) {
                for (int i = threadIdx.x; i < 2 * win.nodes; i += kBlock) words[i] = 0;
                __syncthreads();
            }
            const int passes = (cnt + (32 << sh) - 1) / (32 << sh) << sh;
#pragma unroll 1
            for (int i = warp; i < passes; i += kBlock / 32) {
                const int q = ((i >> sh) << (5 + sh)) + (lane << sh) + (i & ((1 << sh) - 1));
                if (q < cnt) rho_particle<L, DIM>(rd, sp, win, window, org, p + q, k, lo, hi, qw, rho);
            }
            if (!window) continue;
            __syncthreads();
            const double unit = __hiloint2double((1023 + k - 62) << 20, 0);
            const int rows = win.nodes / win.w[0];
            for (int r = warp; r < rows; r += kBlock / 32) {
                const int ry = r % win.w[1], rz = r / win.w[1];
                const int gy = wrap_near(org[1] - win.pre[1] + ry, rd.n[1]);
                const int gz = DIM == 3 ? wrap_near(org[2] - win.pre[2] + rz, rd.n[2]) : 0;
                double *row = rho + gidx(rd, 0, gy, gz);
                for (int i = lane; i < win.w[0]; i += 32) {
                    const int m = r * win.w[0] + i;
                    const uint64_t v = (uint64_t)hi[m] << 32 | lo[m];
                    if (v) atomicAdd(row + wrap_near(org[0] - win.pre[0] + i, rd.n[0]), (double)v * unit * qw);
                }
            }
            __syncthreads();
        }
        p = end;
    }
}

// The window of a tile's charge density: the nodes that particles up to `drift` cells (at most 3)
// away from the tile reach, if they fit the shared memory every launch may use.
RhoWin rho_window(const RunDev &rd)
{
    RhoWin w;
    int64_t nodes = 1;
    for (int a = 0; a < 3; ++a) {
        const bool on = a < rd.dim;
        w.drift[a] = on ? (rd.drift[a] < 3 ? rd.drift[a] : 3) : 0;
        w.pre[a] = on ? w.drift[a] + rd.l / 2 : 0;
        w.w[a] = on ? rd.tile[a] + w.drift[a] + w.pre[a] + rd.l - (rd.l - 1) / 2 : 1;
        nodes *= w.w[a];
    }
    w.nodes = nodes * 8 <= 47 * 1024 ? (int)nodes : 0;  // (48 KB, some of it the kernel's own)
    return w;
}

// Backward-difference divergence at integer node c of a field whose component a sits half a
// cell up along a (E or J on the Yee grid): sum_a (F_a(c) - F_a(c - e_a)) / dx_a.
__device__ __forceinline__ double div_node(const RunDev &rd, const double *const *F, int64_t c)
{
    const int nx = rd.n[0], ny = rd.n[1], nz = rd.n[2];
    const int i = (int)(c % nx);
    const int j = (int)((c / nx) % ny);
    const int k = (int)(c / ((int64_t)nx * ny));
    const int im = (i == 0) ? nx - 1 : i - 1;
    const int jm = (j == 0) ? ny - 1 : j - 1;
    double dv = (F[0][c] - F[0][gidx(rd, im, j, k)]) * rd.idx[0]
                + (F[1][c] - F[1][gidx(rd, i, jm, k)]) * rd.idx[1];
    if (rd.dim == 3) {
        const int km = (k == 0) ? nz - 1 : k - 1;
        dv += (F[2][c] - F[2][gidx(rd, i, j, km)]) * rd.idx[2];
    }
    return dv;
}

// Charge-conservation residuals (App. B, Eq. gauss; Sec. 1 for the continuity equation of the
// Esirkepov deposit), with G = D.E - rho at every node:
//   out[0] = max |G|;
//   gref_out: G written per node (the reference the drift is measured from);
//   gref_in : out[1] = max |G - gref_in|;
//   rho_prev: out[2] = max |(rho - rho_prev) inv_dt + D.J|, J = F[6..8].
__global__ void __launch_bounds__(kBlock) k_gauss(const __grid_constant__ RunDev rd,
                                                  const double *rho, double *out,
                                                  const double *gref_in, double *gref_out,
                                                  const double *rho_prev, double inv_dt)
{
    double m = 0.0, md = 0.0, mc = 0.0;
    for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < rd.ncell;
         c += (int64_t)gridDim.x * blockDim.x) {
        const double g = div_node(rd, rd.F, c) - rho[c];
        m = fmax(m, fabs(g));
        if (gref_out) gref_out[c] = g;
        if (gref_in) md = fmax(md, fabs(g - gref_in[c]));
        if (rho_prev) mc = fmax(mc, fabs((rho[c] - rho_prev[c]) * inv_dt + div_node(rd, rd.F + 6, c)));
    }
    m = block_max(m);
    if (threadIdx.x == 0) atomic_max_nonneg(out, m);
    if (gref_in) {
        md = block_max(md);
        if (threadIdx.x == 0) atomic_max_nonneg(out + 1, md);
    }
    if (rho_prev) {
        mc = block_max(mc);
        if (threadIdx.x == 0) atomic_max_nonneg(out + 2, mc);
    }
}

// Fixed-point current of a deterministic run (RunDev::det) -> FP64, in place.
__global__ void __launch_bounds__(kBlock) k_det_finish(const __grid_constant__ RunDev rd)
{
    const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (c >= rd.ncell) return;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        long long *w = (long long *)rd.F[6 + a];
        if (rd.prec == 1) {
            rd.F[6 + a][c] = (double)w[c] * (rd.det_scale * 0x1p-40);
        } else {
            const double v = (double)w[c] + (double)(long long)rd.Jlo[a][c] * 0x1p-32;
            rd.F[6 + a][c] = v * (rd.det_scale * 0x1p-31);
        }
    }
}

// The padded FP32 current (RunDev::J32) -> F[6..8]: every grid node gets the sum, in FP64, of
// its periodic images in the padded buffer (padded index i + jp_lo + m n along each axis).
__global__ void __launch_bounds__(kBlock) k_j32_finish(const __grid_constant__ RunDev rd)
{
    const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (c >= rd.ncell) return;
    const int i = (int)(c % rd.n[0]);
    const int64_t r = c / rd.n[0];
    const int j = (int)(r % rd.n[1]), k = (int)(r / rd.n[1]);
    double s[3] = {0.0, 0.0, 0.0};
    for (int kp = (k + rd.jp_lo) % rd.n[2]; kp < rd.jp[2]; kp += rd.n[2])
        for (int jq = (j + rd.jp_lo) % rd.n[1]; jq < rd.jp[1]; jq += rd.n[1])
            for (int ip = (i + rd.jp_lo) % rd.n[0]; ip < rd.jp[0]; ip += rd.n[0]) {
                const int64_t q = ((int64_t)kp * rd.jp[1] + jq) * rd.jp[0] + ip;
#pragma unroll
                for (int a = 0; a < 3; ++a) s[a] += (double)rd.J32[a][q];
            }
#pragma unroll
    for (int a = 0; a < 3; ++a) rd.F[6 + a][c] = s[a];
}

inline unsigned grid_for(int64_t n)
{
    return (unsigned)((n + kBlock - 1) / kBlock);
}

}  // namespace

// B's part of an update.  first: the first step of a call (B at integer time -> half a step ahead);
// last: the last one (-> integer time); neither: from half a step behind to half a step ahead
static int yee_b_flags(const RunDev &rd, bool first, bool last)
{
    int flags = (first ? 0 : kYeeFinish) | (last ? 0 : kYeeStart);
    if (rd.prec == 1 && !first) flags |= kYeeShadow;
    if (rd.Bg[0] && !last) flags |= kYeeKeep;
    if (!last && !rd.J32[0]) flags |= kYeeZeroJ;
    return flags;
}

cudaError_t launch_yee_start(const RunDev &rd, cudaStream_t st)
{
    k_yee_b<<<grid_for(rd.ncell), kBlock, 0, st>>>(rd, 0.5 * rd.dt, yee_b_flags(rd, true, false));
    return cudaGetLastError();
}

int yee_step_launches(const RunDev &rd) { return rd.ncell <= kYeeOneCells ? 1 : 2; }

cudaError_t launch_yee_step(const RunDev &rd, bool shadow, bool last, cudaStream_t st)
{
    const int flags = yee_b_flags(rd, false, last);
    if (yee_step_launches(rd) == 1) {
        k_yee_eb<<<kYeeCtas, kBlock, 0, st>>>(rd, 0.5 * rd.dt, shadow ? 1 : 0, flags);
        return cudaGetLastError();
    }
    k_yee_e<<<grid_for(rd.ncell), kBlock, 0, st>>>(rd, shadow ? 1 : 0);
    k_yee_b<<<grid_for(rd.ncell), kBlock, 0, st>>>(rd, 0.5 * rd.dt, flags);
    return cudaGetLastError();
}

cudaError_t launch_shadow(const RunDev &rd, cudaStream_t st)
{
    k_shadow<<<grid_for(rd.ncell), kBlock, 0, st>>>(rd);
    return cudaGetLastError();
}

cudaError_t launch_pack(const RunDev &rd, int s, const double *x, int64_t xs, const double *u,
                        int64_t us, int64_t m, int64_t p0, cudaStream_t st)
{
    if (m == 0) return cudaSuccess;
    k_pack<<<grid_for(m), kBlock, 0, st>>>(rd, s, x, xs, u, us, m, p0);
    return cudaGetLastError();
}

cudaError_t launch_unpack(const RunDev &rd, int s, double *x, double *u, int64_t *cell,
                          int64_t m, int64_t p0, cudaStream_t st)
{
    if (m == 0) return cudaSuccess;
    k_unpack<<<grid_for(m), kBlock, 0, st>>>(rd, s, x, u, cell, m, p0);
    return cudaGetLastError();
}

// rho of all species at their current positions (FP64, into rho, cleared first)
static cudaError_t launch_rho(const RunDev &rd, double *rho, cudaStream_t st)
{
    cudaError_t e = cudaMemsetAsync(rho, 0, rd.ncell * sizeof(double), st);
    if (e != cudaSuccess) return e;
    int64_t n = 0;
    for (int s = 0; s < rd.nsp; ++s) n = rd.sp[s].n > n ? rd.sp[s].n : n;
    if (n == 0) return cudaSuccess;
    int sh = 0;
    while (!rd.slot_major && sh < 5 && (rd.ncell << (sh + 1)) <= n) ++sh;
    RhoWin win = rho_window(rd);
    // zeroing and adding the window costs as much as what it saves below about five to seven
    // contributions per node (pic_diag without it / with it, us: FP64 96x40x36 quadratic 4.8 per node
    // 238 / 235, 7.2 321 / 282, 9.6 406 / 333; 512x256 cubic 7.0 96 / 96, 14 120 / 109; FP32
    // 128x64x64 quadratic 5.2 402 / 418, 10.4 746 / 591): the line lies at eight for the average
    // tile, and at four for a single one of a run that takes windows
    double per = 1.0;
    for (int a = 0; a < rd.dim; ++a) per *= rd.l + 1;
    if ((double)n / rd.ntiles * per < 8.0 * win.nodes) win.nodes = 0;
    win.least = (int64_t)(4.0 * win.nodes / per);
    // enough blocks for a grid of few tiles, each of a thousand particles or more
    const int64_t want = (2048 + rd.ntiles - 1) / rd.ntiles, most = n / rd.ntiles / 1024;
    const int64_t parts = want < most ? want : most;
    const dim3 g((unsigned)(rd.ntiles * (parts > 1 ? parts : 1)), rd.nsp);
    const bool d3 = rd.dim == 3;
    auto k = rd.l == 1 ? (d3 ? k_rho<1, 3> : k_rho<1, 2>)
             : rd.l == 2 ? (d3 ? k_rho<2, 3> : k_rho<2, 2>)
             : rd.l == 3 ? (d3 ? k_rho<3, 3> : k_rho<3, 2>) : (d3 ? k_rho<4, 3> : k_rho<4, 2>);
    k<<<g, kBlock, (size_t)win.nodes * 8, st>>>(rd, win, sh, rho);
    return cudaGetLastError();
}

cudaError_t launch_diag(const RunDev &rd, double *out, double *rho, const double *gref,
                        const double *rho_prev, cudaStream_t st)
{
    cudaError_t e = cudaMemsetAsync(out, 0, 6 * sizeof(double), st);
    if (e != cudaSuccess) return e;
    const unsigned gr = 1024;
    k_field_energy<<<gr, kBlock, 0, st>>>(rd, out + 0);
    for (int s = 0; s < rd.nsp; ++s) k_kinetic<<<gr, kBlock, 0, st>>>(rd, s, out + 1);
    e = launch_rho(rd, rho, st);
    if (e != cudaSuccess) return e;
    k_gauss<<<gr, kBlock, 0, st>>>(rd, rho, out + 2, gref, nullptr, rho_prev, 1.0 / rd.dt);
    return cudaGetLastError();
}

cudaError_t launch_gauss_ref(const RunDev &rd, double *rho, double *gref, double *scratch,
                             cudaStream_t st)
{
    cudaError_t e = cudaMemsetAsync(scratch, 0, 3 * sizeof(double), st);
    if (e != cudaSuccess) return e;
    e = launch_rho(rd, rho, st);
    if (e != cudaSuccess) return e;
    k_gauss<<<1024, kBlock, 0, st>>>(rd, rho, scratch, nullptr, gref, nullptr, 0.0);
    return cudaGetLastError();
}

cudaError_t launch_det_finish(const RunDev &rd, cudaStream_t st)
{
    k_det_finish<<<grid_for(rd.ncell), kBlock, 0, st>>>(rd);
    return cudaGetLastError();
}

cudaError_t launch_j32_finish(const RunDev &rd, cudaStream_t st)
{
    k_j32_finish<<<grid_for(rd.ncell), kBlock, 0, st>>>(rd);
    return cudaGetLastError();
}

cudaError_t launch_load_plasma(const RunDev &rd, int s, const LoadKeys &keys, int64_t per_cell,
                               double gamma, double u_th, double theta, int64_t n, cudaStream_t st)
{
    if (n == 0) return cudaSuccess;
    k_load_plasma<<<grid_for(n), kBlock, 0, st>>>(rd, s, keys, per_cell, gamma, u_th, theta, n);
    return cudaGetLastError();
}


}  // namespace pic
