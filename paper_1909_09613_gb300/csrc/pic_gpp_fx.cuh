// The fused particle pass of the plain FP64 form in 2D: weights, gather and current products in
// 62-bit fixed point (pic_fixed.cuh), Boris push and move in FP64.
//
// What bounds it: an FP64 evaluation is bound by the FP64 pipe (2 operations per clock and SM, 410
// of them per particle for cubic splines).  In fixed point 78 stay there (Boris, move, the
// interpolated fields' conversion) and the rest goes to the integer units; the pipes are then
// about equally loaded (FP64 39%, wide multiplier 54%, ALU 43% of their cycles, 52% of the issue
// slots) and the warps wait on fixed-latency dependencies.  512x256, cubic, 64 per cell: 7.39 ->
// 2.70 ms per pass over 8.4 M particles (now 2.76); 255x130, quartic, 16 per cell: 0.72 -> 0.34 ms.  Three
// CTAs per SM at 80 registers spill (2.90 ms).  The old-position weights, which the FP64
// evaluation read from a per-particle cache (128 B per particle and step), are evaluated.
//
// The gather's signed, rounded sums and the search for tiles whose fields one scale does not resolve
// cost 2 to 9% of it (cubic, 512x256 at 32 and 8 of a species per cell 3.11 -> 3.18 and 0.848 -> 0.905 ms,
// 64x32 at 8 37.6 -> 41.1 us, most of it the search) against biased sums of truncated products, which
// gave a particle a one-signed field of 2^-54 of the tile's largest where its own was zero, and a node
// below 2^-6 of the largest fewer bits than FP64.
#pragma once
#include "pic_fixed.cuh"
#include "pic_gpp_kernels.cuh"

namespace pic {

// Shared-memory layout of a staged tile: the fields in fixed point (field_fixed, units of 2^(E - 60)
// with 2^E above the component's largest magnitude in the tile) as Parts, or, in an exact tile, in
// FP64.
//   pa = (E1, B2), pb = (E2, B1) (16 bytes a node), e3, b3 (8 bytes), then the masks of small
//   fields (mask_words)
struct StageFx {
    uint4 *pa, *pb;
    uint2 *e3, *b3;
    TTable *tt;
    int *emax;   // high word of the largest magnitude, per component (E1..E3, B1..B3)
    int *exact;  // the tile's fields are staged in FP64 and gathered in FP64
    uint32_t *mask;
};

// Warps of a block, two blocks per SM.  Quartic splines spill at the 128 registers of 16 warps per
// SM as they do at the 96 of 20, and the extra warps hide more of the wait (8 / 10 warps, us: 255x130
// at 2, 8 and 32 of a species per cell 105 / 101, 386 / 348, 1334 / 1252; 512x256 at 4 and 16 675 / 657,
// 2523 / 2445; 1024x512 at 16 9580 / 9602; the other way 128x64 at 8 90 / 97, 512x256 at 32 4766 /
// 4952).  Deterministic runs spill with ten warps only and are faster with them all the same (255x130
// at 8 734 / 715, 512x256 at 32 9594 / 9499).  Cubic splines do not spill and lose (134M particles
// 40.7 -> 42.5 ms).
__host__ __device__ constexpr int fx_warps(int l) { return l == 4 ? 10 : 8; }

constexpr int kFxHead = 2 * sizeof(TTable) + 32;  // tables, exponents and the exact flag

__host__ __device__ inline size_t stage_fx_bytes(int64_t nodes)
{
    return (kFxHead + 15) / 16 * 16 + (size_t)nodes * 48;
}

// Words of the masks of small fields: per component and row one bit a node, set where it is small or
// zero.
__host__ __device__ inline int64_t mask_words(const RunDev &rd)
{
    return 6 * (int64_t)rd.reg[1] * ((rd.reg[0] + 31) / 32);
}

// Shared memory of a launch: with the masks where the device has room for them (without them every
// tile is exact).
__host__ __device__ inline size_t stage_fx_launch_bytes(const RunDev &rd)
{
    const size_t b = stage_fx_bytes(rd.reg_nodes), m = b + 4 * mask_words(rd);
    return m <= 227 * 1024 ? m : b;
}

__device__ __forceinline__ StageFx stage_fx_carve(char *smem, const RunDev &rd)
{
    const size_t nodes = rd.reg_nodes;
    StageFx s;
    s.tt = (TTable *)smem;
    s.emax = (int *)(smem + 2 * sizeof(TTable));
    s.exact = s.emax + 6;
    char *p = smem + (kFxHead + 15) / 16 * 16;
    s.pa = (uint4 *)p; p += nodes * 16;
    s.pb = (uint4 *)p; p += nodes * 16;
    s.e3 = (uint2 *)p; p += nodes * 8;
    s.b3 = (uint2 *)p; p += nodes * 8;
    s.mask = stage_fx_launch_bytes(rd) > stage_fx_bytes(nodes) ? (uint32_t *)p : nullptr;
    return s;
}

__device__ __forceinline__ double field_at(const RunDev &rd, int c, int64_t g)
{
    return __ldg((c < 3 ? rd.F[c] : rd.Bg[c - 3]) + g);
}

// A node's six fields into the stage, v(c) the 8 bytes of component c.
template <typename V>
__device__ __forceinline__ void stage_node(const StageFx &st, int n, const V &v)
{
    const uint2 e1 = v(0), e2 = v(1), b1 = v(3), b2 = v(4);
    st.pa[n] = make_uint4(e1.x, e1.y, b2.x, b2.y);
    st.pb[n] = make_uint4(e2.x, e2.y, b1.x, b1.y);
    st.e3[n] = v(2);
    st.b3[n] = v(5);
}

// Whether a staged field (fixed point) is zero, which field_fixed makes of zero alone.
__device__ __forceinline__ bool staged_zero(const StageFx &st, int c, int n)
{
    const uint4 v = c == 0 || c == 4 ? st.pa[n] : st.pb[n];
    if (c == 2 || c == 5) {
        const uint2 w = c == 2 ? st.e3[n] : st.b3[n];
        return (w.x | w.y) == 0;
    }
    return c < 2 ? (v.x | v.y) == 0 : (v.z | v.w) == 0;
}

// Whether some stencil of the tile may hold fields that are all small and not all zero: an
// (L + 1) x (L + 1) window (no stencil is smaller) of small nodes with one that is not zero.
// Thread by thread over component, row and mask word; components of zeros alone are left out.
template <int L>
__device__ __forceinline__ bool small_window(const RunDev &rd, const StageFx &st)
{
    const int RX = rd.reg[0], RY = rd.reg[1], mw = (RX + 31) / 32, rows = RY - L;
    for (int i = threadIdx.x; i < 6 * rows * mw; i += blockDim.x) {
        const int w = i % mw, ry = i / mw % rows, c = i / mw / rows;
        if (st.emax[c] == 0) continue;
        uint64_t s = ~(uint64_t)0;
#pragma unroll
        for (int k = 0; k <= L; ++k) {
            const uint32_t *m = st.mask + (c * RY + ry + k) * mw + w;
            s &= m[0] | (w + 1 < mw ? (uint64_t)m[1] << 32 : 0);
        }
        uint64_t all = s;  // bit b: the window of columns b .. b + L is small
#pragma unroll
        for (int k = 1; k <= L; ++k) all &= s >> k;
        for (uint32_t left = (uint32_t)all; left; left &= left - 1) {
            const int rx = 32 * w + __ffs(left) - 1;
            for (int k = 0; k < (L + 1) * (L + 1); ++k)
                if (!staged_zero(st, c, (ry + k / (L + 1)) * RX + rx + k % (L + 1))) return true;
        }
    }
    return false;
}

// Stage the fields of the tile at (x0, y0): the largest exponent of every component over the staged
// region first, then the fields in its units (the second read comes from L1 or L2).  One warp per row.
// A unit is 2^-60 of the scale, so a stencil whose fields all lie below 2^-7 of it would be summed
// with less than FP64's relative precision, and a non-finite or very small largest field gives no
// scale: such a tile is staged again in FP64 and gathered in FP64 (st.exact).  Smooth and noisy fields
// alike hold no such stencil (a window of l + 1 nodes squared crosses a zero, but is not that flat);
// the edges of pulses and of regions without fields do.
template <int L, int W>
__device__ inline void stage_fx_load(const RunDev &rd, const StageFx &st, int x0, int y0)
{
    const int RX = rd.reg[0], RY = rd.reg[1], lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < (int)(2 * sizeof(TTable) / sizeof(int)); i += blockDim.x)
        ((int *)st.tt)[i] = ((const int *)rd.tt)[i];
    if (threadIdx.x < 7) st.emax[threadIdx.x] = 0;  // (exact among them)
    __syncthreads();
    int em[6] = {0, 0, 0, 0, 0, 0};
    for (int ry = warp; ry < RY; ry += W) {
        const int64_t row = (int64_t)wrap_near(y0 - rd.pre[1] + ry, rd.n[1]) * rd.n[0];
        for (int rx = lane; rx < RX; rx += 32) {
            const int64_t g = row + wrap_near(x0 - rd.pre[0] + rx, rd.n[0]);
#pragma unroll
            for (int c = 0; c < 6; ++c) {
                const double f = field_at(rd, c, g);
                em[c] = max(em[c], (__double2hiint(f) & 0x7fffffff) | (__double2loint(f) != 0 ? 1 : 0));
            }
        }
    }
#pragma unroll
    for (int c = 0; c < 6; ++c) {
        const int m = __reduce_max_sync(0xffffffffu, em[c]);
        if (lane == 0 && m > 0) atomicMax(st.emax + c, m);
    }
    __syncthreads();
    bool exact = st.mask == nullptr;
#pragma unroll
    for (int c = 0; c < 6; ++c) {
        em[c] = st.emax[c];
        exact = exact || em[c] >= 0x7ff00000 || (em[c] > 0 && em[c] < 64 << 20);
        em[c] &= 0x7ff00000;
    }
    if (!exact) {
        const int mw = (RX + 31) / 32;
        for (int ry = warp; ry < RY; ry += W) {
            const int64_t row = (int64_t)wrap_near(y0 - rd.pre[1] + ry, rd.n[1]) * rd.n[0];
            for (int w = 0; w < mw; ++w) {
                const int rx = 32 * w + lane;
                const bool in = rx < RX;
                const int64_t g = row + wrap_near(x0 - rd.pre[0] + (in ? rx : 0), rd.n[0]);
                uint32_t small[6];
                uint2 p[6];
#pragma unroll
                for (int c = 0; c < 6; ++c) {
                    const double f = field_at(rd, c, g);
                    small[c] = __ballot_sync(0xffffffffu, in && (__double2hiint(f) & 0x7fffffff)
                                                                    < em[c] - ((kSmallField - 1) << 20));
                    const Parts q = parts(field_fixed((uint64_t)__double_as_longlong(f), em[c] >> 20));
                    p[c] = make_uint2((uint32_t)q.h, (uint32_t)q.l);
                }
                if (in) stage_node(st, ry * RX + rx, [&](int c) { return p[c]; });
                if (lane == 0) {
#pragma unroll
                    for (int c = 0; c < 6; ++c) st.mask[(c * RY + ry) * mw + w] = small[c];
                }
            }
        }
        __syncthreads();
        exact = __syncthreads_or(small_window<L>(rd, st));
    }
    if (!exact) return;
    if (threadIdx.x == 0) *st.exact = 1;
    for (int ry = warp; ry < RY; ry += W) {
        const int64_t row = (int64_t)wrap_near(y0 - rd.pre[1] + ry, rd.n[1]) * rd.n[0];
        for (int rx = lane; rx < RX; rx += 32) {
            const int64_t g = row + wrap_near(x0 - rd.pre[0] + rx, rd.n[0]);
            stage_node(st, ry * RX + rx, [&](int c) {
                const double f = field_at(rd, c, g);
                return make_uint2((uint32_t)__double2loint(f), (uint32_t)__double2hiint(f));
            });
        }
    }
}

// The FP64 value of a weight.
__device__ __forceinline__ double weight_value(uint64_t v)
{
    return __longlong_as_double((int64_t)weight_bits(v));
}

__device__ __forceinline__ double weight_value(const Parts &w)
{
    return weight_value((uint64_t)((int64_t)w.h * ((int64_t)1 << 32) + w.l));
}

// The FP64 value of an interpolated field; emax as staged, at least 64 << 20 (or a field of zeros).
__device__ __forceinline__ double field_value(int64_t v, int emax)
{
    return (double)v * __hiloint2double((emax & 0x7ff00000) - ((60 - 1) << 20), 0);
}

// A pair of fields (first: parts x, y; second: z, w) with weights wx along x, wy along y.
template <int NX, int NY>
__device__ __forceinline__ void gather_pair_fx(const uint4 *f, int RX, const Parts *wx,
                                               const Parts *wy, int64_t &a, int64_t &b)
{
    GatherSum A, B;
    A.zero();
    B.zero();
#pragma unroll 1
    for (int j = 0; j < NY; ++j) {
        GatherSum ra, rb;
        ra.zero();
        rb.zero();
#pragma unroll
        for (int i = 0; i < NX; ++i) {
            const uint4 v = f[j * RX + i];
            ra.add(wx[i], (int)v.x, (int)v.y);
            rb.add(wx[i], (int)v.z, (int)v.w);
        }
        const Parts la = parts(ra.value()), lb = parts(rb.value());
        A.add(wy[j], la.h, la.l);
        B.add(wy[j], lb.h, lb.l);
    }
    a = A.value();
    b = B.value();
}

template <int NX, int NY>
__device__ __forceinline__ int64_t gather_one_fx(const uint2 *f, int RX, const Parts *wx,
                                                 const Parts *wy)
{
    GatherSum A;
    A.zero();
#pragma unroll 1
    for (int j = 0; j < NY; ++j) {
        GatherSum r;
        r.zero();
#pragma unroll
        for (int i = 0; i < NX; ++i) {
            const uint2 v = f[j * RX + i];
            r.add(wx[i], (int)v.x, (int)v.y);
        }
        const Parts l = parts(r.value());
        A.add(wy[j], l.h, l.l);
    }
    return A.value();
}

// One field of an exact tile, in FP64: p its 8 bytes at the stencil's first node, stride those of a
// node.
template <int NX, int NY>
__device__ __forceinline__ double gather_exact(const char *p, int stride, int RX, const Parts *wx,
                                               const Parts *wy)
{
    double dx[NX], acc = 0.0;
#pragma unroll
    for (int i = 0; i < NX; ++i) dx[i] = weight_value(wx[i]);
#pragma unroll 1
    for (int j = 0; j < NY; ++j) {
        double r = 0.0;
#pragma unroll
        for (int i = 0; i < NX; ++i) r += dx[i] * *(const double *)(p + (size_t)(j * RX + i) * stride);
        acc += weight_value(wy[j]) * r;
    }
    return acc;
}

// One contribution (v in U62, its scale's sign and exponent in top) added to a node of the
// global current.
template <bool DET>
__device__ __forceinline__ void add_current_fx(double *J, unsigned long long *Jlo, int g,
                                               uint64_t v, uint32_t top, double dinv)
{
    if constexpr (DET) {
        if (v == 0) return;
        unsigned long long hi, lo;
        det_words64(__longlong_as_double((int64_t)to_fp64_bits(v, top)), dinv, hi, lo);
        atomicAdd((unsigned long long *)(J + g), hi);
        atomicAdd(Jlo + g, lo);
    } else {
        red_fixed(J + g, v, top);
    }
}

// The Esirkepov window of one particle added to the global FP64 current (reductions performed
// by L2).  With S0, S1 the old and new weights of an axis:
//   W_x = P_x (S0y + S1y) / 2, W_y = P_y (S0x + S1x) / 2 (P: prefix sums of S1 - S0), and
//   W_z = S0y (S0x / 3 + S1x / 6) + S1y (S0x / 6 + S1x / 3)
// (the form of deposit_lane with DS = S1 - S0 written out), whose factors are all non-negative.
// The mantissas of the scales kx, ky, kz go into the y factors, their exponents into the
// conversion of every product.  wide = false when no lane of the warp changed its y window base:
// row l + 1 then carries zeros.  The rows are a rolled loop (their factors in local memory), as
// the gather's are: unrolled, the kernel's code outgrew the instruction cache and waiting for
// instructions was the largest stall (2.1 of 8.8 cycles per issue; 512x256 as above 3.22 -> 2.73
// ms).  Taking J1 and J2 as FP64 products of converted factors instead measured the same.
template <int L, bool DET>
__device__ __forceinline__ void deposit_fx(const Hot2D &h, int gx0, int gy0, double kx, double ky,
                                           double kz, const AxisS62<L> &Sx, const AxisS62<L> &Sy,
                                           bool upx, bool upy, bool wide)
{
    const Scale62 mx = scale62((uint64_t)__double_as_longlong(kx));
    const Scale62 my = scale62((uint64_t)__double_as_longlong(ky));
    const Scale62 mz = scale62((uint64_t)__double_as_longlong(kz));
    // the prefix sums are negative for a move up
    const uint32_t topx = mx.top ^ (upx ? 0x80000000u : 0u);
    const uint32_t topy = my.top ^ (upy ? 0x80000000u : 0u);
    uint64_t ys[4][L + 2];  // (S0y + S1y) / 2, |P_y|, S0y, S1y
    {
        uint64_t qy[L + 1];
        prefix62<L>(Sy, upy, qy);
#pragma unroll
        for (int k = 0; k < L + 2; ++k) {
            ys[0][k] = (Sy.s0[k] + Sy.s1[k]) >> 1;
            ys[1][k] = k <= L ? qy[k <= L ? k : 0] : 0;
            ys[2][k] = Sy.s0[k];
            ys[3][k] = Sy.s1[k];
        }
    }
    Limbs qx[L + 1], Ax[L + 2], Bx[L + 2], Cx[L + 2];
    {
        uint64_t q[L + 1];
        prefix62<L>(Sx, upx, q);
        const Limbs sixth = limbs(frac62(1, 6));
#pragma unroll
        for (int k = 0; k <= L; ++k) qx[k] = limbs(q[k]);
#pragma unroll
        for (int k = 0; k < L + 2; ++k) {
            const uint64_t a = mul62(limbs(Sx.s0[k]), sixth), b = mul62(limbs(Sx.s1[k]), sixth);
            Ax[k] = limbs((Sx.s0[k] + Sx.s1[k]) >> 1);
            Bx[k] = limbs(a + 2 * b);
            Cx[k] = limbs(2 * a + b);
        }
    }
    const Limbs lmx = limbs(mx.m), lmy = limbs(my.m), lmz = limbs(mz.m);
    int gx[L + 2];
#pragma unroll
    for (int k = 0; k < L + 2; ++k) gx[k] = wrap_near(gx0 + k, h.n0);
    const int rows = wide ? L + 2 : L + 1;
#pragma unroll 1
    for (int b = 0; b < rows; ++b) {
        const int gy = wrap_near(gy0 + b, h.n1) * h.n0;  // (at most 2^30 cells)
        const Limbs ay = limbs(mul62(limbs(ys[0][b]), lmx));
        const Limbs py = limbs(mul62(limbs(ys[1][b]), lmy));
        const Limbs z0 = limbs(mul62(limbs(ys[2][b]), lmz));
        const Limbs z1 = limbs(mul62(limbs(ys[3][b]), lmz));
#pragma unroll
        for (int a = 0; a < L + 2; ++a) {
            const int g = gy + gx[a];
            if (a <= L)
                add_current_fx<DET>(h.J0, h.Jlo0, g, mul62(qx[a <= L ? a : 0], ay), topx, h.dinv64);
            add_current_fx<DET>(h.J1, h.Jlo1, g, mul62(Ax[a], py), topy, h.dinv64);
            const uint64_t x = wide_mul(z0.h, Cx[a].l) + wide_mul(z0.l, Cx[a].h)
                               + wide_mul(z1.h, Bx[a].l) + wide_mul(z1.l, Bx[a].h);
            add_current_fx<DET>(h.J2, h.Jlo2, g,
                                wide_mul(z0.h, Cx[a].h) + wide_mul(z1.h, Bx[a].h) + (x >> 31),
                                mz.top, h.dinv64);
        }
    }
}

// Move one axis in cell units: x + delta rounded once to FP64, wrapped into [0, n).  Returns the
// cell shift in {-1, 0, 1} relative to cell c; cn, f: the new cell and offset, decoded from the
// stored value, so that the next step's old-position weights equal this step's new-position
// ones.  A non-finite move (a non-finite momentum) leaves the particle where it is; its
// momentum reports it.
__device__ __forceinline__ int move_axis_fx(double &x, double delta, int c, int n, int &cn,
                                            uint64_t &f)
{
    double X = x + delta;
    if ((__double2hiint(X) & 0x7ff00000) == 0x7ff00000) X = x;
    const double N = (double)n;
    const bool lo = __double2hiint(X) < 0;
    const bool up = !lo && __double_as_longlong(X) >= __double_as_longlong(N);
    X += lo ? N : (up ? -N : 0.0);
    uint64_t bits = (uint64_t)__double_as_longlong(X);
    if ((int64_t)bits < 0) bits = 0;  // -0
    cn = min(decode_position(bits, f), n);
    int sh = cn + (lo ? -n : (up ? n : 0)) - c;
    if (cn >= n) {  // -tiny + n rounded up to n
        cn = 0;
        f = 0;
        bits = 0;
    }
    if (sh > 1) {  // x + delta rounded up to the cell two above: the top of the cell above
        sh = 1;
        f = ~(uint64_t)0;
    }
    if (sh < -1) sh = -1;
    x = __longlong_as_double((int64_t)bits);
    return sh;
}

// One particle per lane.  Called by all 32 lanes of a warp together; lanes with act == false
// carry no particle.
template <int L, int KT, bool DET>
__device__ __forceinline__ void particle_fx(const Hot2D &h, const HotSp<double> &hs,
                                            const StageFx &st, int64_t p, bool act, int x0, int y0)
{
    double x[2] = {0.0, 0.0}, u[3] = {0.0, 0.0, 0.0};
    int c[2], lc[2] = {0, 0};
    uint64_t f[2];
    if (act) {
        x[0] = __ldg((const double *)hs.pos0 + p);
        x[1] = __ldg((const double *)hs.pos1 + p);
        u[0] = __ldg((const double *)hs.mom0 + p);
        u[1] = __ldg((const double *)hs.mom1 + p);
        u[2] = __ldg((const double *)hs.mom2 + p);
        // in [0, n) by construction; the clamp keeps a non-finite position's index valid
        c[0] = min(decode_position((uint64_t)__double_as_longlong(x[0]), f[0]), h.n0 - 1);
        c[1] = min(decode_position((uint64_t)__double_as_longlong(x[1]), f[1]), h.n1 - 1);
        const bool okx = local_coord(c[0], x0, h.tile0, h.drift0, h.n0, lc[0]);
        const bool oky = local_coord(c[1], y0, h.tile1, h.drift1, h.n1, lc[1]);
        if (!(okx && oky)) {
            set_err(h.err, 1);
            act = false;
        }
    }
    if (!act) {  // a harmless stand-in at the tile origin; it deposits and stores nothing
        x[0] = x[1] = 0.0;
        u[0] = u[1] = u[2] = 0.0;
        c[0] = x0;
        c[1] = y0;
        f[0] = f[1] = (uint64_t)1 << 63;
        lc[0] = lc[1] = 0;
    }
    const int RX = h.RX;
    const int sx = lc[0] + h.pre0, sy = lc[1] + h.pre1;

    // ---- gather (Eq. interpolation-EB-real-mod; MC when the tables hold W_l) ----
    double E[3], B[3];
    {
        Parts wh[2][L + 1], wt[2][KT];
        int bh[2], bt[2];
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            uint64_t psi, w[L + 1], t[KT];
            bh[a] = spline_base62<L>(f[a], true, psi);
            bspline62<L>(psi, w);
            bt[a] = ttable_weights62<L, KT>(st.tt[a], f[a], t);
#pragma unroll
            for (int k = 0; k <= L; ++k) wh[a][k] = parts((int64_t)w[k]);
#pragma unroll
            for (int k = 0; k < KT; ++k) wt[a][k] = parts((int64_t)t[k]);
        }
        const int xh = sx + bh[0], xt = sx + bt[0];
        const int yh = (sy + bh[1]) * RX, yt = (sy + bt[1]) * RX;
        const uint4 *pa = st.pa + yt + xh, *pb = st.pb + yh + xt;
        const uint2 *p3 = st.e3 + yt + xt, *q3 = st.b3 + yh + xh;
        if (*st.exact) {  // the whole CTA
            E[0] = gather_exact<L + 1, KT>((const char *)pa, 16, RX, wh[0], wt[1]);
            B[1] = gather_exact<L + 1, KT>((const char *)pa + 8, 16, RX, wh[0], wt[1]);
            E[1] = gather_exact<KT, L + 1>((const char *)pb, 16, RX, wt[0], wh[1]);
            B[0] = gather_exact<KT, L + 1>((const char *)pb + 8, 16, RX, wt[0], wh[1]);
            E[2] = gather_exact<KT, KT>((const char *)p3, 8, RX, wt[0], wt[1]);
            B[2] = gather_exact<L + 1, L + 1>((const char *)q3, 8, RX, wh[0], wh[1]);
        } else {
            int64_t v[6];
            gather_pair_fx<L + 1, KT>(pa, RX, wh[0], wt[1], v[0], v[4]);  // E1, B2
            gather_pair_fx<KT, L + 1>(pb, RX, wt[0], wh[1], v[1], v[3]);  // E2, B1
            v[2] = gather_one_fx<KT, KT>(p3, RX, wt[0], wt[1]);
            v[5] = gather_one_fx<L + 1, L + 1>(q3, RX, wh[0], wh[1]);
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                E[k] = field_value(v[k], st.emax[k]);
                B[k] = field_value(v[3 + k], st.emax[3 + k]);
            }
        }
    }

    // ---- Boris push and move ----
    const double ig = boris<double>(hs.qmdt_half, E, B, u);
    int cn[2], sh[2];
    uint64_t fn[2];
    sh[0] = move_axis_fx(x[0], h.dtt0 * u[0] * ig, c[0], h.n0, cn[0], fn[0]);
    sh[1] = move_axis_fx(x[1], h.dtt1 * u[1] * ig, c[1], h.n1, cn[1], fn[1]);

    // ---- Esirkepov deposit ----
    AxisS62<L> Sx, Sy;
    axis_shapes62<L>(f[0], fn[0], sh[0], Sx);
    axis_shapes62<L>(f[1], fn[1], sh[1], Sy);
    const bool upx = sh[0] > 0 || (sh[0] == 0 && fn[0] >= f[0]);
    const bool upy = sh[1] > 0 || (sh[1] == 0 && fn[1] >= f[1]);
    double kz = hs.kz * u[2] * ig;
    const int gx0 = x0 - h.pre0 + sx + Sx.wb, gy0 = y0 - h.pre1 + sy + Sy.wb;
    if (act && (__double2hiint(kz) & 0x7ff00000) == 0x7ff00000) {
        // a non-finite velocity: its current is reported as such, at the first node; a deterministic
        // run's current holds integers and reports it in the error word
        if (DET) set_err(h.err, 2);
        else atomicAdd(h.J2 + (int64_t)wrap_near(gy0, h.n1) * h.n0 + wrap_near(gx0, h.n0), kz);
        kz = 0.0;
    }
    // a drift along x1 rarely moves the y window: skip its empty last row warp-uniformly
    const bool wide = __any_sync(0xffffffffu, act && Sy.wide);
    if (!act) return;
    deposit_fx<L, DET>(h, gx0, gy0, hs.kx0, hs.kx1, kz, Sx, Sy, upx, upy, wide);

    // ---- store ----
    ((double *)hs.pos0)[p] = x[0];
    ((double *)hs.pos1)[p] = x[1];
    ((double *)hs.mom0)[p] = u[0];
    ((double *)hs.mom1)[p] = u[1];
    ((double *)hs.mom2)[p] = u[2];
}

// All particles of one tile, or the share blockIdx.y of gridDim.y of every species' (tile_parts).
template <int L, int KT, bool DET>
__device__ void tile_fx(const RunDev &rd, char *smem, int64_t tile)
{
    constexpr int W = fx_warps(L);
    const StageFx st = stage_fx_carve(smem, rd);
    const int tx = (int)(tile % rd.ntile[0]), ty = (int)(tile / rd.ntile[0]);
    const int x0 = tx * rd.tile[0], y0 = ty * rd.tile[1];
    stage_fx_load<L, W>(rd, st, x0, y0);
    const Hot2D h = make_hot2d(rd);
    __syncthreads();
    for (int s = 0; s < rd.nsp; ++s) {
        const SpeciesDev &sp = rd.sp[s];
        const HotSp<double> hs = make_hotsp<double>(sp);
        int64_t a = sp.tile_start[tile], b = sp.tile_start[tile + 1];
        split_range(GridSplit(), a, b);
        // warp-uniform trip count: a warp's lanes take 32 consecutive particles.  The species
        // start at different warps, so that a part of few particles does not queue its species
        // one behind the other on the first warps.
        const int w = ((threadIdx.x >> 5) + s * (W / 2)) % W;
        for (int64_t q = a + 32 * w; q < b; q += blockDim.x) {
            const int64_t p = q + (threadIdx.x & 31);
            if (p + blockDim.x < b) prefetch_particle<double>(hs, p + blockDim.x);
            particle_fx<L, KT, DET>(h, hs, st, p, p < b, x0, y0);
        }
    }
}

}  // namespace pic
