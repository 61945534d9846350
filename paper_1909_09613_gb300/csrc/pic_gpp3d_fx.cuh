// The fused particle pass of the plain FP64 form in 3D: weights and current products in 62-bit
// fixed point (pic_fixed.cuh), gather, Boris push and move in FP64.
//
// What bounds it: evaluated in FP64 throughout, a particle of quadratic splines takes about 650
// operations of the FP64 pipe (2 per clock and SM), which set the time.  The weights and the
// current products are bounded by 1 and go to the integer units; the gather (234 operations)
// stays in FP64, because its fields, read through L1 at any distance from the sorted tile, share
// no scale.  96x40x36, quadratic, 8 per cell (1.1 M particles): 1.67 -> 1.09 ms per pass.
#pragma once
#include "pic_gpp3d.cuh"
#include "pic_gpp_fx.cuh"

namespace pic {

// One staggered field component at a particle through L1 from the global field: sum over the
// stencil nodes of wz[c] wy[b] wx[a] F(zi[c], yi[b], xi[a]), wrapped node indices per axis.
template <int NA, int NB, int NC>
__device__ __forceinline__ double gather3_global(const double *f, int nx, int ny, const int *xi,
                                                 const int *yi, const int *zi, const double *wx,
                                                 const double *wy, const double *wz)
{
    double acc = 0.0;
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        double r2 = 0.0;
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            const double *row = f + (zi[c] * ny + yi[b]) * nx;  // (at most 2^30 cells)
            double r1 = 0.0;
#pragma unroll
            for (int a = 0; a < NA; ++a) r1 += wx[a] * __ldg(row + xi[a]);
            r2 += wy[b] * r1;
        }
        acc += wz[c] * r2;
    }
    return acc;
}

// The Esirkepov window of one particle added to the global FP64 current (reductions performed by
// L2).  With S0, S1 the old and new weights of an axis, P the prefix sums of S1 - S0 and (a, b, c)
// the axes in cyclic order,
//   J_a(ka, kb, kc) = kx_a P_a[ka] (S0_b[kb] G0_c[kc] + S1_b[kb] G1_c[kc]),
//   G0 = S0 / 3 + S1 / 6, G1 = S0 / 6 + S1 / 3
// (Sec. 1's W_a with DS = S1 - S0 written out), whose factors are all non-negative.  Along an
// axis on which no lane of the warp moved its window base (mv false), node l + 1 of every window
// and the prefix sum over the whole window are exact zeros: the warp skips those rows together.
// The components and the rows along b are rolled loops (factors in local memory), so that the
// kernel's code stays in the instruction cache.
template <int L, bool DET>
__device__ __forceinline__ void deposit3_fx(const RunDev &rd, const SpeciesDev &sp, const int *g0,
                                            const AxisS62<L> *S, const bool *up, const bool *mv)
{
    uint64_t s0[3][L + 2], s1[3][L + 2], h0[3][L + 2], h1[3][L + 2], q[3][L + 1];
    int off[3][L + 2];
    uint32_t top[3];
    const Limbs sixth = limbs(frac62(1, 6));
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const Scale62 k = scale62((uint64_t)__double_as_longlong(sp.kx[a]));
        top[a] = k.top ^ (up[a] ? 0x80000000u : 0u);  // the prefix sums are negative for a move up
        uint64_t t[L + 1];
        prefix62<L>(S[a], up[a], t);
        const int stride = a == 0 ? 1 : (a == 1 ? rd.n[0] : rd.n[0] * rd.n[1]);
#pragma unroll
        for (int i = 0; i <= L; ++i) q[a][i] = mul62(limbs(t[i]), limbs(k.m));
#pragma unroll
        for (int i = 0; i < L + 2; ++i) {
            const uint64_t x = mul62(limbs(S[a].s0[i]), sixth), y = mul62(limbs(S[a].s1[i]), sixth);
            s0[a][i] = S[a].s0[i];
            s1[a][i] = S[a].s1[i];
            h0[a][i] = 2 * x + y;
            h1[a][i] = x + 2 * y;
            off[a][i] = wrap_near(g0[a] + i, rd.n[a]) * stride;
        }
    }
#pragma unroll 1
    for (int a = 0; a < 3; ++a) {
        const int b = a == 2 ? 0 : a + 1, c = a == 0 ? 2 : a - 1;
        double *J = rd.F[6 + a];
        unsigned long long *Jlo = rd.Jlo[a];
        Limbs p[L + 1];
#pragma unroll
        for (int i = 0; i <= L; ++i) p[i] = limbs(q[a][i]);
        const int nb = L + 1 + (mv[b] ? 1 : 0);
        const bool mc = mv[c], ma = mv[a];
        const uint32_t ta = top[a];
#pragma unroll 1
        for (int kb = 0; kb < nb; ++kb) {
            const Limbs x = limbs(s0[b][kb]), y = limbs(s1[b][kb]);
            const int gb = off[b][kb];
#pragma unroll
            for (int kc = 0; kc < L + 2; ++kc) {
                if (kc == L + 1 && !mc) break;
                const Limbs u = limbs(h0[c][kc]), v = limbs(h1[c][kc]);
                const uint64_t cross = wide_mul(x.h, u.l) + wide_mul(x.l, u.h)
                                       + wide_mul(y.h, v.l) + wide_mul(y.l, v.h);
                const Limbs perp = limbs(wide_mul(x.h, u.h) + wide_mul(y.h, v.h) + (cross >> 31));
                const int g = gb + off[c][kc];
#pragma unroll
                for (int ka = 0; ka <= L; ++ka) {
                    if (ka == L && !ma) break;
                    add_current_fx<DET>(J, Jlo, g + off[a][ka], mul62(p[ka], perp), ta,
                                        rd.det_inv64);
                }
            }
        }
    }
}

// One particle per lane.  Called by all 32 lanes of a warp together; lanes with act == false
// carry no particle.
template <int L, int KT, bool DET>
__device__ __forceinline__ void particle3_fx(const RunDev &rd, const SpeciesDev &sp, int64_t p,
                                             bool act)
{
    double x[3] = {0.0, 0.0, 0.0}, u[3] = {0.0, 0.0, 0.0};
    if (act) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            x[a] = __ldg((const double *)sp.pos[a] + p);
            u[a] = __ldg((const double *)sp.mom[a] + p);
        }
    }
    int c[3];
    uint64_t f[3];
#pragma unroll
    for (int a = 0; a < 3; ++a)  // in [0, n) by construction; the clamp keeps any index valid
        c[a] = min(decode_position((uint64_t)__double_as_longlong(x[a]), f[a]), rd.n[a] - 1);

    // ---- gather (Eq. interpolation-EB-real-mod in 3D):
    // E1: W T T ; E2: T W T ; E3: T T W ; B1: T W W ; B2: W T W ; B3: W W T (x, y, z)
    double E[3], B[3];
    {
        const int nx = rd.n[0], ny = rd.n[1];
        double wh[3][L + 1], wt[3][KT];
        int ih[3][L + 1], it[3][KT];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            uint64_t psi, w[L + 1], t[KT];
            const int bh = spline_base62<L>(f[a], true, psi);
            bspline62<L>(psi, w);
            const int bt = ttable_weights62<L, KT>(rd.tt[a], f[a], t);
#pragma unroll
            for (int k = 0; k <= L; ++k) {
                wh[a][k] = weight_value(w[k]);
                ih[a][k] = wrap_near(c[a] + bh + k, rd.n[a]);
            }
#pragma unroll
            for (int k = 0; k < KT; ++k) {
                wt[a][k] = weight_value(t[k]);
                it[a][k] = wrap_near(c[a] + bt + k, rd.n[a]);
            }
        }
        E[0] = gather3_global<L + 1, KT, KT>(rd.F[0], nx, ny, ih[0], it[1], it[2], wh[0], wt[1], wt[2]);
        E[1] = gather3_global<KT, L + 1, KT>(rd.F[1], nx, ny, it[0], ih[1], it[2], wt[0], wh[1], wt[2]);
        E[2] = gather3_global<KT, KT, L + 1>(rd.F[2], nx, ny, it[0], it[1], ih[2], wt[0], wt[1], wh[2]);
        B[0] = gather3_global<KT, L + 1, L + 1>(rd.Bg[0], nx, ny, it[0], ih[1], ih[2], wt[0], wh[1], wh[2]);
        B[1] = gather3_global<L + 1, KT, L + 1>(rd.Bg[1], nx, ny, ih[0], it[1], ih[2], wh[0], wt[1], wh[2]);
        B[2] = gather3_global<L + 1, L + 1, KT>(rd.Bg[2], nx, ny, ih[0], ih[1], it[2], wh[0], wh[1], wt[2]);
    }

    // ---- Boris push and move ----
    const double ig = boris<double>(sp.qmdt_half, E, B, u);
    int sh[3];
    uint64_t fn[3];
    double dl[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        int cn;
        dl[a] = rd.dtt[a] * u[a] * ig;
        sh[a] = move_axis_fx(x[a], dl[a], c[a], rd.n[a], cn, fn[a]);
    }

    // ---- Esirkepov deposit ----
    AxisS62<L> S[3];
    bool up[3], mv[3];
    int g0[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        axis_shapes62<L>(f[a], fn[a], sh[a], S[a]);
        up[a] = sh[a] > 0 || (sh[a] == 0 && fn[a] >= f[a]);
        mv[a] = __any_sync(0xffffffffu, act && S[a].wide);
        g0[a] = c[a] + S[a].wb;
    }
    if (!act) return;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        // a non-finite velocity is reported as such, at the first node (a deterministic run's
        // current holds integers: in the error word)
        if ((__double2hiint(dl[a]) & 0x7ff00000) != 0x7ff00000) continue;
        if (DET) set_err(rd.err, 2);
        else
            atomicAdd(rd.F[6 + a] + (wrap_near(g0[2], rd.n[2]) * rd.n[1] + wrap_near(g0[1], rd.n[1])) * rd.n[0]
                          + wrap_near(g0[0], rd.n[0]), dl[a]);
    }
    deposit3_fx<L, DET>(rd, sp, g0, S, up, mv);

    // ---- store ----
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        ((double *)sp.pos[a])[p] = x[a];
        ((double *)sp.mom[a])[p] = u[a];
    }
}

// All particles of one 3D tile, or the share blockIdx.y of gridDim.y of every species'.
template <int L, int KT, bool DET>
__device__ void tile3_fx(const RunDev &rd, int64_t tile)
{
    for (int s = 0; s < rd.nsp; ++s) {
        const SpeciesDev &sp = rd.sp[s];
        int64_t a = sp.tile_start[tile], b = sp.tile_start[tile + 1];
        split_range(GridSplit(), a, b);
        // warp-uniform trip count: a warp's lanes take 32 consecutive particles
        for (int64_t q = a + (threadIdx.x & ~31); q < b; q += blockDim.x) {
            const int64_t p = q + (threadIdx.x & 31);
            if (p + blockDim.x < b) prefetch_particle_3d<double>(sp, p + blockDim.x);
            particle3_fx<L, KT, DET>(rd, sp, p, p < b);
        }
    }
}

}  // namespace pic
