// Tile kernels of the fused particle pass in 2D (shared-memory staged) and the per-tile
// driver shared by the single-run and the batched launches (3D: pic_gpp3d.cuh).
#pragma once
#include "pic_gpp.cuh"

namespace pic {

// Shared-memory layout of a staged 2D tile (all arrays reg_nodes long, x fastest):
//   pa = (E1, B2) pairs  [both sit at (i+1/2, j): W along x, T along y]
//   pb = (E2, B1) pairs  [both sit at (i, j+1/2): T along x, W along y]
//   e3 = E3 [(i, j): T T],  b3 = B3 [(i+1/2, j+1/2): W W],  j1, j2, j3 (R), or, for a
//   deterministic run, q1, q2, q3 (64-bit fixed point, RunDev::det) in their place.
//   rec = per-warp factor records of the FP32 deposit (see DepFrame), FP32 form only.
template <typename R>
struct Stage2D {
    typename Vec2<R>::T *pa, *pb;
    R *e3, *b3;
    R *j1, *j2, *j3;
    unsigned long long *q1, *q2, *q3;
    TTable *tt;
    float *rec;
};

// Warps of a 2D tile block (the kernels launch 256 threads).
constexpr int kTileWarps = 8;

// Frame of the FP32 warp deposit.  The Esirkepov current of a group of lanes whose windows
// start at most SXM nodes apart along x and SYM along y is a sum over lanes of outer products
// (J1 = sum px (x) Ay, J2 = sum Ax (x) py, J3 = sum Ax (x) S0y + Bx (x) DSy, in the notation of
// particle_2d) on a common NX x NY block of nodes.  Every lane writes its factor vectors,
// shifted into the block, as a record (x part: px, Ax, Bx over NX nodes; y part: Ay, py, S0y,
// DSy over NY nodes); then the lanes sum the 32 records, each lane one term (J1, J2, or one of
// the two products of J3) on a block of nodes with packed FMAs, every load a shared-memory
// broadcast within its record: on a HALF frame (NY = 2 or 4) the two half warps take the even
// and the odd records, each lane a 2 x NY block from one 64-bit and one 64- or 128-bit load per
// record; otherwise each lane takes a 2 x BY block (BY = NY / 2) over all 32 records, from one
// 64-bit and BY 32-bit loads.  The sums are bound by shared-memory wavefronts and issue, not by
// arithmetic (a 128-bit load takes a wavefront per quarter warp, a 64-bit one per half warp).
// RS (floats per record) is a multiple of 4 with RS / 4 odd, so that the float4 stores of 8
// consecutive lanes fall in distinct banks.  NARROW: no lane of the group moved its y window
// base, so every window's last row (node l + 1) is zero and the frame has l + 1 + SYM rows
// (rounded up to even) instead of l + 2 + SYM.
template <int L, bool NARROW = false>
struct DepFrame {
    // Along y the windows of a group start at most SYM rows apart: for odd l a particle's
    // integer-node window starts at a fixed offset from its cell, so the lanes of one cell row
    // share it (SYM = 0; a warp straddling the end of a tile row takes a second pass); for even
    // l the start moves by one with the in-cell offset (SYM = 1).  Along x, up to SXM nodes.
    static constexpr int SYM = (L % 2 == 0) ? 1 : 0;
    static constexpr int WYN = NARROW ? L + 1 : L + 2;  // y nodes of one lane's window
    static constexpr int PX = (L + 2 + 2 + 1) / 2, PY = (WYN + SYM + 1) / 2;
    static constexpr int NX = 2 * PX, NY = 2 * PY;
    static constexpr int SXM = NX - (L + 2);
    static constexpr int BY = NY / 2;            // y nodes of a lane's sub-block
    static constexpr int NBT = (NX / 2) * 2;     // sub-blocks of one term
    // x part padded to a multiple of 4 floats, so that every term's y factors start 16-byte
    // aligned within the record
    static constexpr int XS = (3 * NX + 3) / 4 * 4, YS = 4 * NY;
    // HALF: the two half warps sum the even and the odd records, each lane one term on a
    // 2 x NY block (one 64-bit and one 64- or 128-bit load and NY packed FMAs per record)
    static constexpr bool HALF = (NY == 2 || NY == 4) && 4 * (NX / 2) <= 16;
    static constexpr int RS0 = XS + YS;
    static constexpr int RS1 = (RS0 + 3) / 4 * 4;
    static constexpr int RS = ((RS1 / 4) % 2 == 0) ? RS1 + 4 : RS1;
    static_assert(4 * NBT <= 32, "one lane per sub-block and term");
};

// Floats of one warp's deposit records for spline order l (host-side sizing).
__host__ __device__ inline int dep_record_floats(int l)
{
    switch (l) {
    case 1: return 32 * DepFrame<1>::RS;
    case 2: return 32 * DepFrame<2>::RS;
    case 3: return 32 * DepFrame<3>::RS;
    default: return 32 * DepFrame<4>::RS;
    }
}

// Bytes per node of the shared current tile: R per component, or (FP32 form of a
// deterministic run) a 64-bit fixed-point word per component.
template <typename R>
__host__ __device__ inline size_t stage2d_j_bytes(bool det)
{
    return (sizeof(R) == 4 && det) ? 8 : sizeof(R);
}

// own_tt: the stage holds its own copy of the two T tables (false when the caller already
// keeps the run descriptor, tables included, in shared memory).
template <typename R>
__host__ __device__ inline size_t stage2d_fields_bytes(int64_t nodes, bool own_tt = true,
                                                       bool det = false)
{
    size_t b = own_tt ? 2 * sizeof(TTable) : 0;
    b += (size_t)nodes * (2 * sizeof(typename Vec2<R>::T) + 2 * sizeof(R)
                          + 3 * stage2d_j_bytes<R>(det));
    return (b + 15) / 16 * 16;
}

// Dynamic shared memory of a 2D tile block: staged fields and current, plus (FP32 form) the
// deposit records of its warps.
template <typename R>
__host__ __device__ inline size_t stage2d_bytes(int64_t nodes, int l, bool own_tt = true,
                                                bool det = false)
{
    size_t b = stage2d_fields_bytes<R>(nodes, own_tt, det);
    if (sizeof(R) == 4) b += (size_t)kTileWarps * dep_record_floats(l) * sizeof(float);
    return b;
}

// tt_shared: T tables already in shared memory (else the stage carries a copy)
template <typename R>
__device__ __forceinline__ Stage2D<R> stage2d_carve(char *smem, int64_t nodes,
                                                    const TTable *tt_shared = nullptr,
                                                    bool det = false)
{
    Stage2D<R> s;
    s.tt = tt_shared ? (TTable *)tt_shared : (TTable *)smem;
    char *p = smem + (tt_shared ? 0 : 2 * sizeof(TTable));
    s.pa = (typename Vec2<R>::T *)p; p += nodes * sizeof(typename Vec2<R>::T);
    s.pb = (typename Vec2<R>::T *)p; p += nodes * sizeof(typename Vec2<R>::T);
    s.e3 = (R *)p; p += nodes * sizeof(R);
    s.b3 = (R *)p; p += nodes * sizeof(R);
    s.j1 = s.j2 = s.j3 = nullptr;
    s.q1 = s.q2 = s.q3 = nullptr;
    if (sizeof(R) == 4 && det) {
        s.q1 = (unsigned long long *)p; p += nodes * 8;
        s.q2 = (unsigned long long *)p; p += nodes * 8;
        s.q3 = (unsigned long long *)p;
    } else {
        s.j1 = (R *)p; p += nodes * sizeof(R);
        s.j2 = (R *)p; p += nodes * sizeof(R);
        s.j3 = (R *)p;
    }
    s.rec = (float *)(smem + stage2d_fields_bytes<R>(nodes, tt_shared == nullptr, det));
    return s;
}

// Stage fields of the tile at (x0, y0) and zero the current tile.  One warp per row, so that the
// periodic wrap and the row offset are formed once per row (a linear node index cost two 64-bit
// remainders per node, which paced the small runs: 64x32 cells 23.4 -> 17.8 us per
// pass, 250x126 44.7 -> 42.7, the batch of 48 uneven runs 2.60 -> 2.51 ms).
template <typename R>
__device__ void stage2d_load(const RunDev &rd, const Stage2D<R> &st, int x0, int y0, int tiles)
{
    const int RX = rd.reg[0], RY = rd.reg[1], lane = threadIdx.x & 31;
    for (int i = threadIdx.x; i < (tiles - 1) * 3 * RX * RY / 2; i += blockDim.x)
        ((float2 *)st.rec)[i] = make_float2(0.0f, 0.0f);
    if (st.tt != rd.tt)
        for (int i = threadIdx.x; i < (int)(2 * sizeof(TTable) / sizeof(int)); i += blockDim.x)
            ((int *)st.tt)[i] = ((const int *)rd.tt)[i];
    for (int ry = threadIdx.x >> 5; ry < RY; ry += kTileWarps) {
        const int64_t row = (int64_t)wrap_near(y0 - rd.pre[1] + ry, rd.n[1]) * rd.n[0];
        for (int rx = lane; rx < RX; rx += 32) {
            const int64_t g = row + wrap_near(x0 - rd.pre[0] + rx, rd.n[0]);
            const int n = ry * RX + rx;
            typename Vec2<R>::T a, b;
            a.x = __ldg(rd.Fs[0] + g); a.y = __ldg(rd.Fs[4] + g);
            b.x = __ldg(rd.Fs[1] + g); b.y = __ldg(rd.Fs[3] + g);
            st.e3[n] = __ldg(rd.Fs[2] + g);
            st.b3[n] = __ldg(rd.Fs[5] + g);
            st.pa[n] = a;
            st.pb[n] = b;
            if (st.q1) {
                st.q1[n] = 0ull;
                st.q2[n] = 0ull;
                st.q3[n] = 0ull;
            } else {
                st.j1[n] = R(0);
                st.j2[n] = R(0);
                st.j3[n] = R(0);
            }
        }
    }
}

// Current tiles of a CTA.  A deterministic run sums integers, exact in any order: one tile for all
// species.  Otherwise the species are added to each other in FP64 only (a neutral plasma's currents
// cancel, and their sum in FP32 would be rounded at the size of one species' current): in the
// slot-major order, which writes no deposit records, every species has a tile of its own, the
// further ones where the records would lie, if they fit; else one tile is flushed once per species.
// (One FP32 tile and one flush for all species is faster by what the second flush takes, us per pass:
// 64x32 quadratic at 2 of a species per cell 17.6 against 19.7 (24.2 with the tiles added in the SM);
// 250x126 cubic at 4 52.6 against 56.2; 512x256 cubic at 16 283 against 294.)
template <int L, bool DET>
__device__ __forceinline__ int current_tiles(const RunDev &rd)
{
    const bool fit = (rd.nsp - 1) * 3 * rd.reg_nodes <= kTileWarps * (int64_t)dep_record_floats(L);
    return !DET && rd.slot_major && fit ? rd.nsp : 1;
}

// Add the current tiles to the global FP64 current; clear: and zero them for another species.  One
// warp per row, two neighbouring nodes per lane (rows hold an even number of nodes).
template <typename R>
__device__ void stage2d_flush(const RunDev &rd, const Stage2D<R> &st, int x0, int y0, int tiles,
                              bool clear)
{
    const int RX = rd.reg[0], RY = rd.reg[1], lane = threadIdx.x & 31;
    const int nodes = RX * RY;
    for (int ry = threadIdx.x >> 5; ry < RY; ry += kTileWarps) {
        const int64_t row = (int64_t)wrap_near(y0 - rd.pre[1] + ry, rd.n[1]) * rd.n[0];
        for (int rx = 2 * lane; rx < RX; rx += 64) {
            const int64_t g0 = row + wrap_near(x0 - rd.pre[0] + rx, rd.n[0]);
            const int64_t g1 = row + wrap_near(x0 - rd.pre[0] + rx + 1, rd.n[0]);
            const int n = ry * RX + rx;
            if (st.q1) {
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    unsigned long long *q = i == 0 ? st.q1 : (i == 1 ? st.q2 : st.q3);
                    unsigned long long *J = (unsigned long long *)rd.F[6 + i];
                    const unsigned long long a = q[n], b = q[n + 1];
                    if (a) atomicAdd(J + g0, a);
                    if (b) atomicAdd(J + g1, b);
                }
                continue;
            }
            float2 v[3] = {*(float2 *)(st.j1 + n), *(float2 *)(st.j2 + n), *(float2 *)(st.j3 + n)};
            if (clear) {
                const float2 z = make_float2(0.0f, 0.0f);
                *(float2 *)(st.j1 + n) = *(float2 *)(st.j2 + n) = *(float2 *)(st.j3 + n) = z;
            }
            for (int k = 1;; ++k) {
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    if (v[i].x != 0.0f) atomicAdd(rd.F[6 + i] + g0, (double)v[i].x);
                    if (v[i].y != 0.0f) atomicAdd(rd.F[6 + i] + g1, (double)v[i].y);
                }
                if (k >= tiles) break;
                const float *j = st.rec + (k - 1) * 3 * nodes + n;
#pragma unroll
                for (int i = 0; i < 3; ++i) v[i] = *(const float2 *)(j + i * nodes);
            }
        }
    }
}

// Add (a, b) to the two FP32 values at p (8-byte aligned: two neighbouring x nodes of a staged
// row that starts at an even node) with one 64-bit compare-and-swap loop and a packed add, each
// half rounded as the scalar add.  Shared-memory FP32 additions are compare-and-swap loops
// either way; this one serves two nodes.
__device__ __forceinline__ void atomic_add_pair(float *p, float a, float b)
{
    unsigned long long *q = (unsigned long long *)p;
    unsigned long long old = *q, got;
    do {
        float2 f = make_float2(__uint_as_float((unsigned)old),
                               __uint_as_float((unsigned)(old >> 32)));
        f = __fadd2_rn(f, make_float2(a, b));
        const unsigned long long nw = (unsigned long long)__float_as_uint(f.x)
                                      | ((unsigned long long)__float_as_uint(f.y) << 32);
        got = atomicCAS(q, old, nw);
        if (got == old) break;
        old = got;
    } while (true);
}

// One lane's Esirkepov window (Sec. 1: W_x = DSx (S0y + DSy/2) summed along x, W_y likewise,
// W_z = S0x S0y + DSx S0y/2 + S0x DSy/2 + DSx DSy/3) added to the shared current tile with
// atomics; WY = false when no
// lane of the warp changed its y window base, so that row l + 1 carries exact zeros; DET: as fixed-point words (RunDev::det).
template <int L, typename R, bool WY = true, bool DET = false>
__device__ __forceinline__ void deposit_lane(const Stage2D<R> &st, int RX, int jx0, int jy0, R kx,
                                             R ky, R kz, const R *px, const R *py, const R *Ax,
                                             const R *Ay, const R *Bx, const AxisS<L, R> &Sy,
                                             float dinv = 0.0f)
{
#pragma unroll
    for (int b = 0; b < (WY ? L + 2 : L + 1); ++b) {
        const int row = (jy0 + b) * RX + jx0;
        const R ayk = kx * Ay[b];
        const R pyk = (b <= L) ? ky * py[b] : R(0);
        const R zs = kz * Sy.s0[b], zd = kz * Sy.ds[b];
#pragma unroll
        for (int a = 0; a < L + 2; ++a) {
            if constexpr (DET) {
                if (a <= L) atomicAdd(st.q1 + row + a, det_word32(ayk * px[a], dinv));
                if (b <= L) atomicAdd(st.q2 + row + a, det_word32(pyk * Ax[a], dinv));
                atomicAdd(st.q3 + row + a, det_word32(zs * Ax[a] + zd * Bx[a], dinv));
            } else {
                if (a <= L) atomicAdd(st.j1 + row + a, ayk * px[a]);
                if (b <= L) atomicAdd(st.j2 + row + a, pyk * Ax[a]);
                atomicAdd(st.j3 + row + a, zs * Ax[a] + zd * Bx[a]);
            }
        }
    }
}

// Scalars the particle loop uses, held in registers for the whole tile (a run descriptor in
// shared or global memory would be re-read for every particle).
struct Hot2D {
    int n0, n1, tile0, tile1, drift0, drift1, pre0, pre1, RX, RY, slot_major;
    double *J0, *J1, *J2;  // global FP64 current (high fixed-point words of a deterministic run)
    double dtt0, dtt1;
    uint64_t dm;  // division by n0 (FastDiv)
    int ds;
    int32_t *err;
    int det;  // RunDev::det and its fixed-point scales and low words
    float dinv32;
    double dinv64;
    unsigned long long *Jlo0, *Jlo1, *Jlo2;
};

template <typename R>
struct HotSp {
    void *pos0, *pos1, *mom0, *mom1, *mom2;
    int32_t *cell;
    double qmdt_half, kx0, kx1, kz;
};

__device__ __forceinline__ Hot2D make_hot2d(const RunDev &rd)
{
    Hot2D h;
    h.n0 = rd.n[0]; h.n1 = rd.n[1];
    h.tile0 = rd.tile[0]; h.tile1 = rd.tile[1];
    h.drift0 = rd.drift[0]; h.drift1 = rd.drift[1];
    h.pre0 = rd.pre[0]; h.pre1 = rd.pre[1];
    h.RX = rd.reg[0];
    h.RY = rd.reg[1];
    h.J0 = rd.F[6]; h.J1 = rd.F[7]; h.J2 = rd.F[8];
    h.slot_major = rd.slot_major;
    h.dtt0 = rd.dtt[0]; h.dtt1 = rd.dtt[1];
    h.dm = rd.div_n0.m; h.ds = rd.div_n0.s;
    h.err = rd.err;
    h.det = rd.det;
    h.dinv32 = rd.det_inv32;
    h.dinv64 = rd.det_inv64;
    h.Jlo0 = rd.Jlo[0]; h.Jlo1 = rd.Jlo[1]; h.Jlo2 = rd.Jlo[2];
    return h;
}

template <typename R>
__device__ __forceinline__ HotSp<R> make_hotsp(const SpeciesDev &sp)
{
    HotSp<R> h;
    h.pos0 = sp.pos[0]; h.pos1 = sp.pos[1];
    h.mom0 = sp.mom[0]; h.mom1 = sp.mom[1]; h.mom2 = sp.mom[2];
    h.cell = sp.cell;
    h.qmdt_half = sp.qmdt_half;
    h.kx0 = sp.kx[0]; h.kx1 = sp.kx[1]; h.kz = sp.kz;
    return h;
}

// Ask the memory system for the particle stream of a later iteration (lines land in L1 while
// the current particle is processed; the particle loop is otherwise stalled on these loads).
template <typename R>
__device__ __forceinline__ void prefetch_particle(const HotSp<R> &hs, int64_t p)
{
    const void *ptrs[6] = {hs.pos0, hs.pos1, hs.mom0, hs.mom1, hs.mom2, hs.cell};
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        if (i == 5 && sizeof(R) == 8) break;  // the FP64 form has no cell array
        const char *a = (const char *)ptrs[i] + p * (i == 5 ? 4 : (int64_t)sizeof(R));
        asm volatile("prefetch.global.L1 [%0];" ::"l"(a));
    }
}

// FP32 gather on packed pairs: __ffma2_rn performs two FP32 fused multiply-adds in one
// instruction (sm_100 and later), each rounded exactly as the scalar FMA, so the result is the
// scalar loop's bit for bit.  (E1, B2) and (E2, B1) are staged as pairs that share their
// weights; E3 (T x T) and B3 (W x W) pair up when the two stencils have the same size.
template <int L, int KT>
__device__ __forceinline__ void gather_2d_x2(const Stage2D<float> &st, const AxisW<L, KT, float> &wx,
                                             const AxisW<L, KT, float> &wy, int sx, int sy,
                                             int RX, float *E, float *B)
{
    const float2 z2 = make_float2(0.0f, 0.0f);
    float2 e1b2 = z2, e2b1 = z2;
#pragma unroll
    for (int b = 0; b < KT; ++b) {  // (E1, B2): W along x (half nodes), T along y
        const int row = (sy + wy.bt + b) * RX + sx + wx.bh;
        float2 r = z2;
#pragma unroll
        for (int a = 0; a <= L; ++a) r = __ffma2_rn(make_float2(wx.wh[a], wx.wh[a]), st.pa[row + a], r);
        e1b2 = __ffma2_rn(make_float2(wy.wt[b], wy.wt[b]), r, e1b2);
    }
#pragma unroll
    for (int b = 0; b <= L; ++b) {  // (E2, B1): T along x, W along y
        const int row = (sy + wy.bh + b) * RX + sx + wx.bt;
        float2 r = z2;
#pragma unroll
        for (int a = 0; a < KT; ++a) r = __ffma2_rn(make_float2(wx.wt[a], wx.wt[a]), st.pb[row + a], r);
        e2b1 = __ffma2_rn(make_float2(wy.wh[b], wy.wh[b]), r, e2b1);
    }
    E[0] = e1b2.x; B[1] = e1b2.y;
    E[1] = e2b1.x; B[0] = e2b1.y;
    if constexpr (KT == L + 1) {
        float2 e3b3 = z2;
#pragma unroll
        for (int b = 0; b < KT; ++b) {  // E3: T T, B3: W W
            const int rt = (sy + wy.bt + b) * RX + sx + wx.bt;
            const int rw = (sy + wy.bh + b) * RX + sx + wx.bh;
            float2 r = z2;
#pragma unroll
            for (int a = 0; a < KT; ++a)
                r = __ffma2_rn(make_float2(wx.wt[a], wx.wh[a]), make_float2(st.e3[rt + a], st.b3[rw + a]), r);
            e3b3 = __ffma2_rn(make_float2(wy.wt[b], wy.wh[b]), r, e3b3);
        }
        E[2] = e3b3.x; B[2] = e3b3.y;
    } else {
        float e3 = 0.0f, b3 = 0.0f;
#pragma unroll
        for (int b = 0; b < KT; ++b) {
            const int row = (sy + wy.bt + b) * RX + sx + wx.bt;
            float r = 0.0f;
#pragma unroll
            for (int a = 0; a < KT; ++a) r += wx.wt[a] * st.e3[row + a];
            e3 += wy.wt[b] * r;
        }
#pragma unroll
        for (int b = 0; b <= L; ++b) {
            const int row = (sy + wy.bh + b) * RX + sx + wx.bh;
            float r = 0.0f;
#pragma unroll
            for (int a = 0; a <= L; ++a) r += wx.wh[a] * st.b3[row + a];
            b3 += wy.wh[b] * r;
        }
        E[2] = e3; B[2] = b3;
    }
}

// One pass of the FP32 warp deposit on frame FR (DepFrame): every lane writes its factor
// record, shifted by (ox, oy) into the frame and scaled by gin (1 for the lanes of this pass's
// group, 0 for the others), then each lane sums its term on its sub-block over the 32 records and
// adds it to the shared current.  The two products of J3 (terms 2 and 3, lanes NBT apart) are
// added together first, so that no two lanes of one atomic instruction address the same node.
// mnx, mny: frame origin (tile-local node); kx, ky, kz: the species' current scales.
template <class FR, int L, bool DET>
__device__ __forceinline__ void warp_frame_pass(const Hot2D &h, const Stage2D<float> &st,
                                                float gin, int ox, int oy, int mnx, int mny,
                                                float kx, float ky, float kz, const float *px,
                                                const float *py, const float *Ax, const float *Ay,
                                                const float *Bx, const AxisS<L, float> &Sy)
{
    const int lane = threadIdx.x & 31;
    // the warp's record area is sized for the widest frame of order l
    float *rec = st.rec + (threadIdx.x >> 5) * (32 * DepFrame<L>::RS);
    float4 *mine = (float4 *)(rec + lane * FR::RS);
    // the record: block node A holds this lane's window node A - ox (zero outside it); the x
    // factors are scaled first, then shifted by ox = 0..SXM in two steps (ox & 1, ox & 2); the
    // y factors are shifted by oy (0 when SYM = 0)
    float r[FR::RS1];
    float sp[L + 2], sa[L + 2], sb2[L + 2];
    const float gkx = gin * kx;
#pragma unroll
    for (int k = 0; k < L + 2; ++k) {
        sp[k] = (k <= L) ? gkx * px[k] : 0.0f;
        sa[k] = gin * Ax[k];
        sb2[k] = gin * Bx[k];
    }
    const bool sh1 = (ox & 1) != 0, sh2 = (ox & 2) != 0;
    float tp[L + 3], ta[L + 3], tb[L + 3];
#pragma unroll
    for (int k = 0; k < L + 3; ++k) {
        const float p0 = (k < L + 2) ? sp[k] : 0.0f, p1 = (k >= 1) ? sp[k - 1] : 0.0f;
        const float a0 = (k < L + 2) ? sa[k] : 0.0f, a1 = (k >= 1) ? sa[k - 1] : 0.0f;
        const float b0 = (k < L + 2) ? sb2[k] : 0.0f, b1 = (k >= 1) ? sb2[k - 1] : 0.0f;
        tp[k] = sh1 ? p1 : p0;
        ta[k] = sh1 ? a1 : a0;
        tb[k] = sh1 ? b1 : b0;
    }
#pragma unroll
    for (int A = 0; A < FR::NX; ++A) {
        const float p0 = (A < L + 3) ? tp[A] : 0.0f;
        const float p2 = (A >= 2 && A - 2 < L + 3) ? tp[A - 2] : 0.0f;
        const float a0 = (A < L + 3) ? ta[A] : 0.0f;
        const float a2 = (A >= 2 && A - 2 < L + 3) ? ta[A - 2] : 0.0f;
        const float b0 = (A < L + 3) ? tb[A] : 0.0f;
        const float b2 = (A >= 2 && A - 2 < L + 3) ? tb[A - 2] : 0.0f;
        r[A] = sh2 ? p2 : p0;
        r[FR::NX + A] = sh2 ? a2 : a0;
        r[2 * FR::NX + A] = sh2 ? b2 : b0;
    }
    float ty[4][L + 2];  // Ay, ky py, kz S0y, kz DSy
#pragma unroll
    for (int k = 0; k < L + 2; ++k) {
        ty[0][k] = Ay[k];
        ty[1][k] = (k <= L) ? ky * py[k] : 0.0f;
        ty[2][k] = kz * Sy.s0[k];
        ty[3][k] = kz * Sy.ds[k];
    }
#pragma unroll
    for (int Bn = 0; Bn < FR::NY; ++Bn) {
#pragma unroll
        for (int f = 0; f < 4; ++f) {
            const float v0 = (Bn <= L + 1) ? ty[f][Bn] : 0.0f;
            if constexpr (FR::SYM == 0) {
                r[FR::XS + f * FR::NY + Bn] = v0;
            } else {
                const float v1 = (Bn >= 1 && Bn - 1 <= L + 1) ? ty[f][Bn - 1] : 0.0f;
                r[FR::XS + f * FR::NY + Bn] = (oy == 1) ? v1 : v0;
            }
        }
    }
#pragma unroll
    for (int k = 3 * FR::NX; k < FR::XS; ++k) r[k] = 0.0f;
#pragma unroll
    for (int k = FR::RS0; k < FR::RS1; ++k) r[k] = 0.0f;
#pragma unroll
    for (int v = 0; v < FR::RS1 / 4; ++v)
        mine[v] = make_float4(r[4 * v], r[4 * v + 1], r[4 * v + 2], r[4 * v + 3]);
    __syncwarp();
    if constexpr (FR::HALF) {
        // lane (half, term, bx): term t (0: J1 = px Ay, 1: J2 = Ax py, 2: J3 from Ax S0y, 3: J3
        // from Bx DSy; lanes past the four terms idle) on the frame columns 2 bx, 2 bx + 1 and
        // all NY rows, summed over the records of parity `half`, as packed pairs (each lane
        // rounded as the scalar FMA)
        constexpr int NBX = FR::NX / 2;
        const int half = lane >> 4, hl = lane & 15;
        const int term = hl / NBX, bx = hl % NBX;
        const bool sums = term < 4;
        const int xo = sums ? (term == 0 ? 0 : (term == 3 ? 2 * FR::NX : FR::NX)) + 2 * bx : 0;
        const int yo = sums ? FR::XS + term * FR::NY : FR::XS;
        float2 o[FR::NY];
#pragma unroll
        for (int j = 0; j < FR::NY; ++j) o[j] = make_float2(0.0f, 0.0f);
#pragma unroll 8
        for (int q = 0; q < 16; ++q) {
            const float *rq = rec + (2 * q + half) * FR::RS;
            const float2 xv = *(const float2 *)(rq + xo);
            float yv[FR::NY];
            if constexpr (FR::NY == 4) {
                const float4 t = *(const float4 *)(rq + yo);
                yv[0] = t.x; yv[1] = t.y; yv[2] = t.z; yv[3] = t.w;
            } else {
                const float2 t = *(const float2 *)(rq + yo);
                yv[0] = t.x; yv[1] = t.y;
            }
#pragma unroll
            for (int j = 0; j < FR::NY; ++j) o[j] = __ffma2_rn(xv, make_float2(yv[j], yv[j]), o[j]);
        }
        // both halves' sums (a + b = b + a: the halves hold the same value), then J3's two
        // products (terms 2 and 3, NBX lanes apart within the half)
#pragma unroll
        for (int j = 0; j < FR::NY; ++j) {
            o[j].x += __shfl_xor_sync(0xffffffffu, o[j].x, 16);
            o[j].y += __shfl_xor_sync(0xffffffffu, o[j].y, 16);
        }
#pragma unroll
        for (int j = 0; j < FR::NY; ++j) {
            const float ox3 = __shfl_down_sync(0xffffffffu, o[j].x, NBX);
            const float oy3 = __shfl_down_sync(0xffffffffu, o[j].y, NBX);
            if (term == 2) {
                o[j].x += ox3;
                o[j].y += oy3;
            }
        }
        // the halves add the lower and the upper NY / 2 rows; with an even frame origin each
        // lane's two x nodes are one aligned pair (the row stride is even)
        if (!DET && (mnx & 1) == 0) {
            if (term < 3) {
                float *t = term == 0 ? st.j1 : (term == 1 ? st.j2 : st.j3);
#pragma unroll
                for (int jj = 0; jj < FR::NY / 2; ++jj) {
                    const float2 v = half ? o[FR::NY / 2 + jj] : o[jj];
                    const int gx = mnx + 2 * bx, gy = mny + (half ? FR::NY / 2 + jj : jj);
                    if (gx >= h.RX || gy >= h.RY || (v.x == 0.0f && v.y == 0.0f)) continue;
                    atomic_add_pair(t + gy * h.RX + gx, v.x, v.y);
                }
            }
        } else if (term < 3) {
#pragma unroll
            for (int i = 0; i < 2; ++i) {
#pragma unroll
                for (int jj = 0; jj < FR::NY / 2; ++jj) {
                    const int j = half ? FR::NY / 2 + jj : jj;
                    const float vlo = i == 0 ? o[jj].x : o[jj].y;
                    const float vhi = i == 0 ? o[FR::NY / 2 + jj].x : o[FR::NY / 2 + jj].y;
                    const float v = half ? vhi : vlo;
                    const int gx = mnx + 2 * bx + i, gy = mny + j;
                    if (gx >= h.RX || gy >= h.RY || v == 0.0f) continue;
                    const int node = gy * h.RX + gx;
                    if (DET) {  // fixed-point words: the warps' sums commute exactly
                        unsigned long long *t = term == 0 ? st.q1 : (term == 1 ? st.q2 : st.q3);
                        atomicAdd(t + node, det_word32(v, h.dinv32));
                    } else {
                        float *t = term == 0 ? st.j1 : (term == 1 ? st.j2 : st.j3);
                        atomicAdd(t + node, v);
                    }
                }
            }
        }
    } else {
        // this lane's sum: term t (0: J1 = px Ay, 1: J2 = Ax py, 2: J3 from Ax S0y, 3: J3 from
        // Bx DSy; lanes past the four terms idle) on the sub-block (bx, by) of the frame, as packed
        // pairs (the sub-block's two x nodes; each lane rounded as the scalar FMA)
        const int term = lane / FR::NBT, sb = lane % FR::NBT;
        const int bx = sb % (FR::NX / 2), by = sb / (FR::NX / 2);
        const bool sums = term < 4;
        const int xo = sums ? (term == 0 ? 0 : (term == 3 ? 2 * FR::NX : FR::NX)) + 2 * bx : 0;
        const int yo = sums ? FR::XS + term * FR::NY + FR::BY * by : FR::XS;
        float2 o[FR::BY];
#pragma unroll
        for (int k = 0; k < FR::BY; ++k) o[k] = make_float2(0.0f, 0.0f);
#pragma unroll 8
        for (int q = 0; q < 32; ++q) {
            const float *rq = rec + q * FR::RS;
            const float2 xv = *(const float2 *)(rq + xo);
#pragma unroll
            for (int k = 0; k < FR::BY; ++k) {
                const float yv = rq[yo + k];
                o[k] = __ffma2_rn(xv, make_float2(yv, yv), o[k]);
            }
        }
#pragma unroll
        for (int k = 0; k < FR::BY; ++k) {
            const float ox3 = __shfl_down_sync(0xffffffffu, o[k].x, FR::NBT);
            const float oy3 = __shfl_down_sync(0xffffffffu, o[k].y, FR::NBT);
            if (term == 2) {
                o[k].x += ox3;
                o[k].y += oy3;
            }
        }
        if (!DET && (mnx & 1) == 0) {
            if (term < 3) {
                float *t = term == 0 ? st.j1 : (term == 1 ? st.j2 : st.j3);
#pragma unroll
                for (int k = 0; k < FR::BY; ++k) {
                    const int gx = mnx + 2 * bx, gy = mny + FR::BY * by + k;
                    if (gx >= h.RX || gy >= h.RY || (o[k].x == 0.0f && o[k].y == 0.0f)) continue;
                    atomic_add_pair(t + gy * h.RX + gx, o[k].x, o[k].y);
                }
            }
        } else if (term < 3) {
#pragma unroll
            for (int i = 0; i < 2; ++i) {
#pragma unroll
                for (int k = 0; k < FR::BY; ++k) {
                    const int gx = mnx + 2 * bx + i, gy = mny + FR::BY * by + k;
                    const float v = i == 0 ? o[k].x : o[k].y;
                    if (gx >= h.RX || gy >= h.RY || v == 0.0f) continue;
                    const int node = gy * h.RX + gx;
                    if (DET) {  // fixed-point words: the warps' sums commute exactly
                        unsigned long long *t = term == 0 ? st.q1 : (term == 1 ? st.q2 : st.q3);
                        atomicAdd(t + node, det_word32(v, h.dinv32));
                    } else {
                        float *t = term == 0 ? st.j1 : (term == 1 ? st.j2 : st.j3);
                        atomicAdd(t + node, v);
                    }
                }
            }
        }
    }
}

// One particle per lane, 2D, staged tile.  Called by all 32 lanes of a warp together (the
// deposit is warp-collective); lanes with act == false carry no particle.  DET: a
// deterministic run (RunDev::det), whose current goes in as fixed-point words; a template
// parameter so that the default instances carry none of its code.
template <int L, int KT, typename R, bool DET = false>
__device__ __forceinline__ void particle_2d(const Hot2D h, const HotSp<R> hs,
                                            const Stage2D<R> &st, int64_t p, bool act, int x0,
                                            int y0)
{
    PState<R> s;
    int lx = 0, ly = 0;
    if (act) {
        const int c = __ldg(hs.cell + p);
        s.c[1] = fast_div(c, h.dm, h.ds);
        s.c[0] = c - s.c[1] * h.n0;
        s.d[0] = __ldg((const float *)hs.pos0 + p);
        s.d[1] = __ldg((const float *)hs.pos1 + p);
        s.c[2] = 0;
        s.u[0] = __ldg((const R *)hs.mom0 + p);
        s.u[1] = __ldg((const R *)hs.mom1 + p);
        s.u[2] = __ldg((const R *)hs.mom2 + p);
        const bool okx = local_coord(s.c[0], x0, h.tile0, h.drift0, h.n0, lx);
        const bool oky = local_coord(s.c[1], y0, h.tile1, h.drift1, h.n1, ly);
        if (!(okx && oky)) {
            set_err(h.err, 1);
            act = false;
        }
    }
    if (!act) {
        // a harmless stand-in particle at the tile origin; its current is weighted by zero
        s.c[0] = x0; s.c[1] = y0; s.c[2] = 0;
        s.d[0] = R(0.5); s.d[1] = R(0.5); s.d[2] = R(0);
        s.u[0] = s.u[1] = s.u[2] = R(0);
        lx = 0; ly = 0;
    }
    const int RX = h.RX;
    const int sx = lx + h.pre0, sy = ly + h.pre1;

    AxisW<L, KT, R> wx, wy;
    axis_weights<L, KT, R>(st.tt[0], s.d[0], wx);
    axis_weights<L, KT, R>(st.tt[1], s.d[1], wy);

    // ---- gather (Eq. interpolation-EB-real-mod; MC when the tables hold W_l) ----
    R E[3], B[3];
    gather_2d_x2<L, KT>(st, wx, wy, sx, sy, RX, E, B);

    // ---- Boris push ----
    const R ig = boris<R>(R(hs.qmdt_half), E, B, s.u);

    // ---- move ----
    R o[2], dl[2];
    int cn[2];
#pragma unroll
    for (int a = 0; a < 2; ++a) {
        dl[a] = R(a == 0 ? h.dtt0 : h.dtt1) * s.u[a] * ig;
        move_axis(s.d[a], dl[a], s.c[a], a == 0 ? h.n0 : h.n1, o[a], cn[a]);
    }

    // ---- Esirkepov deposit ----
    AxisS<L, R> Sx, Sy;
    axis_shapes_dd<L, true>(s.d[0], dl[0], Sx);  // all 32 lanes take part
    axis_shapes_dd<L, true>(s.d[1], dl[1], Sy);
    // the warp-collective deposit carries idle lanes with zero weight
    const R wgt = act ? R(1) : R(0);
    const R kx = wgt * R(hs.kx0);
    const R ky = wgt * R(hs.kx1);
    const R kz = wgt * R(hs.kz) * s.u[2] * ig;
    const R third = R(1) / R(3);
    // W_x = DSx (S0y + DSy/2), prefix along x; W_y = DSy (S0x + DSx/2), prefix along y;
    // W_z = S0x S0y + DSx S0y/2 + S0x DSy/2 + DSx DSy/3 = S0y Ax + DSy Bx.
    R Ax[L + 2], Ay[L + 2], Bx[L + 2], px[L + 2], py[L + 2];
    R acc_x = R(0), acc_y = R(0);
#pragma unroll
    for (int k = 0; k < L + 2; ++k) {
        Ax[k] = Sx.s0[k] + R(0.5) * Sx.ds[k];
        Ay[k] = Sy.s0[k] + R(0.5) * Sy.ds[k];
        Bx[k] = R(0.5) * Sx.s0[k] + third * Sx.ds[k];
        acc_x += Sx.ds[k];
        acc_y += Sy.ds[k];
        px[k] = acc_x;
        py[k] = acc_y;
    }
    const int jx0 = sx + Sx.wb, jy0 = sy + Sy.wb;

    {
        // Warp-collective path (cell-major order): lanes whose windows start at most SXM nodes
        // apart in x and SYM in y (up to three or four neighbouring cells along a row) form a
        // group; the group's current is a sum of per-lane outer products on a common block
        // (DepFrame), which the warp sums through shared memory and adds node by node.
        // Otherwise every lane adds its own window with shared atomics (the slot-major order,
        // lanes in different cells).
        using FR = DepFrame<L>;
        if (h.slot_major) {  // lanes in different cells: per-lane atomics do not collide
            // (shared-memory CAS atomics: measured faster here than global FP64 reductions,
            // which would need an FP32 -> FP64 conversion per node)
            const bool wide = __any_sync(0xffffffffu, act && Sy.wide);
            if (!act) {
            } else if (DET) {
                if (wide)
                    deposit_lane<L, R, true, true>(st, RX, jx0, jy0, kx, ky, kz, px, py, Ax, Ay,
                                                   Bx, Sy, h.dinv32);
                else
                    deposit_lane<L, R, false, true>(st, RX, jx0, jy0, kx, ky, kz, px, py, Ax, Ay,
                                                    Bx, Sy, h.dinv32);
            } else if (wide) {
                deposit_lane<L, R, true>(st, RX, jx0, jy0, kx, ky, kz, px, py, Ax, Ay, Bx, Sy);
            } else {
                deposit_lane<L, R, false>(st, RX, jx0, jy0, kx, ky, kz, px, py, Ax, Ay, Bx, Sy);
            }
        } else {
        // passes over groups of lanes that fit one common block (usually one pass; a warp that
        // straddles the end of a tile row takes two)
        bool todo = act;
        while (__any_sync(0xffffffffu, todo)) {
            const int mny = __reduce_min_sync(0xffffffffu, todo ? jy0 : 0x7fffffff);
            const bool rowok = todo && jy0 <= mny + FR::SYM;
            const int mnx = __reduce_min_sync(0xffffffffu, rowok ? jx0 : 0x7fffffff);
            const bool in = rowok && jx0 <= mnx + FR::SXM;
            todo = todo && !in;
            const int ox = in ? jx0 - mnx : 0, oy = in ? jy0 - mny : 0;
            const R gin = in ? R(1) : R(0);
            __syncwarp();  // the previous pass has read every record
            // a group none of whose lanes moved its y window base leaves row l + 1 of every
            // window at exact zeros (S0y = DSy = 0): its frame is two rows lower
            if (__any_sync(0xffffffffu, in && Sy.wide))
                warp_frame_pass<DepFrame<L, false>, L, DET>(h, st, gin, ox, oy, mnx, mny, kx, ky,
                                                            kz, px, py, Ax, Ay, Bx, Sy);
            else
                warp_frame_pass<DepFrame<L, true>, L, DET>(h, st, gin, ox, oy, mnx, mny, kx, ky,
                                                           kz, px, py, Ax, Ay, Bx, Sy);
        }
        }
    }
    if (!act) return;

    // ---- store ----
    ((R *)hs.mom0)[p] = s.u[0];
    ((R *)hs.mom1)[p] = s.u[1];
    ((R *)hs.mom2)[p] = s.u[2];
    hs.cell[p] = cn[1] * h.n0 + cn[0];
    ((float *)hs.pos0)[p] = o[0];
    ((float *)hs.pos1)[p] = o[1];
}

// Which share of a tile's particles a CTA takes: [from, to) of `of` equal shares of every species'
// range, read where used so that it holds no registers across the tile.  The FP64 form's launch
// puts the part in blockIdx.y (tile_parts chooses how many); the FP32 form's divides the grid's
// tiles evenly over its CTAs, tile borders or not (tile_ctas); the batched kernel keeps the part in
// shared memory beside its work item.
struct GridSplit {
    __device__ __forceinline__ int64_t from() const { return blockIdx.y; }
    __device__ __forceinline__ int64_t to() const { return blockIdx.y + 1; }
    __device__ __forceinline__ int64_t of() const { return gridDim.y; }
};
struct EvenSplit {
    int64_t tile, ntiles;  // CTA k of G takes k ntiles / G .. (k + 1) ntiles / G
    __device__ __forceinline__ int64_t from() const
    {
        return max(blockIdx.x * ntiles - tile * gridDim.x, (int64_t)0);
    }
    __device__ __forceinline__ int64_t to() const
    {
        return min((blockIdx.x + 1) * ntiles - tile * gridDim.x, (int64_t)gridDim.x);
    }
    __device__ __forceinline__ int64_t of() const { return gridDim.x; }
};
struct SharedSplit {
    const int *s;  // (part, parts)
    __device__ __forceinline__ int64_t from() const { return s[0]; }
    __device__ __forceinline__ int64_t to() const { return s[0] + 1; }
    __device__ __forceinline__ int64_t of() const { return s[1]; }
};

template <typename Split>
__device__ __forceinline__ void split_range(const Split &split, int64_t &a, int64_t &b)
{
    const int64_t len = b - a, of = split.of();
    if (split.to() - split.from() == of) return;
    b = a + len * split.to() / of;
    a += len * split.from() / of;
}

// All particles of one tile (both species), 2D FP32 form, or split's share of them: a grid of few
// tiles, or a batch of few particles, is spread over several CTAs per tile, each staging the tile
// and adding its own share of the current.  tt_shared as in stage2d_carve.
template <int L, int KT, typename R, bool DET = false, typename Split>
__device__ void tile_2d(const RunDev &rd, char *smem, int64_t tile, const TTable *tt_shared,
                        const Split split)
{
    Stage2D<R> st = stage2d_carve<R>(smem, rd.reg_nodes, tt_shared, DET);
    const int tx = (int)(tile % rd.ntile[0]);
    const int ty = (int)(tile / rd.ntile[0]);
    const int x0 = tx * rd.tile[0], y0 = ty * rd.tile[1];
    const int tiles = current_tiles<L, DET>(rd);
    const bool once = DET || tiles == rd.nsp;  // one flush, after the last species
    stage2d_load<R>(rd, st, x0, y0, tiles);
    const Hot2D h = make_hot2d(rd);
    __syncthreads();
    for (int s = 0; s < rd.nsp; ++s) {
        const SpeciesDev &sp = rd.sp[s];
        const HotSp<R> hs = make_hotsp<R>(sp);
        int64_t a = sp.tile_start[tile], b = sp.tile_start[tile + 1];
        split_range(split, a, b);
        if (a >= b) continue;  // (the whole CTA)
        Stage2D<R> own = st;
        if (s > 0 && tiles > 1) {
            own.j1 = st.rec + (s - 1) * 3 * (int)rd.reg_nodes;
            own.j2 = own.j1 + (int)rd.reg_nodes;
            own.j3 = own.j2 + (int)rd.reg_nodes;
        }
        // every warp takes a contiguous chunk of the tile's particles of this species (for a
        // uniform plasma in the cell-major order, one row of cells), so that the warps' frames,
        // a row apart, rarely race for the same nodes of the tile: 5.53 -> 5.38 ms on the
        // 134M-particle FP32 step (slot-major runs, whose lanes deposit one by one, lose about
        // 5%; a runtime choice between the two loops cost the dense kernel more).  With
        // one flush, the species of a part of few particles start at different warps, so as not to
        // queue one behind the other on the first warps.
        const int lane = threadIdx.x & 31;
        const int64_t groups = (b - a + 31) / 32;
        const int w = ((threadIdx.x >> 5) + (once && groups < kTileWarps ? s * (kTileWarps / 2) : 0)) % kTileWarps;
        const int64_t gw = (groups + kTileWarps - 1) / kTileWarps;
        const int64_t ca = a + 32 * min(groups, (int64_t)w * gw);
        const int64_t cb = min(b, a + 32 * min(groups, (int64_t)(w + 1) * gw));
        for (int64_t q = ca; q < cb; q += 32) {  // warp-uniform trip count
            const int64_t p = q + lane;
            if (p + 32 < cb) prefetch_particle<R>(hs, p + 32);
            particle_2d<L, KT, R, DET>(h, hs, own, p, p < cb, x0, y0);
        }
        if (!once) {
            const bool more = s + 1 < rd.nsp;
            __syncthreads();
            stage2d_flush<R>(rd, st, x0, y0, 1, more);
            if (more) __syncthreads();
        }
    }
    if (once) {
        __syncthreads();
        stage2d_flush<R>(rd, st, x0, y0, tiles, false);
    }
}

}  // namespace pic
