// Fixed-point evaluation of the interpolation weights, the gather and the current products of
// the plain FP64 form (2D).
//
// This GPU completes 2 FP64 operations per clock and SM, but 25 or more products of 32 x 32 bits with a
// 64-bit accumulation (GB300 at 2.07 GHz: 627 G DFMA/s, and 7,880 G mad.wide/s, signed or unsigned, in a
// loop of four with two other integer operations).
// Everything between the particle's offset and its current is bounded -- offsets, weights and
// their products lie in [0, 1], and a tile's fields lie below their largest magnitude -- so
// 62-bit fixed point carries it with more bits than FP64's 53, at three such products per
// multiplication.  The Boris push and the move, whose range is open, stay in FP64, and so does the
// gather of a tile whose fields differ by more than the fixed point resolves (stage_fx_load).
//
// U62: an unsigned value in units of 2^-62 (1 is 2^62), split for multiplication into limbs of
// 31 bits, v = h 2^31 + l.  A product drops l l' (below one unit) and truncates the rest: it is
// low by less than two units.
#pragma once
#include "pic_common.cuh"

#define PIC_HD __host__ __device__ __forceinline__

namespace pic {

constexpr uint64_t kOne62 = (uint64_t)1 << 62;

// n / d in U62
PIC_HD constexpr uint64_t frac62(uint64_t n, uint64_t d)
{
    return kOne62 / d * n + kOne62 % d * n / d;
}

struct Limbs {
    uint32_t h, l;
};

PIC_HD Limbs limbs(uint64_t v)
{
    Limbs r;
    r.h = (uint32_t)(v >> 31);
    r.l = (uint32_t)v & 0x7fffffffu;
    return r;
}

PIC_HD uint64_t wide_mul(uint32_t a, uint32_t b) { return (uint64_t)a * b; }

PIC_HD uint64_t mul62(const Limbs &a, const Limbs &b)
{
    return wide_mul(a.h, b.h) + ((wide_mul(a.h, b.l) + wide_mul(a.l, b.h)) >> 31);
}

// a s with a signed (|a| <= 2^62) and s a U62 below 1, low by less than two units
PIC_HD int64_t mul62s(int64_t a, const Limbs &s)
{
    const int32_t ah = (int32_t)(a >> 31);
    const uint32_t al = (uint32_t)a & 0x7fffffffu;
    const int64_t x = (int64_t)ah * (int32_t)s.l + (int64_t)wide_mul(al, s.h);
    return (int64_t)ah * (int32_t)s.h + (x >> 31);
}

PIC_HD uint64_t nonneg(uint64_t v) { return (int64_t)v < 0 ? 0 : v; }

PIC_HD int leading_zeros(uint64_t v)  // v != 0
{
#ifdef __CUDA_ARCH__
    return __clzll((long long)v);
#else
    return __builtin_clzll(v);
#endif
}

// Cell and in-cell offset (units of 2^-64) of a position x >= 0 given by its bits; exact for
// offsets of at most 64 bits, else truncated below 2^-64.  A non-finite or huge x gives a cell
// of 2^31 - 1 (the caller clamps it to the grid).
PIC_HD int decode_position(uint64_t bits, uint64_t &frac)
{
    const int e = (int)(bits >> 52) & 0x7ff;
    const uint64_t m = (bits & 0xfffffffffffffull) | ((uint64_t)1 << 52);
    const int s = 1075 - e;  // x = m 2^-s
    if (s < 22) {
        frac = 0;
        return 0x7fffffff;
    }
    const int r = s - 64;
    frac = r <= 0 ? m << -r : (r < 64 ? m >> r : 0);
    return s <= 52 ? (int)(m >> s) : 0;
}

// An FP32 in-cell offset in [0, 1) in units of 2^-64, exact down to offsets of 2^-40.  A
// non-finite offset gives some value.
PIC_HD uint64_t offset_fixed(uint32_t bits)
{
    const int e = (int)(bits >> 23) & 0xff;
    const uint64_t m = (bits & 0x7fffffu) | 0x800000u;
    const int s = e - 86;
    return s >= 0 ? m << (s < 40 ? s : 40) : (s > -24 && e > 0 ? m >> -s : 0);
}

// W_l at the l + 1 nodes (bspline<L> in U62), p = psi in U62, below 1.
template <int L>
PIC_HD void bspline62(uint64_t p, uint64_t *w)
{
    const Limbs P = limbs(p);
    if constexpr (L == 1) {
        w[0] = kOne62 - p;
        w[1] = p;
    } else {
        const uint64_t p2 = mul62(P, P);
        if constexpr (L == 2) {
            w[0] = nonneg(frac62(1, 2) - p + (p2 >> 1));
            w[2] = p2 >> 1;
            w[1] = kOne62 - w[0] - w[2];
        } else if constexpr (L == 3) {
            const uint64_t p3 = mul62(limbs(p2), P);
            w[3] = mul62(limbs(p3), limbs(frac62(1, 6)));
            w[0] = nonneg(frac62(1, 6) - (p >> 1) + (p2 >> 1) - w[3]);
            w[1] = frac62(2, 3) - p2 + (p3 >> 1);
            w[2] = kOne62 - w[0] - w[1] - w[3];
        } else {
            const Limbs P2 = limbs(p2), sixth = limbs(frac62(1, 6));
            const uint64_t a = mul62(P, sixth);
            const uint64_t b = mul62(limbs(mul62(P2, P)), sixth);
            const uint64_t g = mul62(limbs(mul62(P2, P2)), sixth);
            w[4] = g >> 2;
            w[0] = nonneg(frac62(1, 24) - a + (p2 >> 2) - b + w[4]);
            w[1] = frac62(11, 24) - (p >> 1) - (p2 >> 2) + 3 * b - g;
            w[3] = frac62(1, 24) + a + (p2 >> 2) + b - g;
            w[2] = kOne62 - w[0] - w[1] - w[3] - w[4];
        }
    }
}

// spline_base of an offset f in units of 2^-64; psi in U62.
template <int L>
PIC_HD int spline_base62(uint64_t f, bool half, uint64_t &psi)
{
    const int h2 = (half ? 1 : 0) + L - 1;
    const int hi = h2 >> 1;
    if (h2 & 1) {
        psi = (f ^ ((uint64_t)1 << 63)) >> 2;  // +- 1/2
        return (f >> 63) ? -hi : -hi - 1;
    }
    psi = f >> 2;
    return -hi;
}

// Integer-node weights from the table's fixed-point coefficients (ttable_weights in U62): on
// each piece of length h the polynomial in s = t / h, whose coefficients are bounded whatever
// the time step (units 2^-59).  The middle weight is what the others leave of 1, so that their
// truncation, always downwards, and the table's own rounding, which grows as the time step shrinks,
// move weight between nodes and do not scale the field.
template <int L, int KT>
PIC_HD int ttable_weights62(const TTable &t, uint64_t f, uint64_t *w)
{
    const uint64_t phi = f - t.fx.rfrac;
    const int base = (f < t.fx.rfrac ? -1 : 0) - t.Rint + 1;
    const int p = phi >= t.fx.phib ? 1 : 0;
    const uint64_t s0 = ((phi - (p ? t.fx.phib : 0)) << t.fx.shift[p]) >> 2;
    uint64_t sv = s0 + mul62(limbs(s0), limbs(t.fx.invm1[p]));
    if (sv >= kOne62) sv = kOne62 - 1;
    const Limbs s = limbs(sv);
    uint64_t rest = kOne62;
#pragma unroll
    for (int k = 0; k < KT; ++k) {
        if (k == KT / 2) continue;
        int64_t acc = t.ci[p][k][L];
#pragma unroll
        for (int m = L - 1; m >= 0; --m) acc = mul62s(acc, s) + t.ci[p][k][m];
        w[k] = nonneg((uint64_t)acc) << 3;
        rest -= w[k];
    }
    w[KT / 2] = nonneg(rest);
    return base;
}

// A finite FP64 scale s = m 2^k (m in [1/2, 1)) as its mantissa in U62 and the high word an FP64
// value of that sign and exponent starts from (to_fp64).  Scales below 2^-900 count as zero.
struct Scale62 {
    uint64_t m;
    uint32_t top;
};

PIC_HD Scale62 scale62(uint64_t bits)
{
    Scale62 r;
    const int e = (int)(bits >> 52) & 0x7ff;  // k = e - 1022
    r.top = ((uint32_t)(bits >> 32) & 0x80000000u) + ((uint32_t)(e + 1) << 20);
    r.m = e < 122 ? 0 : ((bits & 0xfffffffffffffull) | ((uint64_t)1 << 52)) << 9;
    return r;
}

// The FP64 value v 2^(k - 62) with the sign of the scale that gave top, rounded to nearest (v a
// U62, not zero).
PIC_HD uint64_t to_fp64_bits(uint64_t v, uint32_t top)
{
    uint32_t hi = (uint32_t)(v >> 32), lo = (uint32_t)v;
    if (hi == 0) {
        hi = lo;
        lo = 0;
        top -= 32u << 20;
    }
#ifdef __CUDA_ARCH__
    const int lz = __clz((int)hi);
    hi = __funnelshift_l(lo, hi, lz);
#else
    const int lz = __builtin_clz(hi);
    hi = lz ? (hi << lz) | (lo >> (32 - lz)) : hi;
#endif
    lo <<= lz;
    // v = (hi, lo) 2^-lz with the top bit set: the mantissa is its upper 53 bits, whose leading
    // one adds 1 to the exponent field 1023 + k - lz - 1
    const uint64_t m = (((uint64_t)hi << 32 | lo) >> 11) + ((lo >> 10) & 1);
    return m + ((uint64_t)(top - ((uint32_t)lz << 20)) << 32);
}

#ifdef __CUDACC__
// *p += v (a U62, its scale's sign and exponent in top) as an FP64 reduction performed by L2;
// nothing for v = 0.  Predicated, not branched around: the compiler's branch per contribution
// cost more instructions than the conversion it skips.
__device__ __forceinline__ void red_fixed(double *p, uint64_t v, uint32_t top)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u64 p, %2, 0;\n\t"
                 "@p red.global.add.f64 [%0], %1;\n\t}"
                 ::"l"(p), "d"(__longlong_as_double((int64_t)to_fp64_bits(v, top))), "l"(v)
                 : "memory");
}
#endif

// The FP64 value of a U62, rounded to nearest, by its bits.
PIC_HD uint64_t weight_bits(uint64_t v) { return v ? to_fp64_bits(v, 1023u << 20) : 0; }

// A signed value split for the gather's products, v = h 2^32 + l with |l| <= 2^31: the dropped l l'
// have no sign of their own.
struct Parts {
    int32_t h, l;
};

PIC_HD Parts parts(int64_t v)
{
    Parts r;
    r.l = (int32_t)(uint32_t)v;
    r.h = (int32_t)((uint64_t)v >> 32) + (r.l < 0 ? 1 : 0);
    return r;
}

// Sum of weight x field products, weights U62 (as Parts) that sum to 1 and fields of at most 2^60
// units: the high products and the cross products apart, so that a term costs three multiply-adds.
// Bounds for up to six terms: hi below 2^59, x below 2.5 2^61.  A field of zeros sums to zero exactly,
// and the rounding of the others (about one unit) has no sign of its own.
struct GatherSum {
    int64_t hi, x;
    PIC_HD void zero() { hi = 0; x = 1 << 29; }  // (half of what value() shifts out)
    PIC_HD void add(const Parts &w, int32_t fh, int32_t fl)
    {
        hi += (int64_t)w.h * fh;
        x += (int64_t)w.h * fl;
        x += (int64_t)w.l * fh;
    }
    PIC_HD int64_t value() const { return 4 * hi + (x >> 30); }
};

// A field value in the fixed point of a tile whose largest magnitude has the exponent field emax:
// round(F 2^(60 - E)) with |F| < 2^E, E = emax - 1022.  Only zero gives zero: a value below half a
// unit gives one unit of its sign.
PIC_HD int64_t field_fixed(uint64_t bits, int emax)
{
    const int e = (int)(bits >> 52) & 0x7ff;
    const uint64_t f = bits & 0xfffffffffffffull;
    const uint64_t m = e == 0 ? 0 : (f | ((uint64_t)1 << 52)) << 7;
    const int r = emax - e;
    uint64_t v = r > 61 ? 0 : (r > 0 ? ((m >> (r - 1)) + 1) >> 1 : m);
    if (v == 0 && (e | (f != 0)) != 0) v = 1;
    return (bits >> 63) ? -(int64_t)v : (int64_t)v;
}

// One unit of the gather is at most one FP64 rounding of the largest field in a stencil that holds a
// field of 2^53 units or more, one whose exponent field is less than kSmallField below emax.
constexpr int kSmallField = 7;

// Esirkepov window of one axis in U62: weights of the old (s0) and the new position (s1) on
// l + 2 nodes starting at node wb relative to the old cell (AxisS in fixed point).
template <int L>
struct AxisS62 {
    int wb;
    bool wide;
    uint64_t s0[L + 2], s1[L + 2];
};

template <int L>
PIC_HD void axis_shapes62(uint64_t f_old, uint64_t f_new, int sh, AxisS62<L> &s)
{
    uint64_t p0, p1, w0[L + 1], w1[L + 1];
    const int b0 = spline_base62<L>(f_old, false, p0);
    const int b1 = sh + spline_base62<L>(f_new, false, p1);
    bspline62<L>(p0, w0);
    bspline62<L>(p1, w1);
    s.wb = b0 < b1 ? b0 : b1;
    s.wide = b0 != b1;
    const bool m0 = b0 > s.wb, m1 = b1 > s.wb;
#pragma unroll
    for (int k = 0; k < L + 2; ++k) {
        const uint64_t a0 = k <= L ? w0[k] : 0, a1 = k >= 1 ? w0[k - 1] : 0;
        const uint64_t c0 = k <= L ? w1[k] : 0, c1 = k >= 1 ? w1[k - 1] : 0;
        s.s0[k] = m0 ? a1 : a0;
        s.s1[k] = m1 ? c1 : c0;
    }
}

// Magnitudes of the prefix sums of s1 - s0: a particle that moves up takes charge from the
// nodes below, so every prefix sum has the sign opposite to the move's (up: moved up).
template <int L>
PIC_HD void prefix62(const AxisS62<L> &s, bool up, uint64_t *q)
{
    uint64_t acc = 0;
#pragma unroll
    for (int k = 0; k <= L; ++k) {
        acc += s.s0[k] - s.s1[k];
        q[k] = nonneg(up ? acc : 0 - acc);
    }
}

}  // namespace pic
