// fft_fixed.cuh -- the FP64 plans' shared-memory FFT in 64-bit fixed point.
//
// GB300 issues one FP64 instruction per SM every 16 cycles (two lanes a cycle; measured 1.96 FMA,
// 1.65 additions), but 64-bit integer additions at 50 lanes a cycle and 32 x 32 + 64-bit
// multiply-adds at 32 to 57.  A line of FP64 data is therefore transformed as 64-bit integers that
// share one exponent: additions are integer additions, a twiddle product is twelve multiply-adds
// (30 instructions; measured 14 SM cycles per warp, where the FP64 units take 64).
//
// Precision.  A line's integers are scaled to its largest component, |re|, |im| < 2^61, rounded (a
// dense line then moves down 3 or 4 bits, see fixed_norm).  FP64 butterflies round at 2^-53 of each
// intermediate value, whose size is the line's norm; here the rounding unit is 2^-60 ... 2^-62 of a
// bound on the result: the smaller of (growth so far) x (largest component) and the sum of all
// |components| (the L1 norm, which no unit-modulus combination exceeds).  A stage shifts right only
// as far as that bound needs, so sparse lines, whose L1 norm is small, keep their bits.  Against long
// double convolutions on the plan's own table (period-2 grids, n = 256 ... 4096; log, |x|^-1, |x|^-1/2 and
// Helmholtz kernels; white noise, smooth bumps, a disk's indicator; 18 cases, every output) the errors
// are 0.18 to 0.84 times the FP64 stages' in the 2-norm and 0.25 to 0.84 times in the maximum norm.
// On compact grids the rounding of the compact table, which both share, is the larger part: over 108
// cases (n = 64 ... 1024, period 2, 3 and compact, every io mode) 0.46 times on average and at most
// 0.92 times in the 2-norm; the largest error is above the FP64 stages' in two, both compact (1.2).
//
// Overflow.  Every value obeys |v| <= 2^62 in modulus: partial sums of a butterfly are combinations
// of disjoint inputs with unit-modulus weights, so the bound above covers them; the rotation
// q1 = (x + y, y - x) before its 1/sqrt 2 stays below 2^62.5; a twiddle product's cross sum is below
// 2^31 (sqrt 2 2^30) + 2^31 (sqrt 2 2^30.5) < 2^63, and a constant's below 0.87 2^63.
//
// A line with an infinity or a NaN becomes all NaN (its FP64 transform would be, but for a few
// infinities).  A line whose exponents leave the normal range is converted by scalbn.
#pragma once
#include <climits>

#include "fft_engine.cuh"
#include "wsconv_internal.h"

namespace wsc {

struct __align__(16) c64 { long long x, y; };

#define FIXED_NAN (1 << 20)  // a poisoned line's exponent

// v = h 2^32 + l with l signed
struct split64 { int h, l; };
__device__ __forceinline__ split64 split_of(long long v)
{
    split64 s;
    asm("mov.b64 {%0, %1}, %2;" : "=r"(s.l), "=r"(s.h) : "l"(v));
    s.h += (int)((unsigned)s.l >> 31);
    return s;
}
// The same for a factor whose halves are negated: where l is INT_MIN, whose negation is itself (one
// double in 2^23 ends in that pattern), v moves up by one unit
__device__ __forceinline__ split64 split_negatable(long long v) { return split_of(v + ((int)v == INT_MIN ? 1 : 0)); }
// a b + c, one 32 x 32 + 64-bit multiply-add
__device__ __forceinline__ long long mad_wide(int a, int b, long long c)
{
    long long r;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
}
// Rounding of a cross sum to its high word: 2^31, or with ties down
#define FX_UP 0x80000000ll
#define FX_DOWN 0x7fffffffll
// hi + (cross >> 32)
__device__ __forceinline__ long long add_high(long long hi, long long cross)
{
    int h;
    asm("{\n\t.reg .b32 l;\n\tmov.b64 {l, %0}, %1;\n\t}" : "=r"(h) : "l"(cross));
    long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(h), "r"(h >> 31));
    return hi + r;
}

// High words of the 128-bit products of z and w, without their low x low terms (below a quarter unit),
// rounded to nearest; hx, hy: FX_UP or FX_DOWN, the rounding of a tie in each component.  w's halves
// are negated in 32 bits: its imaginary part's low half must not be INT_MIN (split_negatable, and
// split_scaled for the tables).
//
// Ties matter: at k = 0 the twiddle is 1 and the product a plain shift, a quarter of whose results are
// ties.  Always resolved one way they leave a bias of an eighth of a unit in every such product of
// every line, which the butterfly and then the next pass add up coherently.  So the untwiddled
// input rounds ties to even, the others alternate over the butterfly (Thue-Morse, but for R/2, which
// is left over and goes to even, as do all of an odd radix), and the biases cancel in the sums.
__host__ __device__ constexpr bool ties_up(int q) { return ((q ^ (q >> 1) ^ (q >> 2) ^ (q >> 3)) & 1) != 0; }
__device__ __forceinline__ c64 cmulw(c64 z, int4 w, long long hx, long long hy)
{
    const split64 x = split_of(z.x), y = split_of(z.y);
    const int nih = -w.z, nil = -w.w;
    long long cr = mad_wide(x.l, w.x, hx), ci = mad_wide(y.l, w.x, hy);
    cr = mad_wide(x.h, w.y, cr);
    ci = mad_wide(y.h, w.y, ci);
    cr = mad_wide(y.l, nih, cr);
    ci = mad_wide(x.l, w.z, ci);
    cr = mad_wide(y.h, nil, cr);
    ci = mad_wide(x.h, w.w, ci);
    c64 r;
    r.x = add_high(mad_wide(y.h, nih, mad_wide(x.h, w.x, 0)), cr);
    r.y = add_high(mad_wide(x.h, w.z, mad_wide(y.h, w.x, 0)), ci);
    return r;
}

// Constants c, |c| < 1/2, in units of 2^-64 and split as h 2^32 + l; a factor f above 1/2 is v + v (f - 1).
struct kfix { int h, l; };
#define FX_NEG(k) kfix{-(k).h, -(k).l}
#define FX_C8M1 kfix{-326934918, -1804979899} // cos(pi/8) - 1
#define FX_S8 kfix{1643612827, -1163556025} // sin(pi/8)
#define FX_R2M1 kfix{-1257966796, -102865788} // sqrt(1/2) - 1
#define FX_H3M1 kfix{-575416509, -1033546850} // sin(2 pi/3) - 1
#define FX_C51 kfix{1327217885, -1079689717} // cos(2 pi/5)
#define FX_C52M1 kfix{-820265763, -1079689717} // -cos(4 pi/5) - 1
#define FX_S51M1 kfix{-210210662, 581434099} // sin(2 pi/5) - 1
#define FX_S52M1 kfix{-1770448860, -1429016722} // sin(4 pi/5) - 1
// v c, rounded
__device__ __forceinline__ long long kmul(long long v, kfix c)
{
    const split64 s = split_of(v);
    return add_high(mad_wide(s.h, c.h, 0), mad_wide(s.h, c.l, mad_wide(s.l, c.h, FX_UP)));
}
// z (c + i d)
__device__ __forceinline__ c64 kcmul(c64 z, kfix c, kfix d)
{
    const split64 x = split_of(z.x), y = split_of(z.y);
    long long cr = mad_wide(x.l, c.h, FX_UP), ci = mad_wide(y.l, c.h, FX_UP);
    cr = mad_wide(x.h, c.l, cr);
    ci = mad_wide(y.h, c.l, ci);
    cr = mad_wide(y.l, -d.h, cr);
    ci = mad_wide(x.l, d.h, ci);
    cr = mad_wide(y.h, -d.l, cr);
    ci = mad_wide(x.h, d.l, ci);
    c64 r;
    r.x = add_high(mad_wide(y.h, -d.h, mad_wide(x.h, c.h, 0)), cr);
    r.y = add_high(mad_wide(x.h, d.h, mad_wide(y.h, c.h, 0)), ci);
    return r;
}
// v / 2^s rounded to nearest, ties to even, s >= 1
__device__ __forceinline__ long long sar_round(long long v, int s)
{
    return (v + ((1ll << (s - 1)) - 1) + ((v >> s) & 1)) >> s;
}

// Input q of a butterfly times its twiddle w = w^(qk), over 2^sh (sh >= 2, w from the copy for sh).
template <int R, int Q> __device__ __forceinline__ void twiddle_one(c64 &x, int sh, int4 w)
{
    if constexpr (R % 2 || 2 * Q == R) {
        x = cmulw(x, w, FX_DOWN + ((x.x >> sh) & 1), FX_DOWN + ((x.y >> sh) & 1));
    } else {
        x = cmulw(x, w, ties_up(Q) ? FX_UP : FX_DOWN, ties_up(Q) ? FX_UP : FX_DOWN);
    }
}
// A butterfly's twiddles, w(q) loading w^(qk)
template <int R, int Q = 0, class W> __device__ __forceinline__ void twiddle(c64 *x, int sh, const W &w)
{
    if constexpr (Q == 0) {
        x[0].x = sar_round(x[0].x, sh);
        x[0].y = sar_round(x[0].y, sh);
    } else {
        twiddle_one<R, Q>(x[Q], sh, w(Q));
    }
    if constexpr (Q + 1 < R) twiddle<R, Q + 1>(x, sh, w);
}

// z c for c > 1/2 (k = c - 1), and for c < 1/2
__device__ __forceinline__ c64 cscale_m1(c64 z, kfix k)
{
    c64 r;
    r.x = z.x + kmul(z.x, k);
    r.y = z.y + kmul(z.y, k);
    return r;
}
__device__ __forceinline__ c64 cscale_k(c64 z, kfix k)
{
    c64 r;
    r.x = kmul(z.x, k);
    r.y = kmul(z.y, k);
    return r;
}
__device__ __forceinline__ c64 cmul_r2(c64 z) { return cscale_m1(z, FX_R2M1); }
// z w16^1 and z w16^3 (c - i s and s - i c with c = cos(pi/8), s = sin(pi/8)), z w16^9 = -z w16
__device__ __forceinline__ c64 cmul_w16(c64 z) { return cadd(z, kcmul(z, FX_C8M1, FX_NEG(FX_S8))); }
__device__ __forceinline__ c64 cmul_w48(c64 z)  // s - i c = -i (c + i s)
{
    const c64 t = cadd(z, kcmul(z, FX_C8M1, FX_S8));
    return rot<false>(t);
}

// Forward butterflies (the inverse transform is the forward one with re and im exchanged on both
// sides).  fft_engine.cuh's dft2 and dft4 are additions only and serve as they are.
// 16 points as 4 x 4, as dft16_layer2 of fft_engine.cuh.
__device__ __forceinline__ void fdft16_layer2(c64 (*y)[4], c64 *x)
{
    {
        c64 z[4] = {y[0][0], y[1][0], y[2][0], y[3][0]};
        dft4<false>(z);
        x[0] = z[0];
        x[4] = z[1];
        x[8] = z[2];
        x[12] = z[3];
    }
    {   // w16^r: (c, -s), (1 - i)/sqrt 2, (s, -c)
        const c64 z0 = y[0][1], z1 = cmul_w16(y[1][1]), z3 = cmul_w48(y[3][1]);
        const c64 z2 = cmul_r2(q1<false>(y[2][1]));
        const c64 a0 = cadd(z0, z2), a1 = csub(z0, z2), a2 = cadd(z1, z3), a3 = rot<false>(csub(z1, z3));
        x[1] = cadd(a0, a2);
        x[9] = csub(a0, a2);
        x[5] = cadd(a1, a3);
        x[13] = csub(a1, a3);
    }
    {   // w16^2r: (1 - i)/sqrt 2, -i, (-1 - i)/sqrt 2
        const c64 z0 = y[0][2], z2 = rot<false>(y[2][2]);
        const c64 z1 = cmul_r2(q1<false>(y[1][2])), z3 = cmul_r2(q3<false>(y[3][2]));
        const c64 a0 = cadd(z0, z2), a1 = csub(z0, z2), a2 = cadd(z1, z3), a3 = rot<false>(csub(z1, z3));
        x[2] = cadd(a0, a2);
        x[10] = csub(a0, a2);
        x[6] = cadd(a1, a3);
        x[14] = csub(a1, a3);
    }
    {   // w16^3r: (s, -c), (-1 - i)/sqrt 2, (-c, s)
        const c64 z0 = y[0][3], z1 = cmul_w48(y[1][3]), z3 = cmul_w16(y[3][3]);  // z3: minus w16^9
        const c64 z2 = cmul_r2(q3<false>(y[2][3]));
        const c64 a0 = cadd(z0, z2), a1 = csub(z0, z2), a2 = csub(z1, z3), a3 = rot<false>(cadd(z1, z3));
        x[3] = cadd(a0, a2);
        x[11] = csub(a0, a2);
        x[7] = cadd(a1, a3);
        x[15] = csub(a1, a3);
    }
}

// HALF: x[8..15] are zero (the zero extension of a line with n = L/2)
template <bool HALF> __device__ __forceinline__ void fdft16(c64 *x)
{
    c64 y[4][4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        if constexpr (HALF) {
            const c64 a = x[r], b = x[r + 4], rb = rot<false>(b);
            y[r][0] = cadd(a, b);
            y[r][1] = cadd(a, rb);
            y[r][2] = csub(a, b);
            y[r][3] = csub(a, rb);
        } else {
            y[r][0] = x[r];
            y[r][1] = x[r + 4];
            y[r][2] = x[r + 8];
            y[r][3] = x[r + 12];
            dft4<false>(y[r]);
        }
    }
    fdft16_layer2(y, x);
}

// twiddle<16> and fdft16 with the twiddle products of one first-layer butterfly next to the additions of
// another: the products fill the multiply pipe, the additions the ALU.
template <int RR = 0, class W> __device__ __forceinline__ void fdft16_layer1(c64 (*y)[4], c64 *x, int sh, const W &w)
{
    if constexpr (RR == 0) {
        x[0].x = sar_round(x[0].x, sh);
        x[0].y = sar_round(x[0].y, sh);
    } else {
        twiddle_one<16, RR>(x[RR], sh, w(RR));
    }
    twiddle_one<16, RR + 8>(x[RR + 8], sh, w(RR + 8));
    twiddle_one<16, RR + 4>(x[RR + 4], sh, w(RR + 4));
    twiddle_one<16, RR + 12>(x[RR + 12], sh, w(RR + 12));
    y[RR][0] = x[RR];
    y[RR][1] = x[RR + 4];
    y[RR][2] = x[RR + 8];
    y[RR][3] = x[RR + 12];
    dft4<false>(y[RR]);
    if constexpr (RR < 3) fdft16_layer1<RR + 1>(y, x, sh, w);
}
template <class W> __device__ __forceinline__ void fdft16_twiddled(c64 *x, int sh, const W &w)
{
    c64 y[4][4];
    fdft16_layer1(y, x, sh, w);
    fdft16_layer2(y, x);
}

__device__ __forceinline__ void fdft8(c64 *x)
{
    c64 e[4] = {x[0], x[2], x[4], x[6]}, o[4] = {x[1], x[3], x[5], x[7]};
    dft4<false>(e);
    dft4<false>(o);
    const c64 o1 = cmul_r2(q1<false>(o[1])), o2 = rot<false>(o[2]), o3 = cmul_r2(q3<false>(o[3]));
    x[0] = cadd(e[0], o[0]);
    x[4] = csub(e[0], o[0]);
    x[1] = cadd(e[1], o1);
    x[5] = csub(e[1], o1);
    x[2] = cadd(e[2], o2);
    x[6] = csub(e[2], o2);
    x[3] = cadd(e[3], o3);
    x[7] = csub(e[3], o3);
}

__device__ __forceinline__ void fdft3(c64 *x)
{
    const c64 t = cadd(x[1], x[2]), r = cscale_m1(rot<false>(csub(x[1], x[2])), FX_H3M1);
    c64 m;
    m.x = x[0].x - sar_round(t.x, 1);
    m.y = x[0].y - sar_round(t.y, 1);
    x[0] = cadd(x[0], t);
    x[1] = cadd(m, r);
    x[2] = csub(m, r);
}

__device__ __forceinline__ void fdft5(c64 *x)
{
    const c64 t1 = cadd(x[1], x[4]), t2 = cadd(x[2], x[3]), d1 = csub(x[1], x[4]), d2 = csub(x[2], x[3]);
    const c64 a1 = cadd(x[0], csub(cscale_k(t1, FX_C51), cscale_m1(t2, FX_C52M1)));
    const c64 a2 = cadd(x[0], csub(cscale_k(t2, FX_C51), cscale_m1(t1, FX_C52M1)));
    const c64 r1 = rot<false>(cadd(cscale_m1(d1, FX_S51M1), cscale_m1(d2, FX_S52M1)));
    const c64 r2 = rot<false>(csub(cscale_m1(d1, FX_S52M1), cscale_m1(d2, FX_S51M1)));
    x[0] = cadd(x[0], cadd(t1, t2));
    x[1] = cadd(a1, r1);
    x[4] = csub(a1, r1);
    x[2] = cadd(a2, r2);
    x[3] = csub(a2, r2);
}

template <int R, bool HALF> __device__ __forceinline__ void fdft(c64 *x)
{
    if constexpr (R == 2) dft2<false>(x);
    else if constexpr (R == 3) fdft3(x);
    else if constexpr (R == 4) dft4<false>(x);
    else if constexpr (R == 5) fdft5(x);
    else if constexpr (R == 8) fdft8(x);
    else fdft16<HALF>(x);
}

// ---------------------------------------------------------------------------- FP64 <-> fixed point
// Biased exponent of a double (0 and subnormals count as 1)
__device__ __forceinline__ unsigned dexp(double d)
{
    return max(((unsigned)__double2hiint(d) >> 20) & 0x7ffu, 1u);
}
// d 2^(P + 1022 - xm), rounded to nearest: |result| <= 2^P for exponents up to xm.  (Truncation would
// shrink every small component the same way, and smooth lines have many: the errors of a spectrum's
// tail then add up where the tail itself does.)
template <int P> __device__ __forceinline__ long long to_fixed(double d, int xm)
{
    const int hi = __double2hiint(d), lo = __double2loint(d);
    const int ex = (hi >> 20) & 0x7ff;
    const long long m = ((long long)((hi & 0xfffff) | (ex ? 0x100000 : 0)) << 32) | (unsigned)lo;
    const unsigned long long twice = (unsigned long long)(m << (P - 52)) >> min(xm - max(ex, 1), 63);
    const long long v = (long long)((twice + 1) >> 1), s = hi >> 31;
    return (v ^ s) - s;
}

static __device__ __noinline__ double from_fixed_slow(long long v, int e)
{
    if (e > FIXED_NAN / 2) return __longlong_as_double(0x7ff8000000000000ll);
    return scalbn((double)v, e);
}
// 32 bytes by one access (q 32-byte aligned)
__device__ __forceinline__ void ld32(const double2 *q, double2 &a, double2 &b)
{
    asm volatile("ld.global.v4.f64 {%0, %1, %2, %3}, [%4];" : "=d"(a.x), "=d"(a.y), "=d"(b.x), "=d"(b.y) : "l"(q));
}
__device__ __forceinline__ void st32(double2 *q, double2 a, double2 b)
{
    asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(q), "d"(a.x), "d"(a.y), "d"(b.x), "d"(b.y) : "memory");
}
__device__ __forceinline__ void prefetch_l2(const void *q) { asm volatile("prefetch.global.L2 [%0];" ::"l"(q)); }

// Whether from_fixed's fast path covers every value of a line with exponent e
__device__ __forceinline__ bool fixed_normal(int e) { return e >= -1020 && e <= 950; }
// v 2^e, rounded to nearest (ties away from zero); normal: fixed_normal(e)
__device__ __forceinline__ double from_fixed(long long v, int e, bool normal)
{
    if (!normal) return v == 0 && e < FIXED_NAN / 2 ? 0.0 : from_fixed_slow(v, e);  // empty lines: zeros
    const long long s = v >> 63;
    const unsigned long long m = (unsigned long long)((v ^ s) - s);
    const int z = __clzll((long long)m);
    const unsigned long long r = ((m << (z - 1)) + 0x200) >> 10;  // the leading one at bit 52 (53 on a carry)
    int hi = (int)(r >> 32) + ((1085 + e - z) << 20);
    hi = m == 0 ? 0 : hi | ((int)(s >> 32) & 0x80000000);
    return __hiloint2double(hi, (int)r);
}

}  // namespace wsc
