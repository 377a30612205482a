// passes_fixed_any.cuh -- the fixed-point passes of passes_fixed.cuh for any length L = 2^a 3^b 5^c (and
// any n <= L): stage structure from the table, two buffers per group (a stage reads one and writes the
// other, so a thread can work through as many butterflies as the radix gives it, one barrier a stage).
#pragma once
#include "passes_fixed.cuh"

namespace wsc {

struct FixedAny {
    const FixedArgs &a;
    const int lt, g, tpt, L;
    unsigned *slot;
    c64 *cur, *oth;
    int r = 0;  // the line's first shift, applied by the first stage

    __device__ FixedAny(const FixedArgs &a_, int lt_, int g_, unsigned *slots, c64 *buf)
        : a(a_), lt(lt_), g(g_), tpt(a_.tpt), L(a_.L), slot(slots + FIXED_SLOTS * g_), cur(buf), oth(buf + fixed_padded(a_.L)) {}
    __device__ __forceinline__ void sync() const { group_sync(tpt, g); }
    __device__ __forceinline__ void clear(int i) const
    {
        if (tpt > 32 && lt == 0) slot[i] = slot[i + 1] = 0;
    }
    // sets r; returns t (fixed_norm)
    __device__ __forceinline__ int norm(unsigned l1, int i)
    {
        return fixed_norm(l1, slot + i, tpt, 32 - __clz(a.P.R[0] - 1), r);
    }
    // the line from doubles ld(e), e < nin, into cur (zeros beyond); exponent and total shift
    template <class Ld> __device__ __forceinline__ int load(int nin, int i, int &T, const Ld &ld)
    {
        constexpr int P = 61;
        unsigned xm = 0, s = 0;
#pragma unroll 4
        for (int e = lt; e < nin; e += tpt) {
            const double2 d = ld(e);
            xm = max(xm, max(dexp(d.x), dexp(d.y)));
        }
        xm = fixed_group_max(xm, slot + i, lt, g, tpt);
#pragma unroll 4
        for (int e = lt; e < nin; e += tpt) {
            const double2 d = ld(e);
            const c64 v = fixed_of<P>(d, xm);
            s += l1_of(v);
            cur[fpidx(e)] = v;
        }
        for (int e = nin + lt; e < L; e += tpt) cur[fpidx(e)] = {0, 0};
        const unsigned l1 = fixed_add_l1(s, slot + i + 1, lt, tpt);
        sync();
        T = norm(l1, i + 1);
        return (xm == 0x7ff ? FIXED_NAN : (int)xm - 1022 - P) + r;
    }
    // the products of x(e) 2^e1 and the multiplier, re and im exchanged, into cur (x may read cur)
    template <class X, class Mul> __device__ __forceinline__ int product(int e1, int i, int &T, const X &x, const Mul &mul)
    {
        constexpr int P = 61;
        int km = 0;
        unsigned s = 0;
#pragma unroll 2
        for (int e = lt; e < L; e += tpt) {
            c64 r;
            const int xg = mul(e, x(e), r);
            km = max(km, product_key(r, xg));
            oth[fpidx(e)] = {r.y, r.x};
        }
        km = (int)fixed_group_max((unsigned)km, slot + i, lt, g, tpt);
#pragma unroll 2
        for (int e = lt; e < L; e += tpt) {
            c64 none;
            const int xg = mul(e, c64{0, 0}, none);  // the exponent alone
            const c64 v = product_align(oth[fpidx(e)], P + xg - km);
            s += l1_of(v);
            cur[fpidx(e)] = v;
        }
        const unsigned l1 = fixed_add_l1(s, slot + i + 1, lt, tpt);
        sync();
        T = norm(l1, i + 1);
        return (km >= 4095 ? FIXED_NAN : e1 - 1020 - P + km) + r;
    }
    template <int R> __device__ __forceinline__ void stage(int s, int sh) const
    {
        const int nbf = L / R, Ns = a.P.Ns[s];
        const unsigned long long mag = a.P.mag[s];
        const int up = s ? max(2 - sh, 0) : 0;  // as FixedLine::raise
        sh += up;
        const int4 *tw = a.tw + a.P.toff[s] + (s ? (sh - 2) * (R - 1) * Ns : 0);
#pragma unroll 1
        for (int j = lt; j < nbf; j += tpt) {
            c64 v[R];
#pragma unroll
            for (int q = 0; q < R; ++q) v[q] = cur[fpidx(j + q * nbf)];
            const int jq = (int)(((unsigned long long)j * mag) >> 40), k = j - jq * Ns, o = jq * Ns * R + k;
            if (s) {
#pragma unroll
                for (int q = 0; q < R; ++q) {
                    v[q].x <<= up;
                    v[q].y <<= up;
                }
                twiddle<R>(v, sh, [&](int q) { return __ldg(tw + (q - 1) * Ns + k); });
            }
            else if (r > 0) {
#pragma unroll
                for (int q = 0; q < R; ++q) {
                    v[q].x = sar_round(v[q].x, r);
                    v[q].y = sar_round(v[q].y, r);
                }
            }
            fdft<R, false>(v);
#pragma unroll
            for (int p = 0; p < R; ++p) oth[fpidx(o + p * Ns)] = v[p];
        }
    }
    // the whole transform of cur; returns its cumulative shift
    __device__ __forceinline__ int transform(int T)
    {
        int c = 0;
        const int nst = a.P.nst;
#pragma unroll 1
        for (int s = 0; s < nst; ++s) {
            const int cn = s ? fixed_shift(a.P, T, s) : 0, sh = cn - c;
            c = cn;
            switch (a.P.R[s]) {
            case 16: stage<16>(s, sh); break;
            case 8: stage<8>(s, sh); break;
            case 4: stage<4>(s, sh); break;
            case 2: stage<2>(s, sh); break;
            case 3: stage<3>(s, sh); break;
            default: stage<5>(s, sh); break;
            }
            sync();
            c64 *t = cur;
            cur = oth;
            oth = t;
        }
        return c;
    }
};

#define WSC_FIXED_ANY_PROLOGUE                                                     \
    if (fixed_gives_up(a)) return;                                                 \
    const int tpt = a.tpt, g = threadIdx.x / tpt, lt = threadIdx.x - g * tpt, G = blockDim.x / tpt; \
    const int n = a.n, L = a.L, h = a.h;                                           \
    unsigned *slots;                                                               \
    const int4 *none;                                                              \
    c64 *buf = fixed_smem(a, g, G, 2, 0, slots, none);                             \
    FixedAny ln(a, lt, g, slots, buf);                                             \
    (void)h;

// Pass 1 (kx_rows_fwd)
template <int IN, bool MASK> __global__ void WSC_FIXED_LB ky_rows_fwd(const __grid_constant__ FixedArgs a)
{
    WSC_FIXED_ANY_PROLOGUE
    const int rows = IN == FIN_PAIR ? (n + 1) / 2 : n;
    for (int unit = blockIdx.x * G + g; unit < a.units; unit += gridDim.x * G) {
        const int b = unit / rows, j1 = (IN == FIN_PAIR ? 2 : 1) * (unit - b * rows);
        const bool has2 = IN == FIN_PAIR && j1 + 1 < n;
        const FixedIn<IN, MASK> src(a, n, b, j1, has2);
        int T;
        int e = ln.load(n, 0, T, [&](int i) -> double2 { return src(i); });
        e += ln.transform(T);
        ln.clear(0);
        if constexpr (IN == FIN_PAIR) {
            --e;
            const bool normal = fixed_normal(e);
            double2 *W = reinterpret_cast<double2 *>(a.out) + (size_t)b * h * n + j1;
            for (int k = lt; k < h; k += tpt)
                split_pair(ln.cur[fpidx(k)], ln.cur[fpidx(k == 0 ? 0 : L - k)], e, normal, has2, a.vec32, W + (size_t)k * n);
        } else {
            const bool normal = fixed_normal(e);
            double2 *W = reinterpret_cast<double2 *>(a.out) + (size_t)b * L * n + j1;
            for (int o = lt; o < L; o += tpt) {
                const c64 z = ln.cur[fpidx(o)];
                W[(size_t)o * n] = make_double2(from_fixed(z.x, e, normal), from_fixed(z.y, e, normal));
            }
        }
        ln.sync();
    }
}

// Pass 2 (kx_cols); the split pass always parks the spectrum in its global line
template <int MODE> __global__ void WSC_FIXED_LB ky_cols(const __grid_constant__ FixedArgs a)
{
    WSC_FIXED_ANY_PROLOGUE
    c64 *park = MODE == FCOL_SPLIT ? a.scratch + ((size_t)blockIdx.x * G + g) * L : nullptr;
    const int cols = a.units / a.batch;
    for (int unit = blockIdx.x * G + g; unit < a.units; unit += gridDim.x * G) {
        const int k2 = unit / a.batch, b = unit - k2 * a.batch;
        const size_t co = ((size_t)b * cols + k2) * n;
        const double2 *cin = reinterpret_cast<const double2 *>(a.in) + co;
        double2 *cout = reinterpret_cast<double2 *>(a.out) + (MODE == FCOL_SPLIT ? 2 * co : co);
        const int k2q = k2 < h ? k2 : L - k2;
        const void *gt = a.nsel ? a.gsel[b] : a.ghat;
        int T;
        int e = ln.load(n, 0, T, [&](int i) -> double2 { return cin[i]; });
        ln.clear(2);
        e += ln.transform(T);
        ln.clear(0);
        const int e1 = e;
        if (MODE == FCOL_SPLIT)
            for (int o = lt; o < L; o += tpt) park[o] = ln.cur[fpidx(o)];
#pragma unroll 1
        for (int part = 0; part < (MODE == FCOL_SPLIT ? 2 : 1); ++part) {
            auto x = [&](int o) -> c64 { return MODE == FCOL_SPLIT && part == 1 ? park[o] : ln.cur[fpidx(o)]; };
            auto mul = [&](int o, c64 z, c64 &r) -> int { return multiply<MODE>(a, gt, k2q, o, L, h, part, z, r); };
            e = ln.product(e1, 2, T, x, mul);
            e += ln.transform(T);
            const bool normal = fixed_normal(e);
            for (int o = lt; o < n; o += tpt) {
                const c64 z = ln.cur[fpidx(o)];
                const double2 w = make_double2(from_fixed(z.y, e, normal), from_fixed(z.x, e, normal));
                if constexpr (MODE == FCOL_SPLIT) cout[2 * o + part] = w;
                else cout[o] = w;
            }
            ln.sync();
            if (MODE == FCOL_SPLIT && part == 0) {
                ln.clear(2);
                ln.sync();
            }
        }
    }
}

// Pass 3 (kx_rows_inv)
template <int OUT, bool BETA> __global__ void WSC_FIXED_LB ky_rows_inv(const __grid_constant__ FixedArgs a)
{
    WSC_FIXED_ANY_PROLOGUE
    constexpr bool PAIRS = OUT == FOUT_R2R || OUT == FOUT_SPLIT;
    const int rows = OUT == FOUT_R2R ? (n + 1) / 2 : n;
    for (int unit = blockIdx.x * G + g; unit < a.units; unit += gridDim.x * G) {
        const int b = unit / rows, j1 = (OUT == FOUT_R2R ? 2 : 1) * (unit - b * rows);
        const bool has2 = OUT != FOUT_R2R || j1 + 1 < n;
        int e, T;
        if constexpr (PAIRS) {
            constexpr int P = 60;
            const size_t ld = OUT == FOUT_R2R ? n : 2 * (size_t)n;
            const double2 *W = reinterpret_cast<const double2 *>(a.in) + (size_t)b * h * ld + (OUT == FOUT_R2R ? j1 : 2 * j1);
            const double2 zero = make_double2(0.0, 0.0);
            unsigned xm = 0, s = 0;
#pragma unroll 4
            for (int k = lt; k < h; k += tpt) {
                const double2 *w = W + (size_t)k * ld;
                const double2 A = w[0], B = has2 ? w[1] : zero;
                xm = max(xm, max(max(dexp(A.x), dexp(A.y)), max(dexp(B.x), dexp(B.y))));
            }
            xm = fixed_group_max(xm, slots + FIXED_SLOTS * g, lt, g, tpt);
#pragma unroll 2
            for (int k = lt; k < h; k += tpt) {
                const double2 *w = W + (size_t)k * ld;
                s += merge_pair<P>(w[0], has2 ? w[1] : zero, xm, k, L, ln.cur);
            }
            const unsigned l1 = fixed_add_l1(s, slots + FIXED_SLOTS * g + 1, lt, tpt);
            ln.sync();
            T = ln.norm(l1, 1);
            e = (xm == 0x7ff ? FIXED_NAN : (int)xm - 1022 - P) + ln.r;
        } else {
            const double2 *W = reinterpret_cast<const double2 *>(a.in) + (size_t)b * L * n + j1;
            e = ln.load(L, 0, T, [&](int i) -> double2 {
                const double2 w = W[(size_t)i * n];
                return make_double2(w.y, w.x);
            });
        }
        e += ln.transform(T);
        ln.clear(0);
        const FixedOut<OUT, BETA> put(a, (size_t)b * n * n + (size_t)j1 * n, e, has2);
        for (int o = lt; o < n; o += tpt) put(o, ln.cur[fpidx(o)]);
        ln.sync();
    }
}

}  // namespace wsc
