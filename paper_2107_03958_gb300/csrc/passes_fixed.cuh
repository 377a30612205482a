// passes_fixed.cuh -- the three convolution passes of FP64 plans on the fixed-point transform of
// fft_fixed.cuh.  Layouts, work items and roles are those of passes_fused.cuh (W[k2][j1], row pairs,
// columns batch-fastest, the split R2C pipeline's (Wr, Wi) pairs); global memory holds FP64, each
// line becomes fixed point when it enters shared memory and FP64 again when it leaves.
//
// A group of `tpt` threads (16 elements each) owns one line; a CTA holds up to 512 / tpt groups that
// run independently (each has its own named barrier, or is one warp).  A line's exponent comes from
// the largest biased exponent of its inputs (one warp reduction, one shared-memory maximum, the
// barrier the stage needs anyway), its shifts from the L1 norm summed beside the first stage.
//
// Bound: integer issue.  At L = 8192 a column takes 9400 instructions a thread (5000 on the ALU pipe, 1400
// 64-bit multiply-adds); the ALU pipe is 55 % busy with 16 warps an SM, DRAM at a tenth of its rate.
// n = 4096, batch 16, log kernel, against the same passes on the FP64 units: pass 1 21.8 -> 4.6 ms,
// pass 2 80.5 -> 16.3 ms, pass 3 23 -> 6.4 ms.
//
// LL: the line's length, a power of two with n = L/2: indices fold into constants, the zero half of
// the input and the cropped half of the output drop out.  Other lengths: passes_fixed_any.cuh.
#pragma once
#include <algorithm>

#include "fft_fixed.cuh"
#include "wsconv_internal.h"

namespace wsc {

struct FixedArgs {
    const void *in;        // pass 1: u; passes 2, 3: the spectrum
    const double *mask;    // pass 1: optional n x n multiplier
    void *out;
    const void *ghat;      // pass 2: FP64 multiplier quadrant [k2][k1]
    const void *u;         // pass 3: u for the beta term
    const int4 *tw;        // twiddle table (FixedDesc)
    int n, h, L, tpt, units, batch;
    double2 alpha;         // pass 3 scale, times 1/M^2
    int ah, al, ae;        // alpha.x = (ah 2^32 + al) 2^(ae - 63); ah = 0: complex alpha (FP64 product)
    double beta;
    int *err, give_up;     // injected fault: report a given-up wait and leave
    int odd, nsel, one;    // one: the split pass 2 parks the spectrum in global scratch lines
    int vec32;             // pass 1 output / pass 3 input: the spectrum pairs lie on 32-byte boundaries
    const void *gsel[WSC_MAX_SEL];
    c64 *scratch;
    FixedDesc P;
};

__device__ __forceinline__ int fpidx(int e) { return e + (e >> 3); }
__host__ __device__ inline int fixed_padded(int L) { return L + (L >> 3) + 1; }
// Entries of the twiddle table that the compile-time lengths' CTAs keep in shared memory: stage 1's three
// copies (Ns = 16) and, to L = 2048, the whole table; from L = 4096 the first copy of stage 2 (Ns = 256, 61 KB;
// its other copies, for lines whose L1 norm nears n times their largest value, are read from
// global memory, as is the last stage's table at L = 8192).  Beside the 147 KB of lines the L1 cache
// that is left, 64 KB, would hold neither.
__host__ __device__ constexpr bool fixed_tw_whole(int L) { return L <= 2048; }
__host__ __device__ constexpr int fixed_tw_smem(int L)
{
    return 720 + (L == 512 ? 256 : L == 1024 ? 768 : L == 2048 ? 3584 : 3840);
}
#define FIXED_SLOTS 4  // per group: maxima and L1 sums of the forward and the inverse transform

// ---- group-wide helpers; a group is one warp or whole warps with the named barrier g + 1
__device__ __forceinline__ void group_sync(int tpt, int g)
{
    if (tpt == 32) __syncwarp();
    else asm volatile("bar.sync %0, %1;" ::"r"(g + 1), "r"(tpt) : "memory");
}
// the group's largest v (slot is 0 before); every thread of the group passes a barrier here
__device__ __forceinline__ unsigned fixed_group_max(unsigned v, unsigned *slot, int lt, int g, int tpt)
{
    v = __reduce_max_sync(0xffffffffu, v);
    if (tpt > 32) {
        if ((lt & 31) == 0) atomicMax(slot, v);
        group_sync(tpt, g);
        return *reinterpret_cast<volatile unsigned *>(slot);
    }
    __syncwarp();
    return v;
}
// the line's L1 norm in units of 2^47, rounded up, from the threads' sums of l1_of: in the slot after
// the group's next barrier (one warp: the return value)
__device__ __forceinline__ unsigned fixed_add_l1(unsigned s, unsigned *slot, int lt, int tpt)
{
    const unsigned v = __reduce_add_sync(0xffffffffu, (s >> 10) + 1);
    if (tpt > 32 && (lt & 31) == 0) atomicAdd(slot, v);
    return v;
}
// The line's first shift r and t, the shift that would then bring its L1 norm to 2^62.  Lines start
// with components up to 2^61 and the first stage adds up 2^grow of them: r = grow for a dense line,
// less where the L1 norm is less than that (spectra of smooth densities: the tail's quantisation is
// the transform's largest error, 2^-61 of the largest component instead of 2^-57).
__device__ __forceinline__ int fixed_norm(unsigned l1, const unsigned *slot, int tpt, int grow, int &r)
{
    if (tpt > 32) l1 = *reinterpret_cast<const volatile unsigned *>(slot);
    const int t = 17 - __clz((int)l1);
    r = max(0, min(t, grow));
    return t - r;
}
// Cumulative shift after stage s >= 1, t = fixed_norm.  With the bounds 2^(62 + min(t, lg)) on the
// unshifted values, this keeps every stored value within 2^62, and within 2^60 before a stage that
// shifts by less than the 2 bits of its twiddle product (whose inputs first move up by the rest), so
// that no bit is given up that the bound does not ask for.
__device__ __forceinline__ int fixed_shift(const FixedDesc &P, int t, int s)
{
    return max(min(t, P.lg[s]), min(t, P.lg[s - 1]) + 2);
}
template <int P> __device__ __forceinline__ c64 fixed_of(double2 d, int xm)
{
    return {to_fixed<P>(d.x, xm), to_fixed<P>(d.y, xm)};
}
// |re| + |im| in units of 2^37, rounded up
__device__ __forceinline__ unsigned l1_of(c64 v)
{
    const int x = (int)(v.x >> 32), y = (int)(v.y >> 32);
    return (((unsigned)(x < 0 ? -x : x) + (unsigned)(y < 0 ? -y : y)) >> 5) + 1u;
}
// bound on log2 of a product's components, biased
__device__ __forceinline__ int product_key(c64 r, int xg)
{
    const long long m = (r.x ^ (r.x >> 63)) | (r.y ^ (r.y >> 63));
    return xg + 64 - __clzll(m);
}
// v 2^sh, rounded where sh < 0
__device__ __forceinline__ c64 product_align(c64 v, int sh)
{
    const int up = max(sh, 0), dn = min(max(-sh, 0), 62);
    const long long half = (1ll << dn) >> 1;
    v.x = ((v.x << up) + half) >> dn;
    v.y = ((v.y << up) + half) >> dn;
    return v;
}

// The sign of e in the Rudin-Shapiro sequence, as a bit: the parity of its pairs of adjacent ones.  The
// ties of a line's first shift go by it.  A tie rule leaves a bias of up to a quarter unit with a
// pattern of its own in every line; the transform adds the pattern up at its frequencies, and the next
// pass adds the lines up.  A rule that alternated over the sixteen blocks of a line (46 % of the line's length
// at one frequency) put it into outputs 3 and 5 of every row: white noise at n = 4096 had errors of
// 9.7e-16 of the largest value there.  This pattern (over lt, times the same over q) has 2 % at most at
// any frequency, which is lost in the rounding noise: 3.9e-16.
__device__ __forceinline__ unsigned rs_bit(int e) { return __popc((unsigned)(e & (e >> 1))) & 1; }
__host__ __device__ constexpr int rs_bit_of(int q)  // q < 16
{
    return ((q & (q >> 1)) ^ ((q & (q >> 1)) >> 1) ^ ((q & (q >> 1)) >> 2)) & 1;
}

// One group's line of compile-time length LL = 16^m 2^r.  All members of the group call every
// function together.
template <int LL> struct FixedLine {
    static constexpr int TPT = LL / 16;
    const FixedArgs &a;
    const int lt, g;
    unsigned *slot;
    const int4 *tws;  // shared-memory copy of the table's first fixed_tw_smem(LL) entries

    __device__ FixedLine(const FixedArgs &a_, int lt_, int g_, unsigned *slots, const int4 *tws_)
        : a(a_), lt(lt_), g(g_), slot(slots + FIXED_SLOTS * g_), tws(tws_) {}
    __device__ __forceinline__ void sync() const { group_sync(TPT, g); }
    __device__ __forceinline__ unsigned group_max(unsigned v, int i) const { return fixed_group_max(v, slot + i, lt, g, TPT); }
    __device__ __forceinline__ unsigned add_l1(unsigned s, int i) const { return fixed_add_l1(s, slot + i, lt, TPT); }
    // buffer index of element lt + c, c a multiple of the padding period
    __device__ __forceinline__ int at(int c) const { return fpidx(lt) + c + (c >> 3); }
    // v / 2^r, rounded; ties of element lt + q TPT up or down by the signs of lt and q (rs_bit)
    template <int N> __device__ __forceinline__ void lower(c64 *v, int r) const
    {
        if (r == 0) return;
        const unsigned half = (1u << r) >> 1, s = rs_bit(lt);
        const unsigned h[2] = {half - s, half - (s ^ 1)};
#pragma unroll
        for (int q = 0; q < N; ++q) {
            v[q].x = (v[q].x + h[rs_bit_of(q)]) >> r;
            v[q].y = (v[q].y + h[rs_bit_of(q)]) >> r;
        }
    }
    // first stage (Ns = 1): the butterfly of v, outputs 16 lt + p
    template <bool HALF> __device__ __forceinline__ void store0(c64 *v, c64 *buf) const
    {
        fdft16<HALF>(v);
        c64 *o = buf + 18 * lt;
#pragma unroll
        for (int p = 0; p < 16; ++p) o[p + (p >> 3)] = v[p];
        sync();
    }
    // first stage on doubles ld(e), e < LL/2 (HALF) or e < LL; returns the line's exponent, sets t
    template <bool HALF, class Ld>
    __device__ __forceinline__ int first_doubles(c64 *buf, int &t, int i, const Ld &ld) const
    {
        constexpr int NQ = HALF ? 8 : 16, P = 61;
        c64 v[16];
        unsigned xm = 0;
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const double2 d = ld(lt + q * TPT);
            xm = max(xm, max(dexp(d.x), dexp(d.y)));
            v[q].x = __double_as_longlong(d.x);
            v[q].y = __double_as_longlong(d.y);
        }
        xm = group_max(xm, i);
        unsigned s = 0;
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            v[q] = fixed_of<P>(make_double2(__longlong_as_double(v[q].x), __longlong_as_double(v[q].y)), xm);
            s += l1_of(v[q]);
        }
        const int r = normalise<HALF ? 3 : 4>(s, i + 1, t);
        lower<NQ>(v, r);
        store0<HALF>(v, buf);
        return xm == 0x7ff ? FIXED_NAN : (int)xm - 1022 - P + r;
    }
    // the line's first shift and t from the threads' L1 sums (a barrier)
    template <int GROW> __device__ __forceinline__ int normalise(unsigned s, int i, int &t) const
    {
        int r;
        const unsigned l1 = add_l1(s, i);
        sync();
        t = fixed_norm(l1, slot + i, TPT, GROW, r);
        return r;
    }
    // first stage on fixed-point values already in buf (natural order), their L1 sum added before the
    // last barrier; returns the first shift
    __device__ __forceinline__ int first_smem(c64 *buf, unsigned l1, int &t, int i) const
    {
        int r;
        t = fixed_norm(l1, slot + i, TPT, 4, r);
        c64 v[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) v[q] = buf[at(q * TPT)];
        sync();
        lower<16>(v, r);
        store0<false>(v, buf);
        return r;
    }
    // first stage on the products of the spectrum x(e) 2^e1 and the multiplier, re and im exchanged
    // (the inverse).  mul(e, x, r) gives the product's high words r and returns the multiplier's
    // biased exponent (4095 for an infinity or a NaN).
    template <class X, class Mul>
    __device__ __forceinline__ int first_product(c64 *buf, int e1, int &t, int i, const X &x, const Mul &mul) const
    {
        constexpr int P = 61;
        c64 v[16];
        int xg[16];
        int km = 0;
#pragma unroll
        for (int q = 0; q < 16; ++q) {
            c64 r;
            xg[q] = mul(lt + q * TPT, x(q * TPT), r);
            km = max(km, product_key(r, xg[q]));
            v[q].x = r.y;
            v[q].y = r.x;
        }
        km = (int)group_max((unsigned)km, i);
        unsigned s = 0;
#pragma unroll
        for (int q = 0; q < 16; ++q) {
            v[q] = product_align(v[q], P + xg[q] - km);
            s += l1_of(v[q]);
        }
        const int r = normalise<4>(s, i + 1, t);
        lower<16>(v, r);
        store0<false>(v, buf);
        return km >= 4095 ? FIXED_NAN : e1 - 1020 - P + km + r;
    }
    // v <<= 2 - sh where a stage's shift sh is below the 2 bits of its twiddle product; returns the
    // product's shift
    template <int N> static __device__ __forceinline__ int raise(c64 *v, int sh)
    {
        if (sh < 2) {
#pragma unroll
            for (int q = 0; q < N; ++q) {
                v[q].x <<= 2 - sh;
                v[q].y <<= 2 - sh;
            }
        }
        return max(sh, 2);
    }
    template <int R, class W> static __device__ __forceinline__ void twiddled(c64 *x, int sh, const W &w)
    {
        if constexpr (R == 16) {
            fdft16_twiddled(x, sh, w);
        } else {
            twiddle<R>(x, sh, w);
            fdft<R, false>(x);
        }
    }
    // x[q] *= w^(qk), all over 2^sh (2 + the twiddle copy's),
    // and the butterfly
    template <int R> __device__ __forceinline__ void butterfly(c64 *x, int s, int sh, int Ns, int k) const
    {
        const int o = a.P.toff[s] + (sh - 2) * (R - 1) * Ns + k;
        if constexpr (fixed_tw_whole(LL)) {
            twiddled<R>(x, sh, [&](int q) { return tws[o + (q - 1) * Ns]; });
        } else {
            const int4 *t = (o < fixed_tw_smem(LL) ? tws : a.tw) + o;
            twiddled<R>(x, sh, [&](int q) { return t[(q - 1) * Ns]; });
        }
    }
    // stages 1 ... nst - 2, radix 16; returns the cumulative shift
    __device__ __forceinline__ int mids(c64 *buf, int T) const
    {
        int c = 0;
        const int last = a.P.nst - 1;
#pragma unroll 1
        for (int s = 1; s < last; ++s) {
            const int cn = fixed_shift(a.P, T, s), ls = 4 * s, Ns = 1 << ls;
            int sh = cn - c;
            c = cn;
            c64 v[16];
#pragma unroll
            for (int q = 0; q < 16; ++q) v[q] = buf[at(q * TPT)];
            sync();
            sh = raise<16>(v, sh);
            const int k = lt & (Ns - 1), o = ((lt >> ls) << (ls + 4)) + k, st = Ns + (Ns >> 3);
            butterfly<16>(v, s, sh, Ns, k);
            c64 *ob = buf + fpidx(o);
#pragma unroll
            for (int p = 0; p < 16; ++p) ob[p * st] = v[p];
            sync();
        }
        return c;
    }
    // last stage: outputs to buf (SMEM) and to dst(o, z); HALF: only o < LL/2 are wanted
    template <bool SMEM, bool HALF, class Dst>
    __device__ __forceinline__ void last(c64 *buf, int sh, const Dst &dst) const
    {
        constexpr int l2 = LL == 512 ? 9 : LL == 1024 ? 10 : LL == 2048 ? 11 : LL == 4096 ? 12 : 13;
        constexpr int R = l2 % 4 ? 1 << (l2 % 4) : 16, NB = 16 / R, Ns = LL / R;
        const int s = a.P.nst - 1;
        c64 v[NB][R];
#pragma unroll
        for (int b = 0; b < NB; ++b)
#pragma unroll
            for (int q = 0; q < R; ++q) v[b][q] = buf[at(b * TPT + q * Ns)];
        if constexpr (SMEM) sync();
        sh = raise<16>(&v[0][0], sh);
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            const int j = lt + b * TPT;
            if (LL == 8192 && b >= NB / 2) {  // w^(k + L/4) = -i w^k: the table stops at L/4
                v[b][1] = rot<false>(v[b][1]);
                butterfly<R>(v[b], s, sh, Ns, j - LL / 4);
            } else {
                butterfly<R>(v[b], s, sh, Ns, j);
            }
#pragma unroll
            for (int p = 0; p < (HALF ? R / 2 : R); ++p) {
                if constexpr (SMEM) buf[at(b * TPT + p * Ns)] = v[b][p];
                dst(j + p * Ns, v[b][p]);
            }
            asm volatile("" ::: "memory");
        }
        if constexpr (SMEM) sync();
    }
    // shift of the last stage; adds the whole shift to the line's exponent
    __device__ __forceinline__ int last_shift(int c, int T, int &e) const
    {
        const int cn = fixed_shift(a.P, T, a.P.nst - 1);
        e += cn;
        return cn - c;
    }
    // one thread clears the slots i, i + 1 (between barriers that separate their uses)
    __device__ __forceinline__ void clear(int i) const
    {
        if (TPT > 32 && lt == 0) slot[i] = slot[i + 1] = 0;
    }
};

// Host side (passes_fixed.cu): alpha = (ah 2^32 + al) 2^(ae - 63); ah = 0 where that form does not serve
void fixed_alpha(double re, double im, int &ah, int &al, int &ae);
template <int LL> conv_status run_fixed(conv_plan_s *p, const void *u, const void *mask, void *out, int batch, double are,
                                        double aim, double beta, void *ws, cudaStream_t st);
template <int LL> conv_status set_attrs_fixed(int smem);

struct NoDst {
    __device__ __forceinline__ void operator()(int, c64) const {}
};

// Shared memory: [twiddles][group 0's buffers][group 1's] ... [slots].  Returns this group's first
// buffer, after the CTA has copied ntw twiddle entries and cleared the slots.
__device__ __forceinline__ c64 *fixed_smem(const FixedArgs &a, int g, int G, int nbuf, int ntw, unsigned *&slots, const int4 *&tws)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int4 *t = reinterpret_cast<int4 *>(smem_raw);
    c64 *base = reinterpret_cast<c64 *>(t + ntw);
    const int per = fixed_padded(a.L) * nbuf;
    slots = reinterpret_cast<unsigned *>(base + (size_t)per * G);
    for (int i = threadIdx.x; i < ntw; i += blockDim.x) t[i] = __ldg(a.tw + i);
    for (int i = threadIdx.x; i < FIXED_SLOTS * G; i += blockDim.x) slots[i] = 0;
    __syncthreads();
    pdl_wait();
    tws = t;
    return base + (size_t)per * g;
}

// An injected fault (CONV_FAULT_WAIT): report it and leave, as a given-up wait does elsewhere.
__device__ __forceinline__ bool fixed_gives_up(const FixedArgs &a)
{
    if (!a.give_up) return false;
    pdl_wait();
    if (threadIdx.x == 0) atomicExch(a.err, (int)CONV_ETIMEOUT);
    return true;
}

// The group's next input, `bytes` at base + off, into L2 while this line is transformed
__device__ __forceinline__ void prefetch_line(bool on, const void *base, size_t off, int bytes, int lt, int tpt)
{
    if (!on) return;
    for (int i = 128 * lt; i < bytes; i += 128 * tpt) prefetch_l2(reinterpret_cast<const char *>(base) + off + i);
}

#define WSC_FIXED_LB __launch_bounds__(512, 1)
#define WSC_FIXED_PROLOGUE(NBUF)                                                   \
    if (fixed_gives_up(a)) return;                                                 \
    constexpr int tpt = LL / 16, L = LL, h = LL / 2 + 1, n = LL / 2;               \
    const int g = threadIdx.x / tpt, lt = threadIdx.x - g * tpt, G = blockDim.x / tpt; \
    unsigned *slots;                                                               \
    const int4 *tws;                                                               \
    c64 *buf = fixed_smem(a, g, G, NBUF, fixed_tw_smem(LL), slots, tws);           \
    const FixedLine<LL> ln(a, lt, g, slots, tws);                                  \
    (void)n; (void)L; (void)h;

enum { FIN_PAIR = 0, FIN_REAL = 1, FIN_CPLX = 2 };

// Element i of a line of pass 1: u (times the mask) of row j1, or of the row pair j1, j1 + 1.
template <int IN, bool MASK> struct FixedIn {
    const double *u, *m;
    const int n;
    const bool has2;
    __device__ FixedIn(const FixedArgs &a, int n_, int b, int j1, bool has2_)
        : u(reinterpret_cast<const double *>(a.in) + ((size_t)b * n_ * n_ + (size_t)j1 * n_) * (IN == FIN_CPLX ? 2 : 1)),
          m(a.mask + (size_t)j1 * n_), n(n_), has2(has2_) {}
    __device__ __forceinline__ double2 operator()(int i) const
    {
        double2 z;
        if constexpr (IN == FIN_CPLX) z = reinterpret_cast<const double2 *>(u)[i];
        else z = make_double2(u[i], has2 ? u[n + i] : 0.0);
        if constexpr (MASK) {
            z.x *= m[i];
            if constexpr (IN == FIN_CPLX) z.y *= m[i];
            else if (has2) z.y *= m[n + i];
        }
        return z;
    }
};

// Spectra of the two real rows of a pair from Z_k and Z_(L-k) (values times 2^e, e one below Z's).
__device__ __forceinline__ void split_pair(c64 zk, c64 zm, int e, bool normal, bool has2, bool vec32, double2 *w)
{
    const double2 A = make_double2(from_fixed(zk.x + zm.x, e, normal), from_fixed(zk.y - zm.y, e, normal));
    const double2 B = make_double2(from_fixed(zk.y + zm.y, e, normal), from_fixed(zm.x - zk.x, e, normal));
    if (vec32) {
        st32(w, A, B);
    } else {
        w[0] = A;
        if (has2) w[1] = B;
    }
}

// Pass 1.  FIN_PAIR: two real rows per line, split into their spectra W[k][j1], W[k][j1 + 1] (k <= L/2);
// FIN_REAL, FIN_CPLX: one row, W[o][j1] for every o < L (the C2C layout).
template <int LL, int IN, bool MASK> __global__ void WSC_FIXED_LB kx_rows_fwd(const __grid_constant__ FixedArgs a)
{
    WSC_FIXED_PROLOGUE(1)
    const int rows = IN == FIN_PAIR ? (n + 1) / 2 : n;
    for (int unit = blockIdx.x * G + g; unit < a.units; unit += gridDim.x * G) {
        const int b = unit / rows, j1 = (IN == FIN_PAIR ? 2 : 1) * (unit - b * rows);
        const bool has2 = IN == FIN_PAIR && j1 + 1 < n;
        const FixedIn<IN, MASK> src(a, n, b, j1, has2);
        prefetch_line(unit + gridDim.x * G < a.units, a.in, (size_t)(unit + gridDim.x * G) * n * (IN == FIN_REAL ? 8 : 16),
                      n * (IN == FIN_REAL ? 8 : 16), lt, tpt);
        int T;
        int e = ln.template first_doubles<true>(buf, T, 0, [&](int i) -> double2 { return src(i); });
        const int c = ln.mids(buf, T), sh = ln.last_shift(c, T, e);
        if constexpr (IN == FIN_PAIR) {
            ln.template last<true, false>(buf, sh, NoDst{});
            ln.clear(0);
            --e;  // the halves of the Hermitian split
            const bool normal = fixed_normal(e);
            double2 *W = reinterpret_cast<double2 *>(a.out) + (size_t)b * h * n + j1;
#pragma unroll 2
            for (int k = lt; k < h; k += tpt) {
                split_pair(buf[fpidx(k)], buf[fpidx(k == 0 ? 0 : L - k)], e, normal, has2, a.vec32, W + (size_t)k * n);
            }
            ln.sync();
        } else {
            const bool normal = fixed_normal(e);
            double2 *W = reinterpret_cast<double2 *>(a.out) + (size_t)b * L * n + j1;
            ln.template last<false, false>(buf, sh, [&](int o, c64 z) {
                W[(size_t)o * n] = make_double2(from_fixed(z.x, e, normal), from_fixed(z.y, e, normal));
            });
            ln.sync();
            ln.clear(0);
            ln.sync();
        }
    }
}

// The multiplier as a 62-bit integer: g = m 2^(x - 1084), returns x (4095 for an infinity or NaN).
__device__ __forceinline__ int mult_fixed(double g, long long &m)
{
    const int hi = __double2hiint(g), lo = __double2loint(g);
    const int ex = (hi >> 20) & 0x7ff;
    const long long v = (long long)(((unsigned long long)(unsigned)((hi & 0xfffff) | (ex ? 0x100000 : 0)) << 32 | (unsigned)lo) << 9);
    const long long s = hi >> 31;
    m = (v ^ s) - s;
    return ex == 0x7ff ? 4095 : max(ex, 1);
}
// high word of the product of a spectrum value and the multiplier
__device__ __forceinline__ long long mul_hi(long long v, split64 m)
{
    const split64 s = split_of(v);
    return add_high(mad_wide(s.h, m.h, 0), mad_wide(s.h, m.l, mad_wide(s.l, m.h, FX_UP)));
}

enum { FCOL_REAL = 0, FCOL_SPLIT = 1, FCOL_CPLX = 2 };

// High words r of the spectrum value z at index o times the multiplier's entry (row k2q of the
// quadrant); returns the multiplier's biased exponent.  FCOL_SPLIT: part 0 takes Re, part 1 Im.
template <int MODE>
__device__ __forceinline__ int multiply(const FixedArgs &a, const void *gt, int k2q, int o, int L, int h, int part, c64 z, c64 &r)
{
    const size_t gi = (size_t)k2q * h + (o < h ? o : L - o);
    long long m;
    if constexpr (MODE == FCOL_CPLX) {
        const double2 gk = __ldg(reinterpret_cast<const double2 *>(gt) + gi);
        long long mi;
        const int xr = mult_fixed(gk.x, m), xi = mult_fixed(gk.y, mi), xm = max(xr, xi);
        m >>= min(xm - xr, 63);
        mi >>= min(xm - xi, 63);
        const split64 sr = split_of(m), si = split_negatable(mi);
        r = cmulw(z, make_int4(sr.h, sr.l, si.h, si.l), FX_UP, FX_UP);
        return xm;
    } else {
        const double gk = MODE == FCOL_SPLIT ? __ldg(reinterpret_cast<const double *>(gt) + 2 * gi + part)
                                             : __ldg(reinterpret_cast<const double *>(gt) + gi);
        const int xg = mult_fixed(gk, m);
        if (MODE == FCOL_REAL && a.odd) {  // i sgn(k1) g; 0 at the unpaired Nyquist index
            if (2 * o == L) m = 0;
            if (2 * o > L) m = -m;
            const long long t = z.x;
            z.x = -z.y;
            z.y = t;
        }
        const split64 sm = split_of(m);
        r.x = mul_hi(z.x, sm);
        r.y = mul_hi(z.y, sm);
        return xg;
    }
}

// Pass 2.  Columns k2 < cols of every density, batch-fastest.  FCOL_REAL: real multiplier;
// FCOL_SPLIT: Re and Im of a complex multiplier as two real ones, results side by side;
// FCOL_CPLX: complex multiplier.  c2c: the columns run over all k2 < L.
template <int LL, int MODE> __global__ void WSC_FIXED_LB kx_cols(const __grid_constant__ FixedArgs a)
{
    const int nbuf = MODE == FCOL_SPLIT && !a.one ? 2 : 1;
    WSC_FIXED_PROLOGUE(nbuf)
    c64 *buf2 = buf + (nbuf == 2 ? fixed_padded(L) : 0);
    c64 *park = MODE == FCOL_SPLIT && a.one ? a.scratch + ((size_t)blockIdx.x * G + g) * L : nullptr;
    const int cols = a.units / a.batch;
    for (int unit = blockIdx.x * G + g; unit < a.units; unit += gridDim.x * G) {
        const int k2 = unit / a.batch, b = unit - k2 * a.batch;
        const size_t co = ((size_t)b * cols + k2) * n;
        const double2 *cin = reinterpret_cast<const double2 *>(a.in) + co;
        double2 *cout = reinterpret_cast<double2 *>(a.out) + (MODE == FCOL_SPLIT ? 2 * co : co);
        const int k2q = k2 < h ? k2 : L - k2;
        const void *gt = a.nsel ? a.gsel[b] : a.ghat;
        const int un = unit + gridDim.x * G, kn = un / a.batch;
        prefetch_line(un < a.units, a.in, ((size_t)(un - kn * a.batch) * cols + kn) * n * 16, n * 16, lt, tpt);
        int T;
        int e = ln.template first_doubles<true>(buf, T, 0, [&](int i) -> double2 { return cin[i]; });
        ln.clear(2);
        int c = ln.mids(buf, T), sh = ln.last_shift(c, T, e);
        const int e1 = e;
        if (MODE == FCOL_SPLIT && a.one)
            ln.template last<true, false>(buf, sh, [&](int o, c64 z) { park[o] = z; });
        else
            ln.template last<true, false>(buf, sh, NoDst{});
        ln.clear(0);
#pragma unroll 1
        for (int part = 0; part < (MODE == FCOL_SPLIT ? 2 : 1); ++part) {
            c64 *src = buf, *dstb = buf;
            if (MODE == FCOL_SPLIT && !a.one && part == 0) dstb = buf2;
            auto x = [&](int c) -> c64 {
                if (MODE == FCOL_SPLIT && a.one && part == 1) return park[lt + c];
                return src[ln.at(c)];
            };
            auto mul = [&](int o, c64 z, c64 &r) -> int { return multiply<MODE>(a, gt, k2q, o, L, h, part, z, r); };
            e = ln.first_product(dstb, e1, T, 2, x, mul);
            c = ln.mids(dstb, T);
            sh = ln.last_shift(c, T, e);
            const bool normal = fixed_normal(e);
            ln.template last<false, true>(dstb, sh, [&](int o, c64 z) {
                const double2 w = make_double2(from_fixed(z.y, e, normal), from_fixed(z.x, e, normal));
                if constexpr (MODE == FCOL_SPLIT) cout[2 * o + part] = w;
                else cout[o] = w;
            });
            if (MODE == FCOL_SPLIT && part == 0) {  // the second product reuses the slots and the buffer
                ln.sync();
                ln.clear(2);
                ln.sync();
            }
        }
        // the next line's group_max barrier separates these reads from its first stores
    }
}

enum { FOUT_R2R = 0, FOUT_SPLIT = 1, FOUT_REAL = 2, FOUT_CPLX = 3 };

// Z_k = A + i B and Z_(L-k) = conj A + i conj B, re and im exchanged for the inverse transform, into the
// line's buffer; returns their part of the L1 norm.
template <int P> __device__ __forceinline__ unsigned merge_pair(double2 A, double2 B, int xm, int k, int L, c64 *buf)
{
    const c64 fa = fixed_of<P>(A, xm), fb = fixed_of<P>(B, xm);
    const long long ax = fa.x, ay = fa.y, bx = fb.x, by = fb.y;
    const c64 z = {ay + bx, ax - by};
    buf[fpidx(k)] = z;
    unsigned s = l1_of(z);
    if (k != 0 && 2 * k != L) {
        const c64 y = {bx - ay, ax + by};
        buf[fpidx(L - k)] = y;
        s += l1_of(y);
    }
    return s;
}

// a scale that is no integer factor; out of line, or its FP64 products would run for every output and
// be selected away
static __device__ __noinline__ double2 fixed_alpha_mul(double2 w, double2 alpha) { return cmul(w, alpha); }

// out = alpha z 2^e + beta u at element o of the row(s) at ro.  z has re and im exchanged.  A real
// alpha is an integer factor and an exponent (one rounding; the factor 1/2 an exponent alone).
template <int OUT, bool BETA> struct FixedOut {
    const FixedArgs &a;
    const size_t ro;
    const bool has2, scaled;
    const int e;
    const bool normal;
    __device__ FixedOut(const FixedArgs &a_, size_t ro_, int e_, bool has2_)
        : a(a_), ro(ro_), has2(has2_), scaled(a_.ah && !((a_.ah == (1 << 30)) && a_.al == 0)),
          e(!a_.ah ? e_ : e_ + a_.ae + (scaled ? 1 : -1)), normal(fixed_normal(e)) {}
    __device__ __forceinline__ void operator()(int o, c64 z) const
    {
        if (scaled) {
            const split64 am = {a.ah, a.al};
            z.x = mul_hi(z.x, am);
            z.y = mul_hi(z.y, am);
        }
        double2 w = make_double2(from_fixed(z.y, e, normal), from_fixed(z.x, e, normal));
        if constexpr (OUT == FOUT_R2R) {
            if (!a.ah) w = fixed_alpha_mul(w, make_double2(a.alpha.x, 0.0));
            double *oa = reinterpret_cast<double *>(a.out) + ro;
            if constexpr (BETA) {
                const double *ua = reinterpret_cast<const double *>(a.u) + ro;
                w.x += a.beta * ua[o];
                if (has2) w.y += a.beta * ua[a.n + o];
            }
            oa[o] = w.x;
            if (has2) oa[a.n + o] = w.y;
        } else {
            if (!a.ah) w = fixed_alpha_mul(w, a.alpha);
            if constexpr (BETA) {
                if constexpr (OUT == FOUT_CPLX) {
                    const double2 x = reinterpret_cast<const double2 *>(a.u)[ro + o];
                    w.x += a.beta * x.x;
                    w.y += a.beta * x.y;
                } else {
                    w.x += a.beta * reinterpret_cast<const double *>(a.u)[ro + o];
                }
            }
            reinterpret_cast<double2 *>(a.out)[ro + o] = w;
        }
    }
};

// Pass 3.  FOUT_R2R: a row pair's spectra A, B (k <= L/2) packed as A + i B; FOUT_SPLIT: a row's (Wr, Wi);
// FOUT_REAL / FOUT_CPLX: one row of the C2C layout (u real / complex in the beta term).
template <int LL, int OUT, bool BETA> __global__ void WSC_FIXED_LB kx_rows_inv(const __grid_constant__ FixedArgs a)
{
    WSC_FIXED_PROLOGUE(1)
    constexpr bool PAIRS = OUT == FOUT_R2R || OUT == FOUT_SPLIT;
    const int rows = OUT == FOUT_R2R ? (n + 1) / 2 : n;
    for (int unit = blockIdx.x * G + g; unit < a.units; unit += gridDim.x * G) {
        const int b = unit / rows, j1 = (OUT == FOUT_R2R ? 2 : 1) * (unit - b * rows);
        const bool has2 = OUT != FOUT_R2R || j1 + 1 < n;
        int e, T;
        if constexpr (PAIRS) {
            // load each pair once, then build Z_k and Z_(L-k) from it (re and im exchanged for the
            // inverse): Z_k = A + i B, Z_(L-k) = conj A + i conj B
            constexpr int P = 60, NK = 8;
            const size_t ld = OUT == FOUT_R2R ? n : 2 * (size_t)n;
            const double2 *W = reinterpret_cast<const double2 *>(a.in) + (size_t)b * h * ld + (OUT == FOUT_R2R ? j1 : 2 * j1);
            double2 A[NK + 1], B[NK + 1];
            unsigned xm = 0;
            const int un = unit + gridDim.x * G;
            if (un < a.units) {
                const int bn = un / rows, jn = un - bn * rows;
                const double2 *N = reinterpret_cast<const double2 *>(a.in) + (size_t)bn * h * ld + 2 * jn;
#pragma unroll
                for (int i = 0; i < NK; ++i) prefetch_l2(N + (size_t)(lt + i * tpt) * ld);
            }
#pragma unroll
            for (int i = 0; i <= NK; ++i) {
                const int k = i < NK ? lt + i * tpt : L / 2;
                const bool on = i < NK || lt == 0;
                A[i] = B[i] = make_double2(0.0, 0.0);
                if (on) {
                    const double2 *w = W + (size_t)k * ld;
                    if (a.vec32) {
                        ld32(w, A[i], B[i]);
                    } else {
                        A[i] = w[0];
                        if (has2) B[i] = w[1];
                    }
                }
                xm = max(xm, max(max(dexp(A[i].x), dexp(A[i].y)), max(dexp(B[i].x), dexp(B[i].y))));
            }
            xm = ln.group_max(xm, 0);
            ln.clear(2);
            unsigned s = 0;
#pragma unroll
            for (int i = 0; i <= NK; ++i) {
                const int k = i < NK ? lt + i * tpt : L / 2;
                const bool on = i < NK || lt == 0;
                if (on) s += merge_pair<P>(A[i], B[i], xm, k, L, buf);
            }
            const unsigned l1 = ln.add_l1(s, 1);
            ln.sync();
            e = (xm == 0x7ff ? FIXED_NAN : (int)xm - 1022 - P) + ln.first_smem(buf, l1, T, 1);
        } else {
            const double2 *W = reinterpret_cast<const double2 *>(a.in) + (size_t)b * L * n + j1;
            e = ln.template first_doubles<false>(buf, T, 0, [&](int i) -> double2 {
                const double2 w = W[(size_t)i * n];
                return make_double2(w.y, w.x);
            });
        }
        const int c = ln.mids(buf, T), sh = ln.last_shift(c, T, e);
        const size_t ro = (size_t)b * n * n + (size_t)j1 * n;
        const FixedOut<OUT, BETA> put(a, ro, e, has2);
        ln.template last<false, true>(buf, sh, [&](int o, c64 z) { put(o, z); });
        ln.sync();
        ln.clear(0);
        ln.sync();
    }
}

}  // namespace wsc
