// passes_fixed.cu -- host side of the FP64 plans' fixed-point passes: stage structure, twiddle table,
// launch shapes, dispatch (kernels in passes_fixed.cuh).
#include <cmath>
#include <cstdlib>
#include <vector>

#include "passes_fixed_launch.cuh"

namespace wsc {

// Lengths with kernels of their own (compile-time indices), for n = L/2; 0: any other length.
static int fixed_ll(const conv_plan_s *p)
{
    if (2 * p->n != p->M) return 0;
    for (int l : {512, 1024, 2048, 4096, 8192})
        if (p->M == l) return l;
    return 0;
}

#define WSC_FIXED_DISPATCH(LLV, CALL)                          \
    switch (LLV) {                                             \
    case 512: { constexpr int LL_ = 512; CALL; } break;        \
    case 1024: { constexpr int LL_ = 1024; CALL; } break;      \
    case 2048: { constexpr int LL_ = 2048; CALL; } break;      \
    case 4096: { constexpr int LL_ = 4096; CALL; } break;      \
    case 8192: { constexpr int LL_ = 8192; CALL; } break;      \
    default: { constexpr int LL_ = 0; CALL; } break;           \
    }

// Radices of L: the power of two as 16s (8s, 4s for short lines, whose stages then fill a warp) and
// one stage for the rest of it, then 3s, then 5s.
static bool fixed_factor(int L, FixedDesc &d)
{
    int rem = L, p2 = 0;
    std::vector<int> R;
    while (rem % 2 == 0) { rem /= 2; ++p2; }
    const int lr = L >= 512 ? 4 : (L >= 256 ? 3 : 2);
    for (int i = 0; i < p2 / lr; ++i) R.push_back(1 << lr);
    if (p2 % lr) R.push_back(1 << (p2 % lr));
    while (rem % 3 == 0) { rem /= 3; R.push_back(3); }
    while (rem % 5 == 0) { rem /= 5; R.push_back(5); }
    if (rem != 1 || p2 < 1 || R.size() < 2 || R.size() > FIXED_MAX_STAGES) return false;
    d.L = L;
    d.nst = (int)R.size();
    int Ns = 1, off = 0;
    double growth = 0.0;
    for (int s = 0; s < d.nst; ++s) {
        d.R[s] = R[s];
        d.Ns[s] = Ns;
        d.mag[s] = ((1ULL << 40) + (unsigned long long)Ns - 1) / (unsigned long long)Ns;
        d.toff[s] = off;
        if (s > 0) {
            // the last, radix-2 stage of L = 8192 reads a quarter turn (FixedLine::last)
            off += L == 8192 && R[s] == 2 ? L / 4 : fixed_variants(R[s]) * (R[s] - 1) * Ns;
            growth += std::log2((double)R[s]);
        }
        d.lg[s] = (int)std::ceil(growth - 1e-9);
        Ns *= R[s];
    }
    d.tw_len = off;
    return true;
}

// v / 2^shift, rounded, as h 2^32 + l with l signed and its negation in range
static void split_scaled(long long v, int shift, int &h, int &l)
{
    if (shift) v = (v + (1LL << (shift - 1))) >> shift;
    if ((int)(unsigned)(unsigned long long)v == INT32_MIN) ++v;
    l = (int)(unsigned)(unsigned long long)v;
    h = (int)((v - l) / (1LL << 32));
}

// Twiddle copies of every stage (FixedDesc), as (re h, re l, im h, im l)
void fixed_twiddles(const FixedDesc &d, std::vector<int> &tab)
{
    std::vector<long long> re, im;
    unit_roots(d.L, [](long double x) { return (long long)llroundl(ldexpl(x, 62)); }, re, im);
    tab.assign(4 * (size_t)d.tw_len, 0);
    for (int s = 1; s < d.nst; ++s) {
        const int R = d.R[s], Ns = d.Ns[s];
        const long long step = d.L / ((long long)Ns * R);
        for (int v = 0; v < fixed_variants(R); ++v)
            for (int q = 1; q < R; ++q)
                for (int k = 0; k < (d.L == 8192 && R == 2 ? d.L / 4 : Ns); ++k) {
                    const size_t t = (size_t)(((long long)q * k * step) % d.L);
                    int *e = &tab[4 * ((size_t)d.toff[s] + ((size_t)v * (R - 1) + q - 1) * Ns + k)];
                    split_scaled(re[t], v, e[0], e[1]);
                    split_scaled(im[t], v, e[2], e[3]);
                }
    }
}

void fixed_alpha(double re, double im, int &ah, int &al, int &ae)
{
    ah = al = ae = 0;
    if (im != 0.0 || re == 0.0 || !std::isfinite(re)) return;
    const double m = std::frexp(re, &ae);  // re = m 2^ae, 1/2 <= |m| < 1
    long long v = (long long)std::ldexp(m, 63);
    const long long h = (v >> 32) + ((v >> 31) & 1);
    if (h > INT32_MAX || h < INT32_MIN) return;  // |m| within 2^-32 of 1: the FP64 product
    ah = (int)h;
    al = (int)(unsigned)(unsigned long long)v;
}

// Whether the plan's lines run in fixed point, and its launch shapes: up to 16 elements per thread
// and 512 threads, so L <= 8192.
bool fixed_configure(conv_plan_s *p, int smem_optin, int sms)
{
    FixedDesc d{};
    if (p->prec != CONV_P_FP64 || p->M < 32 || p->M > 8192 || !fixed_factor(p->M, d)) return false;
    const int L = p->M, ll = fixed_ll(p);
    LaunchShape S{};
    S.tpt = ll ? L / 16 : ((L + 15) / 16 + 31) / 32 * 32;
    // compile-time lengths: one buffer per group; others: two
    const size_t line = (size_t)fixed_padded(L) * sizeof(c64) * (ll ? 1 : 2) + FIXED_SLOTS * sizeof(unsigned);
    const size_t tw = ll ? fixed_tw_smem(ll) * sizeof(int4) : 0;
    // named barriers 1 ... 15 where a group is more than one warp
    S.groups = std::min(std::min(512 / S.tpt, S.tpt > 32 ? 15 : 16), (int)(((size_t)smem_optin - tw) / line));
    if (S.groups < 1) return false;
    S.smem = line * S.groups + tw;
    S.max_ctas = sms;
    p->rows = p->cols = p->inv = S;
    // Helmholtz R2C: the spectrum is parked in a global line (L2) while the first product is
    // inverted, unless WSCONV_SPLIT_ONE=0 asks for two buffers per group and they fit
    p->r2c_split = p->io == CONV_IO_R2C && p->complex_ghat;
    p->split_scratch_elems = 0;
    if (p->r2c_split) {
        const char *one_env = getenv("WSCONV_SPLIT_ONE");
        const int two = (int)(((size_t)smem_optin - tw) / (2 * line));
        p->cols.one = !(ll && one_env && atoi(one_env) == 0 && two >= 1);
        if (p->cols.one) p->split_scratch_elems = (size_t)sms * S.groups * L;
        else p->cols.groups = std::min(S.groups, two);
    }
    p->fixed_desc = d;
    p->sms = sms;
    p->fixed = p->fused = true;
    p->elems = 16;
    p->tws = ll != 0;  // the radix-16 stages' (fixed_tw_smem)
    int l2 = 0;
    while ((1 << l2) < L) ++l2;
    p->ed = ll ? 1000 + l2 : 0;
    p->fft = FFTDesc{};
    p->fft.L = L;
    p->fft.nst = d.nst;
    for (int s = 0; s < d.nst; ++s) p->fft.R[s] = d.R[s];
    return true;
}

conv_status set_all_attrs_fixed(int smem)
{
    conv_status rc = CONV_OK;
    for (int l : {0, 512, 1024, 2048, 4096, 8192})
        if (rc == CONV_OK) WSC_FIXED_DISPATCH(l, rc = set_attrs_fixed<LL_>(smem));
    return rc;
}

conv_status launch_fixed(conv_plan_s *p, const void *u, const void *mask, void *out, int batch, double are, double aim,
                         double beta, bool split, void *ws, cudaStream_t st)
{
    conv_status rc = CONV_OK;
    WSC_FIXED_DISPATCH(fixed_ll(p), rc = run_fixed<LL_>(p, u, mask, out, batch, are, aim, beta, split, ws, st));
    return rc;
}

}  // namespace wsc
