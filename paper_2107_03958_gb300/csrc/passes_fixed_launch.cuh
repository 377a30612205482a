// passes_fixed_launch.cuh -- launches of the fixed-point passes (included once per line length).
// LL = 0: passes_fixed_any.cuh's kernels.
#pragma once
#include "passes_fixed_any.cuh"

namespace wsc {

typedef void (*FixedKernel)(FixedArgs);
template <int LL, int IN, bool MASK> FixedKernel fixed_rows_fwd()
{
    if constexpr (LL) return kx_rows_fwd<LL, IN, MASK>;
    else return ky_rows_fwd<IN, MASK>;
}
template <int LL, int MODE> FixedKernel fixed_cols()
{
    if constexpr (LL) return kx_cols<LL, MODE>;
    else return ky_cols<MODE>;
}
template <int LL, int OUT, bool BETA> FixedKernel fixed_rows_inv()
{
    if constexpr (LL) return kx_rows_inv<LL, OUT, BETA>;
    else return ky_rows_inv<OUT, BETA>;
}

template <int LL> conv_status set_attrs_fixed(int smem)
{
#define WSC_ATTR(k) WSC_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem))
    WSC_ATTR((fixed_rows_fwd<LL, FIN_PAIR, false>()));
    WSC_ATTR((fixed_rows_fwd<LL, FIN_PAIR, true>()));
    WSC_ATTR((fixed_rows_fwd<LL, FIN_REAL, false>()));
    WSC_ATTR((fixed_rows_fwd<LL, FIN_REAL, true>()));
    WSC_ATTR((fixed_rows_fwd<LL, FIN_CPLX, false>()));
    WSC_ATTR((fixed_rows_fwd<LL, FIN_CPLX, true>()));
    WSC_ATTR((fixed_cols<LL, FCOL_REAL>()));
    WSC_ATTR((fixed_cols<LL, FCOL_SPLIT>()));
    WSC_ATTR((fixed_cols<LL, FCOL_CPLX>()));
    WSC_ATTR((fixed_rows_inv<LL, FOUT_R2R, false>()));
    WSC_ATTR((fixed_rows_inv<LL, FOUT_R2R, true>()));
    WSC_ATTR((fixed_rows_inv<LL, FOUT_SPLIT, false>()));
    WSC_ATTR((fixed_rows_inv<LL, FOUT_SPLIT, true>()));
    WSC_ATTR((fixed_rows_inv<LL, FOUT_REAL, false>()));
    WSC_ATTR((fixed_rows_inv<LL, FOUT_REAL, true>()));
    WSC_ATTR((fixed_rows_inv<LL, FOUT_CPLX, false>()));
    WSC_ATTR((fixed_rows_inv<LL, FOUT_CPLX, true>()));
#undef WSC_ATTR
    return CONV_OK;
}

template <int LL>
conv_status run_fixed(conv_plan_s *p, const void *u, const void *mask, void *out, int batch, double are, double aim,
                      double beta, bool split, void *ws, cudaStream_t st)
{
    const int n = p->n, L = p->M, h = p->h;
    const double sc = 1.0 / ((double)L * (double)L);
    FixedArgs a{};
    a.err = p->dev_err;
    a.give_up = fault_take(CONV_FAULT_WAIT) ? 1 : 0;
    a.nsel = p->nsel;
    for (int i = 0; i < p->nsel; ++i) a.gsel[i] = p->sel[i];
    a.odd = p->kern.family == CONV_K_DX1LOG ? 1 : 0;
    a.mask = reinterpret_cast<const double *>(mask);
    a.ghat = p->ghat64;
    a.u = u;
    a.tw = reinterpret_cast<const int4 *>(p->tw);
    a.P = p->fixed_desc;
    a.n = n;
    a.h = h;
    a.L = L;
    a.tpt = p->rows.tpt;
    a.batch = batch;
    a.alpha = make_double2(are * sc, aim * sc);
    fixed_alpha(a.alpha.x, a.alpha.y, a.ah, a.al, a.ae);
    a.beta = beta;
    const bool may_early = may_launch_early(st);
    // groups per CTA: as many as fit, fewer when the work items would not reach every SM
    auto launch = [&](auto kern, const LaunchShape &S, int nbuf, int units) {
        a.units = units;
        const int G = std::max(1, std::min(S.groups, (units + p->sms - 1) / p->sms));
        const long long need = (units + G - 1) / G, most = (long long)p->sms * (S.groups / G);
        const size_t smem = ((size_t)fixed_padded(L) * (LL ? nbuf : 2) * sizeof(c64) + FIXED_SLOTS * sizeof(unsigned)) * G +
                            (LL ? fixed_tw_smem(LL) * sizeof(int4) : 0);
        launch_pass(kern, may_early && need <= p->sms, (unsigned)std::min(need, most), (unsigned)(S.tpt * G), smem, st, a);
    };
    cudaEvent_t *ev = timing_slot(p);
    if (ev) cudaEventRecord(ev[0], st);
    const int run = p->run_passes;  // conv_apply_multi runs pass 1 once for several plans
    const bool r2r = p->io == CONV_IO_R2R, in_real = p->io == CONV_IO_R2C;
    auto pairs32 = [&](const void *w) { return n % 2 == 0 && reinterpret_cast<uintptr_t>(w) % 32 == 0; };
    a.in = u;
    a.out = ws;
    a.vec32 = pairs32(ws);
    if (run & 1) {
        if (r2r || split) launch(mask ? fixed_rows_fwd<LL, FIN_PAIR, true>() : fixed_rows_fwd<LL, FIN_PAIR, false>(), p->rows, 1, batch * ((n + 1) / 2));
        else if (in_real) launch(mask ? fixed_rows_fwd<LL, FIN_REAL, true>() : fixed_rows_fwd<LL, FIN_REAL, false>(), p->rows, 1, batch * n);
        else launch(mask ? fixed_rows_fwd<LL, FIN_CPLX, true>() : fixed_rows_fwd<LL, FIN_CPLX, false>(), p->rows, 1, batch * n);
    }
    if (ev) cudaEventRecord(ev[1], st);
    a.in = p->w_in ? p->w_in : ws;
    if (split) {
        // W2 follows W on the next even element, the scratch lines after the batch's 3 h n + 1 values
        double2 *w = reinterpret_cast<double2 *>(ws);
        a.out = w + (((size_t)batch * h * n + 1) & ~(size_t)1);
        a.one = p->cols.one;
        a.scratch = reinterpret_cast<c64 *>(w + (((size_t)batch * (3 * (size_t)h * n + 1) + 1) & ~(size_t)1));
        if (run & 2) launch(fixed_cols<LL, FCOL_SPLIT>(), p->cols, a.one ? 1 : 2, batch * h);
    } else if (run & 2) {
        if (p->complex_ghat) launch(fixed_cols<LL, FCOL_CPLX>(), p->cols, 1, batch * (r2r ? h : L));
        else launch(fixed_cols<LL, FCOL_REAL>(), p->cols, 1, batch * (r2r ? h : L));
    }
    if (ev) cudaEventRecord(ev[2], st);
    if (run & 4) {
        a.in = a.out;
        a.out = out;
        a.vec32 = split ? reinterpret_cast<uintptr_t>(a.in) % 32 == 0 : pairs32(a.in);
        if (r2r) launch(beta != 0.0 ? fixed_rows_inv<LL, FOUT_R2R, true>() : fixed_rows_inv<LL, FOUT_R2R, false>(), p->inv, 1, batch * ((n + 1) / 2));
        else if (split) launch(beta != 0.0 ? fixed_rows_inv<LL, FOUT_SPLIT, true>() : fixed_rows_inv<LL, FOUT_SPLIT, false>(), p->inv, 1, batch * n);
        else if (in_real) launch(beta != 0.0 ? fixed_rows_inv<LL, FOUT_REAL, true>() : fixed_rows_inv<LL, FOUT_REAL, false>(), p->inv, 1, batch * n);
        else launch(beta != 0.0 ? fixed_rows_inv<LL, FOUT_CPLX, true>() : fixed_rows_inv<LL, FOUT_CPLX, false>(), p->inv, 1, batch * n);
    }
    if (ev) cudaEventRecord(ev[3], st);
    WSC_CUDA(cudaGetLastError());
    return CONV_OK;
}

}  // namespace wsc
