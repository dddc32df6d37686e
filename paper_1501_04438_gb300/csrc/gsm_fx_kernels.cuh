// gsm_fx_kernels.cuh -- the fixed-point pass kernels, of any schedule (SC =
// Sched) and of schedules known at compile time (FixedSched).
//
// The general kernels hold every radix and every stage in one function of 64
// registers: the conv pass spills 770 bytes per thread, and a third of its
// instructions are addresses, tests and loops.  FixedPasses<M> are the same
// passes with the default schedule of padded length M as constants, which spill
// 0 to 96 bytes.  Integer issue bounds both.  Passes xf, yf, conv, yi, xi in us,
// general -> fixed: dipolar 120x90x50 17, 31, 111, 40, 46 -> 15, 23, 56, 27, 17;
// 100^3 29, 42, 179, 48, 52 -> 21, 33, 109, 38, 29; 250x216x180 187, 345, 1864,
// 378, 230 -> 150, 240, 1176, 257, 167; 2D (xf, conv, xi) 1024^2 27, 68, 33 -> 25,
// 54, 27; 512^2 15, 27, 31 -> 13, 21, 15.
//
// They are compiled for the even n from 24 to 256 that are products of 2, 3 and 5,
// but for the lengths of gsm_fx3.cuh (faster still), and for n = 512 and 1024; in
// two halves (gsm_fx_conv.cu) for n = 2048 and 4096: up to 256 every length a 3D
// grid usually has, beyond it the powers of two, as each length costs five
// kernels.  All give the general kernels' bits.  Schedules or launch shapes that
// were set or tuned to something else keep the general kernels.
#pragma once

#include "gsm_fx_passes.cuh"

namespace gsm {
namespace {

// ------------------------------------------------------------------ kernels
template <int EMAX, class SC>
__global__ void __launch_bounds__(fx_threads(EMAX), fx_ctas(EMAX))
    k_fx_xf(const double *__restrict__ rho, fxc *__restrict__ W1, FxExps ex, int nx, int ny, int hx, SC sc, int nl,
            const int4 *__restrict__ tw)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int red[kFxRedWords];
    fx_body_xf<EMAX>(fx_thread_of<SC>(), rho, W1, ex, nx, ny, hx, sc, nl, tw, blockIdx.x, blockIdx.y, smem_raw, red);
}

template <int EMAX, class SC>
__global__ void __launch_bounds__(fx_threads(EMAX), fx_ctas(EMAX))
    k_fx_yf(const fxc *__restrict__ W1, fxc *__restrict__ W2, FxExps ex, int ny, int nz, int hx, SC sc, int nl,
            const int4 *__restrict__ tw)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int red[kFxRedWords];
    fx_body_yf<EMAX, false>(fx_thread_of<SC>(), W1, W2, ex, ny, nz, hx, sc, nl, tw, blockIdx.x, blockIdx.y, smem_raw, red);
}

template <int EMAX, class SC>
__global__ void __launch_bounds__(fx_threads(EMAX), fx_ctas(EMAX))
    k_fx_yi(const fxc *__restrict__ W2, fxc *__restrict__ W1, FxExps ex, int ny, int nz, int hx, SC sc, int nl,
            const int4 *__restrict__ tw)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int red[kFxRedWords];
    fx_body_yi<EMAX, false>(fx_thread_of<SC>(), W2, W1, ex, ny, nz, hx, sc, nl, tw, blockIdx.x, blockIdx.y, smem_raw, red);
}

template <int EMAX, class SC>
__global__ void __launch_bounds__(fx_threads(EMAX), fx_ctas(EMAX))
    k_fx_xi(const fxc *__restrict__ W1, double *__restrict__ u, const int *__restrict__ ek, int ek_stride, int nx,
            int ny, int hx, SC sc, int nl, const int4 *__restrict__ tw)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int red[kFxRedWords];
    fx_body_xi<EMAX, false>(fx_thread_of<SC>(), W1, u, ek + (size_t)blockIdx.y * ek_stride, nx, ny, hx, sc, nl, tw, blockIdx.x,
                            blockIdx.y, smem_raw, red);
}

template <int EMAX, class SC, class SCI>
__global__ void __launch_bounds__(fx_threads(EMAX), fx_ctas(EMAX))
    k_fx_conv(fxc *__restrict__ W, const int2 *__restrict__ mult, const int *__restrict__ mrow_exp, FxExps ex,
              int nlines, int n, int is3d, int My, int ny1, SC sc, SCI sci, int nl,
              const int4 *__restrict__ tw, const int4 *__restrict__ twi, int full)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int red[kFxRedWords];
    fx_body_conv<EMAX, false>(fx_thread_of<SC>(), W, mult, mrow_exp, ex, nlines, n, is3d, My, ny1, sc, sci, nl, tw, twi, blockIdx.x,
                              blockIdx.y, smem_raw, full != 0, red);
}

}  // namespace

// The passes of padded length M.  Defined in the translation unit that the length
// belongs to and nowhere else: the kernels have internal linkage, so a second copy
// would have shared-memory limits of its own.
template <int M>
struct FixedPasses {
    static bool serves(const Plan *p, int axis, bool fwd, bool inv, const PassCfg &c);
    // kernels' shared-memory limits for shape c (any that serves() may accept)
    static cudaError_t raise(const Plan *p, int pass, const PassCfg &c);
    // false: not served
    static bool launch(const FxCall &a, int pass, const PassCfg &c);
};

#ifdef GSM_FX_LENGTH_UNIT
template <int M>
bool FixedPasses<M>::serves(const Plan *p, int axis, bool fwd, bool inv, const PassCfg &c)
{
    using F = FixedSched<M>;
    using I = FixedSched<M, true>;
    const bool conv = fwd && inv;
    return c.emax == 8 && c.gthr == fixed_threads<F>() && (!fwd || F::is(p->sched_f[axis])) &&
           (!inv || (conv ? I::is(p->sched_i[axis]) : F::is(p->sched_i[axis])));
}
template <int M>
cudaError_t FixedPasses<M>::raise(const Plan *p, int pass, const PassCfg &c)
{
    using F = FixedSched<M>;
    using I = FixedSched<M, true>;
    const int last = p->d == 3 ? 4 : 2, conv = p->d == 3 ? 2 : 1;
    if (c.emax != 8) return cudaSuccess;
    if (pass == 0) return raise_smem(k_fx_xf<8, F>, c.smem);
    if (pass == last) return raise_smem(k_fx_xi<8, F>, c.smem);
    if (pass == conv) return raise_smem(k_fx_conv<8, F, I>, c.smem);
    if constexpr (M <= kFxLongM) return pass == 1 ? raise_smem(k_fx_yf<8, F>, c.smem) : raise_smem(k_fx_yi<8, F>, c.smem);
    return cudaSuccess;
}
template <int M>
bool FixedPasses<M>::launch(const FxCall &a, int pass, const PassCfg &c)
{
    using F = FixedSched<M>;
    using I = FixedSched<M, true>;
    const Plan *p = a.p;
    const int last = p->d == 3 ? 4 : 2, conv = p->d == 3 ? 2 : 1;
    const int axis = pass == 0 || pass == last ? 0 : pass == conv ? p->d - 1 : 1;
    if (!serves(p, axis, pass <= conv, pass >= conv, c)) return false;
    if constexpr (M > kFxLongM)
        if (pass != 0 && pass != last && pass != conv) return false;
    const int nx = p->n[0], ny = p->n[1], nz = a.nz, hx = nx + 1;
    fxc *W1 = static_cast<fxc *>(a.W1), *W2 = static_cast<fxc *>(a.W2);
    const int4 *tw = static_cast<const int4 *>(p->d_tw[axis]), *twi = static_cast<const int4 *>(p->d_twi[axis]);
    const dim3 gx((ny + 2 * c.nl - 1) / (2 * c.nl), nz), gy((nz + c.nl - 1) / c.nl, hx), b(c.gthr, c.nl);
    if (pass == 0) {
        k_fx_xf<8, F><<<gx, b, c.smem, a.st>>>(a.rho, W1, a.ex, nx, ny, hx, F(), c.nl, tw);
    } else if (pass == last) {
        k_fx_xi<8, F><<<gx, b, c.smem, a.st>>>(W1, a.u, p->d == 3 ? a.ex.yi : a.ex.cv, hx, nx, ny, hx, F(), c.nl, twi);
    } else if (pass == conv) {
        const int My = p->d == 3 ? p->M[1] : 1;
        const dim3 g = p->d == 3 ? dim3((My + c.nl - 1) / c.nl, hx) : dim3((hx + c.nl - 1) / c.nl);
        k_fx_conv<8, F, I><<<g, b, c.smem, a.st>>>(p->d == 3 ? W2 : W1, static_cast<const int2 *>(p->d_mult), p->d_mrow,
                                                   a.ex, p->d == 3 ? hx * My : hx, p->n[axis], p->d == 3, My, ny + 1,
                                                   F(), I(), c.nl, tw, twi, p->mult_full ? 1 : 0);
    } else if constexpr (M <= kFxLongM) {
        if (pass == 1) k_fx_yf<8, F><<<gy, b, c.smem, a.st>>>(W1, W2, a.ex, ny, nz, hx, F(), c.nl, tw);
        else k_fx_yi<8, F><<<gy, b, c.smem, a.st>>>(W2, W1, a.ex, ny, nz, hx, F(), c.nl, twi);
    }
    return true;
}
#endif

// The lengths of each translation unit (gsm_fx_len_*.cu).
#define GSM_FX_LENGTHS_A(X) X(48) X(60) X(72) X(80) X(96) X(100) X(108)
#define GSM_FX_LENGTHS_B(X) X(120) X(144) X(160) X(180) X(200)
#define GSM_FX_LENGTHS_C(X) X(216) X(240) X(288) X(300) X(324)
#define GSM_FX_LENGTHS_D(X) X(360) X(400) X(432) X(480) X(500)
#define GSM_FX_LENGTHS_E(X) X(1024) X(2048)
#define GSM_FX_LENGTHS(X) \
    GSM_FX_LENGTHS_A(X) GSM_FX_LENGTHS_B(X) GSM_FX_LENGTHS_C(X) GSM_FX_LENGTHS_D(X) GSM_FX_LENGTHS_E(X)
#define GSM_FX_DEFINE(M) template struct FixedPasses<M>;
#ifndef GSM_FX_LENGTH_UNIT
inline int fixed_axis(const Plan *p, int pass)
{
    return pass == 0 || pass == (p->d == 3 ? 4 : 2) ? 0 : pass == (p->d == 3 ? 2 : 1) ? p->d - 1 : 1;
}
// A pass on its fixed kernel; false: there is none for this length, schedule or shape.
inline bool fixed_launch(const FxCall &a, int pass, const PassCfg &c)
{
    if ((a.p->opt.debug & 4) != 0) return false;
#define GSM_FX_CASE(M) case M: return FixedPasses<M>::launch(a, pass, c);
    switch (a.p->M[fixed_axis(a.p, pass)]) { GSM_FX_LENGTHS(GSM_FX_CASE) }
#undef GSM_FX_CASE
    return false;
}
inline cudaError_t fixed_raise(const Plan *p, int pass, const PassCfg &c)
{
#define GSM_FX_CASE(M) case M: return FixedPasses<M>::raise(p, pass, c);
    switch (p->M[fixed_axis(p, pass)]) { GSM_FX_LENGTHS(GSM_FX_CASE) }
#undef GSM_FX_CASE
    return cudaSuccess;
}
#endif

}  // namespace gsm
