// gsm_fx_kernels.cuh -- the fixed-point pass kernels, of any schedule (SC =
// Sched) and of schedules known at compile time (FixedSched).
//
// The general kernels hold every radix and every stage in one function of 64
// registers: the conv pass spills 820 bytes per thread, a third of the instructions
// are addresses, tests and loops, and where an SM has few warps (2D) the warps wait
// for instructions: 400x500, warps stalled on fetch per issue 5.5, 6.7, 12.3 (xf,
// conv, xi) against 0.3, 1.2, 0.6 for 512^2 with its schedule compiled in.
// FixedPasses<M> are the same passes with the default schedule of padded length M
// as constants, which spill a tenth of that.  Passes xf, yf, conv, yi, xi in us
// (white noise, L2 cold), general -> fixed: dipolar 120x90x50 32, 43, 127, 47, 45 ->
// 14, 23, 62, 26, 17; 100^3 39, 45, 203, 51, 59 -> 23, 33, 129, 37, 27; 250x216x180
// 205, 381, 2263, 414, 258 -> 160, 248, 1322, 270, 176; 2D (xf, conv, xi) 400x500 28,
// 59, 39 -> 15, 35, 19; 512^2 23, 41, 35 -> 15, 22, 14; 1024^2 31, 76, 39 -> 27, 61, 27;
// 1280x640 62, 96, 92 -> 48, 65, 56.  (Pairs of floats, which FP32X2 once was, took 83
// and 190 us for the whole 400x500 and 1280x640.)
//
// The rule: every even n from 24 to 4096 that is a product of 2, 3 and 5, but for the
// lengths of gsm_fx3.cuh (faster still), in two halves from n = 2048 on
// (gsm_fx_split.cuh).  Over n = 256 there are no y passes (3D grids with such an axis
// are rare; they cost two kernels a length), and below 24 lines are too short to
// gain.  All give the general kernels' bits.  Schedules or launch shapes that were
// set or tuned to something else keep the general kernels.
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
    fx_body_xf<EMAX>(fx_thread_of<SC, EMAX>(), rho, W1, ex, nx, ny, hx, sc, nl, tw, blockIdx.x, blockIdx.y, smem_raw, red);
}

template <int EMAX, class SC>
__global__ void __launch_bounds__(fx_threads(EMAX), fx_ctas(EMAX))
    k_fx_yf(const fxc *__restrict__ W1, fxc *__restrict__ W2, FxExps ex, int ny, int nz, int hx, SC sc, int nl,
            const int4 *__restrict__ tw)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int red[kFxRedWords];
    fx_body_yf<EMAX, false>(fx_thread_of<SC, EMAX>(), W1, W2, ex, ny, nz, hx, sc, nl, tw, blockIdx.x, blockIdx.y, smem_raw, red);
}

template <int EMAX, class SC>
__global__ void __launch_bounds__(fx_threads(EMAX), fx_ctas(EMAX))
    k_fx_yi(const fxc *__restrict__ W2, fxc *__restrict__ W1, FxExps ex, int ny, int nz, int hx, SC sc, int nl,
            const int4 *__restrict__ tw)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int red[kFxRedWords];
    fx_body_yi<EMAX, false>(fx_thread_of<SC, EMAX>(), W2, W1, ex, ny, nz, hx, sc, nl, tw, blockIdx.x, blockIdx.y, smem_raw, red);
}

template <int EMAX, class SC>
__global__ void __launch_bounds__(fx_threads(EMAX), fx_ctas(EMAX))
    k_fx_xi(const fxc *__restrict__ W1, double *__restrict__ u, const int *__restrict__ ek, int ek_stride, int nx,
            int ny, int hx, SC sc, int nl, const int4 *__restrict__ tw)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int red[kFxRedWords];
    fx_body_xi<EMAX, false>(fx_thread_of<SC, EMAX>(), W1, u, ek + (size_t)blockIdx.y * ek_stride, nx, ny, hx, sc, nl, tw, blockIdx.x,
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
    fx_body_conv<EMAX, false>(fx_thread_of<SC, EMAX>(), W, mult, mrow_exp, ex, nlines, n, is3d, My, ny1, sc, sci, nl, tw, twi, blockIdx.x,
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
// values per thread of its kernels: the default shape's (choose_cfg)
constexpr int fixed_emax(int M) { return M <= 8 * fx_threads(8) ? 8 : 16; }

#ifdef GSM_FX_LENGTH_UNIT
template <int M>
bool FixedPasses<M>::serves(const Plan *p, int axis, bool fwd, bool inv, const PassCfg &c)
{
    using F = FixedSched<M>;
    using I = FixedSched<M, true>;
    const bool conv = fwd && inv;
    return c.emax == fixed_emax(M) && c.gthr == fixed_threads<F, fixed_emax(M)>() && (!fwd || F::is(p->sched_f[axis])) &&
           (!inv || (conv ? I::is(p->sched_i[axis]) : F::is(p->sched_i[axis])));
}
template <int M>
cudaError_t FixedPasses<M>::raise(const Plan *p, int pass, const PassCfg &c)
{
    using F = FixedSched<M>;
    using I = FixedSched<M, true>;
    constexpr int E = fixed_emax(M);
    const int last = p->d == 3 ? 4 : 2, conv = p->d == 3 ? 2 : 1;
    if (c.emax != E) return cudaSuccess;
    if (pass == 0) return raise_smem(k_fx_xf<E, F>, c.smem);
    if (pass == last) return raise_smem(k_fx_xi<E, F>, c.smem);
    if (pass == conv) return raise_smem(k_fx_conv<E, F, I>, c.smem);
    if constexpr (M <= kFxLongM) return pass == 1 ? raise_smem(k_fx_yf<E, F>, c.smem) : raise_smem(k_fx_yi<E, F>, c.smem);
    return cudaSuccess;
}
template <int M>
bool FixedPasses<M>::launch(const FxCall &a, int pass, const PassCfg &c)
{
    using F = FixedSched<M>;
    using I = FixedSched<M, true>;
    constexpr int E = fixed_emax(M);
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
        k_fx_xf<E, F><<<gx, b, c.smem, a.st>>>(a.rho, W1, a.ex, nx, ny, hx, F(), c.nl, tw);
    } else if (pass == last) {
        k_fx_xi<E, F><<<gx, b, c.smem, a.st>>>(W1, a.u, p->d == 3 ? a.ex.yi : a.ex.cv, hx, nx, ny, hx, F(), c.nl, twi);
    } else if (pass == conv) {
        const int My = p->d == 3 ? p->M[1] : 1;
        const dim3 g = p->d == 3 ? dim3((My + c.nl - 1) / c.nl, hx) : dim3((hx + c.nl - 1) / c.nl);
        k_fx_conv<E, F, I><<<g, b, c.smem, a.st>>>(p->d == 3 ? W2 : W1, static_cast<const int2 *>(p->d_mult), p->d_mrow,
                                                   a.ex, p->d == 3 ? hx * My : hx, p->n[axis], p->d == 3, My, ny + 1,
                                                   F(), I(), c.nl, tw, twi, p->mult_full ? 1 : 0);
    } else if constexpr (M <= kFxLongM) {
        if (pass == 1) k_fx_yf<E, F><<<gy, b, c.smem, a.st>>>(W1, W2, a.ex, ny, nz, hx, F(), c.nl, tw);
        else k_fx_yi<E, F><<<gy, b, c.smem, a.st>>>(W2, W1, a.ex, ny, nz, hx, F(), c.nl, twi);
    }
    return true;
}
#endif

// The lengths of each translation unit (gsm_fx_len_*.cu).
#define GSM_FX_LENGTHS_A(X) X(48) X(60) X(72) X(80) X(96) X(100) X(108)
#define GSM_FX_LENGTHS_B(X) X(120) X(144) X(160) X(180) X(200)
#define GSM_FX_LENGTHS_C(X) X(216) X(240) X(288) X(300) X(324)
#define GSM_FX_LENGTHS_D(X) X(360) X(400) X(432) X(480) X(500)
#define GSM_FX_LENGTHS_E(X) X(540) X(1152) X(1200) X(2304) X(2400) X(4000)
#define GSM_FX_LENGTHS_F(X) X(576) X(1080) X(1280) X(2160) X(2500) X(3888)
#define GSM_FX_LENGTHS_G(X) X(600) X(1024) X(1296) X(2048) X(2560) X(3840)
#define GSM_FX_LENGTHS_H(X) X(640) X(1000) X(1440) X(2000) X(2592) X(3600)
#define GSM_FX_LENGTHS_I(X) X(648) X(972) X(1500) X(1944) X(2700) X(3456)
#define GSM_FX_LENGTHS_J(X) X(720) X(960) X(1536) X(1920) X(2880) X(3240)
#define GSM_FX_LENGTHS_K(X) X(768) X(900) X(1600) X(1800) X(2916) X(3200)
#define GSM_FX_LENGTHS_L(X) X(800) X(864) X(1620) X(1728) X(3000) X(3072)
#define GSM_FX_LENGTHS(X) \
    GSM_FX_LENGTHS_A(X) GSM_FX_LENGTHS_B(X) GSM_FX_LENGTHS_C(X) GSM_FX_LENGTHS_D(X) GSM_FX_LENGTHS_E(X) \
    GSM_FX_LENGTHS_F(X) GSM_FX_LENGTHS_G(X) GSM_FX_LENGTHS_H(X) GSM_FX_LENGTHS_I(X) GSM_FX_LENGTHS_J(X) GSM_FX_LENGTHS_K(X) GSM_FX_LENGTHS_L(X)
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
