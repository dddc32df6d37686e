// gsm_fx_queue.cuh -- the tiles of the fixed-point batch queue kernel
// (k_batch_queue, gsm_pass_common.cuh); one translation unit per dimension.
#pragma once

#include "gsm_fx_passes.cuh"

namespace gsm {
namespace {

// One tile of pass PASS of one instance.
template <class Pol, int D, int PASS>
__device__ __forceinline__ void queue_tile(const InstDesc &d, int nl, int t, unsigned char *smem_raw, int *red)
{
    using io = typename Pol::io_t;
    using tw = typename Pol::tw_t;
    constexpr int last = D == 3 ? 4 : 2;
    const int gx = d.gx[PASS];
    const int bx = t % gx, by = t / gx;
    const int nx = d.n[0], ny = d.n[1], nz = D == 3 ? d.n[2] : 1, hx = nx + 1;
    S_t<Pol> *W1 = static_cast<S_t<Pol> *>(d.W1);
    S_t<Pol> *W2 = static_cast<S_t<Pol> *>(d.W2);
    const auto *mult = static_cast<const typename Pol::mult_t *>(d.mult);
    auto T = [&](const void *t) { return static_cast<const tw *>(t); };
    if constexpr (PASS == 0) {
        fx_body_xf<kBatchEmax>(fx_warp_line(), static_cast<const io *>(d.rho), W1, d.ex, nx, ny, hx, d.sc[0], nl, T(d.tw[0]), bx,
                               by, smem_raw, red);
    } else if constexpr (PASS == last) {
        fx_body_xi<kBatchEmax, true>(fx_warp_line(), W1, static_cast<io *>(d.u), D == 3 ? d.ex.yi + (size_t)by * hx : d.ex.cv, nx,
                                     ny, hx, d.sci[0], nl, T(d.twi[0]), bx, by, smem_raw, red);
    } else if constexpr (D == 2) {
        fx_body_conv<kBatchEmax, true>(fx_warp_line(), W1, mult, d.mrow, d.ex, hx, ny, 0, 1, ny + 1, d.sc[1], d.sci[1], nl,
                                       T(d.tw[1]), T(d.twi[1]), bx, by, smem_raw, d.full != 0, red);
    } else if constexpr (PASS == 1) {
        fx_body_yf<kBatchEmax, true>(fx_warp_line(), W1, W2, d.ex, ny, nz, hx, d.sc[1], nl, T(d.tw[1]), bx, by, smem_raw, red);
    } else if constexpr (PASS == 2) {
        fx_body_conv<kBatchEmax, true>(fx_warp_line(), W2, mult, d.mrow, d.ex, hx * d.M[1], nz, 1, d.M[1], ny + 1, d.sc[2],
                                       d.sci[2], nl, T(d.tw[2]), T(d.twi[2]), bx, by, smem_raw, d.full != 0,
                                       red);
    } else {
        fx_body_yi<kBatchEmax, true>(fx_warp_line(), W2, W1, d.ex, ny, nz, hx, d.sci[1], nl, T(d.twi[1]), bx, by, smem_raw,
                                     red);
    }
}

}  // namespace
}  // namespace gsm
