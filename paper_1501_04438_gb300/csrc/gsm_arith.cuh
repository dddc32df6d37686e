// gsm_arith.cuh -- arithmetic of the FP32 passes (the FP64 and FP32X2 passes
// compute in block fixed point, gsm_fx.cuh).
//
// The kernels are written against this interface:
//   real  R          scalar type
//   cx<R>            complex in registers
//   Pol::scplx       complex as stored in shared/global memory
//   Pol::tw_t        twiddle-table entry, Pol::mult_t multiplier entry,
//   Pol::io_t        element type of rho and u
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace gsm {

template <class R>
struct cx {
    R re, im;
};

// ------------------------------------------------------------------ float
__device__ __forceinline__ float radd(float a, float b) { return a + b; }
__device__ __forceinline__ float rsub(float a, float b) { return a - b; }
__device__ __forceinline__ float rneg(float a) { return -a; }
__device__ __forceinline__ float rmul(float a, float b) { return a * b; }
__device__ __forceinline__ float rmulk(float a, double k) { return a * (float)k; }

// ------------------------------------------------------------------ complex
template <class R>
__device__ __forceinline__ cx<R> cadd(cx<R> a, cx<R> b) { return {radd(a.re, b.re), radd(a.im, b.im)}; }
template <class R>
__device__ __forceinline__ cx<R> csub(cx<R> a, cx<R> b) { return {rsub(a.re, b.re), rsub(a.im, b.im)}; }
// multiply by -i (forward) or +i (inverse) exactly
template <class R>
__device__ __forceinline__ cx<R> cmul_negi(cx<R> a) { return {a.im, rneg(a.re)}; }
template <class R>
__device__ __forceinline__ cx<R> cmul_posi(cx<R> a) { return {rneg(a.im), a.re}; }
template <class R>
__device__ __forceinline__ cx<R> cconj(cx<R> a) { return {a.re, rneg(a.im)}; }
// a * w or a * conj(w)
template <class R>
__device__ __forceinline__ cx<R> cmul(cx<R> a, cx<R> w)
{
    return {rsub(rmul(a.re, w.re), rmul(a.im, w.im)), radd(rmul(a.re, w.im), rmul(a.im, w.re))};
}
template <class R>
__device__ __forceinline__ cx<R> cmulc(cx<R> a, cx<R> w)
{
    return {radd(rmul(a.re, w.re), rmul(a.im, w.im)), rsub(rmul(a.im, w.re), rmul(a.re, w.im))};
}
__device__ __forceinline__ cx<float> cmul(cx<float> a, cx<float> w)
{
    return {fmaf(a.re, w.re, -a.im * w.im), fmaf(a.re, w.im, a.im * w.re)};
}
__device__ __forceinline__ cx<float> cmulc(cx<float> a, cx<float> w)
{
    return {fmaf(a.re, w.re, a.im * w.im), fmaf(a.im, w.re, -a.re * w.im)};
}
template <class R>
__device__ __forceinline__ cx<R> cscale(cx<R> a, R m) { return {rmul(a.re, m), rmul(a.im, m)}; }
template <class R>
__device__ __forceinline__ cx<R> cmulk(cx<R> a, double k) { return {rmulk(a.re, k), rmulk(a.im, k)}; }

// ------------------------------------------------------------------ policies
struct F32 {
    using real = float;
    using scplx = float2;
    using tw_t = float2;
    using mult_t = float;
    using io_t = float;
    static constexpr int kId = 1;
    static constexpr int kPadShift = 4;   // one pad element per 16 (128 bytes)
    __device__ static __forceinline__ cx<real> ld(const scplx &v) { return {v.x, v.y}; }
    __device__ static __forceinline__ scplx st(cx<real> a) { return make_float2(a.re, a.im); }
    __device__ static __forceinline__ cx<real> tw(const tw_t &v) { return {v.x, v.y}; }
    __device__ static __forceinline__ real mult(mult_t m) { return m; }
    __device__ static __forceinline__ real from_io(io_t x) { return x; }
    __device__ static __forceinline__ io_t to_io(real x) { return x; }
    __device__ static __forceinline__ real zero() { return 0.0f; }
};

}  // namespace gsm
