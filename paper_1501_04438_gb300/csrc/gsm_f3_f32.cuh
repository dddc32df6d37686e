// gsm_f3_f32.cuh -- FP32 passes for padded lengths M = 64 R, R = 1..6, on the
// packed lines and the three stages of gsm_fx3.cuh (n = 256, R = 8, has the
// register-resident kernels of gsm_conv_rr.cu).
//
// The FP32 passes are bound by the instructions around the butterflies
// (addresses, twiddle indices, loop and radix tests) and by the stages' trips
// through shared memory.  Here the length is known at compile time, the first
// stage reads global memory into registers and the last one of the conv and
// inverse passes stores to global memory, twiddles are read in stage order
// (consecutive threads, consecutive entries), and no lane idles where 8 R is
// not a multiple of 32.  Against the kernels of any length: 128^3 FP32 apply 154 -> 93 us
// (conv 77 -> 39), 160^3 420 -> 170, conv pass of 150 x 90 x 64 59 -> 21.
#pragma once

#include "gsm_fx3.cuh"

namespace gsm {
namespace {

using f32c = cx<float>;
__device__ __forceinline__ f32c f3f_ld(const float2 &v) { return {v.x, v.y}; }
__device__ __forceinline__ float2 f3f_st(f32c a) { return make_float2(a.re, a.im); }
template <bool FWD>
__device__ __forceinline__ f32c f3f_rot(f32c a, float2 w)   // w = exp(-i t)
{
    return FWD ? cmul(a, f32c{w.x, w.y}) : cmulc(a, f32c{w.x, w.y});
}

// HALF = 1: inputs t >= 4 are zero; 2: outputs t < 4 only.
template <bool FWD, int HALF>
__device__ __forceinline__ void f3f_bfly8(f32c *v)
{
    if constexpr (HALF == 1) {
        f32c a[4] = {v[0], v[1], v[2], v[3]}, b[4] = {v[0], v[1], v[2], v[3]};
        const f32c z = b[1], y = b[3];
        if (FWD) {
            b[1] = {rmulk(z.re + z.im, kSqrtHalf), rmulk(z.im - z.re, kSqrtHalf)};
            b[3] = {rmulk(y.im - y.re, kSqrtHalf), -rmulk(y.re + y.im, kSqrtHalf)};
        } else {
            b[1] = {rmulk(z.re - z.im, kSqrtHalf), rmulk(z.re + z.im, kSqrtHalf)};
            b[3] = {-rmulk(y.re + y.im, kSqrtHalf), rmulk(y.re - y.im, kSqrtHalf)};
        }
        b[2] = rot_quarter<float, FWD>(b[2]);
        bfly4<float, FWD>(a);
        bfly4<float, FWD>(b);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            v[2 * k] = a[k];
            v[2 * k + 1] = b[k];
        }
    } else {
        bfly<float, 8, FWD, HALF>(v);
    }
}

// Radix 6 = 2 x 3 without twiddles (see fx_bfly6).
template <bool FWD>
__device__ __forceinline__ void f3f_bfly6(f32c *v)
{
    f32c a[3], b[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        a[i] = cadd(v[2 * i], v[(2 * i + 3) % 6]);
        b[i] = csub(v[2 * i], v[(2 * i + 3) % 6]);
    }
    bfly3<float, FWD>(a);
    bfly3<float, FWD>(b);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        v[4 * k % 6] = a[k];
        v[(3 + 4 * k) % 6] = b[k];
    }
}
template <int RC, bool FWD>
__device__ __forceinline__ void f3f_bfly(f32c *v)
{
    if constexpr (RC == 6) f3f_bfly6<FWD>(v);
    else bfly<float, RC, FWD, 0>(v);
}

// ------------------------------------------------------------------ stages
// load(t): input b + t NB of the thread's line
template <int R, bool FWD, int HALF, bool SMEM, class Load>
__device__ __forceinline__ void f3f_first(float2 *s, const F3Thread<R> &th, Load load)
{
    using F = F3<R>;
    f32c v[8];
#pragma unroll
    for (int t = 0; t < (HALF == 1 ? 4 : 8); ++t) v[t] = load(t);
    f3f_bfly8<FWD, HALF>(v);
    if (SMEM) th.sync();   // the inputs come from the line's shared memory
    float2 *d = s + th.line * F::LS + 9 * th.b;
#pragma unroll
    for (int t = 0; t < 8; ++t) d[t] = f3f_st(v[t]);
    th.sync();
}

template <int R, bool FWD>
__device__ __forceinline__ void f3f_second(float2 *s, const F3Thread<R> &th, const float2 *__restrict__ tw)
{
    using F = F3<R>;
    if constexpr (F::TWO) return;
    const int j = th.b & 7;
    float2 *l = s + th.line * F::LS;
    const float2 *p = l + f3_pos(th.b), *w = tw + j;
    f32c v[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) v[t] = f3f_ld(p[t * 9 * R]);
#pragma unroll
    for (int t = 1; t < 8; ++t) v[t] = f3f_rot<FWD>(v[t], w[(t - 1) * 8]);
    f3f_bfly8<FWD, 0>(v);
    th.sync();
    float2 *d = l + 72 * (th.b >> 3) + j;
#pragma unroll
    for (int t = 0; t < 8; ++t) d[9 * t] = f3f_st(v[t]);
    th.sync();
}

template <int R, bool FWD>
__device__ __forceinline__ void f3f_last_in(f32c *v, const float2 *l, int bc, const float2 *__restrict__ tw)
{
    using F = F3<R>;
    const float2 *p = l + f3_pos(bc), *w = tw + (F::NSC - 8) + bc;
#pragma unroll
    for (int t = 0; t < F::RC; ++t) v[t] = f3f_ld(p[t * (F::NSC + F::NSC / 8)]);
#pragma unroll
    for (int t = 1; t < F::RC; ++t) v[t] = f3f_rot<FWD>(v[t], w[(t - 1) * F::NSC]);
}

template <int R, bool FWD, bool CROP, class Out>
__device__ __forceinline__ void f3f_last(const float2 *s, const F3Thread<R> &th, const float2 *__restrict__ tw, Out out)
{
    using F = F3<R>;
    constexpr bool EVEN = F::RC % 2 == 0;
    constexpr int NOUT = CROP ? (F::RC + 1) / 2 : F::RC;
#pragma unroll
    for (int k = 0; k < F::KC; ++k) {
        int ln, bc;
        if (!th.last_bfly(k, &ln, &bc)) break;
        f32c v[F::RC];
        f3f_last_in<R, FWD>(v, s + ln * F::LS, bc, tw);
        if constexpr (CROP && F::RC == 8) f3f_bfly8<FWD, 2>(v);
        else f3f_bfly<F::RC, FWD>(v);
#pragma unroll
        for (int t = 0; t < NOUT; ++t)
            if (!CROP || EVEN || t < F::RC / 2 || bc < F::NSC / 2) out(ln, bc, t, v[t]);
    }
}

template <int R>
__device__ __forceinline__ void f3f_to_smem(float2 *s, int ln, int i, int t, f32c v)
{
    using F = F3<R>;
    s[ln * F::LS + f3_pos(i) + t * (F::NSC + F::NSC / 8)] = f3f_st(v);
}

__device__ __forceinline__ void f3f_copy8(float2 *dst, const float2 *src)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src) : "memory");
}

template <int R>
struct F3F {
    static constexpr size_t SMEM = (size_t)F3<R>::NL * F3<R>::LS * sizeof(float2);
    static constexpr int CTAS = 65536 / (64 * F3<R>::THREADS);   // a 64-register bound
};

// ------------------------------------------------------------------ passes
template <int R, int COUNT>
__global__ void __launch_bounds__(F3<R>::THREADS, F3F<R>::CTAS)
    k_f3f_xf(const __grid_constant__ F3Group<COUNT> g, int ny, const float2 *__restrict__ tw)
{
    const float *__restrict__ rho = static_cast<const float *>(g.at().rho);
    float2 *__restrict__ W1 = static_cast<float2 *>(g.at().W1);
    using F = F3<R>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2 *s = reinterpret_cast<float2 *>(smem_raw);
    constexpr int nx = F::M / 2, hx = nx + 1;
    const F3Thread<R> th;
    const int z = blockIdx.y, y0 = blockIdx.x * 2 * F::NL, ya = y0 + 2 * th.line;
    const float *pa = rho + ((size_t)z * ny + ya) * nx + th.b, *pb = pa + nx;
    f3f_first<R, true, 1, false>(s, th, [&](int t) {
        return f32c{ya < ny ? pa[t * F::NB] : 0.f, ya + 1 < ny ? pb[t * F::NB] : 0.f};
    });
    f3f_second<R, true>(s, th, tw);
    f3f_last<R, true, false>(s, th, tw, [&](int ln, int i, int t, f32c v) { f3f_to_smem<R>(s, ln, i, t, v); });
    __syncthreads();
    // 2A[k] = Z[k] + conj Z[-k], 2B[k] = -i (Z[k] - conj Z[-k]) (see body_xf)
    float2 *out = W1 + (size_t)z * hx * ny + y0;
    constexpr int ROW = 2 * F::NL, STEP = F::THREADS / ROW;
    const int r = th.tid % ROW, ll = r >> 1;
    if (y0 + r < ny) {
        const float2 *l = s + ll * F::LS;
#pragma unroll 4
        for (int k = th.tid / ROW; k < hx; k += STEP) {
            const float2 zk = l[f3_pos(k)], zm = l[f3_pos(k == 0 ? 0 : F::M - k)];
            out[(size_t)k * ny + r] = r & 1 ? make_float2(zk.y + zm.y, zm.x - zk.x) : make_float2(zk.x + zm.x, zk.y - zm.y);
        }
    }
}

template <int R, int COUNT>
__global__ void __launch_bounds__(F3<R>::THREADS, F3F<R>::CTAS)
    k_f3f_yf(const __grid_constant__ F3Group<COUNT> g, int nz, int hx, const float2 *__restrict__ tw)
{
    const float2 *__restrict__ W1 = static_cast<const float2 *>(g.at().W1);
    float2 *__restrict__ W2 = static_cast<float2 *>(g.at().W2);
    using F = F3<R>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2 *s = reinterpret_cast<float2 *>(smem_raw);
    constexpr int ny = F::M / 2;
    const F3Thread<R> th;
    const int kx = blockIdx.y, z0 = blockIdx.x * F::NL, z = z0 + th.line;
    const float2 *p = W1 + ((size_t)(z < nz ? z : 0) * hx + kx) * ny + th.b;
    f3f_first<R, true, 1, false>(s, th, [&](int t) { return z < nz ? f3f_ld(p[t * F::NB]) : f32c{0.f, 0.f}; });
    f3f_second<R, true>(s, th, tw);
    f3f_last<R, true, false>(s, th, tw, [&](int ln, int i, int t, f32c v) { f3f_to_smem<R>(s, ln, i, t, v); });
    __syncthreads();
    const int ll = th.tid % F::NL, zz = z0 + ll;
    if (zz < nz) {
        float2 *out = W2 + (size_t)kx * F::M * nz + zz;
        const float2 *l = s + ll * F::LS;
#pragma unroll 8
        for (int ky = th.tid / F::NL; ky < F::M; ky += F::NB) out[(size_t)ky * nz] = l[f3_pos(ky)];
    }
}

// twi: the table of the inverse (R 8 8)
template <int R, bool IS3D, int COUNT>
__global__ void __launch_bounds__(F3<R>::THREADS, F3F<R>::CTAS)
    k_f3f_conv(const __grid_constant__ F3Group<COUNT> g, int rows, int ny1, const float2 *__restrict__ tw,
               const float2 *__restrict__ twi, int full)
{
    float2 *__restrict__ Wd = static_cast<float2 *>(IS3D ? g.at().W2 : g.at().W1);
    const float *__restrict__ mult = static_cast<const float *>(g.at().mult);
    using F = F3<R>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2 *s = reinterpret_cast<float2 *>(smem_raw);
    constexpr int M = F::M, n = M / 2, RC = F::RC;
    const F3Thread<R> th;
    const int r0 = blockIdx.x * F::NL, by = blockIdx.y, base = IS3D ? by * rows : 0;
    const bool active = r0 + th.line < rows;
    float2 *w = Wd + (size_t)(base + (active ? r0 + th.line : 0)) * n + th.b;
    f3f_first<R, true, 1, false>(s, th, [&](int t) { return active ? f3f_ld(w[t * F::NB]) : f32c{0.f, 0.f}; });
    f3f_second<R, true>(s, th, tw);
    f32c v[F::KC][RC];
#pragma unroll
    for (int k = 0; k < F::KC; ++k) {
        int ln, bc;
        if (!th.last_bfly(k, &ln, &bc)) break;
        f3f_last_in<R, true>(v[k], s + ln * F::LS, bc, tw);
        f3f_bfly<RC, true>(v[k]);
        const int row = min(r0 + ln, rows - 1);   // a line that is not there takes some row
        size_t mr = base + row;
        if (IS3D && !full) mr = (size_t)by * ny1 + min(row, rows - row);
        const float *m = mult + mr * (full ? M : n + 1) + bc;
        const float *mm = full ? m : mult + mr * (n + 1) + (M - bc);
#pragma unroll
        for (int t = 0; t < RC; ++t) {
            float f;
            if (full || 2 * t < RC - 1) f = __ldg(m + t * F::NSC);
            else if (2 * t >= RC) f = __ldg(mm - t * F::NSC);
            else f = __ldg(2 * (bc + t * F::NSC) <= M ? m + t * F::NSC : mm - t * F::NSC);
            v[k][t] = cscale(v[k][t], f);
        }
        f3f_bfly<RC, false>(v[k]);
    }
    th.sync();
    constexpr bool PAD = R != 3 && R != 5 && R != 6;
#pragma unroll
    for (int k = 0; k < F::KC; ++k) {
        int ln, bc;
        if (!th.last_bfly(k, &ln, &bc)) break;
        float2 *d = s + ln * F::LS + (PAD ? f3_pos(RC * bc) : RC * bc);
#pragma unroll
        for (int t = 0; t < RC; ++t) d[t] = f3f_st(v[k][t]);
    }
    th.sync();
    float2 *l = s + th.line * F::LS;
    const float2 *p = l + (PAD ? f3_pos(th.b) : th.b);
    f32c x[8];
    if constexpr (!F::TWO) {
        const int j = th.b % R;
        const float2 *q = twi + j;
#pragma unroll
        for (int t = 0; t < 8; ++t) x[t] = f3f_ld(p[t * (PAD ? 9 * R : 8 * R)]);
#pragma unroll
        for (int t = 1; t < 8; ++t) x[t] = f3f_rot<false>(x[t], q[(t - 1) * R]);
        f3f_bfly8<false, 0>(x);
        th.sync();
        const int d0 = (th.b - j) * 8 + j;
        float2 *d = l + (PAD ? f3_pos(d0) : d0);
#pragma unroll
        for (int t = 0; t < 8; ++t) d[PAD ? t * R + (t * R >> 3) : t * R] = f3f_st(x[t]);
        th.sync();
    }
    const float2 *q = twi + (F::TWO ? 0 : 7 * R) + th.b;
#pragma unroll
    for (int t = 0; t < 8; ++t) x[t] = f3f_ld(p[t * (PAD ? 9 * R : 8 * R)]);
#pragma unroll
    for (int t = 1; t < 8; ++t) x[t] = f3f_rot<false>(x[t], q[(t - 1) * F::NB]);
    f3f_bfly8<false, 2>(x);
    if (active) {
#pragma unroll
        for (int t = 0; t < 4; ++t) w[t * F::NB] = f3f_st(x[t]);
    }
}

template <int R, int COUNT>
__global__ void __launch_bounds__(F3<R>::THREADS, F3F<R>::CTAS)
    k_f3f_yi(const __grid_constant__ F3Group<COUNT> g, int nz, int hx, const float2 *__restrict__ tw)
{
    const float2 *__restrict__ W2 = static_cast<const float2 *>(g.at().W2);
    float2 *__restrict__ W1 = static_cast<float2 *>(g.at().W1);
    using F = F3<R>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2 *s = reinterpret_cast<float2 *>(smem_raw);
    constexpr int ny = F::M / 2;
    const F3Thread<R> th;
    const int kx = blockIdx.y, z0 = blockIdx.x * F::NL;
    {
        const int ll = th.tid % F::NL;
        float2 *l = s + ll * F::LS;
        if (z0 + ll < nz) {
            const float2 *src = W2 + (size_t)kx * F::M * nz + z0 + ll;
#pragma unroll 8
            for (int ky = th.tid / F::NL; ky < F::M; ky += F::NB) f3f_copy8(l + f3_pos(ky), src + (size_t)ky * nz);
        } else {
            for (int ky = th.tid / F::NL; ky < F::M; ky += F::NB) l[f3_pos(ky)] = make_float2(0.f, 0.f);
        }
    }
    fx_copy_wait();
    __syncthreads();
    const float2 *p = s + th.line * F::LS + f3_pos(th.b);
    f3f_first<R, false, 0, true>(s, th, [&](int t) { return f3f_ld(p[t * 9 * R]); });
    f3f_second<R, false>(s, th, tw);
    float2 *out = W1 + ((size_t)z0 * hx + kx) * ny;
    const int lines = nz - z0;
    f3f_last<R, false, true>(s, th, tw, [&](int ln, int i, int t, f32c v) {
        if (ln < lines) (out + (size_t)ln * hx * ny + i)[t * F::NSC] = f3f_st(v);
    });
}

template <int R, int COUNT>
__global__ void __launch_bounds__(F3<R>::THREADS, F3F<R>::CTAS)
    k_f3f_xi(const __grid_constant__ F3Group<COUNT> g, int ny, const float2 *__restrict__ tw)
{
    const float2 *__restrict__ W1 = static_cast<const float2 *>(g.at().W1);
    float *__restrict__ u = static_cast<float *>(g.at().u);
    using F = F3<R>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2 *s = reinterpret_cast<float2 *>(smem_raw);
    constexpr int nx = F::M / 2, hx = nx + 1;
    const F3Thread<R> th;
    const int z = blockIdx.y, y0 = blockIdx.x * 2 * F::NL;
    {
        // Hermitian fill (see body_xi)
        const int ll = th.tid % F::NL, yy = y0 + 2 * ll;
        const float2 *src = W1 + (size_t)z * hx * ny + yy;
        float2 *l = s + ll * F::LS;
        gather_smem<4, float4>(
            th.tid / F::NL, F::NB, hx,
            [&](int k) {
                float2 a = make_float2(0.f, 0.f), b = a;
                if (yy < ny) a = src[(size_t)k * ny];
                if (yy + 1 < ny) b = src[(size_t)k * ny + 1];
                return make_float4(a.x, a.y, b.x, b.y);
            },
            [&](int k, const float4 &v) {
                const bool real = k == 0 || k == nx;
                const float ai = real ? 0.f : v.y, bi = real ? 0.f : v.w;
                l[f3_pos(k)] = make_float2(v.x - bi, ai + v.z);
                if (!real) l[f3_pos(F::M - k)] = make_float2(v.x + bi, v.z - ai);
            });
    }
    __syncthreads();
    const float2 *p = s + th.line * F::LS + f3_pos(th.b);
    f3f_first<R, false, 0, true>(s, th, [&](int t) { return f3f_ld(p[t * 9 * R]); });
    f3f_second<R, false>(s, th, tw);
    float *out = u + ((size_t)z * ny + y0) * nx;
    const int rows = ny - y0;
    f3f_last<R, false, true>(s, th, tw, [&](int ln, int i, int t, f32c v) {
        float *o = out + (size_t)(2 * ln) * nx + i;
        if (2 * ln < rows) o[t * F::NSC] = v.re;
        if (2 * ln + 1 < rows) o[nx + t * F::NSC] = v.im;
    });
}

}  // namespace

// One pass (see f3_launch); the stage-ordered tables follow the M plain twiddles.
template <int R, int COUNT>
void f3f_launch_group(const F3Call &c, int pass)
{
    using F = F3<R>;
    constexpr size_t smem = F3F<R>::SMEM;
    static_assert(smem <= 48 * 1024, "no raised shared-memory limit");
    F3Group<COUNT> g{};
    for (int i = 0; i < c.count; ++i) g.inst[i] = c.inst[i];
    const Plan *p = c.p;
    const int last = p->d == 3 ? 4 : 2, conv = p->d == 3 ? 2 : 1;
    const int ny = p->n[1], hx = p->n[0] + 1, nz = c.nz, full = p->mult_full ? 1 : 0;
    const int axis = pass == 0 || pass == last ? 0 : pass == conv ? p->d - 1 : 1;
    const float2 *tw = static_cast<const float2 *>(p->d_tw[axis]) + F::M;
    const float2 *twi = static_cast<const float2 *>(p->d_twi[axis]) + F::M;
    const dim3 gx((ny + 2 * F::NL - 1) / (2 * F::NL), nz, c.count), gy((nz + F::NL - 1) / F::NL, hx, c.count);
    if (pass == 0) {
        k_f3f_xf<R, COUNT><<<gx, F::THREADS, smem, c.st>>>(g, ny, tw);
    } else if (pass == last) {
        k_f3f_xi<R, COUNT><<<gx, F::THREADS, smem, c.st>>>(g, ny, twi);
    } else if (pass == conv && p->d == 3) {
        const int My = p->M[1];
        k_f3f_conv<R, true, COUNT><<<dim3((My + F::NL - 1) / F::NL, hx, c.count), F::THREADS, smem, c.st>>>(
            g, My, ny + 1, tw, twi, full);
    } else if (pass == conv) {
        k_f3f_conv<R, false, COUNT><<<dim3((hx + F::NL - 1) / F::NL, 1, c.count), F::THREADS, smem, c.st>>>(
            g, hx, ny + 1, tw, twi, full);
    } else if (pass == 1) {
        k_f3f_yf<R, COUNT><<<gy, F::THREADS, smem, c.st>>>(g, nz, hx, tw);
    } else {
        k_f3f_yi<R, COUNT><<<gy, F::THREADS, smem, c.st>>>(g, nz, hx, twi);
    }
}
template <int R>
void f3f_launch(const F3Call &c, int pass)
{
    if (c.count == 1) f3f_launch_group<R, 1>(c, pass);
    else f3f_launch_group<R, kF3Group>(c, pass);
}

}  // namespace gsm
