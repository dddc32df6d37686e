// gsm_fx_passes.cuh -- the passes of the FP64 and FP32X2 precisions in block
// fixed point (gsm_fx.cuh).  Same data flow as the FP32 passes (gsm_passes.cu);
// the workspace holds 64-bit integers, and one exponent per transformed line:
//   xf[z][y/2]   of W1 as the x pass leaves it (one line = rows y, y + 1); in
//                2D [kx parity][y/2] when the x pass is split by parity
//   yf[kx][z]    of W2 as the y pass leaves it
//   cv[kx][ky]   of W2 after the conv pass (2D: cv[kx] of W1)
//   yi[z][kx]    of W1 after the inverse y pass
// Each pass reads lines that run across those of the pass before, so element i
// of a line comes with exponent i of a row of one of these arrays.
//
// A line's first stage takes its inputs straight into registers (in the
// forward passes and the conv pass from global memory: the threads of a warp
// hold consecutive elements), and the last stage of the conv and inverse
// passes stores straight to global memory: a transform of s stages crosses
// shared memory s - 1 times.
#pragma once

#include "gsm_pass_common.cuh"

namespace gsm {
namespace {

// Resident CTAs per SM asked of the compiler for the kernels with EMAX elements
// per thread: 8 elements, four CTAs of 256 threads (64 registers): measured
// 0.30 against 0.33 ms (three) and 0.37 ms (two) for the y and x passes at
// 128^3, 0.139 against 0.162 and 0.164 ms for 1024^2.
constexpr int fx_ctas(int emax) { return emax == 8 ? 4 : 1; }

// A thread's place in its CTA: the line's group, the line of the CTA and the
// thread of the CTA.  The CTAs are gthr x nl blocks (thread x of line y), so
// that none of it costs a division.
struct FxThread {
    Group g;
    int l, tid;
};
__device__ __forceinline__ FxThread fx_thread()
{
    FxThread th;
    th.g.t = threadIdx.x;
    th.g.T = blockDim.x;
    th.g.bar = blockDim.x == 32 ? -1 : blockDim.y == 1 ? 0 : 1 + (int)threadIdx.y;
    th.l = threadIdx.y;
    th.tid = threadIdx.y * blockDim.x + threadIdx.x;
    return th;
}
// the same for a schedule known at compile time
template <class SC, int EMAX>
constexpr int fixed_threads() { return ((SC::M + EMAX - 1) / EMAX + 31) / 32 * 32; }
template <class SC, int EMAX>
__device__ __forceinline__ FxThread fx_thread_of()
{
    FxThread th = fx_thread();
    if constexpr (is_fixed_sched<SC>::value) {
        th.g.T = fixed_threads<SC, EMAX>();
        if (fixed_threads<SC, EMAX>() == 32) th.g.bar = -1;
    }
    return th;
}
// one warp per line in a one-dimensional CTA
__device__ __forceinline__ FxThread fx_warp_line()
{
    return FxThread{Group{(int)(threadIdx.x & 31), 32, -1}, (int)(threadIdx.x >> 5), (int)threadIdx.x};
}

// ------------------------------------------------------------------ inputs and outputs
struct FxNoOut {
    static constexpr bool kSmem = false;
    __device__ __forceinline__ void operator()(int, int, cx<long long>) const {}
};
// output i to the line's own shared memory
struct FxToSmem {
    static constexpr bool kSmem = true;
    fxc *s;
    const FxLine *ln;
    __device__ __forceinline__ void operator()(int b, int off, cx<long long> v) const
    {
        s[fx_pos(b, ln->pad) + fx_pos(off, ln->pad)] = fx_st(v);
    }
};
// output i < n to consecutive global memory
struct FxToGlobal {
    static constexpr bool kSmem = false;
    fxc *p;
    int n;
    __device__ __forceinline__ void operator()(int b, int off, cx<long long> v) const
    {
        if (b + off < n) (p + b)[off] = fx_st(v);
    }
};
// two rows of doubles
struct FxFromRows : FxDoubles {
    const double *a, *b;   // NULL: a row of zeros
    __device__ __forceinline__ raw load(int i, int off) const
    {
        return {a != nullptr ? (a + i)[off] : 0.0, b != nullptr ? (b + i)[off] : 0.0};
    }
};
struct FxToRows {
    static constexpr bool kSmem = false;
    double *a, *b;         // NULL: not stored
    int n;
    const FxLine *ln;
    __device__ __forceinline__ void operator()(int i, int off, cx<long long> v) const
    {
        if (i + off >= n) return;
        if (a != nullptr) (a + i)[off] = fx_out_double(v.re, ln->E);
        if (b != nullptr) (b + i)[off] = fx_out_double(v.im, ln->E);
    }
};
// consecutive global elements, the exponent of element i at e[i >> shift]
template <bool CG>
struct FxFromGlobal : FxInts {
    const fxc *p;          // NULL: a line of zeros
    const int *e;
    int shift;
    __device__ __forceinline__ raw load(int b, int off) const
    {
        if (p == nullptr) return {fxc{0, 0}, kFxZero};
        raw r;
        const longlong2 v = ldw<CG>(reinterpret_cast<const longlong2 *>(p + b) + off);
        r.v = {v.x, v.y};
        r.e = ldw<CG>(e + ((b + off) >> shift));
        return r;
    }
};
// the line's own shared memory, exponent of element i at e[min(i, fold - i)]
template <bool CG>
struct FxFromSmem : FxInts {
    const fxc *s;
    const int *e;
    int fold, pad;
    __device__ __forceinline__ raw load(int b, int off) const
    {
        const int i = b + off;
        raw r;
        r.v = s[fx_pos(i, pad)];
        r.e = ldw<CG>(e + min(i, fold - i));
        return r;
    }
};

// Copies of 16 bytes, global to shared (cp.async through L2, which is what the
// batch queue kernel needs: see ldw).
__device__ __forceinline__ void fx_copy16(fxc *dst, const fxc *src)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void fx_copy_wait()
{
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
}

// ------------------------------------------------------------------ x forward
template <int EMAX, class SC>
__device__ __forceinline__ void fx_body_xf(const FxThread &th, const double *__restrict__ rho, fxc *__restrict__ W1, const FxExps &ex,
                                           int nx, int ny, int hx, const SC &sc, int nl,
                                           const int4 *__restrict__ tw, int bx, int by, unsigned char *smem_raw,
                                           int *red)
{
    const int M = sc.M, LS = line_stride<FX>(M);
    const Group &g = th.g;
    const int l = th.l;
    fxc *s = reinterpret_cast<fxc *>(smem_raw) + l * LS;
    const int z = by, y0 = bx * 2 * nl, ya = y0 + 2 * l;
    const double *slab = rho + (size_t)z * ny * nx;
    FxLine ln{0, 0, M > kFxLongM, red, 1};
    FxFromRows in;
    in.a = ya < ny ? slab + (size_t)ya * nx : nullptr;
    in.b = ya + 1 < ny ? slab + (size_t)(ya + 1) * nx : nullptr;
    fx_transform<true, EMAX, true, false>(s, sc, tw, g, ln, in, FxToSmem{s, &ln});
    if (g.t == 0 && ya < ny) ex.xf[(size_t)z * ((ny + 1) >> 1) + (ya >> 1)] = ln.E;
    __syncthreads();
    // Z = A + iB with A, B the transforms of the two real rows:
    // 2A[k] = Z[k] + conj Z[-k], 2B[k] = -i (Z[k] - conj Z[-k]); the factor 2
    // is removed by the multiplier.  Consecutive threads take consecutive y.
    const fxc *s0 = reinterpret_cast<const fxc *>(smem_raw);
    fxc *out = W1 + (size_t)z * hx * ny;
    // (the CTA's nl g.T threads are whole rows of 2 nl)
    const int nrow = 2 * nl, r = th.tid % nrow, ll = r >> 1;
    for (int k = th.tid / nrow; k < hx; k += g.T >> 1) {
        const cx<long long> zk = fx_ld(s0[ll * LS + fx_pos(k, ln.pad)]);
        const cx<long long> zm = fx_ld(s0[ll * LS + fx_pos(k == 0 ? 0 : M - k, ln.pad)]);
        cx<long long> v;
        if (r & 1) v = {radd(zk.im, zm.im), rsub(zm.re, zk.re)};
        else v = {radd(zk.re, zm.re), rsub(zk.im, zm.im)};
        if (y0 + r < ny) out[(size_t)k * ny + y0 + r] = fx_st(v);
    }
}

// ------------------------------------------------------------------ y forward
template <int EMAX, bool CG, class SC>
__device__ __forceinline__ void fx_body_yf(const FxThread &th, const fxc *__restrict__ W1, fxc *__restrict__ W2, const FxExps &ex, int ny,
                                           int nz, int hx, const SC &sc, int nl,
                                           const int4 *__restrict__ tw, int bx, int by, unsigned char *smem_raw,
                                           int *red)
{
    const int M = sc.M, LS = line_stride<FX>(M);
    const Group &g = th.g;
    const int l = th.l;
    fxc *s = reinterpret_cast<fxc *>(smem_raw) + l * LS;
    const int kx = by, z0 = bx * nl, z = z0 + l;
    FxLine ln{0, 0, M > kFxLongM, red, 0};
    FxFromGlobal<CG> in;
    in.p = z < nz ? W1 + ((size_t)z * hx + kx) * ny : nullptr;
    in.e = ex.xf + (size_t)z * ((ny + 1) >> 1);
    in.shift = 1;
    fx_transform<true, EMAX, true, false>(s, sc, tw, g, ln, in, FxToSmem{s, &ln});
    if (g.t == 0 && z < nz) ex.yf[(size_t)kx * nz + z] = ln.E;
    __syncthreads();
    const fxc *s0 = reinterpret_cast<const fxc *>(smem_raw);
    fxc *out = W2 + (size_t)kx * M * nz;
    const int ll = th.tid % nl, zz = z0 + ll;
    if (zz < nz) {
        for (int ky = th.tid / nl; ky < M; ky += g.T) out[(size_t)ky * nz + zz] = s0[ll * LS + fx_pos(ky, ln.pad)];
    }
}

// ------------------------------------------------------------------ conv
// Lines of n stored values padded to M: forward, multiplier, inverse, crop, in
// place; 3D: line = kx * My + ky, 2D: line = kx (see body_conv).  mrow_exp:
// exponent of each multiplier row.
struct FxMultRow {
    const int2 *row;
    int M, full;
    __device__ __forceinline__ int2 operator()(int k) const { return __ldg(row + (full ? k : min(k, M - k))); }
    // entry b + t nb of a stage of radix R (nb = M / R): its half is known for even R
    template <int R>
    __device__ __forceinline__ int2 at(int b, int t, int nb) const
    {
        if (full || R % 2 != 0) return (*this)(b + t * nb);
        return __ldg(t < R / 2 ? row + b + t * nb : row - b + (M - t * nb));
    }
};
// output k of the forward, multiplied, back to the line (schedules whose
// middle stages are not fused), and from there, scaled to its largest product
struct FxMulToSmem {
    static constexpr bool kSmem = true;
    fxc *s;
    FxMultRow m;
    const FxLine *ln;
    __device__ __forceinline__ void operator()(int b, int off, cx<long long> v) const
    {
        const int2 f = m(b + off);
        s[fx_pos(b, ln->pad) + fx_pos(off, ln->pad)] = {fx_mul(fx_split(v.re), f.x, f.y), fx_mul(fx_split(v.im), f.x, f.y)};
    }
};

struct FxFromProducts : FxInts {
    const fxc *s;
    FxMultRow m;
    int e0, pad;
    __device__ __forceinline__ raw load(int b, int off) const
    {
        return {s[fx_pos(b + off, pad)], -fx_mult_exp(m(b + off))};
    }
    static __device__ __forceinline__ int exponent(const raw &r)
    {
        return fx_bits(fx_abs_high(r.v.re) | fx_abs_high(r.v.im)) + r.e;
    }
    static __device__ __forceinline__ cx<long long> align(const raw &r, int em, bool)   // below 2^62
    {
        return fx_scale2(cx<long long>{r.v.re, r.v.im}, fx_product_shift(em - 30, -r.e));
    }
    __device__ __forceinline__ int line_exponent(int em) const { return e0 + em - 30; }
};

// Forward, multiplication and inverse of the line whose inputs `in` gives;
// the outputs go to `out`.
template <int EMAX, bool ZPAD, bool CROP, class SC, class SCI, class In, class MultF, class MulOut, class Out>
__device__ __forceinline__ void fx_convolve(fxc *s, const SC &sc, const SCI &sci, const int4 *__restrict__ tw,
                                            const int4 *__restrict__ twi, const Group &g, FxLine &ln, In in,
                                            MultF mult, int erow, MulOut mul_out, Out out)
{
    bool fused = true;
    if constexpr (!is_fixed_sched<SC>::value) fused = fused_radix(sc, sci) != 0;
    ln.pad = sc.pad;
    fx_begin<true, EMAX, ZPAD, true>(s, sc, g, ln, in, mul_out);
    if (fused) {
        fx_rest_of<true, EMAX, false, true>(s, sc, tw, g, ln, FxNoOut{});
        fx_mid_of<EMAX>(s, sc, sci, tw, g, ln, mult, erow);
        fx_rest_of<false, EMAX, CROP, false>(s, sci, twi, g, ln, out);
    } else if constexpr (!is_fixed_sched<SC>::value) {
        fx_rest_of<true, EMAX, false, false>(s, sc, tw, g, ln, mul_out);
        group_sync(g);
        FxFromProducts back;
        back.s = s;
        back.m = mult;
        back.e0 = ln.E + erow;
        back.pad = ln.pad;
        fx_transform<false, EMAX, false, CROP>(s, sci, twi, g, ln, back, out);
    }
}

template <int EMAX, bool CG, class SC, class SCI>
__device__ __forceinline__ void fx_body_conv(const FxThread &th, fxc *__restrict__ W, const int2 *__restrict__ mult,
                                             const int *__restrict__ mrow_exp, const FxExps &ex, int nlines, int n,
                                             int is3d, int My, int ny1, const SC &sc, const SCI &sci, int nl,
                                             const int4 *__restrict__ tw, const int4 *__restrict__ twi,
                                             int bx, int by, unsigned char *smem_raw, bool full, int *red)
{
    const int M = sc.M, LS = line_stride<FX>(M);
    const Group &g = th.g;
    const int l = th.l;
    fxc *s = reinterpret_cast<fxc *>(smem_raw) + l * LS;
    // 3D: block row = kx, block column = nl consecutive ky; 2D: nl consecutive kx
    const int ky = bx * nl + l, kx = by;
    if (ky >= (is3d ? My : nlines)) return;   // the whole group leaves; no CTA barrier follows
    const int line = kx * My + ky;
    fxc *w = W + (size_t)line * n;
    size_t row = line;            // of the multiplier: the half spectrum (full) or the octant
    FxFromGlobal<CG> in;
    in.p = w;
    if (is3d) {
        if (!full) row = (size_t)kx * ny1 + min(ky, My - ky);
        in.e = ex.yf + (size_t)kx * n;
        in.shift = 0;
    } else {
        in.e = ex.xf + (line & 1) * ex.xf_par;
        in.shift = 1;
    }
    const FxMultRow m{mult + row * (full ? M : n + 1), M, full ? 1 : 0};
    FxLine ln{0, 0, M > kFxLongM, red, is3d ? 0 : 1};
    fx_convolve<EMAX, true, true>(s, sc, sci, tw, twi, g, ln, in, m, mrow_exp[row], FxMulToSmem{s, m, &ln},
                                  FxToGlobal{w, n});
    if (g.t == 0) ex.cv[line] = ln.E;
}

// ------------------------------------------------------------------ y inverse
template <int EMAX, bool CG, class SC>
__device__ __forceinline__ void fx_body_yi(const FxThread &th, const fxc *__restrict__ W2, fxc *__restrict__ W1, const FxExps &ex, int ny,
                                           int nz, int hx, const SC &sc, int nl,
                                           const int4 *__restrict__ tw, int bx, int by, unsigned char *smem_raw,
                                           int *red)
{
    const int M = sc.M, LS = line_stride<FX>(M);
    const Group &g = th.g;
    const int l = th.l;
    fxc *s0 = reinterpret_cast<fxc *>(smem_raw);
    fxc *s = s0 + l * LS;
    const int pad = sc.pad;
    const int kx = by, z0 = bx * nl;
    const fxc *src = W2 + (size_t)kx * M * nz;
    const int ll = th.tid % nl;
    if (z0 + ll < nz) {
        for (int ky = th.tid / nl; ky < M; ky += g.T)
            fx_copy16(s0 + ll * LS + fx_pos(ky, pad), src + (size_t)ky * nz + z0 + ll);
    }
    fx_copy_wait();
    __syncthreads();
    const int z = z0 + l;
    if (z >= nz) return;          // whole groups; no CTA barrier follows
    FxLine ln{0, 0, M > kFxLongM, red, 1};
    FxFromSmem<CG> in;
    in.s = s;
    in.e = ex.cv + (size_t)kx * M;
    in.fold = INT_MAX;
    in.pad = pad;
    fx_transform<false, EMAX, false, true>(s, sc, tw, g, ln, in, FxToGlobal{W1 + ((size_t)z * hx + kx) * ny, ny});
    if (g.t == 0) ex.yi[(size_t)z * hx + kx] = ln.E;
}

// ------------------------------------------------------------------ x inverse
// ek: exponents of the kx rows of this slab (3D: yi[z], 2D: cv)
template <int EMAX, bool CG, class SC>
__device__ __forceinline__ void fx_body_xi(const FxThread &th, const fxc *__restrict__ W1, double *__restrict__ u,
                                           const int *__restrict__ ek, int nx, int ny, int hx, const SC &sc, int nl,
                                           const int4 *__restrict__ tw, int bx, int by,
                                           unsigned char *smem_raw, int *red)
{
    const int M = sc.M, LS = line_stride<FX>(M);
    const Group &g = th.g;
    const int l = th.l;
    fxc *s0 = reinterpret_cast<fxc *>(smem_raw);
    fxc *s = s0 + l * LS;
    const int pad = sc.pad;
    const int z = by, y0 = bx * 2 * nl;
    const fxc *src = W1 + (size_t)z * hx * ny;
    // Z[k] = A[k] + i B[k] (k = 0..nx), Z[M-k] = conj A[k] + i conj B[k];
    // A, B real at k = 0 and k = nx (DC and Nyquist of real rows)
    struct AB {
        longlong2 a, b;
    };
    const int ll = th.tid % nl, yy = y0 + 2 * ll;
    gather_smem<4, AB>(
        th.tid / nl, g.T, hx,
        [&](int k) {
            const longlong2 *q = reinterpret_cast<const longlong2 *>(src + (size_t)k * ny + yy);
            AB v{{0, 0}, {0, 0}};
            if (yy < ny) v.a = ldw<CG>(q);
            if (yy + 1 < ny) v.b = ldw<CG>(q + 1);
            return v;
        },
        [&](int k, const AB &v) {
            const bool real = k == 0 || k == nx;
            const long long ai = real ? 0 : v.a.y, bi = real ? 0 : v.b.y;
            s0[ll * LS + fx_pos(k, pad)] = {rsub(v.a.x, bi), radd(ai, v.b.x)};
            if (!real) s0[ll * LS + fx_pos(M - k, pad)] = {radd(v.a.x, bi), rsub(v.b.x, ai)};
        });
    __syncthreads();
    const int ya = y0 + 2 * l;
    if (ya >= ny) return;         // whole groups; no CTA barrier follows
    double *slab = u + (size_t)z * ny * nx;
    FxLine ln{0, 0, M > kFxLongM, red, 0};
    FxFromSmem<CG> in;
    in.s = s;
    in.e = ek;
    in.fold = M;
    in.pad = pad;
    FxToRows out{slab + (size_t)ya * nx, ya + 1 < ny ? slab + (size_t)(ya + 1) * nx : nullptr, nx, &ln};
    fx_transform<false, EMAX, false, true>(s, sc, tw, g, ln, in, out);
}

}  // namespace
}  // namespace gsm
