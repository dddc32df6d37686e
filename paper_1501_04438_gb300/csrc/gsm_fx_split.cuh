// gsm_fx_split.cuh -- the fixed-point passes of long 2D lines (padded length >=
// kSplitMinM), each line as two half-length transforms on two CTAs, of any half
// length and of those known at compile time.
#pragma once

#include "gsm_fx_passes.cuh"

namespace gsm {
namespace {

// ------------------------------------------------------------------ conv, long 2D lines
// Threads of a half line and CTAs per SM: a length known at compile time has 8
// values per thread (64 to 85 registers), any other 16 in 128.  FP64, white noise, xf,
// conv, xi in us: whole lines, halves of any length, halves of a length known at
// compile time: 4096^2 436, 1444, 516; 395, 1467, 451; 322, 1178, 369; 3000^2 371, 1452,
// 513; 391, 1438, 440; 233, 880, 258; 2048^2 108, 311, 133; 137, 397, 149; 83, 290, 91.
// (3000^2 in pairs of floats, which FP32X2 once was: 394, 1059, 389.)
template <class SC>
constexpr int split_threads()
{
    if constexpr (is_fixed_sched<SC>::value) return fixed_threads<SC, 8>();
    else return kSplitThreads;
}
template <class SC>
constexpr int split_ctas() { return is_fixed_sched<SC>::value ? 1024 / split_threads<SC>() : 2; }

// A conv line of padded length M = 2 Mh holds Mh values x and zeros; its even
// and odd frequencies are two transforms of length Mh, X[2k] = FFT_Mh(x)[k],
// X[2k + 1] = FFT_Mh(x w_M^n)[k], and the cropped inverse is
//   u[n] = IFFT_Mh(E)[n] + w_M^(-n) IFFT_Mh(O)[n]
// (E, O the multiplied halves): a cluster of two CTAs takes a line, one half
// each, and adds the peer's half through distributed shared memory.  Half
// lines leave room for several CTAs on an SM, whose phases overlap, where a
// whole line of 8192 (147 KB) fills it.  twM: the M twiddles w_M^m.
struct FxFromGlobalRot : FxInts {
    struct raw {
        fxc v;
        int e, i;
    };
    const fxc *p;
    const int *e;
    const int4 *twM;
    int rank;
    __device__ __forceinline__ raw load(int b, int off) const { return {p[b + off], e[(b + off) >> 1], b + off}; }
    __device__ __forceinline__ int exponent(const raw &r) const { return r.e; }
    __device__ __forceinline__ cx<long long> align(const raw &r, int em, bool longm) const
    {
        const cx<long long> x = FxInts::align({r.v, r.e}, em, longm);
        return rank ? fx_rot<true>(x, fx_tw(twM + r.i)) : x;
    }
};
struct FxHalfToSmem {
    static constexpr bool kSmem = true;
    fxc *s;
    const int4 *twM;
    int rank;
    __device__ __forceinline__ void operator()(int b, int off, cx<long long> v) const
    {
        s[pidx<FX>(b + off)] = fx_st(rank ? fx_rot<false>(v, fx_tw(twM + b + off)) : v);
    }
};
struct FxMultHalf {   // output k' of a half is frequency 2 k' + rank
    FxMultRow m;
    int rank;
    template <int R>
    __device__ __forceinline__ int2 at(int b, int t, int nb) const { return m(2 * (b + t * nb) + rank); }
};

template <int EMAX, class SC, class SCI>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(split_threads<SC>(), split_ctas<SC>())
    k_fx_conv_split(fxc *__restrict__ W, const int2 *__restrict__ mult, const int *__restrict__ mrow_exp, FxExps ex,
                    int nlines, int ny1, SC sc, SCI sci, const int4 *__restrict__ tw,
                    const int4 *__restrict__ twi, const int4 *__restrict__ twM, int full)
{
    namespace cg = cooperative_groups;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int red[kFxRedWords];
    __shared__ int line_e;
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank();
    const int line = blockIdx.x >> 1;
    const int Mh = sc.M, M = 2 * Mh;
    const Group g = fx_thread_of<SC, EMAX>().g;
    fxc *s = reinterpret_cast<fxc *>(smem_raw);
    fxc *w = W + (size_t)line * Mh;
    const bool active = line < nlines;   // every CTA of a cluster reaches both cluster barriers
    if (active) {
        FxLine ln{0, 0, Mh > kFxLongM, red, 1};
        FxFromGlobalRot in;
        in.p = w;
        in.e = ex.xf + (line & 1) * ex.xf_par;
        in.twM = twM;
        in.rank = rank;
        const FxMultRow m{mult + (size_t)line * (full ? M : ny1), M, full};
        // the half's schedules always fuse (make_split_tables)
        ln.pad = sc.pad;
        fx_begin<true, EMAX, false, true>(s, sc, g, ln, in, FxNoOut{});
        fx_rest_of<true, EMAX, false, true>(s, sc, tw, g, ln, FxNoOut{});
        fx_mid_of<EMAX>(s, sc, sci, tw, g, ln, FxMultHalf{m, rank}, mrow_exp[line]);
        fx_rest_of<false, EMAX, false, false>(s, sci, twi, g, ln, FxHalfToSmem{s, twM, rank});
        if (threadIdx.x == 0) line_e = ln.E;
    }
    cl.sync();   // both halves transformed
    if (active) {
        const fxc *peer = cl.map_shared_rank(s, rank ^ 1);
        const int e0 = line_e, e1 = *cl.map_shared_rank(&line_e, rank ^ 1);
        const int e = max(e0, e1) + 1, d0 = min(e - e0, 62), d1 = min(e - e1, 62);
        const int h = Mh / 2, n0 = rank * h;
        for (int i = threadIdx.x; i < h; i += blockDim.x) {
            const int n = n0 + i, p = pidx<FX>(n);
            w[n] = fx_st(fx_add(fx_shift(fx_ld(s[p]), d0), fx_shift(fx_ld(peer[p]), d1)));
        }
        if (rank == 0 && threadIdx.x == 0) ex.cv[line] = e;
    }
    cl.sync();   // the peer has read this CTA's half: its shared memory may go
}

// ------------------------------------------------------------------ x forward, long 2D lines
// The same halves for an x line (two real rows).  The forward needs no
// exchange: the Hermitian split pairs Z[k] with Z[M - k], of the parity of k,
// so each CTA of a pair writes the frequencies of its own parity, with its own
// line exponent.
struct FxFromRowsRot : FxDoubles {
    struct raw {
        double a, b;
        int i;
    };
    const double *pa, *pb;
    const int4 *twM;
    int rank;
    __device__ __forceinline__ raw load(int b, int off) const
    {
        const int i = b + off;
        return {pa != nullptr ? pa[i] : 0.0, pb != nullptr ? pb[i] : 0.0, i};
    }
    __device__ __forceinline__ int exponent(const raw &r) const { return FxDoubles::exponent({r.a, r.b}); }
    __device__ __forceinline__ cx<long long> align(const raw &r, int em, bool longm) const
    {
        const cx<long long> x = FxDoubles::align({r.a, r.b}, em, longm);
        return rank ? fx_rot<true>(x, fx_tw(twM + r.i)) : x;
    }
};

template <int EMAX, class SC>
__global__ void __launch_bounds__(split_threads<SC>(), split_ctas<SC>())
    k_fx_xf_split(const double *__restrict__ rho, fxc *__restrict__ W1, FxExps ex, int nx, int ny, SC sc,
                  const int4 *__restrict__ tw, const int4 *__restrict__ twM)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int red[kFxRedWords];
    const int rank = blockIdx.x & 1, ya = 2 * (blockIdx.x >> 1);
    const int Mh = sc.M;   // == nx
    const Group g = fx_thread_of<SC, EMAX>().g;
    fxc *s = reinterpret_cast<fxc *>(smem_raw);
    FxLine ln{0, 0, Mh > kFxLongM, red, 1};
    FxFromRowsRot in;
    in.pa = ya < ny ? rho + (size_t)ya * nx : nullptr;
    in.pb = ya + 1 < ny ? rho + (size_t)(ya + 1) * nx : nullptr;
    in.twM = twM;
    in.rank = rank;
    fx_transform<true, EMAX, false, false>(s, sc, tw, g, ln, in, FxToSmem{s, &ln});
    if (threadIdx.x == 0 && ya < ny) ex.xf[rank * ex.xf_par + (ya >> 1)] = ln.E;
    __syncthreads();
    // frequency k = 2 k' + rank sits at k' of this half; M - k at (Mh - k' - rank) mod Mh
    const int nk = rank ? nx / 2 : nx / 2 + 1;   // k = 0 .. nx of this parity (nx is even)
    for (int i = threadIdx.x; i < 2 * nk; i += blockDim.x) {
        const int kp = i >> 1, r = i & 1, k = 2 * kp + rank;
        int km = Mh - kp - rank;
        if (km == Mh) km = 0;
        const cx<long long> zk = fx_ld(s[fx_pos(kp, ln.pad)]);
        const cx<long long> zm = fx_ld(s[fx_pos(km, ln.pad)]);
        cx<long long> v;
        if (r) v = {radd(zk.im, zm.im), rsub(zm.re, zk.re)};
        else v = {radd(zk.re, zm.re), rsub(zk.im, zm.im)};
        if (ya + r < ny) W1[(size_t)k * ny + ya + r] = fx_st(v);
    }
}

// ------------------------------------------------------------------ x inverse, long 2D lines
// The halves of the inverse x line (two real rows), on a cluster of two CTAs as
// in the conv: the Hermitian fill pairs Z[k] with Z[M - k], of the parity of k,
// so each CTA reads the rows of its own parity only; the halves of the cropped
// line are added through distributed shared memory, and each CTA stores one
// half of both rows.
struct FxFromSmemHalf : FxInts {   // element i of a half is frequency 2 i + rank
    const fxc *s;
    const int *e;
    int M, rank, pad;
    __device__ __forceinline__ raw load(int b, int off) const
    {
        const int i = b + off, f = 2 * i + rank;
        return {s[fx_pos(i, pad)], e[min(f, M - f)]};
    }
};

template <int EMAX, class SC>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(split_threads<SC>(), split_ctas<SC>())
    k_fx_xi_split(const fxc *__restrict__ W1, double *__restrict__ u, const int *__restrict__ ek, int nx, int ny,
                  SC sc, const int4 *__restrict__ tw, const int4 *__restrict__ twM)
{
    namespace cg = cooperative_groups;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int red[kFxRedWords];
    __shared__ int line_e;
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank(), ya = 2 * (blockIdx.x >> 1);   // ya < ny
    const int Mh = sc.M, M = 2 * Mh;   // Mh == nx, even
    const Group g = fx_thread_of<SC, EMAX>().g;
    const bool two = ya + 1 < ny;
    fxc *s = reinterpret_cast<fxc *>(smem_raw);
    struct AB {
        longlong2 a, b;
    };
    // the frequencies k = 2 k' + rank <= nx; M - k sits at Mh - k' - rank
    gather_smem<4, AB>(
        (int)threadIdx.x, (int)blockDim.x, rank ? nx / 2 : nx / 2 + 1,
        [&](int kp) {
            const longlong2 *q = reinterpret_cast<const longlong2 *>(W1 + (size_t)(2 * kp + rank) * ny + ya);
            AB v{q[0], {0, 0}};
            if (two) v.b = q[1];
            return v;
        },
        [&](int kp, const AB &v) {
            const int k = 2 * kp + rank;
            const bool real = k == 0 || k == nx;
            const long long ai = real ? 0 : v.a.y, bi = real ? 0 : v.b.y;
            s[fx_pos(kp, sc.pad)] = {rsub(v.a.x, bi), radd(ai, v.b.x)};
            if (!real) s[fx_pos(Mh - kp - rank, sc.pad)] = {radd(v.a.x, bi), rsub(v.b.x, ai)};
        });
    __syncthreads();
    FxLine ln{0, 0, Mh > kFxLongM, red, 0};
    FxFromSmemHalf in;
    in.s = s;
    in.e = ek;
    in.M = M;
    in.rank = rank;
    in.pad = sc.pad;
    fx_transform<false, EMAX, false, false>(s, sc, tw, g, ln, in, FxHalfToSmem{s, twM, rank});
    if (threadIdx.x == 0) line_e = ln.E;
    cl.sync();   // both halves transformed
    const fxc *peer = cl.map_shared_rank(s, rank ^ 1);
    const int e0 = line_e, e1 = *cl.map_shared_rank(&line_e, rank ^ 1);
    const int e = max(e0, e1) + 1, d0 = min(e - e0, 62), d1 = min(e - e1, 62);
    const int h = Mh / 2;
    double *row = u + (size_t)ya * nx;
    for (int i = threadIdx.x; i < h; i += blockDim.x) {
        const int n = rank * h + i, p = pidx<FX>(n);
        const cx<long long> v = fx_add(fx_shift(fx_ld(s[p]), d0), fx_shift(fx_ld(peer[p]), d1));
        row[n] = fx_out_double(v.re, e);
        if (two) row[nx + n] = fx_out_double(v.im, e);
    }
    cl.sync();   // the peer has read this CTA's half: its shared memory may go
}

// A split pass (0 xf, 1 conv, 2 xi) of a 2D plan, and its kernels' shared-memory limits.
template <int EMAX, class SC, class SCI>
void split_launch(const FxCall &a, int pass, const SC &sc, const SCI &sci)
{
    const Plan *p = a.p;
    const bool conv = pass == 1;
    const int nx = p->n[0], ny = p->n[1], hx = nx + 1;
    fxc *W1 = static_cast<fxc *>(a.W1);
    const int4 *twM = static_cast<const int4 *>(p->d_tw[conv ? 1 : 0]) + p->M[conv ? 1 : 0];   // the plain entries
    const PassCfg &c = conv ? p->cfg_split : p->cfg_xsplit;
    const int b = is_fixed_sched<SC>::value ? split_threads<SC>() : c.nthr;
    const int4 *tw = static_cast<const int4 *>(conv ? p->d_twh : p->d_twxh);
    if (conv)
        k_fx_conv_split<EMAX, SC, SCI><<<2 * hx, b, c.smem, a.st>>>(
            W1, static_cast<const int2 *>(p->d_mult), p->d_mrow, a.ex, hx, ny + 1, sc, sci, tw,
            static_cast<const int4 *>(p->d_twhi), twM, p->mult_full ? 1 : 0);
    else if (pass == 0)
        k_fx_xf_split<EMAX, SC><<<2 * ((ny + 1) / 2), b, c.smem, a.st>>>(a.rho, W1, a.ex, nx, ny, sc, tw, twM);
    else
        k_fx_xi_split<EMAX, SC><<<2 * ((ny + 1) / 2), b, c.smem, a.st>>>(W1, a.u, a.ex.cv, nx, ny, sc, tw, twM);
}
template <int EMAX, class SC, class SCI>
cudaError_t split_raise(bool conv, size_t smem)
{
    if (conv) return raise_smem(k_fx_conv_split<EMAX, SC, SCI>, smem);
    const cudaError_t e = raise_smem(k_fx_xf_split<EMAX, SC>, smem);
    return e == cudaSuccess ? raise_smem(k_fx_xi_split<EMAX, SC>, smem) : e;
}

}  // namespace

// The split passes of half length M, defined in one translation unit (see FixedPasses).
template <int M>
struct FixedSplit {
    static cudaError_t raise(bool conv, size_t smem);
    static void launch(const FxCall &a, int pass);
};
#ifdef GSM_FX_LENGTH_UNIT
template <int M>
cudaError_t FixedSplit<M>::raise(bool conv, size_t smem)
{
    return split_raise<8, FixedSched<M>, FixedSched<M, true>>(conv, smem);
}
template <int M>
void FixedSplit<M>::launch(const FxCall &a, int pass)
{
    split_launch<8>(a, pass, FixedSched<M>(), FixedSched<M, true>());
}
#endif

// The half lengths of each translation unit (gsm_fx_split_*.cu).
#define GSM_FX_HALVES_A(X) X(2304) X(2400) X(3072) X(3200) X(4096)
#define GSM_FX_HALVES_B(X) X(2250) X(2430) X(3000) X(3240) X(4050)
#define GSM_FX_HALVES_C(X) X(2160) X(2500) X(2916) X(3456) X(4000)
#define GSM_FX_HALVES_D(X) X(2048) X(2560) X(2880) X(3600) X(3888)
#define GSM_FX_HALVES_E(X) X(2592) X(2700) X(3750) X(3840)
#define GSM_FX_HALVES(X) \
    GSM_FX_HALVES_A(X) GSM_FX_HALVES_B(X) GSM_FX_HALVES_C(X) GSM_FX_HALVES_D(X) GSM_FX_HALVES_E(X)
#define GSM_FX_DEFINE_HALF(M) template struct FixedSplit<M>;

}  // namespace gsm
