// gsm_fx_conv.cu -- fixed point: the conv pass and the split passes of long 2D lines.
#include "gsm_fx_passes.cuh"

namespace gsm {
namespace {

template <int EMAX>
__global__ void __launch_bounds__(fx_threads(EMAX), fx_ctas(EMAX))
    k_fx_conv(fxc *__restrict__ W, const int2 *__restrict__ mult, const int *__restrict__ mrow_exp, FxExps ex,
              int nlines, int n, int is3d, int My, int ny1, Sched sc, Sched sci, int nl,
              const int4 *__restrict__ tw, const int4 *__restrict__ twi, int full)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int red[kFxRedWords];
    fx_body_conv<EMAX, false>(fx_thread(), W, mult, mrow_exp, ex, nlines, n, is3d, My, ny1, sc, sci, nl, tw, twi, blockIdx.x,
                              blockIdx.y, smem_raw, full != 0, red);
}

// ------------------------------------------------------------------ conv, long 2D lines
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
    __device__ __forceinline__ cx<long long> align(const raw &r, int em) const
    {
        // the x pass leaves values below 2^63: halved before a rotation
        const cx<long long> x = FxInts::align({r.v, r.e}, em + rank);
        return rank ? fx_rot<true>(x, twM[r.i]) : x;
    }
    __device__ __forceinline__ int line_exponent(int em) const { return em + rank; }
};
struct FxHalfToSmem {
    static constexpr bool kSmem = true;
    fxc *s;
    const int4 *twM;
    int rank;
    __device__ __forceinline__ void operator()(int b, int off, cx<long long> v) const
    {
        s[pidx<FX>(b + off)] = fx_st(rank ? fx_rot<false>(v, twM[b + off]) : v);
    }
};
struct FxMultHalf {   // output k' of a half is frequency 2 k' + rank
    FxMultRow m;
    int rank;
    template <int R>
    __device__ __forceinline__ int2 at(int b, int t, int nb) const { return m(2 * (b + t * nb) + rank); }
};

template <int EMAX>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kSplitThreads, 2)
    k_fx_conv_split(fxc *__restrict__ W, const int2 *__restrict__ mult, const int *__restrict__ mrow_exp, FxExps ex,
                    int nlines, int ny1, Sched sc, Sched sci, const int4 *__restrict__ tw,
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
    const Group g = fx_thread().g;
    fxc *s = reinterpret_cast<fxc *>(smem_raw);
    fxc *w = W + (size_t)line * Mh;
    const bool active = line < nlines;   // every CTA of a cluster reaches both cluster barriers
    if (active) {
        FxLine ln{0, 0, Mh > kFxLongM, red};
        FxFromGlobalRot in;
        in.p = w;
        in.e = ex.xf + (line & 1) * ex.xf_par;
        in.twM = twM;
        in.rank = rank;
        const FxMultRow m{mult + (size_t)line * (full ? M : ny1), M, full};
        // the half's schedules always fuse (make_split_tables)
        ln.pad = sc.pad;
        fx_begin<true, EMAX, false>(s, sc, g, ln, in, FxNoOut{});
        fx_rest<true, EMAX, false>(s, sc, tw, g, ln, 1, sc.nst - 1, FxNoOut{});
        const FxMultHalf mh{m, rank};
        const int fr = sci.r[0], er = mrow_exp[line];
        if (fr == 8) fx_mid<8, (EMAX + 7) / 8>(s, sc, sci, tw, g, ln, mh, er);
        else if (fr == 4) fx_mid<4, (EMAX + 3) / 4>(s, sc, sci, tw, g, ln, mh, er);
        else if (fr == 2) fx_mid<2, (EMAX + 1) / 2>(s, sc, sci, tw, g, ln, mh, er);
        else if (fr == 5) fx_mid<5, (EMAX + 4) / 5>(s, sc, sci, tw, g, ln, mh, er);
        else fx_mid<3, (EMAX + 2) / 3>(s, sc, sci, tw, g, ln, mh, er);
        fx_rest<false, EMAX, false>(s, sci, twi, g, ln, 1, -1, FxHalfToSmem{s, twM, rank});
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
    __device__ __forceinline__ cx<long long> align(const raw &r, int em) const
    {
        const cx<long long> x = FxDoubles::align({r.a, r.b}, em);
        return rank ? fx_rot<true>(x, twM[r.i]) : x;
    }
};

template <int EMAX>
__global__ void __launch_bounds__(kSplitThreads, 2)
    k_fx_xf_split(const double *__restrict__ rho, fxc *__restrict__ W1, FxExps ex, int nx, int ny, Sched sc,
                  const int4 *__restrict__ tw, const int4 *__restrict__ twM)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int red[kFxRedWords];
    const int rank = blockIdx.x & 1, ya = 2 * (blockIdx.x >> 1);
    const int Mh = sc.M;   // == nx
    const Group g = fx_thread().g;
    fxc *s = reinterpret_cast<fxc *>(smem_raw);
    FxLine ln{0, 0, Mh > kFxLongM, red};
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

}  // namespace

cudaError_t fx_raise_conv_smem(const PassCfg &c)
{
    cudaError_t e = cudaSuccess;
    with_emax(c, [&](auto E) { e = raise_smem(k_fx_conv<E()>, c.smem); });
    return e;
}

cudaError_t fx_raise_split_smem(bool conv, size_t smem)
{
    return conv ? raise_smem(k_fx_conv_split<16>, smem) : raise_smem(k_fx_xf_split<16>, smem);
}

void fx_launch_conv(const FxCall &a, const PassCfg &c)
{
    const Plan *p = a.p;
    const int z = p->d - 1, ny = p->n[1], hx = p->n[0] + 1, My = p->d == 3 ? p->M[1] : 1;
    const int2 *mult = static_cast<const int2 *>(p->d_mult);
    const int4 *tw = static_cast<const int4 *>(p->d_tw[z]), *twi = static_cast<const int4 *>(p->d_twi[z]);
    fxc *W = static_cast<fxc *>(p->d == 3 ? a.W2 : a.W1);
    const dim3 g = p->d == 3 ? dim3((My + c.nl - 1) / c.nl, hx) : dim3((hx + c.nl - 1) / c.nl), b(c.gthr, c.nl);
    with_emax(c, [&](auto E) {
        k_fx_conv<E()><<<g, b, c.smem, a.st>>>(W, mult, p->d_mrow, a.ex, p->d == 3 ? hx * My : hx, p->n[z], p->d == 3,
                                               My, ny + 1, p->sched_f[z], p->sched_i[z], c.nl, tw, twi,
                                               p->mult_full ? 1 : 0);
    });
}

// The split conv (conv) or the split x forward pass of a 2D plan.
void fx_launch_split(const FxCall &a, bool conv)
{
    const Plan *p = a.p;
    const int nx = p->n[0], ny = p->n[1], hx = nx + 1;
    fxc *W1 = static_cast<fxc *>(a.W1);
    const int4 *twM = static_cast<const int4 *>(p->d_tw[conv ? 1 : 0]) + p->M[conv ? 1 : 0];   // the plain entries
    if (conv) {
        const PassCfg &c = p->cfg_split;
        k_fx_conv_split<16><<<2 * hx, c.nthr, c.smem, a.st>>>(
            W1, static_cast<const int2 *>(p->d_mult), p->d_mrow, a.ex, hx, ny + 1, p->sched_hf, p->sched_hi,
            static_cast<const int4 *>(p->d_twh), static_cast<const int4 *>(p->d_twhi), twM, p->mult_full ? 1 : 0);
    } else {
        const PassCfg &c = p->cfg_xsplit;
        k_fx_xf_split<16><<<2 * ((ny + 1) / 2), c.nthr, c.smem, a.st>>>(
            a.rho, W1, a.ex, nx, ny, p->sched_xh, static_cast<const int4 *>(p->d_twxh), twM);
    }
}

}  // namespace gsm
