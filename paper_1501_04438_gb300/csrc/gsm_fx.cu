// gsm_fx.cu -- fixed point: the x and y passes, the FFT hook and the tables.
#include "gsm_fx_kernels.cuh"

namespace gsm {
namespace {

// ------------------------------------------------------------------ FFT test hook
struct FxFromPairs : FxDoubles {
    const double2 *p;
    __device__ __forceinline__ raw load(int b, int off) const { return {p[b + off].x, p[b + off].y}; }
};
struct FxToPairs {
    static constexpr bool kSmem = false;
    double2 *p;
    const FxLine *ln;
    __device__ __forceinline__ void operator()(int b, int off, cx<long long> v) const
    {
        p[b + off] = make_double2(fx_out_double(v.re, ln->E), fx_out_double(v.im, ln->E));
    }
};

template <bool FWD, int EMAX>
__global__ void __launch_bounds__(fx_threads(EMAX), fx_ctas(EMAX))
    k_fx_hook(const double2 *__restrict__ in, double2 *__restrict__ out, int nlines, Sched sc, int nl,
              const int4 *__restrict__ tw)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int red[kFxRedWords];
    const int M = sc.M;
    const FxThread th = fx_thread();
    const Group &g = th.g;
    const int l = th.l;
    fxc *s = reinterpret_cast<fxc *>(smem_raw) + l * line_stride<FX>(M);
    const int line = blockIdx.x * nl + l;
    if (line >= nlines) return;
    FxLine ln{0, 0, M > kFxLongM, red, 0};
    FxFromPairs src;
    src.p = in + (size_t)line * M;
    fx_transform<FWD, EMAX, false, false>(s, sc, tw, g, ln, src, FxToPairs{out + (size_t)line * M, &ln});
}

// ------------------------------------------------------------------ tables
// Double-double arithmetic (T. J. Dekker 1971; Hida, Li and Bailey 2001) for
// the twiddles, whose 62 bits a double does not hold.
struct dd {
    double h, l;
};
__device__ __forceinline__ dd dd_norm(double a, double b)
{
    const double s = a + b;
    return {s, b - (s - a)};
}
__device__ __forceinline__ dd dd_add(dd a, dd b)
{
    const double s = a.h + b.h, t = s - a.h;
    const double e = (a.h - (s - t)) + (b.h - t);
    return dd_norm(s, e + a.l + b.l);
}
__device__ __forceinline__ dd dd_mul(dd a, dd b)
{
    const double p = a.h * b.h;
    return dd_norm(p, fma(a.h, b.h, -p) + (a.h * b.l + a.l * b.h));
}
__device__ __forceinline__ dd dd_div(dd a, double b)
{
    const double q = a.h / b;
    return dd_norm(q, (fma(-q, b, a.h) + a.l) / b);
}
// cos and sin of 2 pi q / D by their power series on |x| <= pi/4, x = 2 pi q/D
// less the nearest quarter turn (exact in integers)
__device__ void dd_sincos(long q, long D, dd *c, dd *s)
{
    q %= D;
    const long k = (4 * q + D / 2) / D;   // nearest quarter turn
    const long m = 4 * q - k * D;         // x = (pi/2) m / D
    dd x = dd_div(dd{(double)m, 0.0}, (double)D);
    x = dd_mul(x, dd{1.5707963267948966, 6.123233995736766e-17});
    const dd x2 = dd_mul(x, x);
    dd tc{1.0, 0.0}, ts = x, sc = tc, ss = ts;
    for (int i = 1; i <= 14; ++i) {
        tc = dd_div(dd_mul(tc, x2), -(double)((2 * i - 1) * (2 * i)));
        ts = dd_div(dd_mul(ts, x2), -(double)((2 * i) * (2 * i + 1)));
        sc = dd_add(sc, tc);
        ss = dd_add(ss, ts);
    }
    const dd nc{-sc.h, -sc.l}, ns{-ss.h, -ss.l};
    switch ((int)(k & 3)) {
    case 0: *c = sc; *s = ss; break;
    case 1: *c = ns; *s = sc; break;
    case 2: *c = nc; *s = ns; break;
    default: *c = ss; *s = nc; break;
    }
}

__device__ __forceinline__ int4 fx_twiddle(long q, long D)   // exp(-2 pi i q / D)
{
    dd c, s;
    dd_sincos(q, D, &c, &s);
    const int2 a = fx_factor(c.h, c.l), b = fx_factor(s.h, s.l);
    return make_int4(a.x, a.y, b.x, b.y);
}

// Table of a schedule: the stages' twiddles (fx_stage_table), M entries of
// which the last r0 are unused, then `plain` entries w_M2^m with M2 = plain_m.
__global__ void k_fx_twiddles(Sched sc, int plain, int plain_m, int4 *out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < plain) out[sc.M + i] = fx_twiddle(i, plain_m);
    int j = i, Ns = sc.r[0];
    if (i >= sc.M - Ns) return;
    for (int st = 1; st < sc.nst; ++st) {
        const int R = sc.r[st], cnt = (R - 1) * Ns;
        if (j < cnt) {
            const int t = j / Ns + 1, b = j % Ns;
            out[i] = fx_twiddle((long)b * t, (long)R * Ns);
            return;
        }
        j -= cnt;
        Ns *= R;
    }
}
// Multiplier rows of `len` doubles to factors of 2^e, e the row's exponent
// (every |entry| <= 2^e), in place or not; one CTA per row.
__global__ void __launch_bounds__(128) k_fx_mult_rows(const double *in, int2 *out, int len, int *row_exp)
{
    __shared__ double red[4];
    const double *r = in + (size_t)blockIdx.x * len;
    double m = 0.0;
    for (int i = threadIdx.x; i < len; i += blockDim.x) m = fmax(m, fabs(r[i]));
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
    __syncthreads();
    m = fmax(fmax(red[0], red[1]), fmax(red[2], red[3]));
    // m < 2^e; a row of zeros takes no part in the exponents of the lines that cross it
    int e = kFxZero;
    if (m > 0.0) frexp(m, &e);
    if (threadIdx.x == 0) row_exp[blockIdx.x] = e;
    for (int i = threadIdx.x; i < len; i += blockDim.x)
        out[(size_t)blockIdx.x * len + i] = m > 0.0 ? fx_mult_factor(ldexp(r[i], -e)) : make_int2(0, 0);
}

// thread x of a line's group, line y of the CTA
dim3 fx_block(const PassCfg &c) { return dim3(c.gthr, c.nl); }

}  // namespace

size_t fx_table_bytes(int M, int plain) { return sizeof(int4) * ((size_t)M + plain); }

void launch_fx_twiddles(const Sched &sc, int plain, int plain_m, void *out, cudaStream_t st)
{
    const int n = std::max(sc.M, plain);
    k_fx_twiddles<<<(n + 127) / 128, 128, 0, st>>>(sc, plain, plain_m, static_cast<int4 *>(out));
}

gsm_status_t make_mult_rows(Plan *p, void *table, int len, size_t rows, cudaStream_t st)
{
    p->d_mrow = reinterpret_cast<int *>(static_cast<double *>(table) + rows * len);
    k_fx_mult_rows<<<(unsigned)rows, 128, 0, st>>>(static_cast<const double *>(table), static_cast<int2 *>(table), len,
                                                   p->d_mrow);
    GSM_CUDA_TRY(cudaGetLastError());
    return GSM_OK;
}

cudaError_t fx_raise_smem(const Plan *p, int pass, const PassCfg &c)
{
    const int last = p->d == 3 ? 4 : 2;
    if (pass == (p->d == 3 ? 2 : 1)) return fx_raise_conv_smem(p, c);
    cudaError_t e = fixed_raise(p, pass, c);
    if (e != cudaSuccess) return e;
    with_emax(c, [&](auto E) {
        if (pass == 0) e = raise_smem(k_fx_xf<E(), Sched>, c.smem);
        else if (pass == last) e = raise_smem(k_fx_xi<E(), Sched>, c.smem);
        else if (pass == 1) e = raise_smem(k_fx_yf<E(), Sched>, c.smem);
        else e = raise_smem(k_fx_yi<E(), Sched>, c.smem);
    });
    return e;
}

// x forward (pass 0), y forward (1), y inverse (3), x inverse (the last)
void fx_launch_xy(const FxCall &a, int pass, const PassCfg &c)
{
    if (fixed_launch(a, pass, c)) return;
    const Plan *p = a.p;
    const int nx = p->n[0], ny = p->n[1], nz = a.nz, hx = nx + 1, last = p->d == 3 ? 4 : 2;
    fxc *W1 = static_cast<fxc *>(a.W1), *W2 = static_cast<fxc *>(a.W2);
    const auto tw = [&](int axis) { return static_cast<const int4 *>(p->d_tw[axis]); };
    const auto twi = [&](int axis) { return static_cast<const int4 *>(p->d_twi[axis]); };
    const dim3 gx((ny + 2 * c.nl - 1) / (2 * c.nl), nz), gy((nz + c.nl - 1) / c.nl, hx), b = fx_block(c);
    with_emax(c, [&](auto E) {
        if (pass == 0)
            k_fx_xf<E(), Sched><<<gx, b, c.smem, a.st>>>(a.rho, W1, a.ex, nx, ny, hx, p->sched_f[0], c.nl, tw(0));
        else if (pass == last)
            k_fx_xi<E(), Sched><<<gx, b, c.smem, a.st>>>(W1, a.u, p->d == 3 ? a.ex.yi : a.ex.cv, hx, nx, ny, hx,
                                                         p->sched_i[0], c.nl, twi(0));
        else if (pass == 1)
            k_fx_yf<E(), Sched><<<gy, b, c.smem, a.st>>>(W1, W2, a.ex, ny, nz, hx, p->sched_f[1], c.nl, tw(1));
        else
            k_fx_yi<E(), Sched><<<gy, b, c.smem, a.st>>>(W2, W1, a.ex, ny, nz, hx, p->sched_i[1], c.nl, twi(1));
    });
}

cudaError_t fx_launch_hook(const PassCfg &c, int nlines, int sign, const Sched &sc, const double *in, double *out,
                           const void *tw, cudaStream_t st)
{
    cudaError_t e = cudaSuccess;
    with_emax(c, [&](auto E) {
        auto kernel = sign < 0 ? k_fx_hook<true, E()> : k_fx_hook<false, E()>;
        e = raise_smem(kernel, c.smem);
        if (e == cudaSuccess)
            kernel<<<(nlines + c.nl - 1) / c.nl, fx_block(c), c.smem, st>>>(
                reinterpret_cast<const double2 *>(in), reinterpret_cast<double2 *>(out), nlines, sc, c.nl,
                static_cast<const int4 *>(tw));
    });
    return e;
}

}  // namespace gsm
