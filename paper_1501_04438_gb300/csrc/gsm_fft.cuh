// gsm_fft.cuh -- batched line FFTs in shared memory (FP32), and what the
// fixed-point transforms (gsm_fx.cuh) share with them: schedules and groups.
//
// A CTA holds `nl` lines of length M in shared memory, line l at offset
// l * LS, element i at pidx(i) (one pad element every 2^kPadShift elements, so
// that the strided accesses of the early stages spread over the banks); the
// FFT of each line is done by its own group of threads (see Group).
// The transform is a Stockham autosort FFT (self-sorting, no bit reversal):
// for a stage of radix R after stages whose radices multiply to Ns,
// butterfly b (0 <= b < M/R) reads x[b + t M/R], t = 0..R-1, multiplies
// element t by w^(j t) with j = b mod Ns and w = exp(-+2 pi i / (Ns R)),
// applies the radix-R DFT in registers and writes the outputs to
// (b - j) R + j + t Ns.  Every thread first loads all its butterflies,
// the group synchronises, then every thread stores: stages run in place.
//
// Unnormalised: forward uses exp(-2 pi i jk/M), inverse exp(+2 pi i jk/M).
#pragma once

#include <type_traits>

#include "gsm_arith.cuh"

namespace gsm {

constexpr int kMaxStages = 12;

// Radix schedule of one FFT length: stage st has radix r[st] (8, 4, 2, 5 or 3,
// in any order whose product is M).
struct Sched {
    int M;
    int nst;
    unsigned char r[kMaxStages];
    int pad;   // fixed point: layout of the line in shared memory (set_pad)
};

// Layout of a fixed-point line (fx_pos in gsm_fx.cuh): one pad element per 8
// (3) when every stage's accesses then have constant strides, else none (31).
inline void set_pad(Sched *s)
{
    int Ns = 1;
    s->pad = 3;
    for (int st = 0; st < s->nst; ++st) {
        if (st > 0 && (s->M / s->r[st]) % 8 != 0) s->pad = 31;
        Ns *= s->r[st];
        if (st + 1 < s->nst && 8 % Ns != 0 && Ns % 8 != 0) s->pad = 31;
    }
}

template <class Pol>
__host__ __device__ __forceinline__ int pidx(int i) { return i + (i >> Pol::kPadShift); }

template <class Pol>
__host__ __device__ __forceinline__ int line_stride(int M) { return M + (M >> Pol::kPadShift) + 1; }

// math constants (exact decimal expansions, rounded by the compiler)
constexpr double kSqrtHalf = 0.707106781186547524400844362104849039;
constexpr double kSin60 = 0.866025403784438646763723170752936183;  // sqrt(3)/2
constexpr double kC5a = 0.309016994374947424102293417182819059;    // cos(2 pi/5)
constexpr double kC5b = -0.809016994374947424102293417182819059;   // cos(4 pi/5)
constexpr double kS5a = 0.951056516295153572116439333379382143;    // sin(2 pi/5)
constexpr double kS5b = 0.587785252292473129168705954639072769;    // sin(4 pi/5)

// ---------------------------------------------------------------- butterflies
// y_k = sum_t x_t exp(-+ 2 pi i t k / R), in place in v[0..R-1].

template <class R, bool FWD>
__device__ __forceinline__ void bfly2(cx<R> *v)
{
    cx<R> a = v[0];
    v[0] = cadd(a, v[1]);
    v[1] = csub(a, v[1]);
}

template <class R, bool FWD>
__device__ __forceinline__ cx<R> rot_quarter(cx<R> a)   // multiply by -i (fwd) / +i (inv)
{
    return FWD ? cmul_negi(a) : cmul_posi(a);
}

template <class R, bool FWD>
__device__ __forceinline__ void bfly4(cx<R> *v)
{
    cx<R> a0 = cadd(v[0], v[2]), a1 = csub(v[0], v[2]);
    cx<R> a2 = cadd(v[1], v[3]), a3 = rot_quarter<R, FWD>(csub(v[1], v[3]));
    v[0] = cadd(a0, a2);
    v[2] = csub(a0, a2);
    v[1] = cadd(a1, a3);
    v[3] = csub(a1, a3);
}

// Radix 8: the rotations by w8 and w8^3 are formed first.
template <class R, bool FWD>
__device__ __forceinline__ void bfly8(cx<R> *v)
{
    cx<R> a[4], b[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        a[t] = cadd(v[t], v[t + 4]);
        b[t] = csub(v[t], v[t + 4]);
    }
    {
        cx<R> z = b[1];
        if (FWD) b[1] = {rmulk(radd(z.re, z.im), kSqrtHalf), rmulk(rsub(z.im, z.re), kSqrtHalf)};
        else b[1] = {rmulk(rsub(z.re, z.im), kSqrtHalf), rmulk(radd(z.re, z.im), kSqrtHalf)};
    }
    b[2] = rot_quarter<R, FWD>(b[2]);
    {
        cx<R> z = b[3];
        if (FWD) b[3] = {rmulk(rsub(z.im, z.re), kSqrtHalf), rneg(rmulk(radd(z.re, z.im), kSqrtHalf))};
        else b[3] = {rneg(rmulk(radd(z.re, z.im), kSqrtHalf)), rmulk(rsub(z.re, z.im), kSqrtHalf)};
    }
    bfly4<R, FWD>(a);
    bfly4<R, FWD>(b);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        v[2 * k] = a[k];
        v[2 * k + 1] = b[k];
    }
}

// --- pruned butterflies -------------------------------------------------------
// Last stage of a transform of which only the outputs t < 4 are kept (the
// crop): a_t = x_t + x_{t+4} and b_t = x_t - x_{t+4}, of whose radix-4
// transforms the outputs 0 and 1 are formed, the 1/sqrt(2) of w8 and w8^3
// applied in the last additions.
template <class R, bool FWD>
__device__ __forceinline__ void bfly8_half_out(cx<R> *v)
{
    cx<R> a[4], b[4], u1, u3;
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        a[t] = cadd(v[t], v[t + 4]);
        b[t] = csub(v[t], v[t + 4]);
    }
    const cx<R> p = cadd(a[0], a[2]), q = csub(a[0], a[2]);
    const cx<R> s = cadd(a[1], a[3]), d = rot_quarter<R, FWD>(csub(a[1], a[3]));
    if (FWD) {   // sqrt2 w8 = 1 - i, sqrt2 w8^3 = -1 - i
        u1 = {radd(b[1].re, b[1].im), rsub(b[1].im, b[1].re)};
        u3 = {rsub(b[3].im, b[3].re), rneg(radd(b[3].re, b[3].im))};
    } else {     // conjugates
        u1 = {rsub(b[1].re, b[1].im), radd(b[1].re, b[1].im)};
        u3 = {rneg(radd(b[3].re, b[3].im)), rsub(b[3].re, b[3].im)};
    }
    const cx<R> b2 = rot_quarter<R, FWD>(b[2]);
    const cx<R> e = cadd(b[0], b2), f = csub(b[0], b2);
    const cx<R> g = cadd(u1, u3), h = rot_quarter<R, FWD>(csub(u1, u3));
    v[0] = cadd(p, s);
    v[1] = {radd(e.re, rmulk(g.re, kSqrtHalf)), radd(e.im, rmulk(g.im, kSqrtHalf))};
    v[2] = cadd(q, d);
    v[3] = {radd(f.re, rmulk(h.re, kSqrtHalf)), radd(f.im, rmulk(h.im, kSqrtHalf))};
}

// First stage whose inputs x_2, x_3 are zero (zero padding).
template <class R, bool FWD>
__device__ __forceinline__ void bfly4_half_in(cx<R> *v)
{
    const cx<R> x0 = v[0], x1 = v[1], r1 = rot_quarter<R, FWD>(v[1]);
    v[0] = cadd(x0, x1);
    v[1] = cadd(x0, r1);
    v[2] = csub(x0, x1);
    v[3] = csub(x0, r1);
}

template <class R, bool FWD>
__device__ __forceinline__ void bfly3(cx<R> *v)
{
    cx<R> s = cadd(v[1], v[2]);
    cx<R> d = csub(v[1], v[2]);
    cx<R> y0 = cadd(v[0], s);
    cx<R> m = csub(v[0], cmulk(s, 0.5));
    cx<R> r = rot_quarter<R, FWD>(cmulk(d, kSin60));   // -+ i (sqrt3/2)(x1 - x2)
    v[0] = y0;
    v[1] = cadd(m, r);
    v[2] = csub(m, r);
}

template <class R, bool FWD>
__device__ __forceinline__ void bfly5(cx<R> *v)
{
    cx<R> a1 = cadd(v[1], v[4]), b1 = csub(v[1], v[4]);
    cx<R> a2 = cadd(v[2], v[3]), b2 = csub(v[2], v[3]);
    cx<R> x0 = v[0];
    cx<R> p1 = cadd(x0, cadd(cmulk(a1, kC5a), cmulk(a2, kC5b)));
    cx<R> p2 = cadd(x0, cadd(cmulk(a1, kC5b), cmulk(a2, kC5a)));
    cx<R> q1 = rot_quarter<R, FWD>(cadd(cmulk(b1, kS5a), cmulk(b2, kS5b)));   // -+ i (s1 b1 + s2 b2)
    cx<R> q2 = rot_quarter<R, FWD>(csub(cmulk(b1, kS5b), cmulk(b2, kS5a)));   // -+ i (s2 b1 - s1 b2)
    v[0] = cadd(x0, cadd(a1, a2));
    v[1] = cadd(p1, q1);
    v[4] = csub(p1, q1);
    v[2] = cadd(p2, q2);
    v[3] = csub(p2, q2);
}

// HALF = 0: full radix-RAD DFT; 1: inputs t >= RAD/2 are zero (radix 4); 2:
// only the outputs t < RAD/2 are formed (radix 8).
template <class R, int RAD, bool FWD, int HALF>
__device__ __forceinline__ void bfly(cx<R> *v)
{
    static_assert(HALF == 0 || (HALF == 1 && RAD == 4) || (HALF == 2 && RAD == 8), "no such pruned butterfly");
    if constexpr (RAD == 2) {
        bfly2<R, FWD>(v);
    } else if constexpr (RAD == 3) {
        bfly3<R, FWD>(v);
    } else if constexpr (RAD == 4) {
        if constexpr (HALF == 1) bfly4_half_in<R, FWD>(v);
        else bfly4<R, FWD>(v);
    } else if constexpr (RAD == 5) {
        bfly5<R, FWD>(v);
    } else {
        if constexpr (HALF == 2) bfly8_half_out<R, FWD>(v);
        else bfly8<R, FWD>(v);
    }
}

// ---------------------------------------------------------------- groups
// The FFT of one line is done by a group of T threads (a multiple of 32).
// The group synchronises with __syncwarp (one warp), with __syncthreads
// (the group is the whole CTA) or with a named barrier of its own, so groups
// of one CTA never wait for each other between stages.
struct Group {
    int t;      // thread index in the group
    int T;      // threads in the group
    int bar;    // -1: one warp; 0: whole CTA; > 0: named barrier id
};

__device__ __forceinline__ void group_sync(const Group &g)
{
    if (g.bar < 0) __syncwarp();
    else if (g.bar == 0) __syncthreads();
    else asm volatile("bar.sync %0, %1;" ::"r"(g.bar), "r"(g.T) : "memory");
}

// Group of the calling thread when the CTA holds nl groups of T threads each.
__device__ __forceinline__ Group make_group(int T, int nl)
{
    Group g;
    g.t = threadIdx.x % T;
    g.T = T;
    g.bar = (T == 32) ? -1 : (nl == 1 ? 0 : 1 + (int)(threadIdx.x / T));
    return g;
}

// b mod Ns; the radix-8/4/2 stages come first, so Ns is usually a power of two
__device__ __forceinline__ int stage_mod(int b, int Ns)
{
    return (Ns & (Ns - 1)) == 0 ? (b & (Ns - 1)) : b % Ns;
}

// ---------------------------------------------------------------- one stage
// One Stockham stage on one line s[pidx(0..M-1)] by the group.  NB = upper
// bound of butterflies per thread (compile time); every thread first loads
// its butterflies, the group synchronises, then every thread stores.
template <class Pol, int RAD, bool FWD, int NB>
__device__ __forceinline__ void fft_stage(typename Pol::scplx *s, int M, int Ns,
                                          const typename Pol::tw_t *__restrict__ tw, const Group &g)
{
    using R = typename Pol::real;
    const int nb = M / RAD;
    const int step = M / (Ns * RAD);   // twiddle-table stride of this stage
    cx<R> v[NB][RAD];
#pragma unroll
    for (int i = 0; i < NB; ++i) {
        const int b = g.t + i * g.T;
        if (b < nb) {
#pragma unroll
            for (int t = 0; t < RAD; ++t) v[i][t] = Pol::ld(s[pidx<Pol>(b + t * nb)]);
            if (Ns > 1) {
                const int j = stage_mod(b, Ns);
#pragma unroll
                for (int t = 1; t < RAD; ++t) {
                    cx<R> w = Pol::tw(tw[j * t * step]);
                    v[i][t] = FWD ? cmul(v[i][t], w) : cmulc(v[i][t], w);
                }
            }
            bfly<R, RAD, FWD, 0>(v[i]);
        }
    }
    group_sync(g);
#pragma unroll
    for (int i = 0; i < NB; ++i) {
        const int b = g.t + i * g.T;
        if (b < nb) {
            const int j = stage_mod(b, Ns);
            const int d0 = (b - j) * RAD + j;
#pragma unroll
            for (int t = 0; t < RAD; ++t) s[pidx<Pol>(d0 + t * Ns)] = Pol::st(v[i][t]);
        }
    }
    group_sync(g);
}

// Rank of a radix in the order the stages of a schedule run in: 8, 4, 2, 5, 3.
__host__ __device__ __forceinline__ int radix_rank(int R)
{
    return R == 8 ? 0 : R == 4 ? 1 : R == 2 ? 2 : R == 5 ? 3 : R == 3 ? 4 : 99;
}

// Whether stages [from, nst) of sc are in the order 8, 4, 2, 5, 3 (radices of
// equal rank together), the only order fft_line runs.
__host__ __device__ inline bool sched_sorted_from(const Sched &sc, int from)
{
    for (int i = from; i < sc.nst; ++i) {
        if (radix_rank(sc.r[i]) > 4) return false;
        if (i > from && radix_rank(sc.r[i]) < radix_rank(sc.r[i - 1])) return false;
    }
    return true;
}

// All stages of the FFT of one line by one group.  EMAX bounds the elements
// per thread (M <= EMAX * T).  The caller synchronises the group (or CTA)
// after writing the line; the last stage ends with a group barrier, so the
// group may read the result right away.  The stages from st_begin on must be
// in the order 8, 4, 2, 5, 3 (sched_sorted_from, checked on the host): each
// radix gets one loop of its own, once (a loop mixing several large stage
// bodies, or one loop around these loops, costs the register allocator
// dearly).  Schedules that start
// with another radix (the inverse of a conv pass whose first stage is fused,
// fft_fused_mid) run from st_begin = 1.
// Stages [st_begin, st_end) run (st_end < 0: to the last).
template <class Pol, bool FWD, int EMAX>
__device__ __forceinline__ void fft_line(typename Pol::scplx *s, const Sched &sc,
                                         const typename Pol::tw_t *__restrict__ tw, const Group &g,
                                         int st_begin = 0, int st_end = -1)
{
    const int M = sc.M;
    const int nend = st_end < 0 ? sc.nst : st_end;
    int Ns = 1, st = st_begin;
    for (int i = 0; i < st_begin; ++i) Ns *= sc.r[i];
#define GSM_STAGE(RAD) fft_stage<Pol, RAD, FWD, (EMAX + RAD - 1) / RAD>(s, M, Ns, tw, g)
    for (; st < nend && sc.r[st] == 8; ++st, Ns *= 8) GSM_STAGE(8);
    for (; st < nend && sc.r[st] == 4; ++st, Ns *= 4) GSM_STAGE(4);
    for (; st < nend && sc.r[st] == 2; ++st, Ns *= 2) GSM_STAGE(2);
    for (; st < nend && sc.r[st] == 5; ++st, Ns *= 5) GSM_STAGE(5);
    for (; st < nend && sc.r[st] == 3; ++st, Ns *= 3) GSM_STAGE(3);
#undef GSM_STAGE
}

// The radix of the stage that fft_fused_mid can fuse for a transform whose
// forward schedule is scf and inverse schedule sci: the forward's last radix
// when the inverse starts with the same radix and both have at least two
// stages; 0 when they cannot be fused.
__host__ __device__ __forceinline__ int fused_radix(const Sched &scf, const Sched &sci)
{
    if (scf.nst < 2 || sci.nst < 2) return 0;
    const int R = scf.r[scf.nst - 1];
    return R == sci.r[0] ? R : 0;
}

// The last forward stage (radix R, schedule scf), a pointwise multiplication
// by mult(k) and the first inverse stage (radix R, schedule sci) of a line, in
// registers.  The forward stage's butterfly b (Ns = M/R = nb, so j = b and the
// twiddles are w_M^(b t)) leaves its outputs at the natural indices b + t M/R,
// which are exactly the inputs of the inverse's untwiddled butterfly b; that
// one writes to R b + t.  Saves two shared-memory round trips and a barrier
// over running the two transforms and the multiplication apart.  Follow with
// fft_line<Pol, false, ...>(..., sci, ..., st_begin = 1).
template <class Pol, int R, int NB, class MultF>
__device__ __forceinline__ void fft_fused_mid(typename Pol::scplx *s, const Sched &scf,
                                              const typename Pol::tw_t *__restrict__ tw, const Group &g, MultF mult)
{
    using Rl = typename Pol::real;
    const int M = scf.M, nb = M / R;
    cx<Rl> v[NB][R];
#pragma unroll
    for (int i = 0; i < NB; ++i) {
        const int b = g.t + i * g.T;
        if (b < nb) {
#pragma unroll
            for (int t = 0; t < R; ++t) v[i][t] = Pol::ld(s[pidx<Pol>(b + t * nb)]);
#pragma unroll
            for (int t = 1; t < R; ++t) v[i][t] = cmul(v[i][t], Pol::tw(tw[b * t]));   // twiddle step 1
            bfly<Rl, R, true, 0>(v[i]);
#pragma unroll
            for (int t = 0; t < R; ++t) v[i][t] = cscale(v[i][t], mult(b + t * nb));
            bfly<Rl, R, false, 0>(v[i]);
        }
    }
    group_sync(g);
#pragma unroll
    for (int i = 0; i < NB; ++i) {
        const int b = g.t + i * g.T;
        if (b < nb) {
#pragma unroll
            for (int t = 0; t < R; ++t) s[pidx<Pol>(R * b + t)] = Pol::st(v[i][t]);
        }
    }
    group_sync(g);
}

}  // namespace gsm
