// gsm_fx.cuh -- line FFTs in block fixed point, the arithmetic of the FP64 and
// FP32X2 passes.
//
// GB300 executes 2 FP64 operations per SM and clock against 128 32-bit integer
// additions and 32 32 x 32 -> 64-bit multiply-adds, so an FFT of doubles is
// bound by its FP64 pipe alone (95 % busy, everything else idle).  Here a line
// is a block of 64-bit integers with one common exponent:
//   value = (re + i im) 2^E,   re, im: signed 64-bit, E one per line.
// A complex addition is two 64-bit integer additions (4 instructions), a
// rotation 12 multiply-adds on 32-bit halves and two 64-bit shifts.  Measured per
// warp and SM sub-partition (2.0 GHz): a 64-bit addition 2.4 cycles, a 32 x 32 + 64
// multiply-add 4, a DFMA 64.  FP64 apply at 256^3: 8.88 ms in FP64 arithmetic,
// 1.80 ms here (1.67 ms before the products and shifts were rounded without bias
// and the multiplier had exponents of its own, see below).
//
// Accuracy.  A line is scaled when it is loaded, and again after the
// multiplication, so that the sum of |re| + |im| over the line is below 2^62 (2^61
// if outputs are added in pairs after it): every value of every stage is a
// partial sum of the inputs with factors of modulus one, so nothing overflows
// and the full range is used, with an absolute rounding of half a unit or so per
// product, 2^-62 of that sum, where FP64 rounds every operation to 2^-53 of
// its result.  Lines longer than kFxLongM, whose sum is far above their
// values, are rescaled from their actual maximum after every stage instead
// (block floating point).  Roundings have no preferred side: a bias of half a unit
// per value adds up to M/2 units in one output, and where that is frequency zero
// the multiplier makes it the result's error.  Multiplied lines (forward, 1/k^2,
// inverse) against long double, maximum norm, here and with a plain FFT in doubles:
// smooth 1.1e-16 / 2.6e-16 (n = 256), 1.1e-16 / 3.3e-16 (n = 2048); a point 9e-17 /
// 2.7e-16, 1.8e-16 / 2.7e-16; white noise 2.2e-16 / 5.6e-16, 2.1e-16 / 5.9e-16;
// Gaussian times a wave at 0.9 of Nyquist 2.6e-14 / 7.6e-14, 1.8e-13 / 1.7e-12.  A
// host test holds such lines to the error of doubles.
//
// The functions here compile for the host too (one thread per line), which is
// what those comparisons run.
#pragma once

#include <limits.h>
#include <math.h>
#include <string.h>

#include "gsm_fft.cuh"

namespace gsm {

#define GSM_HD __host__ __device__ __forceinline__

// ---------------------------------------------------------------- policy
struct alignas(16) fxc {
    long long re, im;
};
struct FX {
    using real = long long;
    using scplx = fxc;      // complex as stored in shared and global memory
    using tw_t = int4;      // exp(-i t): (cos high, cos low, sin high, sin low), see fx_mul
    using mult_t = int2;    // multiplier entry (high, low), in units of its row's 2^exponent
    using io_t = double;
    static constexpr int kId = 2;
    static constexpr int kPadShift = 3;   // one pad element per 8 (128 bytes), see fx_pos
};

// Line exponents: beyond +-kFxBig they mark a line whose input held an
// infinity or a NaN (its outputs are NaN) and a line that is not there (zeros).
constexpr int kFxNan = 1 << 28, kFxZero = -(1 << 28), kFxBig = 1 << 27;
constexpr int kFxTop = 62;         // bound of a line's sum, as a power of two (FxLine::paired: one less)
constexpr int kFxLongM = 512;      // lines longer than this are rescaled after every stage

// ---------------------------------------------------------------- arithmetic
GSM_HD long long radd(long long a, long long b) { return (long long)((unsigned long long)a + (unsigned long long)b); }
GSM_HD long long rsub(long long a, long long b) { return (long long)((unsigned long long)a - (unsigned long long)b); }
GSM_HD long long rneg(long long a) { return rsub(0, a); }

// x = h 2^32 + l with -2^31 <= l < 2^31: l is x's low word, so that the part of
// a product that is dropped below has no preferred sign
struct fxh {
    int h, l;
};
GSM_HD fxh fx_split(long long x) { return {(int)(x >> 32) + (int)((unsigned)x >> 31), (int)x}; }

// A factor c, |c| <= 1, is (h, l) with c = h 2^-30 + l 2^-62, |l| < 2^31, so that
// 1 is exact.  x c = 4 hx hc + (hx lc + lx hc) 2^-30 + lx lc 2^-62; the cross
// terms are rounded (kFxHalf), the last term, one unit at most, is dropped.  A
// factor of 1, -1, i or -i is exact, and no product leans to one side: a bias of
// half a unit per product would add up in the output of frequency zero of what
// follows, where the multiplier is largest.
constexpr long long kFxHalf = 1ll << 29;
// a b + c, one instruction (spelled out: the compiler would widen a factor that
// it knows not to be negative unsigned, which makes the product a 64 x 64-bit one)
GSM_HD long long fx_mad(int a, int b, long long c)
{
#ifdef __CUDA_ARCH__
    long long r;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
#else
    return (long long)a * b + c;
#endif
}
GSM_HD long long fx_join(long long acc, long long mid) { return radd((long long)((unsigned long long)acc << 2), mid >> 30); }
GSM_HD long long fx_mul(fxh x, int ch, int cl)
{
    return fx_join(fx_mad(x.h, ch, 0), fx_mad(x.l, ch, fx_mad(x.h, cl, kFxHalf)));
}
// a constant given as round(c 2^62)
template <long long K62>
GSM_HD long long fx_mulc(long long x)
{
    constexpr int h = (int)((K62 + (1ll << 31)) >> 32);
    constexpr int l = (int)(K62 - h * (1ll << 32));
    return fx_mul(fx_split(x), h, l);
}

// A table entry, loaded by one instruction: of the plain loads of the radix-3 stage
// after 48 of padded length 432, unrolled, nvcc 13.0 took the low halves of the
// factors t = 1 from the entries t = 2 (results 1e-10 off), with every other
// stage and length as written.
GSM_HD int4 fx_tw(const int4 *p)
{
#ifdef __CUDA_ARCH__
    int4 w;
    asm("ld.global.nc.v4.s32 {%0, %1, %2, %3}, [%4];" : "=r"(w.x), "=r"(w.y), "=r"(w.z), "=r"(w.w) : "l"(p));
    return w;
#else
    return *p;
#endif
}

// x exp(-i t) (FWD) or x exp(+i t)
template <bool FWD>
GSM_HD cx<long long> fx_rot(cx<long long> x, int4 w)
{
    const fxh a = fx_split(x.re), b = fx_split(x.im);
    const int sh = FWD ? w.z : -w.z, sl = FWD ? w.w : -w.w, nh = -sh, nl = -sl;
    const long long re = fx_mad(b.h, sh, fx_mad(a.h, w.x, 0)), im = fx_mad(a.h, nh, fx_mad(b.h, w.x, 0));
    const long long mr = fx_mad(b.l, sh, fx_mad(b.h, sl, fx_mad(a.l, w.x, fx_mad(a.h, w.y, kFxHalf))));
    const long long mi = fx_mad(a.l, nh, fx_mad(a.h, nl, fx_mad(b.l, w.x, fx_mad(b.h, w.y, kFxHalf))));
    return {fx_join(re, mr), fx_join(im, mi)};
}

GSM_HD cx<long long> fx_add(cx<long long> a, cx<long long> b) { return {radd(a.re, b.re), radd(a.im, b.im)}; }
GSM_HD cx<long long> fx_sub(cx<long long> a, cx<long long> b) { return {rsub(a.re, b.re), rsub(a.im, b.im)}; }
// a + (-+ i) b and a - (-+ i) b without forming the negation
template <bool FWD>
GSM_HD cx<long long> fx_addq(cx<long long> a, cx<long long> b)
{
    return FWD ? cx<long long>{radd(a.re, b.im), rsub(a.im, b.re)} : cx<long long>{rsub(a.re, b.im), radd(a.im, b.re)};
}
template <bool FWD>
GSM_HD cx<long long> fx_subq(cx<long long> a, cx<long long> b) { return fx_addq<!FWD>(a, b); }

GSM_HD cx<long long> fx_ld(const fxc &v) { return {v.re, v.im}; }
GSM_HD fxc fx_st(cx<long long> a) { return {a.re, a.im}; }

// x 2^-s, 0 < s <= 62, rounded to nearest, ties to even (a preferred side would
// add up like the products' above)
GSM_HD long long fx_shift(long long x, int s)
{
    return (x + ((1ll << (s - 1)) - 1) + ((unsigned)(x >> s) & 1u)) >> s;
}
GSM_HD cx<long long> fx_shift(cx<long long> a, int s) { return {fx_shift(a.re, s), fx_shift(a.im, s)}; }
// x 2^-s for either sign of s, |s| <= 62 (x 2^-s must fit)
GSM_HD long long fx_scale2(long long x, int s) { return s > 0 ? fx_shift(x, s) : (long long)((unsigned long long)x << -s); }
GSM_HD cx<long long> fx_scale2(cx<long long> a, int s) { return {fx_scale2(a.re, s), fx_scale2(a.im, s)}; }

GSM_HD unsigned fx_abs_high(long long x)
{
    const int h = (int)(x >> 32);
    return (unsigned)(h < 0 ? -h : h);
}
GSM_HD int fx_bits(unsigned v)   // v < 2^fx_bits(v)
{
#ifdef __CUDA_ARCH__
    return 32 - __clz((int)v);
#else
    return v ? 32 - __builtin_clz(v) : 0;
#endif
}

// ---------------------------------------------------------------- butterflies
// constants as round(c 2^62)
constexpr long long kFxSqrtHalf = 3260954456333195553ll;    // sqrt(1/2)
constexpr long long kFxSin60 = 3993837246235628775ll;       // sqrt(3)/2
constexpr long long kFxSqrt5Quarter = 2578010857022246787ll;   // sqrt(5)/4
constexpr long long kFxS1 = 4385974038932618941ll;          // sin(2 pi/5)
constexpr long long kFxS1mS2 = 1675293009097605857ll;       // sin(2 pi/5) - sin(4 pi/5)
constexpr long long kFxS1pS2m1 = 2484969050340244120ll;     // sin(2 pi/5) + sin(4 pi/5) - 1

template <long long K62>
GSM_HD cx<long long> fx_scale(cx<long long> a) { return {fx_mulc<K62>(a.re), fx_mulc<K62>(a.im)}; }

// Radix RAD, HALF = 0: full; 1: the inputs t >= RAD/2 are zero; 2: only the
// outputs t < RAD/2 are formed (even RAD only).
// TURN: v[2] still has its quarter turn before it.
template <bool FWD, int HALF, bool TURN = false>
GSM_HD void fx_bfly4(cx<long long> *v)
{
    if (HALF == 1) {
        const cx<long long> a = v[0], b = v[1];
        v[0] = fx_add(a, b);
        v[1] = fx_addq<FWD>(a, b);
        v[2] = fx_sub(a, b);
        v[3] = fx_subq<FWD>(a, b);
        return;
    }
    const cx<long long> a0 = TURN ? fx_addq<FWD>(v[0], v[2]) : fx_add(v[0], v[2]);
    const cx<long long> a1 = TURN ? fx_subq<FWD>(v[0], v[2]) : fx_sub(v[0], v[2]);
    const cx<long long> a2 = fx_add(v[1], v[3]), a3 = fx_sub(v[1], v[3]);
    v[0] = fx_add(a0, a2);
    v[1] = fx_addq<FWD>(a1, a3);
    if (HALF == 2) return;
    v[2] = fx_sub(a0, a2);
    v[3] = fx_subq<FWD>(a1, a3);
}

template <bool FWD, int HALF>
GSM_HD void fx_bfly8(cx<long long> *v)
{
    cx<long long> a[4], b[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        a[t] = HALF == 1 ? v[t] : fx_add(v[t], v[t + 4]);
        b[t] = HALF == 1 ? v[t] : fx_sub(v[t], v[t + 4]);
    }
    // b1 w8, b2 w8^2, b3 w8^3
    {
        const cx<long long> z = b[1];
        const long long p = radd(z.re, z.im), q = rsub(z.im, z.re);
        b[1] = FWD ? cx<long long>{fx_mulc<kFxSqrtHalf>(p), fx_mulc<kFxSqrtHalf>(q)}
                   : cx<long long>{fx_mulc<-kFxSqrtHalf>(q), fx_mulc<kFxSqrtHalf>(p)};
    }
    {
        const cx<long long> z = b[3];
        const long long p = radd(z.re, z.im), q = rsub(z.im, z.re);
        b[3] = FWD ? cx<long long>{fx_mulc<kFxSqrtHalf>(q), fx_mulc<-kFxSqrtHalf>(p)}
                   : cx<long long>{fx_mulc<-kFxSqrtHalf>(p), fx_mulc<-kFxSqrtHalf>(q)};
    }
    constexpr int H4 = HALF == 2 ? 2 : 0;
    fx_bfly4<FWD, H4>(a);
    fx_bfly4<FWD, H4, true>(b);
#pragma unroll
    for (int k = 0; k < (HALF == 2 ? 2 : 4); ++k) {
        v[2 * k] = a[k];
        v[2 * k + 1] = b[k];
    }
}

template <bool FWD>
GSM_HD void fx_bfly3(cx<long long> *v)
{
    const cx<long long> s = fx_add(v[1], v[2]);
    const cx<long long> r = fx_scale<kFxSin60>(fx_sub(v[1], v[2]));
    const cx<long long> m = fx_sub(v[0], fx_shift(s, 1));
    v[0] = fx_add(v[0], s);
    v[1] = fx_addq<FWD>(m, r);
    v[2] = fx_subq<FWD>(m, r);
}

// cos(2 pi/5) = (-1 + sqrt 5)/4, cos(4 pi/5) = (-1 - sqrt 5)/4, and the sine
// terms s1 b1 + s2 b2 = s1 (b1 + b2) - (s1 - s2) b2, s2 b1 - s1 b2 =
// (s1 + s2) b1 - s1 (b1 + b2): four products per component (S. Winograd, Math.
// Comp. 32 (1978)).
template <bool FWD>
GSM_HD void fx_bfly5(cx<long long> *v)
{
    const cx<long long> a1 = fx_add(v[1], v[4]), b1 = fx_sub(v[1], v[4]);
    const cx<long long> a2 = fx_add(v[2], v[3]), b2 = fx_sub(v[2], v[3]);
    const cx<long long> t = fx_add(a1, a2), d = fx_scale<kFxSqrt5Quarter>(fx_sub(a1, a2));
    const cx<long long> m = fx_sub(v[0], fx_shift(t, 2));
    const cx<long long> p1 = fx_add(m, d), p2 = fx_sub(m, d);
    const cx<long long> u = fx_scale<kFxS1>(fx_add(b1, b2));
    const cx<long long> q1 = fx_sub(u, fx_scale<kFxS1mS2>(b2));
    const cx<long long> q2 = fx_sub(fx_add(b1, fx_scale<kFxS1pS2m1>(b1)), u);
    v[0] = fx_add(v[0], t);
    v[1] = fx_addq<FWD>(p1, q1);
    v[4] = fx_subq<FWD>(p1, q1);
    v[2] = fx_addq<FWD>(p2, q2);
    v[3] = fx_subq<FWD>(p2, q2);
}

// Radix 6 = 2 x 3 without twiddles (prime factors: I. J. Good 1958): inputs
// 3 n1 + 2 n2, outputs 3 k1 + 4 k2 mod 6.
template <bool FWD>
GSM_HD void fx_bfly6(cx<long long> *v)
{
    cx<long long> a[3], b[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        a[i] = fx_add(v[2 * i], v[(2 * i + 3) % 6]);
        b[i] = fx_sub(v[2 * i], v[(2 * i + 3) % 6]);
    }
    fx_bfly3<FWD>(a);
    fx_bfly3<FWD>(b);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        v[4 * k % 6] = a[k];
        v[(3 + 4 * k) % 6] = b[k];
    }
}

template <int RAD, bool FWD, int HALF>
GSM_HD void fx_bfly(cx<long long> *v)
{
    if constexpr (RAD == 6) {
        fx_bfly6<FWD>(v);
    } else if constexpr (RAD == 8) {
        fx_bfly8<FWD, HALF>(v);
    } else if constexpr (RAD == 4) {
        fx_bfly4<FWD, HALF>(v);
    } else if constexpr (RAD == 2) {
        const cx<long long> a = v[0];
        if (HALF == 1) {
            v[1] = a;
        } else {
            v[0] = fx_add(a, v[1]);
            if (HALF == 0) v[1] = fx_sub(a, v[1]);
        }
    } else if constexpr (RAD == 5) {
        fx_bfly5<FWD>(v);
    } else {
        fx_bfly3<FWD>(v);
    }
}

// ---------------------------------------------------------------- group reductions
GSM_HD void fx_sync(const Group &g)
{
#ifdef __CUDA_ARCH__
    group_sync(g);
#else
    (void)g;
#endif
}

// Maximum (MAX) or sum over the group.  buf: one word per warp of the CTA; a
// group of several warps passes one barrier, after which every thread reads
// the group's words; the next call must use another buffer or come after a
// further barrier of the group.
template <bool MAX>
GSM_HD int fx_reduce(int v, const Group &g, int *buf)
{
#ifdef __CUDA_ARCH__
    v = MAX ? __reduce_max_sync(0xffffffffu, v) : (int)__reduce_add_sync(0xffffffffu, (unsigned)v);
    if (g.bar < 0) return v;
    // groups of several warps: a CTA of T x nl threads, one row each
    const int nw = g.T >> 5, w0 = threadIdx.y * nw;
    if ((g.t & 31) == 0) buf[w0 + (g.t >> 5)] = v;
    group_sync(g);
    if (nw > 4) {   // one load and one more warp reduction
        const int lane = g.t & 31;
        v = lane < nw ? buf[w0 + lane] : MAX ? INT_MIN : 0;
        return MAX ? __reduce_max_sync(0xffffffffu, v) : (int)__reduce_add_sync(0xffffffffu, (unsigned)v);
    }
    v = buf[w0];
    for (int i = 1; i < nw; ++i) v = MAX ? max(v, buf[w0 + i]) : (int)((unsigned)v + (unsigned)buf[w0 + i]);
    return v;
#else
    (void)g;
    (void)buf;
    return v;
#endif
}

// What a transform keeps of its line: the exponent and the mode.
struct FxLine {
    int E;        // value = integer 2^E
    int pad;      // layout in shared memory (fx_pos)
    bool longm;   // rescale after every stage
    int *red;     // two buffers of one word per warp of the CTA
    int paired;   // 1: sums and differences of two outputs are formed from them
};
constexpr int kFxRedWarps = 16;
constexpr int kFxRedWords = 2 * kFxRedWarps;

// Bound (as a power of two) of re and im before a stage of a long line that adds
// `terms` values: its outputs, terms sqrt(2) times that at most, stay below 2^63
// or, out > 0 (1 + FxLine::paired), those of a line's last stage below 2^(63 - out).
// So every value in the workspace, pairs included, is below 2^62 (see FxInts).
GSM_HD constexpr int fx_bound(int terms, int out) { return (terms > 5 ? 59 : terms > 2 ? 60 : 61) - out; }

// The shift that brings a line into range, from the group's sum of
// (|high word| >> 12) + 1 over re and im (kFxTop), or from its maximum high
// word (long lines: 2^bound); the same for every thread of the group.
// fx_weight: one value's part of that sum or maximum.
GSM_HD unsigned fx_weight(cx<long long> x, bool longm)
{
    const unsigned a = fx_abs_high(x.re), b = fx_abs_high(x.im);
    return longm ? (a > b ? a : b) : (a >> 12) + (b >> 12) + 2u;
}
GSM_HD unsigned fx_weigh(unsigned acc, unsigned w, bool longm) { return longm ? (acc > w ? acc : w) : acc + w; }
GSM_HD int fx_shift_of(unsigned acc, const FxLine &ln, const Group &g, int *buf, int bound)
{
    // sum: below acc 2^44, so acc - 1 < 2^b gives sum <= 2^(44 + b); maximum: high word + 1
    int s;
    if (ln.longm) s = fx_bits((unsigned)fx_reduce<true>((int)acc, g, buf)) - (bound - 32);
    else s = fx_bits((unsigned)fx_reduce<false>((int)acc, g, buf)) - (kFxTop - ln.paired - 44);
    return s > 0 ? s : 0;
}

// ---------------------------------------------------------------- schedules
// A schedule known at compile time: the default order of make_sched (INV: the
// fused inverse, the last radix first).  The functions below take it in the
// place of a Sched; strides, tests, barriers' counts and loops are then
// constants.
template <int M_, bool INV = false>
struct FixedSched {
    struct List {
        int n, r[kMaxStages];
    };
    static constexpr List list()
    {
        List l{};
        int m = M_;
        const int order[5] = {8, 4, 2, 5, 3};
        for (int k = 0; k < 5; ++k)
            for (; m % order[k] == 0; m /= order[k]) l.r[l.n++] = order[k];
        if (INV) {
            const int last = l.r[l.n - 1];
            for (int i = l.n - 1; i > 0; --i) l.r[i] = l.r[i - 1];
            l.r[0] = last;
        }
        return l;
    }
    static constexpr int padding()   // set_pad
    {
        const List l = list();
        int Ns = 1, pad = 3;
        for (int st = 0; st < l.n; ++st) {
            if (st > 0 && (M_ / l.r[st]) % 8 != 0) pad = 31;
            Ns *= l.r[st];
            if (st + 1 < l.n && 8 % Ns != 0 && Ns % 8 != 0) pad = 31;
        }
        return pad;
    }
    static constexpr int M = M_, nst = list().n, pad = padding();
    template <int ST>
    static constexpr int radix() { return list().r[ST]; }
    static constexpr int product(int st)   // of the radices before stage st
    {
        const List l = list();
        int Ns = 1;
        for (int i = 0; i < st; ++i) Ns *= l.r[i];
        return Ns;
    }
    static bool is(const Sched &s)
    {
        const List l = list();
        if (s.M != M || s.nst != nst || s.pad != pad) return false;
        for (int i = 0; i < nst; ++i)
            if (s.r[i] != l.r[i]) return false;
        return true;
    }
};
template <class SC>
struct is_fixed_sched {
    static constexpr bool value = true;
};
template <>
struct is_fixed_sched<Sched> {
    static constexpr bool value = false;
};
template <class SC>
GSM_HD int first_radix(const SC &sc)
{
    if constexpr (is_fixed_sched<SC>::value) return SC::template radix<0>();
    else return sc.r[0];
}
// bound of a long line before stage ST (Sched: st); out: see fx_bound, should it be the last
template <int ST, class SC>
GSM_HD int fx_bound_before(const SC &sc, int st, int out)
{
    if constexpr (is_fixed_sched<SC>::value) return fx_bound(SC::template radix<(ST < SC::nst ? ST : 0)>(), ST == SC::nst - 1 ? out : 0);
    else return fx_bound(sc.r[st], st == sc.nst - 1 ? out : 0);
}

// ---------------------------------------------------------------- stages
// First radix of the stage-ordered table: the twiddles of stage st (radix R
// after stages of product Ns) are exp(-2 pi i j t / (R Ns)), j < Ns, t = 1..R-1,
// at offset Ns - r0 + (t - 1) Ns + j: consecutive j, the threads of a warp,
// read consecutive entries (a table indexed by j t scattered them over as many
// 128-byte lines as threads).  M - r0 entries for the whole transform.
template <class SC>
GSM_HD const int4 *fx_stage_table(const int4 *tw, const SC &sc, int Ns) { return tw + (Ns - first_radix(sc)); }

GSM_HD int fx_mod(int b, int Ns) { return (Ns & (Ns - 1)) == 0 ? (b & (Ns - 1)) : b % Ns; }

// Position of element i of a line in shared memory: one pad element per 8
// (pad = 3: the strided stores of the first stages would otherwise meet in the
// same banks), or none (pad = 31).  Sched::pad says which: padded
// when every access of a stage then has a constant stride, i.e. fx_pos(i + t S)
// = fx_pos(i) + fx_pos(t S), so that a thread's 8 addresses cost one addition
// each.  That needs the input strides M / R of all stages but the first to be
// multiples of 8, and the products Ns to divide 8 or be multiples of it.  The
// other schedules start with an odd radix or have a factor 4 only; their
// strides spread over the banks by themselves, or nearly.
GSM_HD int fx_pos(int i, int pad) { return i + (i >> pad); }
// Inputs and outputs of a transform are functors; element b + off, off the
// same for all threads:
//   in.load(b, off)       raw element (In::raw) of the line
//   in.exponent(r)        its exponent
//   in.align(r, e, longm) it as integers of exponent e >= its own
//   in.line_exponent(e)   exponent of the line whose largest is e
//   out(b, off, v)        takes an output of the transform
//   Out::kSmem            stores it in the line's own shared memory
// First stage (radix RAD, untwiddled), HALF = 1: inputs t >= RAD/2 are zero.
// next: bound of a long line before the second stage.
template <int RAD, bool FWD, int NB, int HALF, class SC, class In, class Out>
GSM_HD void fx_first(fxc *s, const SC &sc, const Group &g, FxLine &ln, int next, In in, Out out)
{
    constexpr int NIN = HALF == 1 ? RAD / 2 : RAD;
    const int nb = sc.M / RAD;
    const bool last = sc.nst == 1;
    cx<long long> v[NB][RAD];
    int em = kFxZero;
    unsigned acc = 0;
    {
        typename In::raw raw[NB][NIN];
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            const int b = g.t + i * g.T;
            if (b < nb) {
#pragma unroll
                for (int t = 0; t < NIN; ++t) raw[i][t] = in.load(b, t * nb);
            }
        }
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            if (g.t + i * g.T < nb) {
#pragma unroll
                for (int t = 0; t < NIN; ++t) {
                    const int e = in.exponent(raw[i][t]);
                    em = em > e ? em : e;
                }
            }
        }
        em = fx_reduce<true>(em, g, ln.red);
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            if (g.t + i * g.T < nb) {
#pragma unroll
                for (int t = 0; t < NIN; ++t) {
                    v[i][t] = in.align(raw[i][t], em, ln.longm);
                    acc = fx_weigh(acc, fx_weight(v[i][t], ln.longm), ln.longm);
                }
            }
        }
    }
    const int sn = fx_shift_of(acc, ln, g, ln.red + kFxRedWarps, fx_bound(NIN, last ? 1 + ln.paired : 0));
    ln.E = in.line_exponent(em) + sn;
    acc = 0;
#pragma unroll
    for (int i = 0; i < NB; ++i) {
        if (g.t + i * g.T < nb) {
            if (sn > 0) {
#pragma unroll
                for (int t = 0; t < NIN; ++t) v[i][t] = fx_shift(v[i][t], sn);
            }
            fx_bfly<RAD, FWD, HALF>(v[i]);
            if (ln.longm && !last) {
#pragma unroll
                for (int t = 0; t < RAD; ++t) acc = fx_weigh(acc, fx_weight(v[i][t], true), true);
            }
        }
    }
    int sh = 0;
    if (ln.longm && !last) {
        sh = fx_shift_of(acc, ln, g, ln.red, next);
        ln.E += sh;
    } else if (g.bar < 0) {
        fx_sync(g);   // one warp: the reductions passed no barrier since the line was read
    }
#pragma unroll
    for (int i = 0; i < NB; ++i) {
        const int b = g.t + i * g.T;
        if (b < nb) {
            if (sh > 0) {
#pragma unroll
                for (int t = 0; t < RAD; ++t) v[i][t] = fx_shift(v[i][t], sh);
            }
            fxc *d = s + fx_pos(b * RAD, ln.pad);
#pragma unroll
            for (int t = 0; t < RAD; ++t) {
                if (last) out(b * RAD, t, v[i][t]);
                else d[t] = fx_st(v[i][t]);   // b RAD is a multiple of 8, 4 or 2, or there are no pads
            }
        }
    }
    fx_sync(g);
}

// Stage of radix RAD after stages of product Ns > 1: s -> s, or -> out when it
// is the last one.  CROP: of the last stage only the outputs t < RAD/2 (even
// radices).  next: bound of a long line before the next stage.
template <int RAD, bool FWD, int NB, bool CROP, class Out>
GSM_HD void fx_stage(fxc *s, int M, int Ns, bool last, const int4 *__restrict__ tws, const Group &g, FxLine &ln,
                     int next, Out out)
{
    const int nb = M / RAD;
    cx<long long> v[NB][RAD];
    unsigned acc = 0;
#pragma unroll
    for (int i = 0; i < NB; ++i) {
        const int b = g.t + i * g.T;
        if (b < nb) {
            const int j = fx_mod(b, Ns);
#pragma unroll
            for (int t = 0; t < RAD; ++t) v[i][t] = fx_ld(s[fx_pos(b, ln.pad) + t * fx_pos(nb, ln.pad)]);
#pragma unroll
            for (int t = 1; t < RAD; ++t) v[i][t] = fx_rot<FWD>(v[i][t], fx_tw(tws + (t - 1) * Ns + j));
            if (CROP && (RAD % 2) == 0 && last) fx_bfly<RAD, FWD, (CROP && (RAD % 2) == 0) ? 2 : 0>(v[i]);
            else fx_bfly<RAD, FWD, 0>(v[i]);
            if (ln.longm && !last) {
#pragma unroll
                for (int t = 0; t < RAD; ++t) acc = fx_weigh(acc, fx_weight(v[i][t], true), true);
            }
        }
    }
    if (last) {
        if (Out::kSmem) fx_sync(g);
        constexpr int NOUT = (CROP && (RAD % 2) == 0) ? RAD / 2 : RAD;
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            const int b = g.t + i * g.T;
            if (b < nb) {
#pragma unroll
                for (int t = 0; t < NOUT; ++t) out(b, t * Ns, v[i][t]);   // Ns = M / RAD: j = b
            }
        }
        return;
    }
    int sh = 0;
    if (ln.longm) {   // several warps: the reduction passes a barrier
        sh = fx_shift_of(acc, ln, g, ln.red + kFxRedWarps, next);
        ln.E += sh;
    } else {
        fx_sync(g);
    }
#pragma unroll
    for (int i = 0; i < NB; ++i) {
        const int b = g.t + i * g.T;
        if (b < nb) {
            const int j = fx_mod(b, Ns);
            fxc *d = s + fx_pos((b - j) * RAD + j, ln.pad);
            if (sh > 0) {
#pragma unroll
                for (int t = 0; t < RAD; ++t) v[i][t] = fx_shift(v[i][t], sh);
            }
#pragma unroll
            for (int t = 0; t < RAD; ++t) d[fx_pos(t * Ns, ln.pad)] = fx_st(v[i][t]);
        }
    }
    fx_sync(g);
}

// The stages [st_begin, st_end) (st_end < 0: to the last) after the first, in
// the order 8, 4, 2, 5, 3, each radix one loop of its own; the transform's
// last stage hands its outputs to `out`.
template <bool FWD, int EMAX, bool CROP, bool MID, int ST, int END, class SC, class Out>
GSM_HD void fx_rest_fixed(fxc *s, const int4 *__restrict__ tw, const Group &g, FxLine &ln, Out out)
{
    if constexpr (ST < END) {
        constexpr int RAD = SC::template radix<ST>(), Ns = SC::product(ST);
        fx_stage<RAD, FWD, (EMAX + RAD - 1) / RAD, CROP>(s, SC::M, Ns, ST == SC::nst - 1, fx_stage_table(tw, SC{}, Ns), g,
                                                         ln, fx_bound_before<ST + 1>(SC{}, 0, MID ? 0 : 1 + ln.paired), out);
        fx_rest_fixed<FWD, EMAX, CROP, MID, ST + 1, END, SC>(s, tw, g, ln, out);
    }
}
// MID: up to the last stage, which is fused with the multiplication
template <bool FWD, int EMAX, bool CROP, bool MID, class SC, class Out>
GSM_HD void fx_rest_of(fxc *s, const SC &sc, const int4 *__restrict__ tw, const Group &g, FxLine &ln, Out out);

template <bool FWD, int EMAX, bool CROP, class Out>
GSM_HD void fx_rest(fxc *s, const Sched &sc, const int4 *__restrict__ tw, const Group &g, FxLine &ln, int st_begin,
                    int st_end, int out_bound, Out out)
{
    const int last = sc.nst - 1, nend = st_end < 0 ? sc.nst : st_end;
    int Ns = 1, st = st_begin;
    for (int i = 0; i < st_begin; ++i) Ns *= sc.r[i];
#define GSM_FX_STAGES(RAD)                                                                      \
    for (; st < nend && sc.r[st] == RAD; ++st, Ns *= RAD)                                       \
        fx_stage<RAD, FWD, (EMAX + RAD - 1) / RAD, CROP>(s, sc.M, Ns, st == last, fx_stage_table(tw, sc, Ns), g, ln, \
                                                         st < last ? fx_bound_before<0>(sc, st + 1, out_bound) : 0, out)
    GSM_FX_STAGES(8);
    GSM_FX_STAGES(4);
    GSM_FX_STAGES(2);
    GSM_FX_STAGES(5);
    GSM_FX_STAGES(3);
#undef GSM_FX_STAGES
}
template <bool FWD, int EMAX, bool CROP, bool MID, class SC, class Out>
GSM_HD void fx_rest_of(fxc *s, const SC &sc, const int4 *__restrict__ tw, const Group &g, FxLine &ln, Out out)
{
    if constexpr (is_fixed_sched<SC>::value) fx_rest_fixed<FWD, EMAX, CROP, MID, 1, MID ? SC::nst - 1 : SC::nst, SC>(s, tw, g, ln, out);
    else fx_rest<FWD, EMAX, CROP>(s, sc, tw, g, ln, 1, MID ? sc.nst - 1 : -1, MID ? 0 : 1 + ln.paired, out);
}

// First stage by the schedule's first radix.  ZPAD: the second half of the
// line is zero (forward transforms; their first radix is even).  MID: the last
// stage is fused with the multiplication.
template <bool FWD, int EMAX, bool ZPAD, bool MID, class SC, class In, class Out>
GSM_HD void fx_begin(fxc *s, const SC &sc, const Group &g, FxLine &ln, In in, Out out)
{
    constexpr int H = ZPAD ? 1 : 0;
    const int next = sc.nst > 1 ? fx_bound_before<1>(sc, 1, MID ? 0 : 1 + ln.paired) : 0;
    if constexpr (is_fixed_sched<SC>::value) {
        constexpr int RAD = SC::template radix<0>();
        fx_first<RAD, FWD, (EMAX + RAD - 1) / RAD, H>(s, sc, g, ln, next, in, out);
    } else {
        const int r = sc.r[0];
        if (r == 8) fx_first<8, FWD, (EMAX + 7) / 8, H>(s, sc, g, ln, next, in, out);
        else if (r == 4) fx_first<4, FWD, (EMAX + 3) / 4, H>(s, sc, g, ln, next, in, out);
        else if (r == 2) fx_first<2, FWD, (EMAX + 1) / 2, H>(s, sc, g, ln, next, in, out);
        else if constexpr (!ZPAD) {
            if (r == 5) fx_first<5, FWD, (EMAX + 4) / 5, 0>(s, sc, g, ln, next, in, out);
            else fx_first<3, FWD, (EMAX + 2) / 3, 0>(s, sc, g, ln, next, in, out);
        }
    }
}

template <bool FWD, int EMAX, bool ZPAD, bool CROP, class SC, class In, class Out>
GSM_HD void fx_transform(fxc *s, const SC &sc, const int4 *__restrict__ tw, const Group &g, FxLine &ln, In in,
                         Out out)
{
    ln.pad = sc.pad;
    fx_begin<FWD, EMAX, ZPAD, false>(s, sc, g, ln, in, out);
    fx_rest_of<FWD, EMAX, CROP, false>(s, sc, tw, g, ln, out);
}

// A multiplier entry is a factor of at least 1/2 in modulus, of 56 bits, and in its
// low six bits the distance d of its exponent from the row's, so that a small
// entry keeps its bits, and so does the product: a line whose weight sits where
// the multiplier is small (an oscillating density) is scaled up by it.
GSM_HD int fx_mult_exp(int2 m) { return m.y & 63; }

// The product p 2^-d of a line's value and an entry: what it has for the maximum
// over the line, all products being below 2^(32 + T) with T the bits of that, and
// for the sum (T >= kFxProductT), whose unit is 2^(14 + T).
constexpr int kFxProductT = 18;
GSM_HD unsigned fx_product_top(cx<long long> p, int d)
{
    const unsigned a = fx_abs_high(p.re) | fx_abs_high(p.im);
    return d < 32 ? a >> d : 0;
}
GSM_HD unsigned fx_product_weight(cx<long long> p, int d, int T)
{
    const int s = d + T - kFxProductT;
    return s < 32 ? ((fx_abs_high(p.re) + fx_abs_high(p.im) + 2u) >> s) + 1u : 1u;
}
// shift of a product of exponent distance d in a line of total shift sn
GSM_HD int fx_product_shift(int sn, int d)
{
    const int s = sn + d;
    return s > 62 ? 62 : s < -62 ? -62 : s;
}

// The forward's last stage (radix R), the multiplication by mult(k) (entries of
// a row in units of 2^erow), the scaling of the product and the inverse's
// first stage, in registers (see fft_fused_mid).
template <int R, int NB, class SC, class SCI, class MultF>
GSM_HD void fx_mid(fxc *s, const SC &scf, const SCI &sci, const int4 *__restrict__ tw, const Group &g, FxLine &ln,
                   MultF mult, int erow)
{
    const int M = scf.M, nb = M / R;
    const int4 *tws = fx_stage_table(tw, scf, nb);
    cx<long long> v[NB][R];
    int d[NB][R];
    unsigned tops = 0;
#pragma unroll
    for (int i = 0; i < NB; ++i) {
        const int b = g.t + i * g.T;
        if (b < nb) {
#pragma unroll
            for (int t = 0; t < R; ++t) v[i][t] = fx_ld(s[fx_pos(b, ln.pad) + t * fx_pos(nb, ln.pad)]);
#pragma unroll
            for (int t = 1; t < R; ++t) v[i][t] = fx_rot<true>(v[i][t], fx_tw(tws + (t - 1) * nb + b));
            fx_bfly<R, true, 0>(v[i]);
#pragma unroll
            for (int t = 0; t < R; ++t) {
                const int2 m = mult.template at<R>(b, t, nb);
                v[i][t] = {fx_mul(fx_split(v[i][t].re), m.x, m.y), fx_mul(fx_split(v[i][t].im), m.x, m.y)};
                d[i][t] = fx_mult_exp(m);
                tops = fx_weigh(tops, fx_product_top(v[i][t], d[i][t]), true);
            }
        }
    }
    int top = fx_bits((unsigned)fx_reduce<true>((int)tops, g, ln.red)), sn;
    if (ln.longm) {
        sn = top + 32 - fx_bound(R, 0);
    } else {
        top = top > kFxProductT ? top : kFxProductT;
        unsigned acc = 0;
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            if (g.t + i * g.T < nb) {
#pragma unroll
                for (int t = 0; t < R; ++t) acc += fx_product_weight(v[i][t], d[i][t], top);
            }
        }
        sn = top + 14 + fx_bits((unsigned)fx_reduce<false>((int)acc, g, ln.red + kFxRedWarps)) - (kFxTop - ln.paired);
    }
    ln.E += erow + sn;
    unsigned acc = 0;
#pragma unroll
    for (int i = 0; i < NB; ++i) {
        if (g.t + i * g.T < nb) {
#pragma unroll
            for (int t = 0; t < R; ++t) v[i][t] = fx_scale2(v[i][t], fx_product_shift(sn, d[i][t]));
            fx_bfly<R, false, 0>(v[i]);
            if (ln.longm) {
#pragma unroll
                for (int t = 0; t < R; ++t) acc = fx_weigh(acc, fx_weight(v[i][t], true), true);
            }
        }
    }
    int sh = 0;
    if (ln.longm) {
        sh = fx_shift_of(acc, ln, g, ln.red + kFxRedWarps, fx_bound_before<1>(sci, 1, 1 + ln.paired));
        ln.E += sh;
    }
    if (g.bar < 0) fx_sync(g);   // one warp: the reductions passed no barrier
    ln.pad = sci.pad;
#pragma unroll
    for (int i = 0; i < NB; ++i) {
        const int b = g.t + i * g.T;
        if (b < nb) {
            if (sh > 0) {
#pragma unroll
                for (int t = 0; t < R; ++t) v[i][t] = fx_shift(v[i][t], sh);
            }
            fxc *o = s + fx_pos(R * b, ln.pad);
#pragma unroll
            for (int t = 0; t < R; ++t) o[t] = fx_st(v[i][t]);
        }
    }
    fx_sync(g);
}

// The same by the inverse's first radix.
template <int EMAX, class SC, class SCI, class MultF>
GSM_HD void fx_mid_of(fxc *s, const SC &scf, const SCI &sci, const int4 *__restrict__ tw, const Group &g, FxLine &ln,
                      MultF mult, int erow)
{
    if constexpr (is_fixed_sched<SCI>::value) {
        constexpr int R = SCI::template radix<0>();
        fx_mid<R, (EMAX + R - 1) / R>(s, scf, sci, tw, g, ln, mult, erow);
    } else {
        const int fr = sci.r[0];
        if (fr == 8) fx_mid<8, (EMAX + 7) / 8>(s, scf, sci, tw, g, ln, mult, erow);
        else if (fr == 4) fx_mid<4, (EMAX + 3) / 4>(s, scf, sci, tw, g, ln, mult, erow);
        else if (fr == 2) fx_mid<2, (EMAX + 1) / 2>(s, scf, sci, tw, g, ln, mult, erow);
        else if (fr == 5) fx_mid<5, (EMAX + 4) / 5>(s, scf, sci, tw, g, ln, mult, erow);
        else fx_mid<3, (EMAX + 2) / 3>(s, scf, sci, tw, g, ln, mult, erow);
    }
}

// ---------------------------------------------------------------- doubles
GSM_HD int fx_field(double x)   // biased exponent, sign dropped
{
#ifdef __CUDA_ARCH__
    return (__double2hiint(x) >> 20) & 0x7ff;
#else
    unsigned long long u;
    memcpy(&u, &x, 8);
    return (int)(u >> 52) & 0x7ff;
#endif
}

// x as an integer of exponent e - 1083, rounded, e >= the field of x and >= 1 (|result| < 2^61)
GSM_HD long long fx_from_double(double x, int e)
{
    unsigned long long u;
#ifdef __CUDA_ARCH__
    u = (unsigned long long)__double_as_longlong(x);
#else
    memcpy(&u, &x, 8);
#endif
    const int f = (int)(u >> 52) & 0x7ff;
    const unsigned long long m = (u & 0xfffffffffffffull) | (f ? 1ull << 52 : 0ull);
    int s = e - (f ? f : 1);
    s = s < 63 ? s : 63;
    const long long a = (long long)(((m << 8) + ((1ull << s) >> 1)) >> s), sg = (long long)u >> 63;
    return (a ^ sg) - sg;
}
constexpr int kFxDoubleBias = 1083;

// v 2^E rounded to double (half away from zero at exact ties)
GSM_HD double fx_to_double(long long v, int E)
{
    const long long sg = v >> 63;
    unsigned long long m = (unsigned long long)((v ^ sg) - sg);
#ifdef __CUDA_ARCH__
    const int lz = __clzll((long long)m);
#else
    const int lz = m ? __builtin_clzll(m) : 64;
#endif
    if (m == 0) return 0.0;
    m <<= lz;
    int be = E + 63 - lz + 1023;   // biased exponent of the leading bit
    unsigned long long r;
    if (be > 0 && be < 2046) {
        r = ((unsigned long long)(be - 1) << 52) + (m >> 11) + ((m >> 10) & 1);
    } else if (be >= 2046) {
        const unsigned long long t = (m >> 11) + ((m >> 10) & 1);
        r = be == 2046 && t < (1ull << 53) ? (2045ull << 52) + t : 0x7ffull << 52;
    } else {                       // subnormal: the last bit is 2^-1074
        const int s = 12 - be;     // be <= 0
        r = s <= 64 ? (s < 64 ? (m >> s) : 0) + ((m >> (s - 1)) & 1) : 0;
    }
    r |= (unsigned long long)sg & (1ull << 63);
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)r);
#else
    double d;
    memcpy(&d, &r, 8);
    return d;
#endif
}
GSM_HD double fx_nan()
{
#ifdef __CUDA_ARCH__
    return __longlong_as_double(0x7ff8000000000000ll);
#else
    return __builtin_nan("");
#endif
}
GSM_HD double fx_out_double(long long v, int E)
{
    if (E > kFxBig) return fx_nan();
    return fx_to_double(v, E);
}

// Raw complex value of two doubles (an x line of two real rows).
struct FxDoubles {
    struct raw {
        double a, b;
    };
    static GSM_HD int exponent(const raw &r)
    {
        const int p = fx_field(r.a), q = fx_field(r.b);
        return p > q ? p : q;
    }
    static GSM_HD cx<long long> align(const raw &r, int e, bool)
    {
        if (e == 0x7ff) return {0, 0};
        e = e < 1 ? 1 : e;
        return {fx_from_double(r.a, e), fx_from_double(r.b, e)};
    }
    static GSM_HD int line_exponent(int em)
    {
        return em == 0x7ff ? kFxNan : em < 0 ? kFxZero : (em < 1 ? 1 : em) - kFxDoubleBias;
    }
};

// Raw complex value of integers below 2^62 with their own exponent.  Aligned, they
// are rounded in long lines: dropping the bits lowers every value by half a unit,
// which the transform adds up, up to 2^11 units of a line whose largest value may
// be 2^61 (an FP64 sum has that much from 2^8 units on); short lines stay below.
struct FxInts {
    struct raw {
        fxc v;
        int e;
    };
    static GSM_HD int exponent(const raw &r) { return r.e; }
    static GSM_HD cx<long long> align(const raw &r, int e, bool longm)
    {
        int s = e - r.e;
        s = s < 63 ? s : 63;
        const long long half = longm ? (long long)((1ull << s) >> 1) : 0;
        return {(r.v.re + half) >> s, (r.v.im + half) >> s};
    }
    static GSM_HD int line_exponent(int em) { return em; }
};

// Entry of the fixed-point tables from hi + lo (|hi + lo| <= 1).
GSM_HD int2 fx_factor(double hi, double lo)
{
    long long T = llrint(hi * 4611686018427387904.0) + llrint(lo * 4611686018427387904.0);
    const long long top = 1ll << 62;
    T = T > top ? top : T < -top ? -top : T;
    const long long h = (T + (1ll << 31)) >> 32, l = T - h * (1ll << 32);
    return make_int2((int)h, l == INT_MIN ? INT_MIN + 1 : (int)l);   // -l must exist too
}

// Multiplier entry c in units of its row's 2^e (|c| <= 1), see fx_mult_exp.
GSM_HD int2 fx_mult_factor(double c)
{
    if (c == 0.0) return make_int2(0, 0);
    int x;
    frexp(c, &x);
    const int d = x > 0 ? 0 : x < -63 ? 63 : -x;
    const long long T = (llrint(ldexp(c, d + 62)) & ~63ll) + d, h = (T + (1ll << 31)) >> 32;
    return make_int2((int)h, (int)(T - h * (1ll << 32)));
}

}  // namespace gsm
