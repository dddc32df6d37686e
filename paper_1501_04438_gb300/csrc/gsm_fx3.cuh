// gsm_fx3.cuh -- fixed-point passes for padded lengths M = 64 R, R = 1, 2, 3, 4,
// 5, 6 or 8 (n = 32, 64, 96, 128, 160, 192, 256), on the transforms of
// gsm_fx.cuh with everything about the length known at compile time: two
// radix-8 stages and one of radix R (R = 1: two of radix 8).
//
// A CTA holds NL lines of 8 R threads each, packed: every thread of every warp
// has one radix-8 butterfly, whatever 8 R is (a whole number of warps per line
// leaves 16 of 32 lanes idle at M = 128, 24 of 64 at M = 320).  Lines that
// share a warp synchronise together: sync groups of SG = lcm(8 R, 32) threads.
// The 64 butterflies of radix R per line are dealt over the group's threads
// anew, so a thread may hold another line there.
//
// Measured against the kernels of any length (FP64, white noise, L2 cold, us): 256^3
// passes xf 190 -> 142, yf 375 -> 282, conv 1363 -> 992, yi 420 -> 309, xi 248 -> 166 (a
// third of the instructions there are addresses, tests and loops), apply 2590 -> 1884;
// 192^3 (8 8 6 instead of 8 8 2 3) 1940 -> 953; 160^3 1060 -> 582; 32^3 80 -> 35.  The line
// is drawn at three stages and 8 values per thread: 64 registers, four CTAs per SM.
#pragma once

#include "gsm_fx_passes.cuh"

namespace gsm {
namespace {

template <int R>
struct F3 {
    static constexpr int M = 64 * R, NB = 8 * R;            // NB: radix-8 butterflies (threads) per line
    static constexpr int LS = M + M / 8 + 1;                // line stride in shared memory (odd)
    static constexpr int W = R % 4 == 0 ? 32 : R % 2 == 0 ? 16 : 8;   // lanes of a line that a shuffle reaches
    static constexpr int SEG = NB / W;
    static constexpr int SG = R == 1 || R == 2 || R == 4 ? 32 : R == 8 ? 64 : R == 5 ? 160 : 96;
    static constexpr int LG = SG / NB;                      // lines of a sync group
    static constexpr int NL = R == 1 ? 32 : R == 2 ? 16 : R == 3 ? 12 : R == 4 ? 8 : R == 5 ? 8 : R == 6 ? 6 : 4;
    static constexpr int THREADS = NL * NB;                 // 256, 288 or 320
    static constexpr bool TWO = R == 1;
    static constexpr int RC = TWO ? 8 : R;                  // radix and butterflies per line of the last forward stage
    static constexpr int BC = M / RC, NSC = BC;
    static constexpr int KC = (BC * LG + SG - 1) / SG;      // of them per thread
    static constexpr size_t SMEM = (size_t)NL * LS * sizeof(fxc);
    // Words of the shared arrays r0, r1 (F3Shared): each line has its own, for the
    // reduction of its threads (SEG of them) and the conv's sums of two warps
    // alike, so that a sync group touches no other group's words: nothing but its
    // own barriers orders the two uses.
    static constexpr int LW = SEG > 2 ? SEG : 2;
    __host__ __device__ static constexpr int reduce_word(int line, int seg) { return line * LW + seg; }
    __host__ __device__ static constexpr int conv_word(int line, int half) { return line * LW + half; }
    static_assert(SG % NB == 0 && THREADS % SG == 0 && SG % 32 == 0, "whole lines and warps per sync group");
};
template <int R>
struct F3Thread {
    int tid, line, b;   // thread of the CTA; its line and butterfly in the radix-8 stages
    __device__ __forceinline__ F3Thread() : tid(threadIdx.x), line(tid / F3<R>::NB), b(tid % F3<R>::NB) {}
    __device__ __forceinline__ void sync() const
    {
        using F = F3<R>;
        if constexpr (F::SG == 32) __syncwarp();
        else if constexpr (F::SG == F::THREADS) __syncthreads();
        else asm volatile("bar.sync %0, %1;" ::"r"(1 + tid / F::SG), "n"(F::SG) : "memory");
    }
    // butterfly k of this thread in the stage of radix RC: its line (of the CTA) and index; false: none
    __device__ __forceinline__ bool last_bfly(int k, int *ln, int *bc) const
    {
        using F = F3<R>;
        if constexpr (F::KC == 1 && F::BC * F::LG == F::SG) {   // R = 8, 1: the thread's own line
            *ln = line;
            *bc = b;
            return true;
        }
        const int g = tid / F::SG, q = tid % F::SG + k * F::SG;
        *ln = g * F::LG + q / F::BC;
        *bc = q % F::BC;
        return F::BC * F::LG % F::SG == 0 || q < F::BC * F::LG;
    }
    // maximum or sum over the threads of the line; buf: NL * LW words
    template <bool MAX>
    __device__ __forceinline__ int reduce(int v, int *buf) const
    {
        using F = F3<R>;
        if constexpr (F::W == 32) {
            v = MAX ? __reduce_max_sync(0xffffffffu, v) : (int)__reduce_add_sync(0xffffffffu, (unsigned)v);
        } else {
#pragma unroll
            for (int o = F::W / 2; o > 0; o >>= 1) {
                const int w = __shfl_xor_sync(0xffffffffu, v, o);
                v = MAX ? max(v, w) : (int)((unsigned)v + (unsigned)w);
            }
        }
        if constexpr (F::SEG == 1) return v;
        if (b % F::W == 0) buf[F::reduce_word(line, b / F::W)] = v;
        sync();
        v = buf[F::reduce_word(line, 0)];
#pragma unroll
        for (int i = 1; i < F::SEG; ++i) {
            const int w = buf[F::reduce_word(line, i)];
            v = MAX ? max(v, w) : (int)((unsigned)v + (unsigned)w);
        }
        return v;
    }
};

// shared words of the reductions and line exponents
template <int R>
struct F3Shared {
    int r0[F3<R>::NL * F3<R>::LW], r1[F3<R>::NL * F3<R>::LW];
    int e[F3<R>::NL];
};

// padded position
__device__ __forceinline__ constexpr int f3_pos(int i) { return i + (i >> 3); }

// First stage: radix 8, HALF = 1: inputs t >= 4 are zero.  In and PAIRED as in gsm_fx.cuh.
// Leaves the line's exponent in sh.e (read it after the next sync).
template <int R, bool FWD, int HALF, bool PAIRED, class In>
__device__ __forceinline__ void f3_first(fxc *s, const F3Thread<R> &th, F3Shared<R> &sh, const In &in)
{
    using F = F3<R>;
    constexpr int NIN = HALF == 1 ? 4 : 8;
    typename In::raw raw[NIN];
    cx<long long> v[8];
    int em = kFxZero;
#pragma unroll
    for (int t = 0; t < NIN; ++t) raw[t] = in.load(th.b, t * F::NB);
#pragma unroll
    for (int t = 0; t < NIN; ++t) em = max(em, in.exponent(raw[t]));
    em = th.template reduce<true>(em, sh.r0);
    unsigned acc = 0;
#pragma unroll
    for (int t = 0; t < NIN; ++t) {
        v[t] = in.align(raw[t], em, false);
        acc += fx_weight(v[t], false);
    }
    const int sn = max(0, fx_bits((unsigned)th.template reduce<false>((int)acc, sh.r1)) - (kFxTop - PAIRED - 44));
    if (th.b == 0) sh.e[th.line] = in.line_exponent(em) + sn;
    if (sn > 0) {
#pragma unroll
        for (int t = 0; t < NIN; ++t) v[t] = fx_shift(v[t], sn);
    }
    fx_bfly8<FWD, HALF>(v);
    if (F::SEG == 1) th.sync();   // the reductions passed no barrier since the line was read
    fxc *d = s + th.line * F::LS + 9 * th.b;
#pragma unroll
    for (int t = 0; t < 8; ++t) d[t] = fx_st(v[t]);
    th.sync();
}

// Second stage of 8 8 R: radix 8 after 8.
template <int R, bool FWD>
__device__ __forceinline__ void f3_second(fxc *s, const F3Thread<R> &th, const int4 *__restrict__ tw)
{
    using F = F3<R>;
    if constexpr (F::TWO) return;
    const int j = th.b & 7;
    fxc *l = s + th.line * F::LS;
    const fxc *p = l + f3_pos(th.b);
    const int4 *w = tw + j;
    cx<long long> v[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) v[t] = fx_ld(p[t * 9 * R]);
#pragma unroll
    for (int t = 1; t < 8; ++t) v[t] = fx_rot<FWD>(v[t], fx_tw(w + (t - 1) * 8));
    fx_bfly8<FWD, 0>(v);
    th.sync();
    fxc *d = l + 72 * (th.b >> 3) + j;
#pragma unroll
    for (int t = 0; t < 8; ++t) d[9 * t] = fx_st(v[t]);
    th.sync();
}

// Inputs of butterfly bc of the last stage of a line, twiddled.
template <int R, bool FWD>
__device__ __forceinline__ void f3_last_in(cx<long long> *v, const fxc *l, int bc, const int4 *__restrict__ tw)
{
    using F = F3<R>;
    const fxc *p = l + f3_pos(bc);
    const int4 *w = tw + (F::NSC - 8) + bc;
#pragma unroll
    for (int t = 0; t < F::RC; ++t) v[t] = fx_ld(p[t * (F::NSC + F::NSC / 8)]);
#pragma unroll
    for (int t = 1; t < F::RC; ++t) v[t] = fx_rot<FWD>(v[t], fx_tw(w + (t - 1) * F::NSC));
}

// Last stage; out(line, i, t, v) takes output i + t NSC of a line.  CROP: only
// the outputs below M / 2.
template <int R, bool FWD, bool CROP, class Out>
__device__ __forceinline__ void f3_last(const fxc *s, const F3Thread<R> &th, const int4 *__restrict__ tw, const Out &out)
{
    using F = F3<R>;
    constexpr bool EVEN = F::RC % 2 == 0;
    constexpr int NOUT = CROP ? (F::RC + 1) / 2 : F::RC;
#pragma unroll
    for (int k = 0; k < F::KC; ++k) {
        int ln, bc;
        if (!th.last_bfly(k, &ln, &bc)) break;
        cx<long long> v[F::RC];
        f3_last_in<R, FWD>(v, s + ln * F::LS, bc, tw);
        fx_bfly<F::RC, FWD, (CROP && EVEN) ? 2 : 0>(v);
#pragma unroll
        for (int t = 0; t < NOUT; ++t)
            if (!CROP || EVEN || t < F::RC / 2 || bc < F::NSC / 2) out(ln, bc, t, v[t]);
    }
}

// The same position in shared memory as the inputs it comes from, so no barrier
// before it.
template <int R>
struct F3ToSmem {
    fxc *s;
    __device__ __forceinline__ void operator()(int ln, int i, int t, cx<long long> v) const
    {
        using F = F3<R>;
        s[ln * F::LS + f3_pos(i) + t * (F::NSC + F::NSC / 8)] = fx_st(v);
    }
};

// ------------------------------------------------------------------ x forward
template <int R>
__device__ __forceinline__ void f3_body_xf(const double *__restrict__ rho, fxc *__restrict__ W1, const FxExps &ex,
                                           int ny, const int4 *__restrict__ tw, int bx, int by, fxc *s,
                                           F3Shared<R> &sh)
{
    using F = F3<R>;
    constexpr int nx = F::M / 2, hx = nx + 1;
    const F3Thread<R> th;
    const int z = by, y0 = bx * 2 * F::NL, ya = y0 + 2 * th.line;
    const double *slab = rho + (size_t)z * ny * nx;
    FxFromRows in;
    in.a = ya < ny ? slab + (size_t)ya * nx : nullptr;
    in.b = ya + 1 < ny ? slab + (size_t)(ya + 1) * nx : nullptr;
    f3_first<R, true, 1, true>(s, th, sh, in);
    f3_second<R, true>(s, th, tw);
    f3_last<R, true, false>(s, th, tw, F3ToSmem<R>{s});
    if (th.b == 0 && ya < ny) ex.xf[(size_t)z * ((ny + 1) >> 1) + (ya >> 1)] = sh.e[th.line];
    __syncthreads();
    // Hermitian split, as in fx_body_xf; threads run over whole rows of 2 NL
    fxc *out = W1 + (size_t)z * hx * ny + y0;
    constexpr int ROW = 2 * F::NL, STEP = F::THREADS / ROW;
    const int r = th.tid % ROW, ll = r >> 1;
    if (th.tid < ROW * STEP && y0 + r < ny) {
        const fxc *l = s + ll * F::LS;
#pragma unroll 4
        for (int k = th.tid / ROW; k < hx; k += STEP) {
            const cx<long long> zk = fx_ld(l[f3_pos(k)]), zm = fx_ld(l[f3_pos(k == 0 ? 0 : F::M - k)]);
            cx<long long> v;
            if (r & 1) v = {radd(zk.im, zm.im), rsub(zm.re, zk.re)};
            else v = {radd(zk.re, zm.re), rsub(zk.im, zm.im)};
            out[(size_t)k * ny + r] = fx_st(v);
        }
    }
}

// ------------------------------------------------------------------ y forward
template <int R, bool CG>
__device__ __forceinline__ void f3_body_yf(const fxc *__restrict__ W1, fxc *__restrict__ W2, const FxExps &ex, int nz,
                                           int hx, const int4 *__restrict__ tw, int bx, int by, fxc *s,
                                           F3Shared<R> &sh)
{
    using F = F3<R>;
    constexpr int ny = F::M / 2;
    const F3Thread<R> th;
    const int kx = by, z0 = bx * F::NL, z = z0 + th.line;
    FxFromGlobal<CG> in;
    in.p = z < nz ? W1 + ((size_t)z * hx + kx) * ny : nullptr;
    in.e = ex.xf + (size_t)z * (ny / 2);
    in.shift = 1;
    f3_first<R, true, 1, false>(s, th, sh, in);
    f3_second<R, true>(s, th, tw);
    f3_last<R, true, false>(s, th, tw, F3ToSmem<R>{s});
    if (th.b == 0 && z < nz) ex.yf[(size_t)kx * nz + z] = sh.e[th.line];
    __syncthreads();
    constexpr int STEP = F::NB;   // THREADS / NL
    const int ll = th.tid % F::NL, zz = z0 + ll;
    if (zz < nz) {
        fxc *out = W2 + (size_t)kx * F::M * nz + zz;
        const fxc *l = s + ll * F::LS;
#pragma unroll 8
        for (int ky = th.tid / F::NL; ky < F::M; ky += STEP) out[(size_t)ky * nz] = l[f3_pos(ky)];
    }
}

// ------------------------------------------------------------------ conv
// Lines (kx = by, ky = bx NL + line) in 3D, kx = bx NL + line in 2D.
template <int R, bool CG, bool IS3D>
__device__ __forceinline__ void f3_body_conv(fxc *__restrict__ Wd, const int2 *__restrict__ mult,
                                             const int *__restrict__ mrow_exp, const FxExps &ex, int rows, int ny1,
                                             const int4 *__restrict__ tw, const int4 *__restrict__ twi, int bx, int by,
                                             bool full, fxc *s, F3Shared<R> &sh)
{
    using F = F3<R>;
    constexpr int M = F::M, n = M / 2;
    const F3Thread<R> th;
    // rows: ky per kx (3D), kx (2D)
    const int r0 = bx * F::NL, base = IS3D ? by * rows : 0;
    {
        const int row = r0 + th.line, line = base + row;
        FxFromGlobal<CG> in;
        in.p = row < rows ? Wd + (size_t)line * n : nullptr;
        in.e = IS3D ? ex.yf + (size_t)by * n : ex.xf + (row & 1) * ex.xf_par;
        in.shift = IS3D ? 0 : 1;
        f3_first<R, true, 1, !IS3D>(s, th, sh, in);
    }
    f3_second<R, true>(s, th, tw);
    // last forward stage, multiplier, scaling, first inverse stage (see fx_mid)
    constexpr int RC = F::RC, BC = F::BC;
    cx<long long> v[F::KC][RC];
    int d[F::KC][RC], T[F::KC], er[F::KC];
    unsigned top[F::KC], acc[F::KC];
#pragma unroll
    for (int k = 0; k < F::KC; ++k) {
        int ln, bc;
        const bool have = th.last_bfly(k, &ln, &bc);
        top[k] = 0;
        er[k] = 0;
        if (have) {
            f3_last_in<R, true>(v[k], s + ln * F::LS, bc, tw);
            fx_bfly<RC, true, 0>(v[k]);
            const int row = min(r0 + ln, rows - 1);   // a line that is not there takes some row
            size_t mr = base + row;
            if (IS3D && !full) mr = (size_t)by * ny1 + min(row, rows - row);
            er[k] = mrow_exp[mr];
            const int2 *m = mult + mr * (full ? M : n + 1) + bc;
            const int2 *mm = full ? m : mult + mr * (n + 1) + (M - bc);
#pragma unroll
            for (int t = 0; t < RC; ++t) {
                int2 f;
                if (full || 2 * t < RC - 1) f = __ldg(m + t * F::NSC);
                else if (2 * t >= RC) f = __ldg(mm - t * F::NSC);
                else f = __ldg(2 * (bc + t * F::NSC) <= M ? m + t * F::NSC : mm - t * F::NSC);   // middle of an odd radix
                v[k][t] = {fx_mul(fx_split(v[k][t].re), f.x, f.y), fx_mul(fx_split(v[k][t].im), f.x, f.y)};
                d[k][t] = fx_mult_exp(f);
                top[k] = max(top[k], fx_product_top(v[k][t], d[k][t]));
            }
        }
        // 32 lanes of one line (two warps per line), or 8 lanes (R = 1)
        if constexpr (F::TWO) {
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) top[k] = max(top[k], __shfl_xor_sync(0xffffffffu, top[k], o));
        } else {
            top[k] = __reduce_max_sync(0xffffffffu, top[k]);
            if (have && (bc & 31) == 0) sh.r0[F::conv_word(ln, bc >> 5)] = (int)top[k];
        }
    }
    if constexpr (!F::TWO) th.sync();
#pragma unroll
    for (int k = 0; k < F::KC; ++k) {
        int ln, bc;
        const bool have = th.last_bfly(k, &ln, &bc);
        acc[k] = 0;
        T[k] = kFxProductT;
        if (have) {
            if constexpr (!F::TWO) top[k] = (unsigned)max(sh.r0[F::conv_word(ln, 0)], sh.r0[F::conv_word(ln, 1)]);
            T[k] = max(kFxProductT, fx_bits(top[k]));
#pragma unroll
            for (int t = 0; t < RC; ++t) acc[k] += fx_product_weight(v[k][t], d[k][t], T[k]);
        }
        if constexpr (F::TWO) {
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) acc[k] += __shfl_xor_sync(0xffffffffu, acc[k], o);
        } else {
            acc[k] = __reduce_add_sync(0xffffffffu, acc[k]);
            if (have && (bc & 31) == 0) sh.r1[F::conv_word(ln, bc >> 5)] = (int)acc[k];
        }
    }
    th.sync();
    constexpr bool PAD = R != 3 && R != 5 && R != 6;   // radices that keep constant strides (see fx_pos)
#pragma unroll
    for (int k = 0; k < F::KC; ++k) {
        int ln, bc;
        if (!th.last_bfly(k, &ln, &bc)) break;
        const unsigned a = F::TWO ? acc[k] : (unsigned)sh.r1[F::conv_word(ln, 0)] + (unsigned)sh.r1[F::conv_word(ln, 1)];
        const int sn = T[k] + 14 + fx_bits(a) - (kFxTop - (IS3D ? 0 : 1));
        if (bc == 0 && r0 + ln < rows) ex.cv[base + r0 + ln] = sh.e[ln] + er[k] + sn;
#pragma unroll
        for (int t = 0; t < RC; ++t) v[k][t] = fx_scale2(v[k][t], fx_product_shift(sn, d[k][t]));
        fx_bfly<RC, false, 0>(v[k]);
        fxc *o = s + ln * F::LS + (PAD ? f3_pos(RC * bc) : RC * bc);
#pragma unroll
        for (int t = 0; t < RC; ++t) o[t] = fx_st(v[k][t]);
    }
    th.sync();
    fxc *l = s + th.line * F::LS;
    cx<long long> x[8];
    if constexpr (!F::TWO) {
        // radix 8 after R
        const int j = th.b % R;
        const fxc *p = l + (PAD ? f3_pos(th.b) : th.b);
        const int4 *w = twi + j;
#pragma unroll
        for (int t = 0; t < 8; ++t) x[t] = fx_ld(p[t * (PAD ? 9 * R : 8 * R)]);
#pragma unroll
        for (int t = 1; t < 8; ++t) x[t] = fx_rot<false>(x[t], fx_tw(w + (t - 1) * R));
        fx_bfly8<false, 0>(x);
        th.sync();
        const int d0 = (th.b - j) * 8 + j;
        fxc *d = l + (PAD ? f3_pos(d0) : d0);
#pragma unroll
        for (int t = 0; t < 8; ++t) d[PAD ? t * R + (t * R >> 3) : t * R] = fx_st(x[t]);
        th.sync();
    }
    // radix 8 after 8 R (R = 1: after 8), the first half of the outputs
    {
        constexpr bool P = PAD;
        const fxc *p = l + (P ? f3_pos(th.b) : th.b);
        const int4 *w = twi + (F::TWO ? 0 : 7 * R) + th.b;
#pragma unroll
        for (int t = 0; t < 8; ++t) x[t] = fx_ld(p[t * (P ? 9 * R : 8 * R)]);
#pragma unroll
        for (int t = 1; t < 8; ++t) x[t] = fx_rot<false>(x[t], fx_tw(w + (t - 1) * F::NB));
        fx_bfly8<false, 2>(x);
        if (r0 + th.line < rows) {
            fxc *o = Wd + (size_t)(base + r0 + th.line) * n + th.b;
#pragma unroll
            for (int t = 0; t < 4; ++t) o[t * F::NB] = fx_st(x[t]);
        }
    }
}

// ------------------------------------------------------------------ y inverse
template <int R>
struct F3FromSmemBase : FxInts {
    const fxc *l;
    const int *e;
};
template <int R, bool CG, bool FOLD>
struct F3FromSmem : F3FromSmemBase<R> {
    __device__ __forceinline__ typename FxInts::raw load(int b, int off) const
    {
        // off is a multiple of 8 R: no carry into the padding
        typename FxInts::raw r;
        r.v = this->l[f3_pos(b) + off + off / 8];
        const int i = b + off;
        r.e = ldw<CG>(this->e + (FOLD ? min(i, F3<R>::M - i) : i));
        return r;
    }
};
template <int R>
struct F3ToLines {   // output i + t NSC < M / 2 of a line to its place in W1
    fxc *p;
    size_t stride;   // of the CTA's lines
    int lines;
    __device__ __forceinline__ void operator()(int ln, int i, int t, cx<long long> v) const
    {
        if (ln < lines) (p + ln * stride + i)[t * F3<R>::NSC] = fx_st(v);
    }
};

template <int R, bool CG>
__device__ __forceinline__ void f3_body_yi(const fxc *__restrict__ W2, fxc *__restrict__ W1, const FxExps &ex, int nz,
                                           int hx, const int4 *__restrict__ tw, int bx, int by, fxc *s,
                                           F3Shared<R> &sh)
{
    using F = F3<R>;
    constexpr int ny = F::M / 2;
    const F3Thread<R> th;
    const int kx = by, z0 = bx * F::NL;
    {
        const int ll = th.tid % F::NL;
        if (z0 + ll < nz) {
            const fxc *src = W2 + (size_t)kx * F::M * nz + z0 + ll;
            fxc *l = s + ll * F::LS;
#pragma unroll 8
            for (int ky = th.tid / F::NL; ky < F::M; ky += F::NB) fx_copy16(l + f3_pos(ky), src + (size_t)ky * nz);
        } else {
            fxc *l = s + ll * F::LS;   // a line that is not there: zeros
            for (int ky = th.tid / F::NL; ky < F::M; ky += F::NB) l[f3_pos(ky)] = fxc{0, 0};
        }
    }
    fx_copy_wait();
    __syncthreads();
    F3FromSmem<R, CG, false> in;
    in.l = s + th.line * F::LS;
    in.e = ex.cv + (size_t)kx * F::M;
    f3_first<R, false, 0, true>(s, th, sh, in);
    f3_second<R, false>(s, th, tw);
    F3ToLines<R> out{W1 + ((size_t)z0 * hx + kx) * ny, (size_t)hx * ny, nz - z0};
    f3_last<R, false, true>(s, th, tw, out);
    if (th.b == 0 && z0 + th.line < nz) ex.yi[(size_t)(z0 + th.line) * hx + kx] = sh.e[th.line];
}

// ------------------------------------------------------------------ x inverse
template <int R>
struct F3ToRows {
    double *u;       // row y0 of the slab
    int rows;        // rows from y0 on
    const int *e;    // line exponents (shared memory)
    __device__ __forceinline__ void operator()(int ln, int i, int t, cx<long long> v) const
    {
        constexpr int nx = F3<R>::M / 2;
        double *p = u + (size_t)(2 * ln) * nx + i;
        if (2 * ln < rows) p[t * F3<R>::NSC] = fx_out_double(v.re, e[ln]);
        if (2 * ln + 1 < rows) p[nx + t * F3<R>::NSC] = fx_out_double(v.im, e[ln]);
    }
};

template <int R, bool CG>
__device__ __forceinline__ void f3_body_xi(const fxc *__restrict__ W1, double *__restrict__ u,
                                           const int *__restrict__ ek, int ny, const int4 *__restrict__ tw, int bx,
                                           int by, fxc *s, F3Shared<R> &sh)
{
    using F = F3<R>;
    constexpr int nx = F::M / 2, hx = nx + 1;
    const F3Thread<R> th;
    const int z = by, y0 = bx * 2 * F::NL;
    {
        // Hermitian fill, as in fx_body_xi
        const int ll = th.tid % F::NL, yy = y0 + 2 * ll;
        const longlong2 *src = reinterpret_cast<const longlong2 *>(W1 + (size_t)z * hx * ny + yy);
        fxc *l = s + ll * F::LS;
        struct AB {
            longlong2 a, b;
        };
        gather_smem<4, AB>(
            th.tid / F::NL, F::NB, hx,
            [&](int k) {
                AB v{{0, 0}, {0, 0}};
                if (yy < ny) v.a = ldw<CG>(src + (size_t)k * ny);
                if (yy + 1 < ny) v.b = ldw<CG>(src + (size_t)k * ny + 1);
                return v;
            },
            [&](int k, const AB &v) {
                const bool real = k == 0 || k == nx;
                const long long ai = real ? 0 : v.a.y, bi = real ? 0 : v.b.y;
                l[f3_pos(k)] = {rsub(v.a.x, bi), radd(ai, v.b.x)};
                if (!real) l[f3_pos(F::M - k)] = {radd(v.a.x, bi), rsub(v.b.x, ai)};
            });
    }
    __syncthreads();
    F3FromSmem<R, CG, true> in;
    in.l = s + th.line * F::LS;
    in.e = ek;
    f3_first<R, false, 0, false>(s, th, sh, in);
    f3_second<R, false>(s, th, tw);
    F3ToRows<R> out{u + ((size_t)z * ny + y0) * nx, ny - y0, sh.e};
    f3_last<R, false, true>(s, th, tw, out);
}

// ------------------------------------------------------------------ kernels
constexpr int f3_ctas(int threads) { return 65536 / (64 * threads); }   // a 64-register bound
// the conv holds KC radix-R butterflies at once: 10 and 12 complex values for R = 5, 6
template <int R>
constexpr int f3_conv_ctas() { return R == 5 || R == 6 ? 2 : f3_ctas(F3<R>::THREADS); }

// COUNT = 1: one plan; kF3Group: up to that many of one size, instance blockIdx.z.
// A batch of small grids is bound by launches and half-empty grids when its plans
// are applied one by one; 48 plans in one launch per pass instead: FP64 64^3 2.82 ->
// 1.40 ms, 160^3 28.9 -> 26.1, FP32 32^3 1.13 -> 0.21, 2D 64^2 0.73 -> 0.15.
template <int COUNT>
struct F3Group {
    F3Inst inst[COUNT];
    __device__ __forceinline__ const F3Inst &at() const { return inst[COUNT > 1 ? blockIdx.z : 0]; }
};

template <int R, int COUNT>
__global__ void __launch_bounds__(F3<R>::THREADS, f3_ctas(F3<R>::THREADS))
    k_f3_xf(const __grid_constant__ F3Group<COUNT> g, int ny, const int4 *__restrict__ tw)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ F3Shared<R> sh;
    const F3Inst &q = g.at();
    f3_body_xf<R>(static_cast<const double *>(q.rho), static_cast<fxc *>(q.W1), q.ex, ny, tw, blockIdx.x, blockIdx.y,
                  reinterpret_cast<fxc *>(smem_raw), sh);
}
template <int R, int COUNT>
__global__ void __launch_bounds__(F3<R>::THREADS, f3_ctas(F3<R>::THREADS))
    k_f3_yf(const __grid_constant__ F3Group<COUNT> g, int nz, int hx, const int4 *__restrict__ tw)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ F3Shared<R> sh;
    const F3Inst &q = g.at();
    f3_body_yf<R, false>(static_cast<const fxc *>(q.W1), static_cast<fxc *>(q.W2), q.ex, nz, hx, tw, blockIdx.x,
                         blockIdx.y, reinterpret_cast<fxc *>(smem_raw), sh);
}
template <int R, bool IS3D, int COUNT>
__global__ void __launch_bounds__(F3<R>::THREADS, f3_conv_ctas<R>())
    k_f3_conv(const __grid_constant__ F3Group<COUNT> g, int rows, int ny1, const int4 *__restrict__ tw,
              const int4 *__restrict__ twi, int full)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ F3Shared<R> sh;
    const F3Inst &q = g.at();
    f3_body_conv<R, false, IS3D>(static_cast<fxc *>(IS3D ? q.W2 : q.W1), static_cast<const int2 *>(q.mult), q.mrow, q.ex,
                                 rows, ny1, tw, twi, blockIdx.x, blockIdx.y, full != 0,
                                 reinterpret_cast<fxc *>(smem_raw), sh);
}
template <int R, int COUNT>
__global__ void __launch_bounds__(F3<R>::THREADS, f3_ctas(F3<R>::THREADS))
    k_f3_yi(const __grid_constant__ F3Group<COUNT> g, int nz, int hx, const int4 *__restrict__ tw)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ F3Shared<R> sh;
    const F3Inst &q = g.at();
    f3_body_yi<R, false>(static_cast<const fxc *>(q.W2), static_cast<fxc *>(q.W1), q.ex, nz, hx, tw, blockIdx.x,
                         blockIdx.y, reinterpret_cast<fxc *>(smem_raw), sh);
}
// ek_stride: 3D hx, the exponents are yi; 2D 0, they are cv
template <int R, int COUNT>
__global__ void __launch_bounds__(F3<R>::THREADS, f3_ctas(F3<R>::THREADS))
    k_f3_xi(const __grid_constant__ F3Group<COUNT> g, int ek_stride, int ny, const int4 *__restrict__ tw)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ F3Shared<R> sh;
    const F3Inst &q = g.at();
    f3_body_xi<R, false>(static_cast<const fxc *>(q.W1), static_cast<double *>(q.u),
                         (ek_stride ? q.ex.yi : q.ex.cv) + (size_t)blockIdx.y * ek_stride, ny, tw, blockIdx.x,
                         blockIdx.y, reinterpret_cast<fxc *>(smem_raw), sh);
}

}  // namespace
// One pass (3D: 0..4 = xf, yf, conv, yi, xi; 2D: 0..2 = xf, conv, xi).  Dynamic and
// static shared memory together stay below the 48 KB that need no raised limit.
template <int R, int COUNT>
void f3_launch_group(const F3Call &c, int pass)
{
    using F = F3<R>;
    static_assert(F::SMEM + sizeof(F3Shared<R>) <= 48 * 1024, "no raised shared-memory limit");
    F3Group<COUNT> g{};
    for (int i = 0; i < c.count; ++i) g.inst[i] = c.inst[i];
    const Plan *p = c.p;
    const int last = p->d == 3 ? 4 : 2, conv = p->d == 3 ? 2 : 1;
    const int ny = p->n[1], hx = p->n[0] + 1, nz = c.nz, full = p->mult_full ? 1 : 0;
    const int axis = pass == 0 || pass == last ? 0 : pass == conv ? p->d - 1 : 1;
    const int4 *tw = static_cast<const int4 *>(p->d_tw[axis]), *twi = static_cast<const int4 *>(p->d_twi[axis]);
    const dim3 gx((ny + 2 * F::NL - 1) / (2 * F::NL), nz, c.count), gy((nz + F::NL - 1) / F::NL, hx, c.count);
    if (pass == 0) {
        k_f3_xf<R, COUNT><<<gx, F::THREADS, F::SMEM, c.st>>>(g, ny, tw);
    } else if (pass == last) {
        k_f3_xi<R, COUNT><<<gx, F::THREADS, F::SMEM, c.st>>>(g, p->d == 3 ? hx : 0, ny, twi);
    } else if (pass == conv && p->d == 3) {
        const int My = p->M[1];
        k_f3_conv<R, true, COUNT><<<dim3((My + F::NL - 1) / F::NL, hx, c.count), F::THREADS, F::SMEM, c.st>>>(
            g, My, ny + 1, tw, twi, full);
    } else if (pass == conv) {
        k_f3_conv<R, false, COUNT><<<dim3((hx + F::NL - 1) / F::NL, 1, c.count), F::THREADS, F::SMEM, c.st>>>(
            g, hx, ny + 1, tw, twi, full);
    } else if (pass == 1) {
        k_f3_yf<R, COUNT><<<gy, F::THREADS, F::SMEM, c.st>>>(g, nz, hx, tw);
    } else {
        k_f3_yi<R, COUNT><<<gy, F::THREADS, F::SMEM, c.st>>>(g, nz, hx, twi);
    }
}
template <int R>
void f3_launch(const F3Call &c, int pass)
{
    if (c.count == 1) f3_launch_group<R, 1>(c, pass);
    else f3_launch_group<R, kF3Group>(c, pass);
}

}  // namespace gsm
