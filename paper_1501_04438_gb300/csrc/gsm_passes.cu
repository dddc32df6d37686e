// gsm_passes.cu -- Algorithm 1, "Actual computation": the zero-padded FFT
// convolution with the stored multiplier (Eq. I1FFT with the Taylor
// correction of Sec. 2.3 folded in), for each precision.
//
// Data flow in 3D (n = grid points per axis, M = 2n the padded lengths,
// hx = nx + 1 the non-negative x frequencies of the real transform):
//   pass xf   rho[z][y][x]        -> W1[z][kx][y]      two real rows per complex
//                                                      line, length Mx, zero pad
//   pass yf   W1[z][kx][y]        -> W2[kx][ky][z]     length My, zero pad
//   pass conv W2[kx][ky][0..nz)   -> same, in place    length Mz: forward,
//                                                      multiply, inverse, crop
//   pass yi   W2[kx][ky][z]       -> W1[z][kx][y]      length My, crop
//   pass xi   W1[z][kx][y]        -> u[z][y][x]        Hermitian fill, crop
// Each pass reads contiguous lines or writes them, and does the transposition
// in shared memory; the other side of each pass moves chunks of 2nl (xf, xi)
// or nl (yf, yi) consecutive complex values.  In 2D: xf (one slab), conv on
// W[kx][y] along y, xi.
#include "gsm_pass_common.cuh"

namespace gsm {
namespace {

// Launch shape (see PassCfg): a CTA holds nl lines; line l is transformed by
// group l of gthr threads (blockDim.x = nl * gthr).  Loads and stores that
// touch one line are done by its group; the transposed side of a pass is
// done by the whole CTA, with one __syncthreads between it and the FFTs.

// ------------------------------------------------------------------ pass xf
// Each pass is a __device__ body taking its tile (bx, by) explicitly, so that
// the single-plan kernels and the grouped batch kernels share it.
template <class Pol, int EMAX>
__device__ __forceinline__ void body_xf(const typename Pol::io_t *__restrict__ rho, S_t<Pol> *__restrict__ W1,
                                        int nx, int ny, int hx, const Sched &sc, int nl, int gthr,
                                        const typename Pol::tw_t *__restrict__ tw, int bx, int by,
                                        unsigned char *smem_raw)
{
    using R = typename Pol::real;
    const int M = sc.M, LS = line_stride<Pol>(M);
    const Group g = make_group(gthr, nl);
    const int l = threadIdx.x / gthr;
    S_t<Pol> *s = reinterpret_cast<S_t<Pol> *>(smem_raw) + l * LS;
    const int z = by;
    const int y0 = bx * 2 * nl;
    const int ya = y0 + 2 * l;
    const typename Pol::io_t *slab = rho + (size_t)z * ny * nx;
    // x >= nx is zero padding
    gather_smem<4, cx<R>>(
        g.t, g.T, M,
        [&](int x) {
            cx<R> v{Pol::zero(), Pol::zero()};
            if (x < nx) {
                if (ya < ny) v.re = Pol::from_io(slab[(size_t)ya * nx + x]);
                if (ya + 1 < ny) v.im = Pol::from_io(slab[(size_t)(ya + 1) * nx + x]);
            }
            return v;
        },
        [&](int x, const cx<R> &v) { s[pidx<Pol>(x)] = Pol::st(v); });
    group_sync(g);
    fft_line<Pol, true, EMAX>(s, sc, tw, g);
    __syncthreads();
    // Z = A + iB with A, B the transforms of the two real rows:
    // 2A[k] = Z[k] + conj Z[-k], 2B[k] = -i (Z[k] - conj Z[-k]); the factor 2
    // is removed by the multiplier.
    const S_t<Pol> *s0 = reinterpret_cast<const S_t<Pol> *>(smem_raw);
    S_t<Pol> *out = W1 + (size_t)z * hx * ny;
    // (a thread keeps its line: the CTA's nl gthr threads are whole rows of nl)
    const int ll = threadIdx.x % nl, yy = y0 + 2 * ll;
    for (int k = threadIdx.x / nl; k < hx; k += gthr) {
        const cx<R> zk = Pol::ld(s0[ll * LS + pidx<Pol>(k)]);
        const cx<R> zm = cconj(Pol::ld(s0[ll * LS + pidx<Pol>(k == 0 ? 0 : M - k)]));
        if (yy < ny) out[(size_t)k * ny + yy] = Pol::st(cadd(zk, zm));
        if (yy + 1 < ny) out[(size_t)k * ny + yy + 1] = Pol::st(cmul_negi(csub(zk, zm)));
    }
}

template <class Pol, int EMAX>
__global__ void __launch_bounds__(kMaxThreads)
    k_xf(const typename Pol::io_t *__restrict__ rho, S_t<Pol> *__restrict__ W1, int nx, int ny, int hx,
         Sched sc, int nl, int gthr, const typename Pol::tw_t *__restrict__ tw)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    body_xf<Pol, EMAX>(rho, W1, nx, ny, hx, sc, nl, gthr, tw, blockIdx.x, blockIdx.y, smem_raw);
}

// ------------------------------------------------------------------ pass yf
template <class Pol, int EMAX, bool CG = false>
__device__ __forceinline__ void body_yf(const S_t<Pol> *__restrict__ W1, S_t<Pol> *__restrict__ W2, int ny,
                                        int nz, int hx, const Sched &sc, int nl, int gthr,
                                        const typename Pol::tw_t *__restrict__ tw, int bx, int by,
                                        unsigned char *smem_raw)
{
    using R = typename Pol::real;
    const int M = sc.M, LS = line_stride<Pol>(M);
    const Group g = make_group(gthr, nl);
    const int l = threadIdx.x / gthr;
    S_t<Pol> *s = reinterpret_cast<S_t<Pol> *>(smem_raw) + l * LS;
    const int kx = by;
    const int z0 = bx * nl;
    const int z = z0 + l;
    const S_t<Pol> *in = W1 + ((size_t)z * hx + kx) * ny;
    gather_smem<4, S_t<Pol>>(   // y >= ny: zero padding
        g.t, g.T, M,
        [&](int y) {
            S_t<Pol> v = Pol::st(cx<R>{Pol::zero(), Pol::zero()});
            if (y < ny && z < nz) v = ldw<CG>(in + y);
            return v;
        },
        [&](int y, const S_t<Pol> &v) { s[pidx<Pol>(y)] = v; });
    group_sync(g);
    fft_line<Pol, true, EMAX>(s, sc, tw, g);
    __syncthreads();
    const S_t<Pol> *s0 = reinterpret_cast<const S_t<Pol> *>(smem_raw);
    S_t<Pol> *out = W2 + (size_t)kx * M * nz;
    const int ll = threadIdx.x % nl, zz = z0 + ll;
    if (zz < nz)
        for (int ky = threadIdx.x / nl; ky < M; ky += gthr) out[(size_t)ky * nz + zz] = s0[ll * LS + pidx<Pol>(ky)];
}

template <class Pol, int EMAX>
__global__ void __launch_bounds__(kMaxThreads)
    k_yf(const S_t<Pol> *__restrict__ W1, S_t<Pol> *__restrict__ W2, int ny, int nz, int hx, Sched sc,
         int nl, int gthr, const typename Pol::tw_t *__restrict__ tw)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    body_yf<Pol, EMAX>(W1, W2, ny, nz, hx, sc, nl, gthr, tw, blockIdx.x, blockIdx.y, smem_raw);
}

// ------------------------------------------------------------------ pass conv
// Lines of length n (stored) padded to M: forward, multiply by the real
// multiplier mult[row + min(k, M - k)], inverse, keep the first n.
// 3D: line = kx * My + ky, row = (kx * (ny + 1) + min(ky, My - ky)) * (nz + 1).
// 2D: line = kx, row = kx * (ny + 1).  Entirely group-local: no CTA barrier.
// full: the multiplier is stored for the whole half spectrum, row line * M.
template <class Pol, int EMAX, bool CG = false>
__device__ __forceinline__ void body_conv(S_t<Pol> *__restrict__ W, const typename Pol::mult_t *__restrict__ mult,
                                          int nlines, int n, int is3d, int My, int ny1, const Sched &sc,
                                          const Sched &sci, int nl, int gthr,
                                          const typename Pol::tw_t *__restrict__ tw,
                                          const typename Pol::tw_t *__restrict__ twi, int bx,
                                          unsigned char *smem_raw, bool full = false)
{
    using R = typename Pol::real;
    const int M = sc.M, LS = line_stride<Pol>(M);
    const Group g = make_group(gthr, nl);
    const int l = threadIdx.x / gthr;
    S_t<Pol> *s = reinterpret_cast<S_t<Pol> *>(smem_raw) + l * LS;
    const int line = bx * nl + l;
    if (line >= nlines) return;   // the whole group leaves; no CTA barrier follows
    S_t<Pol> *w = W + (size_t)line * n;
    gather_smem<4, S_t<Pol>>(   // z >= n: zero padding
        g.t, g.T, M, [&](int z) { return z < n ? ldw<CG>(w + z) : Pol::st(cx<R>{Pol::zero(), Pol::zero()}); },
        [&](int z, const S_t<Pol> &v) { s[pidx<Pol>(z)] = v; });
    group_sync(g);
    // multiplier of frequency k: the whole half spectrum is stored (full), or
    // the octant, read at min(k, M - k) (the multiplier is even)
    const typename Pol::mult_t *mrow;
    if (full) {
        mrow = mult + (size_t)line * M;
    } else if (is3d) {
        const int kx = line / My, ky = line - kx * My;
        mrow = mult + ((size_t)kx * ny1 + min(ky, My - ky)) * (n + 1);
    } else {
        mrow = mult + (size_t)line * (n + 1);
    }
    auto mult_of = [&](int k) -> R { return Pol::mult(mrow[full ? k : min(k, M - k)]); };
    const int fr = fused_radix(sc, sci);
    if (fr != 0) {
        // forward up to its last stage; last forward stage, multiplication and
        // first inverse stage in registers; the rest of the inverse
        fft_line<Pol, true, EMAX>(s, sc, tw, g, 0, sc.nst - 1);
        if (fr == 8) fft_fused_mid<Pol, 8, (EMAX + 7) / 8>(s, sc, tw, g, mult_of);
        else if (fr == 4) fft_fused_mid<Pol, 4, (EMAX + 3) / 4>(s, sc, tw, g, mult_of);
        else if (fr == 2) fft_fused_mid<Pol, 2, (EMAX + 1) / 2>(s, sc, tw, g, mult_of);
        else if (fr == 5) fft_fused_mid<Pol, 5, (EMAX + 4) / 5>(s, sc, tw, g, mult_of);
        else fft_fused_mid<Pol, 3, (EMAX + 2) / 3>(s, sc, tw, g, mult_of);
        fft_line<Pol, false, EMAX>(s, sci, twi, g, 1);
    } else {
        fft_line<Pol, true, EMAX>(s, sc, tw, g);
        for (int k = g.t; k < M; k += g.T) {
            const int p = pidx<Pol>(k);
            s[p] = Pol::st(cscale(Pol::ld(s[p]), mult_of(k)));
        }
        group_sync(g);
        fft_line<Pol, false, EMAX>(s, sci, twi, g);
    }
    for (int z = g.t; z < n; z += g.T) w[z] = s[pidx<Pol>(z)];
}

// Registers: with 56 an SM holds three CTAs of 384 threads (M = 80 with 12 lines, M =
// 1536, M = 3000), with the 61 that the compiler takes by itself two.  Conv pass in us
// with 61, 56, 48, 40: 768^2 36.9, 26.6, 26.6, 26.7; 648x1500 67.6, 55.3, 55.3, 57.3; 1536^2
// 106.5, 88.1, 88.1, 86.0; 1500x648 69.6, 69.6, 69.6, 75.8; 300x48x40 73.0, 61.5, 61.4, 61.4.
template <class Pol, int EMAX>
__global__ void __maxnreg__(EMAX == 8 ? 56 : 80)
    k_conv(S_t<Pol> *__restrict__ W, const typename Pol::mult_t *__restrict__ mult,
                                                      int nlines, int n, int is3d, int My, int ny1, Sched sc,
                                                      Sched sci, int nl, int gthr,
                                                      const typename Pol::tw_t *__restrict__ tw,
                                                      const typename Pol::tw_t *__restrict__ twi, int full)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    body_conv<Pol, EMAX>(W, mult, nlines, n, is3d, My, ny1, sc, sci, nl, gthr, tw, twi, blockIdx.x, smem_raw,
                         full != 0);
}

// ------------------------------------------------------------------ pass yi
template <class Pol, int EMAX, bool CG = false>
__device__ __forceinline__ void body_yi(const S_t<Pol> *__restrict__ W2, S_t<Pol> *__restrict__ W1, int ny,
                                        int nz, int hx, const Sched &sc, int nl, int gthr,
                                        const typename Pol::tw_t *__restrict__ tw, int bx, int by,
                                        unsigned char *smem_raw)
{
    const int M = sc.M, LS = line_stride<Pol>(M);
    const Group g = make_group(gthr, nl);
    const int l = threadIdx.x / gthr;
    S_t<Pol> *s0 = reinterpret_cast<S_t<Pol> *>(smem_raw);
    S_t<Pol> *s = s0 + l * LS;
    const int kx = by;
    const int z0 = bx * nl;
    const S_t<Pol> *in = W2 + (size_t)kx * M * nz;
    const int ll = threadIdx.x % nl;
    if (z0 + ll < nz)
        gather_smem<4, S_t<Pol>>(
            threadIdx.x / nl, gthr, M, [&](int ky) { return ldw<CG>(in + (size_t)ky * nz + z0 + ll); },
            [&](int ky, const S_t<Pol> &v) { s0[ll * LS + pidx<Pol>(ky)] = v; });
    __syncthreads();
    const int z = z0 + l;
    fft_line<Pol, false, EMAX>(s, sc, tw, g);
    if (z < nz) {
        S_t<Pol> *out = W1 + ((size_t)z * hx + kx) * ny;
        for (int y = g.t; y < ny; y += g.T) out[y] = s[pidx<Pol>(y)];
    }
}

template <class Pol, int EMAX>
__global__ void __launch_bounds__(kMaxThreads)
    k_yi(const S_t<Pol> *__restrict__ W2, S_t<Pol> *__restrict__ W1, int ny, int nz, int hx, Sched sc,
         int nl, int gthr, const typename Pol::tw_t *__restrict__ tw)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    body_yi<Pol, EMAX>(W2, W1, ny, nz, hx, sc, nl, gthr, tw, blockIdx.x, blockIdx.y, smem_raw);
}

// ------------------------------------------------------------------ pass xi
template <class Pol, int EMAX, bool CG = false>
__device__ __forceinline__ void body_xi(const S_t<Pol> *__restrict__ W1, typename Pol::io_t *__restrict__ u, int nx,
                                        int ny, int hx, const Sched &sc, int nl, int gthr,
                                        const typename Pol::tw_t *__restrict__ tw, int bx, int by,
                                        unsigned char *smem_raw)
{
    using R = typename Pol::real;
    const int M = sc.M, LS = line_stride<Pol>(M);
    const Group g = make_group(gthr, nl);
    const int l = threadIdx.x / gthr;
    S_t<Pol> *s0 = reinterpret_cast<S_t<Pol> *>(smem_raw);
    S_t<Pol> *s = s0 + l * LS;
    const int z = by;
    const int y0 = bx * 2 * nl;
    const S_t<Pol> *in = W1 + (size_t)z * hx * ny;
    // Z[k] = A[k] + i B[k] (k = 0..nx), Z[M-k] = conj A[k] + i conj B[k];
    // A, B real at k = 0 and k = nx (DC and Nyquist of real rows)
    struct AB {
        S_t<Pol> a, b;
    };
    const int ll = threadIdx.x % nl, yy = y0 + 2 * ll;
    gather_smem<4, AB>(
        threadIdx.x / nl, gthr, hx,
        [&](int k) {
            AB v{Pol::st(cx<R>{Pol::zero(), Pol::zero()}), Pol::st(cx<R>{Pol::zero(), Pol::zero()})};
            if (yy < ny) v.a = ldw<CG>(in + (size_t)k * ny + yy);
            if (yy + 1 < ny) v.b = ldw<CG>(in + (size_t)k * ny + yy + 1);
            return v;
        },
        [&](int k, const AB &v) {
            cx<R> A = Pol::ld(v.a), B = Pol::ld(v.b);
            if (k == 0 || k == nx) {
                A.im = Pol::zero();
                B.im = Pol::zero();
            }
            s0[ll * LS + pidx<Pol>(k)] = Pol::st(cadd(A, cmul_posi(B)));
            if (k > 0 && k < nx) s0[ll * LS + pidx<Pol>(M - k)] = Pol::st(cadd(cconj(A), cmul_posi(cconj(B))));
        });
    __syncthreads();
    fft_line<Pol, false, EMAX>(s, sc, tw, g);
    const int ya = y0 + 2 * l;
    typename Pol::io_t *slab = u + (size_t)z * ny * nx;
    for (int x = g.t; x < nx; x += g.T) {
        const cx<R> c = Pol::ld(s[pidx<Pol>(x)]);
        if (ya < ny) slab[(size_t)ya * nx + x] = Pol::to_io(c.re);
        if (ya + 1 < ny) slab[(size_t)(ya + 1) * nx + x] = Pol::to_io(c.im);
    }
}

template <class Pol, int EMAX>
__global__ void __launch_bounds__(kMaxThreads)
    k_xi(const S_t<Pol> *__restrict__ W1, typename Pol::io_t *__restrict__ u, int nx, int ny, int hx,
         Sched sc, int nl, int gthr, const typename Pol::tw_t *__restrict__ tw)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    body_xi<Pol, EMAX>(W1, u, nx, ny, hx, sc, nl, gthr, tw, blockIdx.x, blockIdx.y, smem_raw);
}

// ------------------------------------------------------------------ pass conv, long 2D lines
// The FP32 form of the split conv: see k_fx_conv_split (gsm_fx_passes.cuh) for
// the method.  rank 0 takes the even, rank 1 the odd frequencies; schedules and
// tables of length Mh (sched_hf, sched_hi, twh, twhi); twM: the M twiddles
// w_M^m.  The kernels keep the engine's usual bound (a 256-thread bound made
// the conv slower, 0.50 -> 0.53 ms at 4096^2).
template <class Pol, int EMAX>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kMaxThreads)
    k_conv_split(S_t<Pol> *__restrict__ W, const typename Pol::mult_t *__restrict__ mult, int nlines, int ny1,
                 Sched sc, Sched sci, const typename Pol::tw_t *__restrict__ tw,
                 const typename Pol::tw_t *__restrict__ twi, const typename Pol::tw_t *__restrict__ twM, int full)
{
    using R = typename Pol::real;
    namespace cg = cooperative_groups;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank();
    const int line = blockIdx.x >> 1;
    const int Mh = sc.M, M = 2 * Mh;
    const Group g = make_group(blockDim.x, 1);
    S_t<Pol> *s = reinterpret_cast<S_t<Pol> *>(smem_raw);
    S_t<Pol> *w = W + (size_t)line * Mh;
    const bool active = line < nlines;   // every CTA of a cluster reaches both cluster barriers
    if (active) {
        for (int i = g.t; i < Mh; i += g.T) {
            cx<R> v = Pol::ld(w[i]);
            if (rank) v = cmul(v, Pol::tw(twM[i]));   // x w_M^n
            s[pidx<Pol>(i)] = Pol::st(v);
        }
        group_sync(g);
        const typename Pol::mult_t *mrow = mult + (size_t)line * (full ? M : ny1);
        // output k' of this half is frequency k = 2 k' + rank
        auto mult_of = [&](int kk) -> R {
            const int k = 2 * kk + rank;
            return Pol::mult(mrow[full ? k : min(k, M - k)]);
        };
        const int fr = fused_radix(sc, sci);
        if (fr != 0) {
            fft_line<Pol, true, EMAX>(s, sc, tw, g, 0, sc.nst - 1);
            if (fr == 8) fft_fused_mid<Pol, 8, (EMAX + 7) / 8>(s, sc, tw, g, mult_of);
            else if (fr == 4) fft_fused_mid<Pol, 4, (EMAX + 3) / 4>(s, sc, tw, g, mult_of);
            else if (fr == 2) fft_fused_mid<Pol, 2, (EMAX + 1) / 2>(s, sc, tw, g, mult_of);
            else if (fr == 5) fft_fused_mid<Pol, 5, (EMAX + 4) / 5>(s, sc, tw, g, mult_of);
            else fft_fused_mid<Pol, 3, (EMAX + 2) / 3>(s, sc, tw, g, mult_of);
            fft_line<Pol, false, EMAX>(s, sci, twi, g, 1);
        } else {
            fft_line<Pol, true, EMAX>(s, sc, tw, g);
            for (int k = g.t; k < Mh; k += g.T) {
                const int p = pidx<Pol>(k);
                s[p] = Pol::st(cscale(Pol::ld(s[p]), mult_of(k)));
            }
            group_sync(g);
            fft_line<Pol, false, EMAX>(s, sci, twi, g);
        }
        if (rank) {
            for (int i = g.t; i < Mh; i += g.T) {
                const int p = pidx<Pol>(i);
                s[p] = Pol::st(cmulc(Pol::ld(s[p]), Pol::tw(twM[i])));   // w_M^(-n)
            }
        }
    }
    cl.sync();   // both halves transformed
    if (active) {
        const S_t<Pol> *peer = cl.map_shared_rank(s, rank ^ 1);
        const int h = Mh / 2, n0 = rank * h;
        for (int i = g.t; i < h; i += g.T) {
            const int n = n0 + i, p = pidx<Pol>(n);
            w[n] = Pol::st(cadd(Pol::ld(s[p]), Pol::ld(peer[p])));
        }
    }
    cl.sync();   // the peer has read this CTA's half: its shared memory may go
}

// ------------------------------------------------------------------ x forward, long 2D lines
// The FP32 form of the split x forward (k_fx_xf_split): each CTA of a pair
// transforms one parity of the frequencies and writes it.  The x inverse stays
// one line per CTA: split by output parity, each CTA reads the whole half
// spectrum and writes every other output, which was slower (4096^2).
// sc: length Mh; tw: its tables; twM: the M twiddles w_M^m.
template <class Pol, int EMAX>
__global__ void __launch_bounds__(kMaxThreads)
    k_xf_split(const typename Pol::io_t *__restrict__ rho, S_t<Pol> *__restrict__ W1, int nx, int ny, int hx,
               Sched sc, const typename Pol::tw_t *__restrict__ tw, const typename Pol::tw_t *__restrict__ twM)
{
    using R = typename Pol::real;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int rank = blockIdx.x & 1, ya = 2 * (blockIdx.x >> 1);
    const int Mh = sc.M;   // == nx
    const Group g = make_group(blockDim.x, 1);
    S_t<Pol> *s = reinterpret_cast<S_t<Pol> *>(smem_raw);
    for (int x = g.t; x < nx; x += g.T) {
        R a = Pol::zero(), b = Pol::zero();
        if (ya < ny) a = Pol::from_io(rho[(size_t)ya * nx + x]);
        if (ya + 1 < ny) b = Pol::from_io(rho[(size_t)(ya + 1) * nx + x]);
        cx<R> v{a, b};
        if (rank) v = cmul(v, Pol::tw(twM[x]));   // x w_M^x: the odd frequencies
        s[pidx<Pol>(x)] = Pol::st(v);
    }
    group_sync(g);
    fft_line<Pol, true, EMAX>(s, sc, tw, g);
    // frequency k = 2 k' + rank sits at k' of this half; M - k at (Mh - k' - rank) mod Mh
    const int nk = rank ? nx / 2 : nx / 2 + 1;   // k = 0 .. nx of this parity (nx is even)
    for (int kp = threadIdx.x; kp < nk; kp += blockDim.x) {
        const int k = 2 * kp + rank;
        int km = Mh - kp - rank;
        if (km == Mh) km = 0;
        const cx<R> zk = Pol::ld(s[pidx<Pol>(kp)]);
        const cx<R> zm = cconj(Pol::ld(s[pidx<Pol>(km)]));
        if (ya < ny) W1[(size_t)k * ny + ya] = Pol::st(cadd(zk, zm));
        if (ya + 1 < ny) W1[(size_t)k * ny + ya + 1] = Pol::st(cmul_negi(csub(zk, zm)));
    }
}

// ------------------------------------------------------------------ FFT test hook
template <class Pol, bool FWD, int EMAX>
__global__ void __launch_bounds__(kMaxThreads) k_fft_hook(const double2 *__restrict__ in, double2 *__restrict__ out,
                                                          int nlines, Sched sc, int nl, int gthr,
                                                          const typename Pol::tw_t *__restrict__ tw)
{
    using R = typename Pol::real;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int M = sc.M, LS = line_stride<Pol>(M);
    const Group g = make_group(gthr, nl);
    const int l = threadIdx.x / gthr;
    S_t<Pol> *s = reinterpret_cast<S_t<Pol> *>(smem_raw) + l * LS;
    const int line = blockIdx.x * nl + l;
    if (line >= nlines) return;
    for (int k = g.t; k < M; k += g.T) {
        const double2 v = in[(size_t)line * M + k];
        s[pidx<Pol>(k)] = Pol::st(cx<R>{Pol::from_io((typename Pol::io_t)v.x), Pol::from_io((typename Pol::io_t)v.y)});
    }
    group_sync(g);
    fft_line<Pol, FWD, EMAX>(s, sc, tw, g);
    for (int k = g.t; k < M; k += g.T) {
        const cx<R> c = Pol::ld(s[pidx<Pol>(k)]);
        out[(size_t)line * M + k] = make_double2((double)Pol::to_io(c.re), (double)Pol::to_io(c.im));
    }
}

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
        body_xf<Pol, kBatchEmax>(static_cast<const io *>(d.rho), W1, nx, ny, hx, d.sc[0], nl, 32, T(d.tw[0]), bx,
                                 by, smem_raw);
    } else if constexpr (PASS == last) {
        body_xi<Pol, kBatchEmax, true>(W1, static_cast<io *>(d.u), nx, ny, hx, d.sci[0], nl, 32, T(d.twi[0]), bx,
                                       by, smem_raw);
    } else if constexpr (D == 2) {
        body_conv<Pol, kBatchEmax, true>(W1, mult, hx, ny, 0, 1, ny + 1, d.sc[1], d.sci[1], nl, 32, T(d.tw[1]),
                                         T(d.twi[1]), bx, smem_raw, d.full != 0);
    } else if constexpr (PASS == 1) {
        body_yf<Pol, kBatchEmax, true>(W1, W2, ny, nz, hx, d.sc[1], nl, 32, T(d.tw[1]), bx, by, smem_raw);
    } else if constexpr (PASS == 2) {
        body_conv<Pol, kBatchEmax, true>(W2, mult, hx * d.M[1], nz, 1, d.M[1], ny + 1, d.sc[2], d.sci[2], nl, 32,
                                         T(d.tw[2]), T(d.twi[2]), bx, smem_raw, d.full != 0);
    } else {
        body_yi<Pol, kBatchEmax, true>(W2, W1, ny, nz, hx, d.sci[1], nl, 32, T(d.twi[1]), bx, by, smem_raw);
    }
}

// ------------------------------------------------------------------ tables
// w[m] = exp(-2 pi i m / M) from sincospi in FP64, rounded to FP32.
__global__ void k_twiddles(int M, float2 *out)
{
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= M) return;
    double sn, cs;
    sincospi(2.0 * m / M, &sn, &cs);
    out[m] = make_float2((float)cs, (float)-sn);
}

__global__ void k_mult_convert(const double *in, size_t count, float *out)
{
    const size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (i < count) out[i] = (float)in[i];
}

// Twiddle table of a schedule in the precision of Pol: bytes, and its filling.
// FX: in stage order, then `plain` entries w_plain_m^i for the split 2D passes;
// FP32: the M twiddles in order, then, with plain = M, the same in stage order
// for the fixed-length kernels.
template <class Pol>
size_t table_bytes(const Sched &sc, int plain)
{
    if constexpr (std::is_same<Pol, FX>::value) return fx_table_bytes(sc.M, plain);
    else return sizeof(float2) * (sc.M + (size_t)plain);
}
template <class Pol>
void fill_table(const Sched &sc, int plain, int plain_m, void *out, cudaStream_t st)
{
    if constexpr (std::is_same<Pol, FX>::value) launch_fx_twiddles(sc, plain, plain_m, out, st);
    else k_twiddles<<<(sc.M + 255) / 256, 256, 0, st>>>(sc.M, static_cast<float2 *>(out));
    if (std::is_same<Pol, F32>::value && plain > 0) launch_f32_stage_twiddles(sc, static_cast<float2 *>(out) + sc.M, st);
}
size_t plan_table_bytes(const Plan *p, const Sched &sc, int plain)
{
    return p->opt.precision == GSM_FP32 ? table_bytes<F32>(sc, plain) : table_bytes<FX>(sc, plain);
}
void fill_plan_table(const Plan *p, const Sched &sc, int plain, int plain_m, void *out, cudaStream_t st)
{
    if (p->opt.precision == GSM_FP32) fill_table<F32>(sc, plain, plain_m, out, st);
    else fill_table<FX>(sc, plain, plain_m, out, st);
}

// ------------------------------------------------------------------ Hartree energy
template <class T>
__global__ void k_psi_to_rho(const T *__restrict__ psi, T *__restrict__ rho, size_t N)
{
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < N; i += (size_t)gridDim.x * blockDim.x) {
        const T a = psi[2 * i], b = psi[2 * i + 1];
        rho[i] = a * a + b * b;
    }
}

// partial[block] = sum |psi|^2 u ; grad = 2 h^3 u psi
template <class T>
__global__ void k_energy_grad(const T *__restrict__ psi, const T *__restrict__ u, T *__restrict__ grad,
                              double cell, size_t N, double *partial)
{
    __shared__ double red[256];
    double acc = 0.0;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < N; i += (size_t)gridDim.x * blockDim.x) {
        const double a = psi[2 * i], b = psi[2 * i + 1], v = u[i];
        acc += (a * a + b * b) * v;
        if (grad) {
            grad[2 * i] = (T)(2.0 * cell * v * a);
            grad[2 * i + 1] = (T)(2.0 * cell * v * b);
        }
    }
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int off = blockDim.x / 2; off > 0; off >>= 1) {
        if (threadIdx.x < off) red[threadIdx.x] += red[threadIdx.x + off];
        __syncthreads();
    }
    if (threadIdx.x == 0) partial[blockIdx.x] = red[0];
}

template <class T>
__global__ void k_energy_final(const double *partial, int nparts, double cell, T *energy)
{
    __shared__ double red[256];
    double acc = 0.0;
    for (int i = threadIdx.x; i < nparts; i += blockDim.x) acc += partial[i];
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int off = blockDim.x / 2; off > 0; off >>= 1) {
        if (threadIdx.x < off) red[threadIdx.x] += red[threadIdx.x + off];
        __syncthreads();
    }
    if (threadIdx.x == 0) *energy = (T)(0.5 * cell * red[0]);
}

constexpr int kEnergyBlocks = 1024;

// Launch shape for lines of length M: emax elements per thread (8 or 16),
// gthr = threads per line (a multiple of 32 with gthr * emax >= M), nl lines
// (groups) per CTA, nthr = nl * gthr <= kMaxThreads.  Groups larger than a
// warp in a CTA of several groups use named barriers 1..nl (nl <= 15).
template <class Pol>
constexpr int max_threads(int emax) { return std::is_same<Pol, FX>::value ? fx_threads(emax) : kMaxThreads; }

inline int round32(int x) { return ((x + 31) / 32) * 32; }

template <class Pol>
bool make_cfg(int M, int nl, int emax, PassCfg *c)
{
    const int gthr = std::max(32, round32((M + emax - 1) / emax));
    const int maxt = max_threads<Pol>(emax);
    if (gthr > maxt || nl < 1 || nl * gthr > maxt) return false;
    if (gthr > 32 && nl > 1 && nl > 15) return false;
    if (pass_smem<Pol>(M, nl) > 200 * 1024) return false;
    c->nl = nl;
    c->gthr = gthr;
    c->nthr = nl * gthr;
    c->emax = emax;
    c->smem = pass_smem<Pol>(M, nl);
    return true;
}

// Default shape before any tuning: 8 elements per thread when a line fits
// 512 threads that way, else 16; as many lines as requested that fit.
template <class Pol>
PassCfg choose_cfg(int M, int nl_want)
{
    PassCfg c;
    const int emax = (M <= 8 * max_threads<Pol>(8)) ? 8 : 16;
    for (int nl = std::max(1, nl_want); nl >= 1; nl /= 2)
        if (make_cfg<Pol>(M, nl, emax, &c)) return c;
    make_cfg<Pol>(M, 1, 16, &c);
    return c;
}

// Shared-memory limit of the kernel of a pass with shape c.
template <class Pol>
cudaError_t raise_pass_smem(const Plan *p, int pass, const PassCfg &c)
{
    if constexpr (std::is_same<Pol, FX>::value) {
        return fx_raise_smem(p, pass, c);
    } else {
        const int last = p->d == 3 ? 4 : 2;
        cudaError_t e = cudaSuccess;
        with_emax(c, [&](auto E) {
            if (pass == 0) e = raise_smem(k_xf<Pol, E()>, c.smem);
            else if (pass == last) e = raise_smem(k_xi<Pol, E()>, c.smem);
            else if (p->d == 2 || pass == 2) e = raise_smem(k_conv<Pol, E()>, c.smem);
            else if (pass == 1) e = raise_smem(k_yf<Pol, E()>, c.smem);
            else e = raise_smem(k_yi<Pol, E()>, c.smem);
        });
        return e;
    }
}
template <class Pol>
cudaError_t raise_split_smem(bool conv, int half, size_t smem)
{
    if constexpr (std::is_same<Pol, FX>::value) return fx_raise_split_smem(conv, half, smem);
    else if (conv) return raise_smem(k_conv_split<Pol, 16>, smem);
    else return raise_smem(k_xf_split<Pol, 16>, smem);
}

// Line exponents of a fixed-point plan: they follow the values of W1 in its
// allocation.
size_t fx_exp_count(const Plan *p)
{
    const size_t ny2 = (p->n[1] + 1) / 2, hx = p->n[0] + 1;
    if (p->d == 2) return 2 * ny2 + hx;
    return p->n[2] * ny2 + hx * p->n[2] + hx * p->M[1] + p->n[2] * hx;
}
FxExps fx_exps(const Plan *p)
{
    const size_t ny2 = (p->n[1] + 1) / 2, hx = p->n[0] + 1, nz = p->d == 3 ? p->n[2] : 1;
    FxExps e;
    e.xf = reinterpret_cast<int *>(static_cast<fxc *>(p->d_work1) + nz * hx * p->n[1]);
    e.xf_par = 0;
    if (p->d == 2) {
        e.xf_par = p->split_x ? (int)ny2 : 0;
        e.cv = e.xf + 2 * ny2;
        e.yf = e.yi = nullptr;
        return e;
    }
    e.yf = e.xf + nz * ny2;
    e.cv = e.yf + hx * nz;
    e.yi = e.cv + hx * p->M[1];
    return e;
}

template <class Pol>
gsm_status_t configure_t(Plan *p)
{
    const int cw = (int)(128 / sizeof(S_t<Pol>));   // complex values per 128 bytes
    const int d = p->d;
    p->cfg_xf = choose_cfg<Pol>(p->M[0], std::max(1, cw / 2));
    p->cfg_xi = p->cfg_xf;
    if (d == 3) {
        p->cfg_yf = choose_cfg<Pol>(p->M[1], cw);
        p->cfg_yi = p->cfg_yf;
        p->cfg_conv = choose_cfg<Pol>(p->M[2], std::max(1, 4096 / p->M[2]));
    } else {
        p->cfg_conv = choose_cfg<Pol>(p->M[1], std::max(1, 4096 / p->M[1]));
        // long lines: two half-length transforms per line on a cluster of two CTAs
        // (options.debug bit 1 keeps one CTA per line, for comparisons)
        p->split_conv = p->M[1] >= kSplitMinM && (p->opt.debug & 2) == 0;
        if (p->split_conv) {
            if (!make_cfg<Pol>(p->M[1] / 2, 1, 16, &p->cfg_split) || p->cfg_split.nthr > kSplitThreads) {
                set_error("no launch shape for the split conv pass");
                return GSM_ERR_UNSUPPORTED_SIZE;
            }
            GSM_CUDA_TRY(raise_split_smem<Pol>(true, p->M[1] / 2, p->cfg_split.smem));
        }
        // the same for the x forward pass
        p->split_x = p->M[0] >= kSplitMinM && p->M[0] == 2 * p->n[0] && (p->opt.debug & 2) == 0;
        if (p->split_x) {
            if (!make_cfg<Pol>(p->M[0] / 2, 1, 16, &p->cfg_xsplit) || p->cfg_xsplit.nthr > kSplitThreads) {
                set_error("no launch shape for the split x pass");
                return GSM_ERR_UNSUPPORTED_SIZE;
            }
            GSM_CUDA_TRY(raise_split_smem<Pol>(false, p->M[0] / 2, p->cfg_xsplit.smem));
        }
    }
    cudaError_t e = cudaSuccess;
    auto chk = [&](cudaError_t x) { if (e == cudaSuccess) e = x; };
    if (d == 3) {
        const PassCfg *c[5] = {&p->cfg_xf, &p->cfg_yf, &p->cfg_conv, &p->cfg_yi, &p->cfg_xi};
        for (int pass = 0; pass < 5; ++pass) chk(raise_pass_smem<Pol>(p, pass, *c[pass]));
    } else {
        const PassCfg *c[3] = {&p->cfg_xf, &p->cfg_conv, &p->cfg_xi};
        for (int pass = 0; pass < 3; ++pass) chk(raise_pass_smem<Pol>(p, pass, *c[pass]));
    }
    GSM_CUDA_TRY(e);
    // workspace
    const size_t cb = sizeof(S_t<Pol>);
    const size_t hx = p->n[0] + 1;
    if (d == 3) {
        p->work1_bytes = cb * (size_t)p->n[2] * hx * p->n[1];
        p->work2_bytes = cb * hx * (size_t)p->M[1] * p->n[2];
    } else {
        p->work1_bytes = cb * hx * p->n[1];
        p->work2_bytes = 0;
    }
    if constexpr (std::is_same<Pol, FX>::value) p->work1_bytes += sizeof(int) * fx_exp_count(p);
    GSM_CUDA_TRY(dev_alloc(&p->d_work1, p->work1_bytes));
    if (p->work2_bytes) GSM_CUDA_TRY(dev_alloc(&p->d_work2, p->work2_bytes));
    return GSM_OK;
}

// One pass of the apply: 3D passes 0..4 = xf, yf, conv, yi, xi; 2D 0..2 = xf, conv, xi.
PassCfg *pass_cfg(Plan *p, int pass);
bool pass_uses_f3(const Plan *p, int pass);
bool pass_is_split(const Plan *p, int pass);
int f3_radix(int M);
int pass_len(const Plan *p, int pass);
// Calls f(std::integral_constant<int, R>) with the R of padded length M.
template <class F>
void with_f3(int M, F &&f)
{
    switch (f3_radix(M)) {
    case 1: f(std::integral_constant<int, 1>()); break;
    case 2: f(std::integral_constant<int, 2>()); break;
    case 3: f(std::integral_constant<int, 3>()); break;
    case 4: f(std::integral_constant<int, 4>()); break;
    case 5: f(std::integral_constant<int, 5>()); break;
    case 6: f(std::integral_constant<int, 6>()); break;
    case 8: f(std::integral_constant<int, 8>()); break;
    default: break;
    }
}
// What the kernels of the lengths 64 R take of plan p, and one of its passes on
// them; FP32: R <= 6 (n = 256 has the register-resident kernels).
F3Inst f3_inst(const Plan *p, const void *rho, void *u)
{
    return {rho, u, p->d_work1, p->d_work2, p->d_mult, p->d_mrow, p->opt.precision == GSM_FP32 ? FxExps() : fx_exps(p)};
}
void launch_f3(const F3Call &c, int pass)
{
    with_f3(pass_len(c.p, pass), [&](auto R) {
        if (c.p->opt.precision != GSM_FP32) f3_launch<R()>(c, pass);
        else if constexpr (R() != 8) f3f_launch<R()>(c, pass);
    });
}
void launch_f3(const Plan *p, int pass, const void *rho, void *u, cudaStream_t st)
{
    const F3Inst inst = f3_inst(p, rho, u);
    launch_f3({p, &inst, 1, p->d == 3 ? p->n[2] : 1, st}, pass);
}

void launch_pass_f32(const Plan *p, int pass, const void *rho_v, void *u_v, cudaStream_t st)
{
    using Pol = F32;
    using io = typename Pol::io_t;
    using tw = typename Pol::tw_t;
    const io *rho = static_cast<const io *>(rho_v);
    io *u = static_cast<io *>(u_v);
    const int nx = p->n[0], ny = p->n[1], nz = p->d == 3 ? p->n[2] : 1;
    const int hx = nx + 1;
    S_t<Pol> *W1 = static_cast<S_t<Pol> *>(p->d_work1);
    S_t<Pol> *W2 = static_cast<S_t<Pol> *>(p->d_work2);
    const auto *mult = static_cast<const typename Pol::mult_t *>(p->d_mult);
    const tw *twx = static_cast<const tw *>(p->d_tw[0]);
    const tw *twy = static_cast<const tw *>(p->d_tw[1]);
    const tw *twxi = static_cast<const tw *>(p->d_twi[0]);
    const tw *twyi = static_cast<const tw *>(p->d_twi[1]);
    const int last = p->d == 3 ? 4 : 2;
    if (pass_uses_f3(p, pass)) {
        launch_f3(p, pass, rho, u, st);
        return;
    }
    if ((pass == 0 || pass == last) && p->M[0] == 512 && p->rr_conv) {
        if (pass == 0) launch_x_rr512_f32(false, rho, W1, ny, nz, twx, st);
        else launch_x_rr512_f32(true, W1, u, ny, nz, twx, st);
        return;
    }
    if (pass == 0 && p->split_x) {
        const PassCfg &c = p->cfg_xsplit;
        const tw *twh = static_cast<const tw *>(p->d_twxh);
        k_xf_split<Pol, 16><<<2 * ((ny + 1) / 2), c.nthr, c.smem, st>>>(rho, W1, nx, ny, hx, p->sched_xh, twh, twx);
        return;
    }
    if (pass == 0) {
        const PassCfg &c = p->cfg_xf;
        dim3 g((ny + 2 * c.nl - 1) / (2 * c.nl), nz);
        with_emax(c, [&](auto E) {
            k_xf<Pol, E()><<<g, c.nthr, c.smem, st>>>(rho, W1, nx, ny, hx, p->sched_f[0], c.nl, c.gthr, twx);
        });
    } else if (pass == last) {
        const PassCfg &c = p->cfg_xi;
        dim3 g((ny + 2 * c.nl - 1) / (2 * c.nl), nz);
        with_emax(c, [&](auto E) {
            k_xi<Pol, E()><<<g, c.nthr, c.smem, st>>>(W1, u, nx, ny, hx, p->sched_i[0], c.nl, c.gthr, twxi);
        });
    } else if (p->d == 2) {
        const PassCfg &c = p->cfg_conv;
        if (p->M[1] == 512 && p->rr_conv) {
            launch_conv_rr512_f32(W1, mult, hx, 0, 1, ny + 1, p->mult_full, twy, st);
            return;
        }
        if (p->split_conv) {
            const PassCfg &cs = p->cfg_split;
            const tw *th = static_cast<const tw *>(p->d_twh), *thi = static_cast<const tw *>(p->d_twhi);
            k_conv_split<Pol, 16><<<2 * hx, cs.nthr, cs.smem, st>>>(W1, mult, hx, ny + 1, p->sched_hf, p->sched_hi,
                                                                    th, thi, twy, p->mult_full ? 1 : 0);
            return;
        }
        with_emax(c, [&](auto E) {
            k_conv<Pol, E()><<<(hx + c.nl - 1) / c.nl, c.nthr, c.smem, st>>>(
                W1, mult, hx, ny, 0, 1, ny + 1, p->sched_f[1], p->sched_i[1], c.nl, c.gthr, twy, twyi,
                p->mult_full ? 1 : 0);
        });
    } else {
        const tw *twz = static_cast<const tw *>(p->d_tw[2]);
        const tw *twzi = static_cast<const tw *>(p->d_twi[2]);
        const int My = p->M[1];
        if (pass == 1) {
            if (p->M[1] == 512 && p->rr_conv) {
                launch_y_rr512_f32(false, W1, W2, nz, hx, twy, st);
                return;
            }
            const PassCfg &c = p->cfg_yf;
            dim3 g((nz + c.nl - 1) / c.nl, hx);
            with_emax(c, [&](auto E) {
                k_yf<Pol, E()><<<g, c.nthr, c.smem, st>>>(W1, W2, ny, nz, hx, p->sched_f[1], c.nl, c.gthr, twy);
            });
        } else if (pass == 2) {
            const PassCfg &c = p->cfg_conv;
            const int nlines = hx * My;
            if (p->M[2] == 512 && p->rr_conv) {
                launch_conv_rr512_f32(W2, mult, nlines, 1, My, ny + 1, p->mult_full, twz, st);
                return;
            }
            with_emax(c, [&](auto E) {
                k_conv<Pol, E()><<<(nlines + c.nl - 1) / c.nl, c.nthr, c.smem, st>>>(
                    W2, mult, nlines, nz, 1, My, ny + 1, p->sched_f[2], p->sched_i[2], c.nl, c.gthr, twz, twzi,
                    p->mult_full ? 1 : 0);
            });
        } else {
            if (p->M[1] == 512 && p->rr_conv) {
                launch_y_rr512_f32(true, W2, W1, nz, hx, twy, st);
                return;
            }
            const PassCfg &c = p->cfg_yi;
            dim3 g((nz + c.nl - 1) / c.nl, hx);
            with_emax(c, [&](auto E) {
                k_yi<Pol, E()><<<g, c.nthr, c.smem, st>>>(W2, W1, ny, nz, hx, p->sched_i[1], c.nl, c.gthr, twyi);
            });
        }
    }
}

// Fixed point: the kernels are in gsm_fx.cu, gsm_fx_conv.cu and gsm_fx3_*.cu.
void launch_pass_fx(const Plan *p, int pass, const void *rho, void *u, cudaStream_t st)
{
    const FxCall c{p,           fx_exps(p),   static_cast<const double *>(rho), static_cast<double *>(u), p->d_work1,
                   p->d_work2, p->d == 3 ? p->n[2] : 1, st};
    const int conv = p->d == 3 ? 2 : 1;
    if (pass_uses_f3(p, pass)) launch_f3(p, pass, rho, u, st);
    else if (pass_is_split(p, pass)) fx_launch_split(c, pass);
    else if (pass == conv) fx_launch_conv(c, p->cfg_conv);
    else fx_launch_xy(c, pass, *pass_cfg(const_cast<Plan *>(p), pass));
}

template <class Pol>
void launch_pass_t(const Plan *p, int pass, const void *rho_v, void *u_v, cudaStream_t st)
{
    if constexpr (std::is_same<Pol, FX>::value) {
        launch_pass_fx(p, pass, rho_v, u_v, st);
    } else {
        launch_pass_f32(p, pass, rho_v, u_v, st);
    }
}
template <class Pol>
gsm_status_t apply_t(const Plan *p, const void *rho, void *u, cudaStream_t st)
{
    const int np = p->d == 3 ? 5 : 3;
    for (int pass = 0; pass < np; ++pass) launch_pass_t<Pol>(p, pass, rho, u, st);
    GSM_CUDA_TRY(cudaGetLastError());
    return GSM_OK;
}

template <class Pol>
gsm_status_t pass_t(const Plan *p, int pass, const void *rho, void *u, cudaStream_t st)
{
    launch_pass_t<Pol>(p, pass, rho, u, st);
    GSM_CUDA_TRY(cudaGetLastError());
    return GSM_OK;
}

// ------------------------------------------------------------------ autotuning
// Each pass has its own launch shape; the tuner times candidate shapes of
// one pass at a time (the others keep theirs) and keeps the fastest.
PassCfg *pass_cfg(Plan *p, int pass)
{
    if (p->d == 3) {
        PassCfg *c[5] = {&p->cfg_xf, &p->cfg_yf, &p->cfg_conv, &p->cfg_yi, &p->cfg_xi};
        return c[pass];
    }
    PassCfg *c[3] = {&p->cfg_xf, &p->cfg_conv, &p->cfg_xi};
    return c[pass];
}

int pass_len(const Plan *p, int pass)
{
    if (p->d == 3) {
        const int m[5] = {p->M[0], p->M[1], p->M[2], p->M[1], p->M[0]};
        return m[pass];
    }
    const int m[3] = {p->M[0], p->M[1], p->M[0]};
    return m[pass];
}

std::mutex g_tune_mutex;

bool same_sched(const Sched &a, const Sched &b)
{
    if (a.M != b.M || a.nst != b.nst) return false;
    for (int i = 0; i < a.nst; ++i)
        if (a.r[i] != b.r[i]) return false;
    return true;
}

std::string tune_key(const Plan *p, int pass)
{
    cudaDeviceProp prop;
    int dev = 0;
    cudaGetDevice(&dev);
    std::string name = "gpu";
    if (cudaGetDeviceProperties(&prop, dev) == cudaSuccess) name = prop.name;
    for (char &ch : name)
        if (ch == ' ') ch = '_';
    char buf[256];
    // (the version: entries of another were timed on other kernels or another density)
    snprintf(buf, sizeof(buf), "v6 %s p%d d%d n%d,%d,%d pass%d", name.c_str(), (int)p->opt.precision, p->d, p->n[0],
             p->n[1], p->d == 3 ? p->n[2] : 1, pass);
    return buf;
}

std::string sched_str(const Sched &sc)
{
    std::string out;
    for (int i = 0; i < sc.nst; ++i) {
        if (i) out += '.';
        out += std::to_string((int)sc.r[i]);
    }
    return out;
}

bool sched_parse(const char *txt, int M, bool forward, Sched *sc)
{
    int r[kMaxStages], n = 0;
    const char *c = txt;
    while (*c && n < kMaxStages) {
        char *end = nullptr;
        const long v = strtol(c, &end, 10);
        if (end == c) break;
        r[n++] = (int)v;
        c = end;
        if (*c != '.') break;
        ++c;
    }
    return make_sched_order(M, r, n, forward, sc);
}

// The axis whose schedules pass `pass` uses, and which of them: 3D xf, yf
// the forward, xi, yi the inverse, conv both (axis z); 2D xf, xi and conv
// (both, axis y).
void pass_axis(const Plan *p, int pass, int *axis, bool *fwd, bool *inv)
{
    const int last = p->d == 3 ? 4 : 2;
    const int conv = p->d == 3 ? 2 : 1;
    *fwd = *inv = false;
    if (pass == 0) { *axis = 0; *fwd = true; }
    else if (pass == last) { *axis = 0; *inv = true; }
    else if (pass == conv) { *axis = p->d - 1; *fwd = *inv = true; }
    else if (pass == 1) { *axis = 1; *fwd = true; }
    else { *axis = 1; *inv = true; }
}

// FP32 passes with padded length 512 run register-resident kernels with a
// fixed decomposition: no schedule to choose.
bool pass_uses_rr(const Plan *p, int pass)
{
    int axis;
    bool f, i;
    pass_axis(p, pass, &axis, &f, &i);
    return p->opt.precision == GSM_FP32 && p->rr_conv && p->M[axis] == 512;
}

// The split 2D passes have a fixed launch shape and half-length schedules of
// their own.  The inverse x pass is split in fixed point only (a whole FP32 line
// takes half the shared memory), and not with a schedule that was set or tuned.
bool pass_is_split(const Plan *p, int pass)
{
    if (p->d != 2) return false;
    Sched def;
    if (pass == 2)
        return p->split_x && p->opt.precision != GSM_FP32 && make_sched(p->M[0], &def) && same_sched(p->sched_i[0], def);
    return pass == 1 ? p->split_conv : p->split_x;
}

// Factorisations of M into radices 8, 4, 2, 5, 3 in the order fft_line runs
// them, with at most one stage more than the default schedule; the default
// first, at most `cap`.
void factorise(int M, int from_rank, std::vector<int> &cur, int max_st, std::vector<std::vector<int>> &out)
{
    static const int radices[5] = {8, 4, 2, 5, 3};
    if (M == 1) {
        out.push_back(cur);
        return;
    }
    if ((int)cur.size() >= max_st) return;
    for (int k = from_rank; k < 5; ++k)
        if (M % radices[k] == 0) {
            cur.push_back(radices[k]);
            factorise(M / radices[k], k, cur, max_st, out);
            cur.pop_back();
        }
}

std::vector<Sched> sched_factorisations(int M, size_t cap)
{
    Sched def;
    std::vector<Sched> out;
    if (!make_sched(M, &def)) return out;
    out.push_back(def);
    std::vector<std::vector<int>> all;
    std::vector<int> cur;
    factorise(M, 0, cur, def.nst + 1, all);
    std::sort(all.begin(), all.end(), [](const std::vector<int> &x, const std::vector<int> &y) {
        return x.size() < y.size();
    });
    for (const auto &f : all) {
        if (out.size() >= cap) break;
        Sched sc;
        if (!make_sched_order(M, f.data(), (int)f.size(), true, &sc)) continue;
        bool seen = false;
        for (const Sched &o : out) seen |= same_sched(o, sc);
        if (!seen) out.push_back(sc);
    }
    return out;
}

// The inverse schedule whose first stage fuses with the last stage of the
// forward f: f's last radix, then f's other radices in run order.
Sched fused_inverse(const Sched &f)
{
    Sched i = f;
    i.r[0] = f.r[f.nst - 1];
    for (int k = 0; k + 1 < f.nst; ++k) i.r[k + 1] = f.r[k];
    set_pad(&i);
    return i;
}

// Default schedules of an axis: engine order; the conv axis's inverse starts
// with the forward's last radix (fused with the multiplication) in fixed point.
Sched default_sched(const Plan *p, int axis, bool inverse)
{
    Sched sc;
    make_sched(p->M[axis], &sc);
    if (inverse && axis == p->d - 1 && p->opt.precision != GSM_FP32) return fused_inverse(sc);
    return sc;
}

// R of the fixed-length kernels (gsm_fx3.cuh) for padded length M (0: none)
int f3_radix(int M)
{
    const int R = M / 64;
    return M % 64 == 0 && (R == 1 || R == 2 || R == 3 || R == 4 || R == 5 || R == 6 || R == 8) ? R : 0;
}

// Their stages: 8 8 R forward and in the inverse x and y passes, R 8 8 in the conv's inverse.
Sched f3_sched(int M, bool conv_inverse)
{
    const int R = f3_radix(M);
    Sched sc{};
    sc.M = M;
    sc.nst = R == 1 ? 2 : 3;
    for (int i = 0; i < sc.nst; ++i) sc.r[i] = 8;
    if (R > 1) sc.r[conv_inverse ? 0 : 2] = (unsigned char)R;
    set_pad(&sc);
    return sc;
}

// Whether the passes of (axis, inverse?) run them: a length of theirs and the
// default schedules (schedules that were set or tuned run the
// general kernels).  options.debug bit 2 turns them off, for comparisons.  The
// conv pass takes both directions.
bool uses_f3(const Plan *p, int axis, bool inverse)
{
    if ((p->opt.debug & 4) != 0 || f3_radix(p->M[axis]) == 0) return false;
    // FP32: n = 256 has the register-resident kernels, or the shared-memory engine asked for
    if (p->opt.precision == GSM_FP32 && (p->M[axis] == 512 || !p->rr_conv)) return false;
    // (a conv inverse in engine order is what plans saved by earlier versions hold)
    const bool f = same_sched(p->sched_f[axis], default_sched(p, axis, false));
    const bool i = same_sched(p->sched_i[axis], default_sched(p, axis, true)) ||
                   same_sched(p->sched_i[axis], default_sched(p, axis, false));
    return axis == p->d - 1 ? f && i : inverse ? i : f;
}
bool pass_uses_f3(const Plan *p, int pass)
{
    int axis;
    bool f, i;
    pass_axis(p, pass, &axis, &f, &i);
    return uses_f3(p, axis, i);
}

// Candidate (forward, inverse) schedules of pass `pass`, the current pair
// first: single-direction passes vary their own direction over the
// factorisations of M; the conv pass tries, for each factorisation, the
// inverse whose first stage fuses with the forward's last, and the same
// order both ways.
std::vector<std::pair<Sched, Sched>> sched_candidates(const Plan *p, int pass)
{
    int axis;
    bool f, i;
    pass_axis(p, pass, &axis, &f, &i);
    const int M = p->M[axis];
    std::vector<std::pair<Sched, Sched>> out;
    out.push_back({p->sched_f[axis], p->sched_i[axis]});
    auto add = [&](const Sched &a, const Sched &b) {
        if (!axis_pair_ok(p, axis, a, b)) return;
        for (const auto &o : out)
            if (same_sched(o.first, a) && same_sched(o.second, b)) return;
        out.push_back({a, b});
    };
    const std::vector<Sched> fz = sched_factorisations(M, 6);
    if (f && i) {
        for (const Sched &a : fz) {
            if (a.nst >= 2) add(a, fused_inverse(a));
            add(a, a);
        }
    } else if (f) {
        for (const Sched &a : fz) add(a, p->sched_i[axis]);
    } else {
        for (const Sched &b : fz) add(p->sched_f[axis], b);
    }
    return out;
}

gsm_status_t apply_axis_pair(Plan *p, int axis, const Sched &a, const Sched &b, cudaStream_t st)
{
    if (same_sched(p->sched_f[axis], a) && same_sched(p->sched_i[axis], b)) return GSM_OK;
    return set_axis_pair(p, axis, a, b, st);
}

bool cache_lookup(const char *path, const std::string &key, int *nl, int *emax, std::string *fs, std::string *is)
{
    FILE *f = fopen(path, "r");
    if (!f) return false;
    char line[512];
    bool hit = false;
    while (fgets(line, sizeof(line), f)) {
        const size_t kl = key.size();
        if (strncmp(line, key.c_str(), kl) == 0 && line[kl] == ' ') {
            int a = 0, b = 0;
            char sf[64] = {0}, si[64] = {0};
            if (sscanf(line + kl, " nl=%d emax=%d f=%63s i=%63s", &a, &b, sf, si) == 4) {
                *nl = a;
                *emax = b;
                *fs = sf;
                *is = si;
                hit = true;
            }
        }
    }
    fclose(f);
    return hit;
}

template <class Pol>
float time_pass(const Plan *p, int pass, const void *rho, void *u, cudaStream_t st, cudaEvent_t e0, cudaEvent_t e1,
                cudaError_t *err)
{
    launch_pass_t<Pol>(p, pass, rho, u, st);
    cudaEventRecord(e0, st);
    for (int r = 0; r < 3; ++r) launch_pass_t<Pol>(p, pass, rho, u, st);
    cudaEventRecord(e1, st);
    *err = cudaEventSynchronize(e1);
    if (*err == cudaSuccess) *err = cudaGetLastError();
    float ms = 0.f;
    if (*err == cudaSuccess) cudaEventElapsedTime(&ms, e0, e1);
    return ms / 3.f;
}

// The density that candidates are timed on: white noise in [-1, 1).  On zeros the
// fixed-point passes would skip the shifts that bring a line into range.
template <class T>
__global__ void k_noise(T *rho, size_t N)
{
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < N; i += (size_t)gridDim.x * blockDim.x) {
        unsigned h = (unsigned)i * 2654435761u;
        h ^= h >> 15;
        h *= 2246822519u;
        h ^= h >> 13;
        rho[i] = (T)((double)(int)h * 0x1p-31);
    }
}

template <class Pol>
gsm_status_t autotune_t(Plan *p, cudaStream_t st, std::string *report)
{
    using io = typename Pol::io_t;
    size_t N = 1;
    for (int a = 0; a < p->d; ++a) N *= (size_t)p->n[a];
    DevTemp rho_buf, u_buf;
    GSM_CUDA_TRY(dev_alloc(&rho_buf.p, N * sizeof(io)));
    GSM_CUDA_TRY(dev_alloc(&u_buf.p, N * sizeof(io)));
    void *rho = rho_buf.p, *u = u_buf.p;
    k_noise<<<1024, 256, 0, st>>>(static_cast<io *>(rho), N);
    GSM_CUDA_TRY(cudaGetLastError());
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    cudaError_t e = cudaEventCreate(&e0);
    if (e == cudaSuccess) e = cudaEventCreate(&e1);
    const char *cache = getenv("GSM_AUTOTUNE_CACHE");
    const int np = p->d == 3 ? 5 : 3;
    char buf[320];
    gsm_status_t s = GSM_OK;
    Sched keep_f[3], keep_i[3];   // put back if the tuning fails part-way
    for (int a = 0; a < p->d; ++a) {
        keep_f[a] = p->sched_f[a];
        keep_i[a] = p->sched_i[a];
    }
    if (e == cudaSuccess)
        for (int pass = 0; pass < np; ++pass) launch_pass_t<Pol>(p, pass, rho, u, st);
    for (int pass = 0; pass < np && e == cudaSuccess && s == GSM_OK; ++pass) {
        PassCfg *cfg = pass_cfg(p, pass);
        const int M = pass_len(p, pass);
        int axis;
        bool df, di;
        pass_axis(p, pass, &axis, &df, &di);
        const std::string key = tune_key(p, pass);
        int cnl = 0, cem = 0;
        std::string cf, ci;
        if (cache) {
            std::lock_guard<std::mutex> lock(g_tune_mutex);
            PassCfg c;
            Sched a, b;
            if (cache_lookup(cache, key, &cnl, &cem, &cf, &ci) && make_cfg<Pol>(M, cnl, cem, &c) &&
                sched_parse(cf.c_str(), p->M[axis], true, &a) && sched_parse(ci.c_str(), p->M[axis], false, &b) &&
                raise_pass_smem<Pol>(p, pass, c) == cudaSuccess) {
                s = apply_axis_pair(p, axis, df ? a : p->sched_f[axis], di ? b : p->sched_i[axis], st);
                if (s != GSM_OK) break;
                *cfg = c;
                snprintf(buf, sizeof(buf), "pass %d M=%d cached nl=%d gthr=%d emax=%d fwd=%s inv=%s\n", pass, M, c.nl,
                         c.gthr, c.emax, sched_str(p->sched_f[axis]).c_str(), sched_str(p->sched_i[axis]).c_str());
                *report += buf;
                continue;
            }
        }
        if (pass_uses_f3(p, pass)) {
            snprintf(buf, sizeof(buf), "pass %d M=%d fixed-length kernel (fixed schedule and shape)\n", pass, M);
            *report += buf;
            continue;
        }
        if (pass_is_split(p, pass)) {
            snprintf(buf, sizeof(buf), "pass %d M=%d split into two halves on a CTA pair (fixed shape)\n", pass, M);
            *report += buf;
            continue;
        }
        // 1. the radix schedule, with the current launch shape
        if (!pass_uses_rr(p, pass)) {
            const auto cands = sched_candidates(p, pass);
            size_t best_i = 0;
            float best_ms = 1e30f;
            for (size_t ci2 = 0; ci2 < cands.size() && e == cudaSuccess; ++ci2) {
                s = apply_axis_pair(p, axis, cands[ci2].first, cands[ci2].second, st);
                if (s != GSM_OK) break;
                const float ms = time_pass<Pol>(p, pass, rho, u, st, e0, e1, &e);
                if (e != cudaSuccess) break;
                snprintf(buf, sizeof(buf), "pass %d M=%d schedule fwd=%s inv=%s: %.4f ms\n", pass, M,
                         sched_str(cands[ci2].first).c_str(), sched_str(cands[ci2].second).c_str(), ms);
                *report += buf;
                if (ms < best_ms) {
                    best_ms = ms;
                    best_i = ci2;
                }
            }
            if (s != GSM_OK || e != cudaSuccess) break;
            s = apply_axis_pair(p, axis, cands[best_i].first, cands[best_i].second, st);
            if (s != GSM_OK) break;
        }
        // 2. the launch shape (elements per thread, lines per CTA) with that schedule
        PassCfg best = *cfg;
        float best_ms = 1e30f;
        const int nls[] = {1, 2, 3, 4, 6, 8, 12, 16};
        for (int emax : {8, 16}) {
            for (int nl : nls) {
                PassCfg c;
                if (!make_cfg<Pol>(M, nl, emax, &c)) continue;
                if (raise_pass_smem<Pol>(p, pass, c) != cudaSuccess) continue;
                *cfg = c;
                const float ms = time_pass<Pol>(p, pass, rho, u, st, e0, e1, &e);
                if (e != cudaSuccess) break;
                snprintf(buf, sizeof(buf), "pass %d M=%d nl=%d gthr=%d emax=%d smem=%zu: %.4f ms\n", pass, M, c.nl,
                         c.gthr, c.emax, c.smem, ms);
                *report += buf;
                if (ms < best_ms) {
                    best_ms = ms;
                    best = c;
                }
            }
            if (e != cudaSuccess) break;
        }
        *cfg = best;
        if (cache && e == cudaSuccess) {
            std::lock_guard<std::mutex> lock(g_tune_mutex);
            FILE *f = fopen(cache, "a");
            if (f) {
                fprintf(f, "%s nl=%d emax=%d f=%s i=%s\n", key.c_str(), best.nl, best.emax,
                        sched_str(p->sched_f[axis]).c_str(), sched_str(p->sched_i[axis]).c_str());
                fclose(f);
            }
        }
    }
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    if (s != GSM_OK || e != cudaSuccess) {
        const std::string msg = gsm_last_error();
        for (int a = 0; a < p->d; ++a) apply_axis_pair(p, a, keep_f[a], keep_i[a], st);
        set_error(msg);
    }
    if (s != GSM_OK) return s;
    GSM_CUDA_TRY(e);
    GSM_CUDA_TRY(cudaGetLastError());
    return GSM_OK;
}

template <class Pol>
cudaError_t launch_hook(const PassCfg &c, int nlines, int sign, const Sched &sc, const double *in, double *out,
                        const void *d_tw, cudaStream_t st)
{
    if constexpr (std::is_same<Pol, FX>::value) {
        return fx_launch_hook(c, nlines, sign, sc, in, out, d_tw, st);
    } else {
        const auto *tw = static_cast<const typename Pol::tw_t *>(d_tw);
        const int blocks = (nlines + c.nl - 1) / c.nl;
        const double2 *x = reinterpret_cast<const double2 *>(in);
        double2 *y = reinterpret_cast<double2 *>(out);
        cudaError_t e = cudaSuccess;
        with_emax(c, [&](auto E) {
            auto kernel = sign < 0 ? k_fft_hook<Pol, true, E()> : k_fft_hook<Pol, false, E()>;
            e = raise_smem(kernel, c.smem);
            if (e == cudaSuccess) kernel<<<blocks, c.nthr, c.smem, st>>>(x, y, nlines, sc, c.nl, c.gthr, tw);
        });
        return e;
    }
}

template <class Pol>
gsm_status_t fft_hook_t(int M, int nlines, int sign, const double *in, double *out, cudaStream_t st)
{
    Sched sc;
    if (!make_sched(M, &sc)) {
        set_error("FFT length must be a product of 2, 3, 5 between 2 and 8192");
        return GSM_ERR_UNSUPPORTED_SIZE;
    }
    void *d_tw = nullptr;
    GSM_CUDA_TRY(dev_alloc_async_bytes(&d_tw, table_bytes<Pol>(sc, 0), st));
    fill_table<Pol>(sc, 0, 1, d_tw, st);
    const PassCfg c = choose_cfg<Pol>(M, std::max(1, 2048 / M));
    cudaError_t e = cudaSuccess;
    e = launch_hook<Pol>(c, nlines, sign, sc, in, out, d_tw, st);
    if (e == cudaSuccess) e = cudaGetLastError();
    dev_free_async(d_tw, st);
    GSM_CUDA_TRY(e);
    return GSM_OK;
}

}  // namespace

// ------------------------------------------------------------------ exported
bool make_sched(int M, Sched *s)
{
    if (M < 2 || M > kMaxM) return false;
    s->M = M;
    s->nst = 0;
    int m = M;
    const int order[5] = {8, 4, 2, 5, 3};
    for (int r : order) {
        while (m % r == 0) {
            if (s->nst >= kMaxStages) return false;
            s->r[s->nst++] = r;
            m /= r;
        }
    }
    set_pad(s);
    return m == 1;
}

size_t cplx_bytes(gsm_precision_t prec) { return prec == GSM_FP32 ? 8 : 16; }

namespace {

// The stages that the passes of (axis, inverse?) run: those of the schedule, or
// those of the fixed-length kernels where they serve.
Sched run_sched(const Plan *p, int axis, bool inverse)
{
    if (uses_f3(p, axis, inverse)) return f3_sched(p->M[axis], inverse && axis == p->d - 1);
    return inverse ? p->sched_i[axis] : p->sched_f[axis];
}

// Whether the table made for (M, schedule a) serves (M, schedule b): equal M
// and, where tables are in stage order, equal schedules.
bool table_serves(const Plan *p, const Sched &a, const Sched &b)
{
    return a.M == b.M && ((p->opt.precision == GSM_FP32 && (f3_radix(a.M) == 0 || a.M == 512)) || same_sched(a, b));
}

// Entries after the first M of the table of (axis, inverse?), see fill_table:
// FP32, the stage-ordered ones of the fixed-length kernels; fixed point, the
// first M / 2 twiddles in order for the split 2D passes.
int table_plain(const Plan *p, int axis, bool inverse)
{
    const int M = p->M[axis];
    if (p->opt.precision == GSM_FP32) return uses_f3(p, axis, inverse) ? M : 0;
    return p->d == 2 && M >= kSplitMinM ? M / 2 : 0;
}

// The table of (axis, inverse?): an existing table that serves it, or a new one.
gsm_status_t table_for(Plan *p, int axis, bool inverse, cudaStream_t st, void **out)
{
    const Sched want = run_sched(p, axis, inverse);
    const int plain = table_plain(p, axis, inverse);
    for (int b = 0; b < p->d; ++b) {
        if (p->d_tw[b] && table_serves(p, run_sched(p, b, false), want) && table_plain(p, b, false) >= plain && !(b == axis && inverse == false)) {
            *out = p->d_tw[b];
            return GSM_OK;
        }
        if (p->d_twi[b] && table_serves(p, run_sched(p, b, true), want) && table_plain(p, b, true) >= plain && !(b == axis && inverse == true)) {
            *out = p->d_twi[b];
            return GSM_OK;
        }
    }
    const int M = want.M;
    void *t = nullptr;
    GSM_CUDA_TRY(dev_alloc(&t, plan_table_bytes(p, want, plain)));
    fill_plan_table(p, want, plain, M, t, st);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        dev_free(t);
        GSM_CUDA_TRY(e);
    }
    *out = t;
    return GSM_OK;
}

// Frees the table t unless a table slot of the plan still holds it.
void release_table(Plan *p, void *t)
{
    if (!t) return;
    for (int b = 0; b < 3; ++b)
        if (p->d_tw[b] == t || p->d_twi[b] == t) return;
    dev_free(t);
}

}  // namespace

gsm_status_t make_twiddles(Plan *p, int axis, cudaStream_t st)
{
    void *old_f = p->d_tw[axis], *old_i = p->d_twi[axis];
    p->d_tw[axis] = p->d_twi[axis] = nullptr;
    void *tf = nullptr, *ti = nullptr;
    gsm_status_t s = table_for(p, axis, false, st, &tf);
    if (s != GSM_OK) {
        p->d_tw[axis] = old_f;
        p->d_twi[axis] = old_i;
        return s;
    }
    p->d_tw[axis] = tf;
    s = table_for(p, axis, true, st, &ti);
    if (s != GSM_OK) {
        p->d_tw[axis] = old_f;
        p->d_twi[axis] = old_i;
        release_table(p, tf);
        return s;
    }
    p->d_twi[axis] = ti;
    // the device may still run work that reads the old tables: wait before freeing
    if ((old_f && old_f != tf && old_f != ti) || (old_i && old_i != tf && old_i != ti)) {
        GSM_CUDA_TRY(cudaStreamSynchronize(st));
        release_table(p, old_f);
        if (old_i != old_f) release_table(p, old_i);
    }
    return GSM_OK;
}

gsm_status_t make_xsplit_tables(Plan *p, cudaStream_t st)
{
    const int Mh = p->M[0] / 2;
    if (!make_sched(Mh, &p->sched_xh)) {
        set_error("half length of the split x pass is not a product of 2, 3 and 5");
        return GSM_ERR_UNSUPPORTED_SIZE;
    }
    GSM_CUDA_TRY(dev_alloc(&p->d_twxh, plan_table_bytes(p, p->sched_xh, 0)));
    fill_plan_table(p, p->sched_xh, 0, 1, p->d_twxh, st);
    GSM_CUDA_TRY(cudaGetLastError());
    return GSM_OK;
}

gsm_status_t make_split_tables(Plan *p, cudaStream_t st)
{
    const int Mh = p->M[1] / 2;
    if (!make_sched(Mh, &p->sched_hf)) {
        set_error("half length of the split conv is not a product of 2, 3 and 5");
        return GSM_ERR_UNSUPPORTED_SIZE;
    }
    // the inverse starts with the forward's last radix: fused with the multiplication
    p->sched_hi = fused_inverse(p->sched_hf);
    const Sched *sc[2] = {&p->sched_hf, &p->sched_hi};
    void **dst[2] = {&p->d_twh, &p->d_twhi};
    for (int k = 0; k < 2; ++k) {
        if (k == 1 && table_serves(p, p->sched_hf, p->sched_hi)) {
            p->d_twhi = p->d_twh;
            break;
        }
        GSM_CUDA_TRY(dev_alloc(dst[k], plan_table_bytes(p, *sc[k], 0)));
        fill_plan_table(p, *sc[k], 0, 1, *dst[k], st);
        GSM_CUDA_TRY(cudaGetLastError());
    }
    return GSM_OK;
}

bool make_sched_order(int M, const int *radices, int count, bool forward, Sched *s)
{
    if (M < 2 || M > kMaxM || count < 1 || count > kMaxStages || !radices) return false;
    long prod = 1;
    for (int i = 0; i < count; ++i) {
        const int r = radices[i];
        if (r != 8 && r != 4 && r != 2 && r != 5 && r != 3) return false;
        prod *= r;
    }
    if (prod != M) return false;
    if (forward && (radices[0] % 2) != 0) return false;   // the pruned first stage of the zero-padded transform
    s->M = M;
    s->nst = count;
    for (int i = 0; i < kMaxStages; ++i) s->r[i] = (unsigned char)(i < count ? radices[i] : 0);
    set_pad(s);
    return true;
}

// Whether (forward f, inverse i) can run on axis `axis`: the forward and,
// except on the conv axis with a fused middle stage, the inverse in the order
// fft_line runs (8, 4, 2, 5, 3); on the conv axis the inverse may instead
// start with the forward's last radix, that stage being fused.
bool axis_pair_ok(const Plan *p, int axis, const Sched &f, const Sched &i)
{
    if (!sched_sorted_from(f, 0)) return false;
    if (sched_sorted_from(i, 0)) return true;
    return axis == p->d - 1 && fused_radix(f, i) != 0 && sched_sorted_from(i, 1);
}

gsm_status_t set_axis_pair(Plan *p, int axis, const Sched &f, const Sched &i, cudaStream_t st)
{
    if (axis < 0 || axis >= p->d || f.M != p->M[axis] || i.M != p->M[axis]) {
        set_error("schedule does not fit the axis");
        return GSM_ERR_INVALID_ARG;
    }
    if (!axis_pair_ok(p, axis, f, i)) {
        set_error("radices must run in the order 8, 4, 2, 5, 3; only the inverse of the conv axis may start "
                  "with the forward's last radix (fused with the multiplication)");
        return GSM_ERR_INVALID_ARG;
    }
    const Sched old_f = p->sched_f[axis], old_i = p->sched_i[axis];
    p->sched_f[axis] = f;
    p->sched_i[axis] = i;
    gsm_status_t s = make_twiddles(p, axis, st);
    if (s != GSM_OK) {
        p->sched_f[axis] = old_f;
        p->sched_i[axis] = old_i;
    }
    return s;
}

gsm_status_t set_axis_schedule(Plan *p, int axis, bool inverse, const Sched &sc, cudaStream_t st)
{
    if (axis < 0 || axis >= p->d) {
        set_error("axis out of range");
        return GSM_ERR_INVALID_ARG;
    }
    return set_axis_pair(p, axis, inverse ? p->sched_f[axis] : sc, inverse ? sc : p->sched_i[axis], st);
}

gsm_status_t make_pass_multiplier(Plan *p, cudaStream_t st)
{
    if (p->opt.precision != GSM_FP32) {
        // the octant's rows (kx, ky) in 3D, kx in 2D, converted in place
        const int len = p->n[p->d - 1] + 1;
        p->d_mult = p->d_mult64;
        return make_mult_rows(p, p->d_mult64, len, p->mult_elems / len, st);
    }
    GSM_CUDA_TRY(dev_alloc(&p->d_mult, sizeof(float) * p->mult_elems));
    k_mult_convert<<<(p->mult_elems + 255) / 256, 256, 0, st>>>(p->d_mult64, p->mult_elems,
                                                                static_cast<float *>(p->d_mult));
    GSM_CUDA_TRY(cudaGetLastError());
    return GSM_OK;
}

gsm_status_t configure_passes(Plan *p)
{
    for (int a = 0; a < p->d; ++a) {
        if (!make_sched(p->M[a], &p->sched_f[a])) {
            set_error("padded length 2n must be a product of 2, 3 and 5");
            return GSM_ERR_UNSUPPORTED_SIZE;
        }
        p->sched_i[a] = default_sched(p, a, true);
    }
    return p->opt.precision == GSM_FP32 ? configure_t<F32>(p) : configure_t<FX>(p);
}

gsm_status_t launch_apply(const Plan *p, const void *rho, void *u, cudaStream_t st)
{
    return p->opt.precision == GSM_FP32 ? apply_t<F32>(p, rho, u, st) : apply_t<FX>(p, rho, u, st);
}

template <class Pol>
gsm_status_t x_slabs_t(const Plan *p, bool inverse, int z0, int z1, const void *rho_v, void *u_v,
                       cudaStream_t st)
{
    using io = typename Pol::io_t;
    using tw = typename Pol::tw_t;
    const int nx = p->n[0], ny = p->n[1], hx = nx + 1;
    const size_t in_off = (size_t)z0 * ny * nx, w_off = (size_t)z0 * hx * ny;
    S_t<Pol> *W1 = static_cast<S_t<Pol> *>(p->d_work1) + w_off;
    const tw *twx = static_cast<const tw *>(p->d_tw[0]);
    const tw *twxi = static_cast<const tw *>(p->d_twi[0]);
    if (z1 <= z0) return GSM_OK;
    if (pass_uses_f3(p, inverse ? 4 : 0)) {
        F3Inst inst = f3_inst(p, static_cast<const io *>(rho_v) + in_off, static_cast<io *>(u_v) + in_off);
        inst.W1 = W1;
        if constexpr (std::is_same<Pol, FX>::value) {
            inst.ex.xf += (size_t)z0 * ((ny + 1) / 2);
            inst.ex.yi += (size_t)z0 * hx;
        }
        launch_f3({p, &inst, 1, z1 - z0, st}, inverse ? 4 : 0);
        GSM_CUDA_TRY(cudaGetLastError());
        return GSM_OK;
    }
    if constexpr (std::is_same<Pol, FX>::value) {
        FxCall c{p, fx_exps(p), static_cast<const io *>(rho_v) + in_off, static_cast<io *>(u_v) + in_off, W1, nullptr,
                 z1 - z0, st};
        c.ex.xf += (size_t)z0 * ((ny + 1) / 2);
        c.ex.yi += (size_t)z0 * hx;
        fx_launch_xy(c, inverse ? 4 : 0, inverse ? p->cfg_xi : p->cfg_xf);
        GSM_CUDA_TRY(cudaGetLastError());
        return GSM_OK;
    } else {
        if (p->M[0] == 512 && p->rr_conv) {
            if (!inverse) launch_x_rr512_f32(false, static_cast<const io *>(rho_v) + in_off, W1, ny, z1 - z0, twx, st);
            else launch_x_rr512_f32(true, W1, static_cast<io *>(u_v) + in_off, ny, z1 - z0, twx, st);
            GSM_CUDA_TRY(cudaGetLastError());
            return GSM_OK;
        }
        if (!inverse) {
            const PassCfg &c = p->cfg_xf;
            dim3 g((ny + 2 * c.nl - 1) / (2 * c.nl), z1 - z0);
            const io *rho = static_cast<const io *>(rho_v) + in_off;
            with_emax(c, [&](auto E) {
                k_xf<Pol, E()><<<g, c.nthr, c.smem, st>>>(rho, W1, nx, ny, hx, p->sched_f[0], c.nl, c.gthr, twx);
            });
        } else {
            const PassCfg &c = p->cfg_xi;
            dim3 g((ny + 2 * c.nl - 1) / (2 * c.nl), z1 - z0);
            io *u = static_cast<io *>(u_v) + in_off;
            with_emax(c, [&](auto E) {
                k_xi<Pol, E()><<<g, c.nthr, c.smem, st>>>(W1, u, nx, ny, hx, p->sched_i[0], c.nl, c.gthr, twxi);
            });
        }
        GSM_CUDA_TRY(cudaGetLastError());
        return GSM_OK;
    }
}

gsm_status_t launch_x_slabs(const Plan *p, bool inverse, int z0, int z1, const void *rho, void *u, cudaStream_t st)
{
    if (p->d != 3 || z0 < 0 || z1 > p->n[2]) {
        set_error("x slabs: 3D plans and 0 <= z0 <= z1 <= nz only");
        return GSM_ERR_INVALID_ARG;
    }
    return p->opt.precision == GSM_FP32 ? x_slabs_t<F32>(p, inverse, z0, z1, rho, u, st) : x_slabs_t<FX>(p, inverse, z0, z1, rho, u, st);
}

gsm_status_t launch_pass(const Plan *p, int pass, const void *rho, void *u, cudaStream_t st)
{
    return p->opt.precision == GSM_FP32 ? pass_t<F32>(p, pass, rho, u, st) : pass_t<FX>(p, pass, rho, u, st);
}

template <class Pol>
gsm_status_t set_pass_shape_t(Plan *p, int pass, int nl, int emax)
{
    PassCfg c;
    if (!make_cfg<Pol>(pass_len(p, pass), nl, emax, &c)) {
        set_error("launch shape not valid for this pass");
        return GSM_ERR_INVALID_ARG;
    }
    GSM_CUDA_TRY(raise_pass_smem<Pol>(p, pass, c));
    *pass_cfg(p, pass) = c;
    return GSM_OK;
}

gsm_status_t set_pass_shape(Plan *p, int pass, int nl, int emax)
{
    if (pass < 0 || pass >= (p->d == 3 ? 5 : 3)) {
        set_error("pass out of range");
        return GSM_ERR_INVALID_ARG;
    }
    return p->opt.precision == GSM_FP32 ? set_pass_shape_t<F32>(p, pass, nl, emax) : set_pass_shape_t<FX>(p, pass, nl, emax);
}

gsm_status_t autotune_plan(Plan *p, cudaStream_t st, std::string *report)
{
    return p->opt.precision == GSM_FP32 ? autotune_t<F32>(p, st, report) : autotune_t<FX>(p, st, report);
}

gsm_status_t launch_fft_lines(int M, int nlines, int sign, gsm_precision_t prec, const double *in,
                              double *out, cudaStream_t st)
{
    return prec == GSM_FP32 ? fft_hook_t<F32>(M, nlines, sign, in, out, st) : fft_hook_t<FX>(M, nlines, sign, in, out, st);
}

template <class T>
static gsm_status_t hartree_t(Plan *p, const T *psi, T *u, T *energy, T *grad, cudaStream_t st)
{
    size_t N = 1;
    double cell = 1.0;
    for (int a = 0; a < p->d; ++a) {
        N *= (size_t)p->n[a];
        cell *= 2.0 * p->L * p->eta[a] / p->n[a];
    }
    if (!p->d_scratch) {
        GSM_CUDA_TRY(dev_alloc(&p->d_scratch, sizeof(double) * kEnergyBlocks));
        p->scratch_elems = kEnergyBlocks;
    }
    k_psi_to_rho<T><<<kEnergyBlocks, 256, 0, st>>>(psi, u, N);
    gsm_status_t s = launch_apply(p, u, u, st);
    if (s != GSM_OK) return s;
    k_energy_grad<T><<<kEnergyBlocks, 256, 0, st>>>(psi, u, grad, cell, N, p->d_scratch);
    k_energy_final<T><<<1, 256, 0, st>>>(p->d_scratch, kEnergyBlocks, cell, energy);
    GSM_CUDA_TRY(cudaGetLastError());
    return GSM_OK;
}

gsm_status_t launch_hartree(Plan *p, const void *psi, void *u, void *energy, void *grad, cudaStream_t st)
{
    if (p->opt.precision == GSM_FP32)
        return hartree_t<float>(p, (const float *)psi, (float *)u, (float *)energy, (float *)grad, st);
    return hartree_t<double>(p, (const double *)psi, (double *)u, (double *)energy, (double *)grad, st);
}

// ------------------------------------------------------------------ no-allocation FFT
// Scratch of gsm_fft_lines_noalloc: the table of one transform length exactly
// as gsm_fft_lines builds it in its own allocation (16-byte entries in fixed
// point, 8-byte in FP32); the largest, M = 8192, is 131072 bytes.  A
// file-scope __device__ array, so every GPU that loads this library holds these
// 128 KiB until the process exits; every call shares it.
namespace {

constexpr size_t kStaticScratchBytes = 128 * 1024;
__device__ __align__(256) unsigned char g_static_scratch[kStaticScratchBytes];

typedef CUresult (*CtxGetCurrentFn)(CUcontext *);
typedef CUresult (*CtxGetIdFn)(CUcontext, unsigned long long *);

// Identifier of the calling thread's current context (unique for the life of
// the process), or 0 if the driver does not give one.
unsigned long long current_context_id()
{
    static CtxGetCurrentFn get_current = nullptr;
    static CtxGetIdFn get_id = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            get_current = reinterpret_cast<CtxGetCurrentFn>(f);
        f = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            get_id = reinterpret_cast<CtxGetIdFn>(f);
        cudaGetLastError();
    });
    CUcontext ctx = nullptr;
    unsigned long long id = 0;
    if (!get_current || !get_id || get_current(&ctx) != CUDA_SUCCESS || !ctx || get_id(ctx, &id) != CUDA_SUCCESS)
        return 0;
    return id;
}

std::mutex g_static_mutex;
std::vector<std::pair<unsigned long long, void *>> g_static_addr;   // (context id, device address)

// The host-side name g_static_scratch is not a device address.  The device
// address is looked up with cudaGetSymbolAddress, with the caller's device
// current, once per context (device, or a new primary context after
// cudaDeviceReset), and remembered; while no context id is available (before
// the runtime has made one current) it is looked up on every call.
cudaError_t static_scratch_address(void **out)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long ctx = current_context_id();
    std::lock_guard<std::mutex> lock(g_static_mutex);
    if (ctx != 0)
        for (const auto &kv : g_static_addr)
            if (kv.first == ctx) {
                *out = kv.second;
                return cudaSuccess;
            }
    void *p = nullptr;
    e = cudaGetSymbolAddress(&p, g_static_scratch);
    if (e != cudaSuccess) return e;
    if (ctx != 0) g_static_addr.emplace_back(ctx, p);
    *out = p;
    return cudaSuccess;
}

template <class Pol>
gsm_status_t fft_hook_static_t(int M, int nlines, int sign, const double *in, double *out, cudaStream_t st)
{
    Sched sc;
    if (!make_sched(M, &sc)) {
        set_error("FFT length must be a product of 2, 3, 5 between 2 and 8192");
        return GSM_ERR_UNSUPPORTED_SIZE;
    }
    if (table_bytes<Pol>(sc, 0) > kStaticScratchBytes) {
        set_error("FFT tables exceed the 128 KiB static scratch (M <= 8192)");
        return GSM_ERR_UNSUPPORTED_SIZE;
    }
    void *d_tw = nullptr;
    GSM_CUDA_TRY(static_scratch_address(&d_tw));
    // the same tables gsm_fft_lines builds, so the same arithmetic and the same
    // bits; every entry the FFT reads is written here first: nothing needs clearing
    fill_table<Pol>(sc, 0, 1, d_tw, st);
    const PassCfg c = choose_cfg<Pol>(M, std::max(1, 2048 / M));
    cudaError_t e = cudaSuccess;
    e = launch_hook<Pol>(c, nlines, sign, sc, in, out, d_tw, st);
    GSM_CUDA_TRY(e);
    GSM_CUDA_TRY(cudaGetLastError());
    return GSM_OK;
}

}  // namespace

gsm_status_t launch_fft_lines_noalloc(int M, int nlines, int sign, gsm_precision_t prec, const double *in,
                                      double *out, cudaStream_t st)
{
    return prec == GSM_FP32 ? fft_hook_static_t<F32>(M, nlines, sign, in, out, st) : fft_hook_static_t<FX>(M, nlines, sign, in, out, st);
}


// ------------------------------------------------------------------ grouped batch, host side
namespace {

// How a batch applies a plan.
enum class BatchWay { queue, group, alone };

// Padded elements of the conv pass below which a fixed-point plan goes to the
// queue: its kernel runs the transforms of any length, and from there on one launch
// saves less than the kernels of compiled-in lengths do.  Through the queue against
// alone on four streams (Fork), FP64, ms: 3D, 48 of 16^3 (1.7e4 elements) 0.45 / 0.91, 24^3
// (5.8e4) 0.93 / 0.80, 32 of four sizes about 32^3 (1.3e5) 0.96 / 0.61; 2D, with three
// passes instead of five, 48 of 200^2 (8e4) 0.56 / 0.84, 16 of 100x250 (5e4) 0.30 / 0.37.
constexpr size_t queue_max_elems(int d) { return d == 3 ? 1 << 16 : 1 << 18; }

size_t conv_elems(const Plan *p) { return (size_t)(p->n[0] + 1) * p->M[1] * (p->d == 3 ? p->M[2] : 1); }

// Every way gives the bits of gsm_apply.  The queue does for lengths whose kernels
// of their own run the same operations as those of any length: fixed point but for
// n = 192 (stages 8 8 6 instead of 8 8 2 3), FP32 only where there are no such
// kernels.  Plans all of whose passes run on the kernels of the lengths 64 R are
// grouped by size, one launch per pass and size (batch_ways: from kGroupMin plans on
// before the queue).
BatchWay group_way(const Plan *p)
{
    for (int pass = 0; pass < (p->d == 3 ? 5 : 3); ++pass)
        if (!pass_uses_f3(p, pass)) return BatchWay::alone;
    return BatchWay::group;
}
BatchWay batch_way(const Plan *p)
{
    const bool fp32 = p->opt.precision == GSM_FP32;
    const int np = p->d == 3 ? 5 : 3;
    bool some_f3 = false, r6 = false;
    for (int a = 0; a < p->d; ++a)
        if (p->M[a] > kBatchMaxM || (fp32 && p->rr_conv && p->M[a] == 512)) return group_way(p);
    for (int pass = 0; pass < np; ++pass) {
        const bool f3 = pass_uses_f3(p, pass);
        some_f3 |= f3;
        r6 |= f3 && f3_radix(pass_len(p, pass)) == 6;
    }
    return r6 || (fp32 ? some_f3 : conv_elems(p) >= queue_max_elems(p->d)) ? group_way(p) : BatchWay::queue;
}
// whether two plans may be in one group: the same launches but for the arrays
bool same_f3_group(const Plan *a, const Plan *b)
{
    return a->d == b->d && a->n[0] == b->n[0] && a->n[1] == b->n[1] && a->n[2] == b->n[2] &&
           (a->opt.precision == GSM_FP32) == (b->opt.precision == GSM_FP32) && a->mult_full == b->mult_full;
}

// The ways of a batch's plans: plans that may be grouped are, from kGroupMin of one
// size on, also where they could go through the queue, whose kernel runs the
// transforms of any length: 48 plans grouped against queued, FP64, ms: 32^3 0.40 / 1.16,
// 2D 64^2 0.25 / 0.32, 256^2 0.38 / 0.52.  (Fewer cost a launch per pass and size.)
constexpr int kGroupMin = 4;
std::vector<BatchWay> batch_ways(int count, const Plan *const *plans)
{
    std::vector<BatchWay> way(count);
    std::vector<int> can;   // queue or group
    for (int i = 0; i < count; ++i) {
        way[i] = batch_way(plans[i]);
        if (way[i] == BatchWay::queue && group_way(plans[i]) == BatchWay::group) can.push_back(i);
    }
    while (!can.empty()) {   // one size after another
        std::vector<int> same, rest;
        for (int i : can) (same_f3_group(plans[can[0]], plans[i]) ? same : rest).push_back(i);
        if ((int)same.size() >= kGroupMin)
            for (int i : same) way[i] = BatchWay::group;
        can.swap(rest);
    }
    return way;
}

// Streams beside the caller's, for plans that are applied alone and do not fill the
// GPU: forked from the caller's stream and joined to it again within the call (or
// the capture), so that every order the caller sees is that of its own stream.  One
// after another against on four streams, ms: FP32, 32 of four sizes about 32^3 0.97 ->
// 0.52, 8 of 64x36x48 0.50 -> 0.35, 6 of 324^2 0.38 -> 0.26; FP64, 48 of 48^3 2.29 -> 1.24, 16
// of 100^3 3.95 -> 3.43, 4 of 2000^2 (8e6 elements) 3.00 -> 2.65.  Four of 200x128x160
// (1.6e7) fill the GPU each (2.5).
constexpr size_t kForkMaxElems = 1 << 23;
struct Fork {
    static constexpr int kStreams = 4;
    cudaStream_t s[kStreams] = {};
    cudaEvent_t start = nullptr, done[kStreams] = {};
    int n = 0;   // 0: there are none
    ~Fork()
    {
        for (cudaStream_t t : s)
            if (t) cudaStreamDestroy(t);   // once what was queued on it has finished
        for (cudaEvent_t e : done)
            if (e) cudaEventDestroy(e);
        if (start) cudaEventDestroy(start);
    }
    // up to `want` streams that go on where st is; on failure everything stays on st
    cudaError_t open(cudaStream_t st, int want)
    {
        const int k = std::min(want, kStreams);
        bool made = k > 1 && cudaEventCreateWithFlags(&start, cudaEventDisableTiming) == cudaSuccess;
        for (int i = 0; i < k && made; ++i)
            made = cudaStreamCreateWithFlags(&s[i], cudaStreamNonBlocking) == cudaSuccess &&
                   cudaEventCreateWithFlags(&done[i], cudaEventDisableTiming) == cudaSuccess;
        if (!made) {
            cudaGetLastError();
            return cudaSuccess;
        }
        cudaError_t e = cudaEventRecord(start, st);
        for (; n < k && e == cudaSuccess; ++n) e = cudaStreamWaitEvent(s[n], start, 0);
        return e;
    }
    cudaError_t join(cudaStream_t st)
    {
        cudaError_t e = cudaSuccess;
        for (int i = 0; i < n; ++i) {
            cudaError_t x = cudaEventRecord(done[i], s[i]);
            if (x == cudaSuccess) x = cudaStreamWaitEvent(st, done[i], 0);
            if (e == cudaSuccess) e = x;
        }
        n = 0;
        return e;
    }
};

// Tile grid of pass `pass` of plan p for lines-per-CTA nl: (gx, gy).
void pass_grid(const Plan *p, int pass, int nl, int *gx, int *gy)
{
    const int nx = p->n[0], ny = p->n[1], nz = p->d == 3 ? p->n[2] : 1, hx = nx + 1;
    const int last = p->d == 3 ? 4 : 2;
    if (pass == 0 || pass == last) {
        *gx = (ny + 2 * nl - 1) / (2 * nl);
        *gy = nz;
    } else if (p->d == 2) {
        *gx = (hx + nl - 1) / nl;
        *gy = 1;
    } else if (pass == 2 && p->opt.precision != GSM_FP32) {
        *gx = (p->M[1] + nl - 1) / nl;
        *gy = hx;
    } else if (pass == 2) {
        *gx = (hx * p->M[1] + nl - 1) / nl;
        *gy = 1;
    } else {
        *gx = (nz + nl - 1) / nl;
        *gy = hx;
    }
}

std::atomic<unsigned long long> g_batch_wait_ns{kBatchWaitDefaultNs};
std::atomic<int> g_batch_hold{-1};

template <class Pol>
cudaError_t launch_queue_kernel(const QueueArgs &a, size_t smem, cudaStream_t st, bool dry)
{
    if constexpr (std::is_same<Pol, FX>::value) return a.d == 3 ? launch_queue_fx3(a, smem, st, dry) : launch_queue_fx2(a, smem, st, dry);
    else return a.d == 3 ? launch_queue_d<Pol, 3>(a, smem, st, dry) : launch_queue_d<Pol, 2>(a, smem, st, dry);
}

template <class Pol>
gsm_status_t launch_queue_t(QueueArgs &a, const std::vector<const Plan *> &plans, const void *const *rho,
                              void *const *u, cudaStream_t st, bool dry)
{
    const int np = a.d == 3 ? 5 : 3;
    a.npass = np;
    size_t smem = 0;
    for (size_t i = 0; i < plans.size(); ++i) {
        const Plan *p = plans[i];
        InstDesc &d = a.inst[i];
        d.rho = rho[i];
        d.u = u[i];
        d.W1 = p->d_work1;
        d.W2 = p->d_work2;
        d.mult = p->d_mult;
        d.mrow = p->d_mrow;
        if constexpr (std::is_same<Pol, FX>::value) d.ex = fx_exps(p);
        d.full = p->mult_full ? 1 : 0;
        for (int ax = 0; ax < 3; ++ax) {
            d.n[ax] = ax < p->d ? p->n[ax] : 1;
            d.M[ax] = ax < p->d ? p->M[ax] : 1;
            d.tw[ax] = ax < p->d ? p->d_tw[ax] : nullptr;
            d.twi[ax] = ax < p->d ? p->d_twi[ax] : nullptr;
            if (ax < p->d) {
                d.sc[ax] = run_sched(p, ax, false);   // what the tables are made for
                d.sci[ax] = run_sched(p, ax, true);
            }
            if (ax < p->d) smem = std::max(smem, pass_smem<Pol>(p->M[ax], a.nl));
        }
        for (int pass = 0; pass < np; ++pass) {
            int gx, gy;
            pass_grid(p, pass, a.nl, &gx, &gy);
            d.gx[pass] = gx;
        }
    }
    // the queue: pass-major, instances in order within a pass, tiles in order
    int item = 0;
    for (int pass = 0; pass < np; ++pass) {
        a.start[pass] = item;
        a.tiles[pass][0] = 0;
        for (int i = 0; i < a.count; ++i) {
            int gx, gy;
            pass_grid(plans[i], pass, a.nl, &gx, &gy);
            a.tiles[pass][i + 1] = a.tiles[pass][i] + gx * gy;
        }
        item += a.tiles[pass][a.count];
    }
    for (int pass = np; pass <= kBatchPasses; ++pass) a.start[pass] = item;
    a.total = item;
    GSM_CUDA_TRY(launch_queue_kernel<Pol>(a, smem, st, dry));
    return GSM_OK;
}

}  // namespace

size_t batch_state_bytes(int count) { return sizeof(unsigned) * kStateWords * (size_t)std::max(count, 1); }

void set_batch_wait(unsigned long long wait_ns, int hold)
{
    g_batch_wait_ns.store(wait_ns == 0 ? kBatchWaitDefaultNs : wait_ns);
    g_batch_hold.store(hold < 0 ? -1 : hold);
}

namespace {
// The plans that are not done yet.
gsm_status_t launch_rest(int count, const Plan *const *plans, const void *const *rho, void *const *u, int nl,
                         cudaStream_t st, bool dry, unsigned *state, const std::vector<BatchWay> &ways, std::vector<int> &done)
{
    int group = 0;
    for (int i = 0; i < count; ++i) {
        if (done[i]) continue;
        const BatchWay way = ways[i];
        if (way == BatchWay::alone) {
            gsm_status_t s = dry ? GSM_OK : launch_apply(plans[i], rho[i], u[i], st);
            if (s != GSM_OK) return s;
            done[i] = 1;
            continue;
        }
        if (way == BatchWay::group) {
            std::vector<F3Inst> inst;
            for (int j = i; j < count && (int)inst.size() < kF3Group; ++j) {
                if (done[j] || ways[j] != BatchWay::group || !same_f3_group(plans[i], plans[j])) continue;
                inst.push_back(f3_inst(plans[j], rho[j], u[j]));
                done[j] = 1;
            }
            const F3Call c{plans[i], inst.data(), (int)inst.size(), plans[i]->d == 3 ? plans[i]->n[2] : 1, st};
            for (int pass = 0; !dry && pass < (c.p->d == 3 ? 5 : 3); ++pass) launch_f3(c, pass);
            GSM_CUDA_TRY(cudaGetLastError());
            continue;
        }
        std::vector<const Plan *> grp;
        std::vector<const void *> r;
        std::vector<void *> w;
        for (int j = i; j < count && (int)grp.size() < kBatchMax; ++j) {
            if (done[j] || ways[j] != BatchWay::queue) continue;
            if (plans[j]->opt.precision != plans[i]->opt.precision || plans[j]->d != plans[i]->d) continue;
            grp.push_back(plans[j]);
            r.push_back(rho[j]);
            w.push_back(u[j]);
            done[j] = 1;
        }
        QueueArgs *a = new (std::nothrow) QueueArgs();
        if (!a) {
            set_error("host allocation failed");
            return GSM_ERR_OOM;
        }
        a->count = (int)grp.size();
        a->d = plans[i]->d;
        a->nl = nl;
        a->state = state + (size_t)group * kStateWords;
        a->wait_ns = g_batch_wait_ns.load();
        a->hold = g_batch_hold.load();
        ++group;
        gsm_status_t s;
        if (plans[i]->opt.precision == GSM_FP32) s = launch_queue_t<F32>(*a, grp, r.data(), w.data(), st, dry);
        else s = launch_queue_t<FX>(*a, grp, r.data(), w.data(), st, dry);
        delete a;
        if (s != GSM_OK) return s;
    }
    return GSM_OK;
}
}  // namespace

// u[i] = U_i * rho[i]: each plan the way batch_way says, queue launches
// (k_batch_queue) by (precision, dimension) of up to kBatchMax instances, launches
// of up to kF3Group plans of one size, or alone, small ones on streams beside st
// (Fork).  Queue launch g keeps its queue
// state at state + g * kStateWords (batch_state_bytes(count) bytes in all,
// zeroed here first).  dry: only prepare the kernels (shared-memory limits),
// launch nothing.
gsm_status_t launch_batched(int count, const Plan *const *plans, const void *const *rho, void *const *u,
                            int nl, cudaStream_t st, bool dry, unsigned *state)
{
    if (!dry) GSM_CUDA_TRY(cudaMemsetAsync(state, 0, batch_state_bytes(count), st));
    const std::vector<BatchWay> ways = batch_ways(count, plans);
    std::vector<int> done(count, 0), small;
    for (int i = 0; i < count && !dry; ++i)
        if (ways[i] == BatchWay::alone && conv_elems(plans[i]) < kForkMaxElems) small.push_back(i);
    Fork fork;
    cudaError_t forked = fork.open(st, (int)small.size());
    gsm_status_t alone = GSM_OK;
    for (int k = 0; k < (int)small.size() && fork.n > 0 && forked == cudaSuccess && alone == GSM_OK; ++k) {
        const int i = small[k];
        alone = launch_apply(plans[i], rho[i], u[i], fork.s[k % fork.n]);
        done[i] = 1;
    }
    gsm_status_t s = alone;
    if (s == GSM_OK && forked == cudaSuccess) s = launch_rest(count, plans, rho, u, nl, st, dry, state, ways, done);
    const cudaError_t joined = fork.join(st);
    if (s != GSM_OK) return s;
    GSM_CUDA_TRY(forked);
    GSM_CUDA_TRY(joined);
    return GSM_OK;
}

// Status of the queue launches whose queue state is at `state`, read
// after everything queued on `st`: GSM_ERR_TIMEOUT if a bounded wait ran out.
gsm_status_t batch_status(const unsigned *state, int count, cudaStream_t st)
{
    std::vector<unsigned> h(batch_state_bytes(count) / sizeof(unsigned));
    GSM_CUDA_TRY(cudaMemcpyAsync(h.data(), state, batch_state_bytes(count), cudaMemcpyDeviceToHost, st));
    GSM_CUDA_TRY(cudaStreamSynchronize(st));
    for (size_t g = 0; g * kStateWords < h.size(); ++g)
        if (h[g * kStateWords + 1] != 0) {
            set_error("a bounded wait of the batch kernel ran out; this batch's outputs are not valid");
            return GSM_ERR_TIMEOUT;
        }
    return GSM_OK;
}

}  // namespace gsm
