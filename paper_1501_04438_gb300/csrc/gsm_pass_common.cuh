// gsm_pass_common.cuh -- what the pass kernels of both arithmetics share:
// helpers of the kernels, shared-memory limits, and the batch queue kernel.
#pragma once

#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <atomic>
#include <mutex>
#include <new>
#include <string>
#include <vector>
#include <type_traits>

#include <cooperative_groups.h>
#include <cuda.h>

#include "gsm_internal.h"
#include "gsm_fx.cuh"

namespace gsm {

namespace {

constexpr int kMaxThreads = 512;   // CTA size cap: leaves 128 registers per thread

template <class Pol>
using S_t = typename Pol::scplx;

// Read of workspace data.  CG = true (the batch queue kernel, in which the
// workspace is written and read again by other CTAs of the same launch): the
// load bypasses L1 and the read-only path (ld.global.cg), so it sees what
// other CTAs stored before they signalled completion.
template <bool CG, class T>
__device__ __forceinline__ T ldw(const T *p)
{
    if constexpr (CG) return __ldcg(p);
    else return *p;
}

// Copies `count` elements into shared memory with U global loads in flight
// per thread (all U loads are issued before the first store waits for its
// data): for i = t, t + T, ... < count, dst(i, src(i)).  The short FP32 passes
// wait on these loads: 2D 1500x648 takes 98.8 us with U = 1 and a division per
// element, 96.5 with U = 4 and the line fixed per thread.
template <int U, class Val, class Src, class Dst>
__device__ __forceinline__ void gather_smem(int t, int T, int count, Src src, Dst dst)
{
    for (int i0 = t; i0 < count; i0 += U * T) {
        Val v[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (i0 + u * T < count) v[u] = src(i0 + u * T);
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (i0 + u * T < count) dst(i0 + u * T, v[u]);
    }
}

// ------------------------------------------------------------------ batch: one launch, a device work queue
// One launch applies up to kBatchMax plans of different sizes (one precision,
// one dimension).  The work is a queue of items (pass, instance, tile), a
// tile being one CTA's share of that instance's pass grid, in pass-major
// order: every item of pass p comes before every item of pass p + 1.  The
// launch has one CTA per item.  When a CTA starts, its thread 0 takes a ticket
// from an atomic counter (so items go to CTAs in the order the CTAs start,
// whatever their block index), waits until the instance's previous pass is
// complete (a counter of finished tiles per instance and pass), the CTA runs
// the tile with the same pass bodies as the single-plan kernels, and counts it
// as finished.  Each item's dependencies were taken earlier, by CTAs that are
// already resident and whose own dependencies were taken earlier still, so
// the waits always end, however many CTAs are resident.  Passes of different
// instances overlap and no launch boundary drains the GPU between passes.
// Each wait is bounded all the same: when it runs out the CTA records
// GSM_ERR_TIMEOUT in the status word and raises the abort flag, and every
// later CTA returns at once.  Every line is done by one warp holding up to 16
// elements per thread (M <= 512), nl lines per CTA, so one CTA shape serves
// all sizes and passes.  (A loop over items inside long-lived CTAs was tried
// first: with the pass bodies inside a loop the compiler no longer kept their
// butterfly arrays in registers, 3 to 13 KB of stack per thread.)
}  // namespace

constexpr int kBatchMax = 48;
constexpr int kBatchEmax = 16;
constexpr int kBatchMaxM = 32 * kBatchEmax;
constexpr int kBatchPasses = 5;

struct InstDesc {
    const void *rho;
    void *u;
    void *W1, *W2;
    const void *mult;
    const int *mrow;              // FX: exponents of the multiplier rows
    FxExps ex;                    // FX: line exponents
    const void *tw[3], *twi[3];   // forward and inverse tables per axis
    int n[3], M[3];
    Sched sc[3], sci[3];          // forward and inverse schedules per axis
    int gx[kBatchPasses];   // x extent of each pass's tile grid
    int full;               // multiplier over the whole half spectrum
};

// Queue state of one launch in device memory, zeroed before the launch: the
// next item, the status word (0 or GSM_ERR_TIMEOUT), the abort flag, one
// unused word, then the finished-tile counter of each (instance, pass).
constexpr int kStateHeader = 4;
constexpr int kStateWords = kStateHeader + kBatchMax * kBatchPasses;

struct QueueArgs {
    int count, d, nl, npass;
    int total;                                  // items in the queue
    int start[kBatchPasses + 1];                // first item of each pass
    int tiles[kBatchPasses][kBatchMax + 1];     // within a pass: first tile of each instance
    unsigned *state;                            // kStateWords words
    unsigned long long wait_ns;                 // bound of every wait
    int hold;                                   // test hook: this instance's first pass never
                                                // counts as complete (-1: none)
    InstDesc inst[kBatchMax];
};

namespace {

__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ unsigned ld_acquire_gpu(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ unsigned ld_relaxed_gpu(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Thread 0 of the CTA: take the next item and wait for its dependency.
// Returns false when the queue is empty, the batch was aborted or the wait ran
// out; otherwise the item's pass, instance and tile.
__device__ __forceinline__ bool take_item(const QueueArgs &a, int *pass, int *inst, int *tile)
{
    unsigned *next = a.state, *status = a.state + 1, *abort_flag = a.state + 2;
    const unsigned *done = a.state + kStateHeader;
    if (ld_relaxed_gpu(abort_flag) != 0) return false;
    const int item = (int)atomicAdd(next, 1u);
    if (item >= a.total) return false;
    int p = 0;
    while (item >= a.start[p + 1]) ++p;
    const int r = item - a.start[p];
    int i = 0;
    while (r >= a.tiles[p][i + 1]) ++i;
    *pass = p;
    *inst = i;
    *tile = r - a.tiles[p][i];
    if (p == 0) return true;
    const unsigned need = (unsigned)(a.tiles[p - 1][i + 1] - a.tiles[p - 1][i]) + (p == 1 && i == a.hold ? 1u : 0u);
    const unsigned *cnt = done + i * kBatchPasses + (p - 1);
    if (ld_acquire_gpu(cnt) >= need) return true;
    const unsigned long long t0 = global_ns();
    unsigned sleep_ns = 32;
    while (ld_acquire_gpu(cnt) < need) {
        if (ld_relaxed_gpu(abort_flag) != 0) return false;
        if (global_ns() - t0 > a.wait_ns) {
            atomicExch(status, (unsigned)GSM_ERR_TIMEOUT);
            atomicExch(abort_flag, 1u);
            return false;
        }
        __nanosleep(sleep_ns);
        if (sleep_ns < 1024) sleep_ns *= 2;
    }
    return true;
}

// One tile of pass PASS of one instance (defined beside the pass bodies of Pol).
template <class Pol, int D, int PASS>
__device__ __forceinline__ void queue_tile(const InstDesc &d, int nl, int t, unsigned char *smem_raw, int *red);

// Item of a CTA (shared): valid if go != 0.
struct QueueItem {
    int go, pass, inst, tile;
};

// The tile of pass PASS if the CTA's item belongs to that pass, then one
// release of the instance's count for the pass.
template <class Pol, int D, int PASS>
__device__ __forceinline__ void queue_pass(const QueueArgs &a, const QueueItem &it, unsigned char *smem_raw, int *red)
{
    if (it.go && it.pass == PASS) {
        const int i = it.inst;
        queue_tile<Pol, D, PASS>(a.inst[i], a.nl, it.tile, smem_raw, red);
        // every thread's stores of the tile, then one release of the count
        __syncthreads();
        if (threadIdx.x == 0) {
            unsigned *cnt = a.state + kStateHeader + i * kBatchPasses + PASS;
            asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(cnt) : "memory");
        }
    }
}

template <class Pol, int D>
// Resident CTAs per SM asked of the compiler: fixed point 2 (a 128-register
// cap), FP32 5 (51 registers; its tiles are short, and more
// resident CTAs cover their ticket and acquire: measured 4 % faster with 4
// than with 3, 2 % faster again with 5, slower with 6)
__global__ void __launch_bounds__(32 * kBatchMaxLines, std::is_same<Pol, F32>::value ? 5 : 2)
    k_batch_queue(const __grid_constant__ QueueArgs a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ QueueItem it;
    __shared__ int red[kFxRedWords];
    if (threadIdx.x == 0) {
        int p = 0, i = 0, t = 0;
        it.go = take_item(a, &p, &i, &t) ? 1 : 0;
        it.pass = p;
        it.inst = i;
        it.tile = t;
    }
    __syncthreads();
    if (!it.go) return;
    queue_pass<Pol, D, 0>(a, it, smem_raw, red);
    queue_pass<Pol, D, 1>(a, it, smem_raw, red);
    queue_pass<Pol, D, 2>(a, it, smem_raw, red);
    if constexpr (D == 3) {
        queue_pass<Pol, D, 3>(a, it, smem_raw, red);
        queue_pass<Pol, D, 4>(a, it, smem_raw, red);
    }
}

// ------------------------------------------------------------------ launching
// The dynamic shared-memory limit is per kernel function, shared by every
// plan; it is always raised to the device's opt-in maximum (never lowered) so
// that one plan cannot shrink the limit another plan launches with.
template <class K>
cudaError_t raise_smem(K kernel, size_t smem)
{
    if (smem <= 48 * 1024) return cudaSuccess;
    int dev = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return e;
    cudaFuncAttributes fa;
    e = cudaFuncGetAttributes(&fa, kernel);
    if (e != cudaSuccess) return e;
    optin -= (int)fa.sharedSizeBytes;   // the kernel's static shared memory counts too
    if (optin < 0 || (size_t)optin < smem) return cudaErrorInvalidValue;
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
}

template <class Pol>
size_t pass_smem(int M, int nl) { return (size_t)nl * line_stride<Pol>(M) * sizeof(S_t<Pol>); }

// Calls f(std::integral_constant<int, E>) with E = c.emax.
template <class F>
void with_emax(const PassCfg &c, F &&f)
{
    if (c.emax == 8) f(std::integral_constant<int, 8>());
    else f(std::integral_constant<int, 16>());
}

// Launches the queue kernel of Pol (dry: only prepares it).
template <class Pol, int D>
cudaError_t launch_queue_d(const QueueArgs &a, size_t smem, cudaStream_t st, bool dry)
{
    auto kernel = k_batch_queue<Pol, D>;
    cudaError_t e = raise_smem(kernel, smem);
    if (e == cudaSuccess && !dry) {
        // one CTA per item
        kernel<<<std::max(1, a.total), a.nl * 32, smem, st>>>(a);
        e = cudaGetLastError();
    }
    return e;
}

}  // namespace

// its fixed-point form (gsm_fx_queue2d.cu, gsm_fx_queue3d.cu)
cudaError_t launch_queue_fx2(const QueueArgs &a, size_t smem, cudaStream_t st, bool dry);
cudaError_t launch_queue_fx3(const QueueArgs &a, size_t smem, cudaStream_t st, bool dry);

}  // namespace gsm
