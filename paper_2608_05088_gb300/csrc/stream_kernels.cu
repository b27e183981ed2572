// stream_kernels.cu -- standalone launches of the HBM-bound stages of the
// MALT / MALTER step (stats, finalize, prescale, norms, scalars, apply; the
// block bodies and their paper references are in stream_blocks.cuh), plus
// pointer binding and the bounded-wait probe.
//
// All reductions run in a fixed order (no atomics), so a step is bitwise
// reproducible.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <cstdint>

#include "chain.cuh"
#include "common.cuh"
#include "kernels.h"
#include "ptx.cuh"
#include "stream_blocks.cuh"

namespace malt {

namespace {

__device__ __forceinline__ int find_mat(const int32_t* __restrict__ pref, int nmat, int32_t x) {
    int lo = 0, hi = nmat - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(pref + mid) <= x) lo = mid; else hi = mid - 1;
    }
    return lo;
}

}  // namespace

// ---------------------------------------------------------------- binding
__global__ void bind_kernel(const __grid_constant__ BindParams P, UserPtrs* __restrict__ table) {
    chain_wait();
    const int i = after_wait(static_cast<int>(threadIdx.x));
    if (i < P.count) table[P.offset + i] = P.p[i];
}

// ------------------------------------------------------------ pad / unpad
// A block copies kPadRows rows x kPadCols columns of one matrix, a warp per row,
// and the blocks of the matrix's first row band also its l and r.  The rows start at
// any element, so accesses are single elements, coalesced across the lanes; every
// lane has kPadCols / 32 of them in flight per buffer, so that a block waits for
// memory once (a row at a time with one in flight, the two launches of six matrices
// of 77 to 515 rows took 42 us).
// Row segments of W (or G) in either type: 16-bit elements in the low halves of v.
__device__ __forceinline__ void load_any(const void* p, bool half, size_t off, int n, int lane,
                                         uint32_t (&v)[kPadCols / 32]) {
#pragma unroll
    for (int k = 0; k < kPadCols / 32; ++k) {
        const int j = lane + 32 * k;
        if (j < n) v[k] = half ? static_cast<const uint16_t*>(p)[off + j] : static_cast<const uint32_t*>(p)[off + j];
    }
}

__device__ __forceinline__ void store_any(void* p, bool half, size_t off, int n, int lane,
                                          const uint32_t (&v)[kPadCols / 32]) {
#pragma unroll
    for (int k = 0; k < kPadCols / 32; ++k) {
        const int j = lane + 32 * k;
        if (j >= n) continue;
        if (half)
            static_cast<uint16_t*>(p)[off + j] = static_cast<uint16_t>(v[k]);
        else
            static_cast<uint32_t*>(p)[off + j] = v[k];
    }
}

template <bool kIn>
__global__ void __launch_bounds__(32 * kPadRows) pad_kernel(const __grid_constant__ PadParams P) {
    chain_wait();
    int k = 0;
    while (k + 1 < P.count && P.e[k + 1].block_begin <= static_cast<int32_t>(blockIdx.x)) ++k;
    const PadEntry& e = P.e[k];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int local = static_cast<int>(blockIdx.x) - e.block_begin;
    const int segs = (e.n + kPadCols - 1) / kPadCols;
    const int band = local / segs, col = (local - band * segs) * kPadCols;
    const int row = band * kPadRows + warp;
    const int n = min(kPadCols, e.n - col);                       // columns of this block
    if (row < e.m) {
        const size_t u = static_cast<size_t>(row) * e.n + col;      // caller layout, ld = n
        const size_t q = static_cast<size_t>(row) * e.n8 + col;     // padded layout, ld = n8
        uint32_t w[kPadCols / 32], g[kPadCols / 32], m[kPadCols / 32];
        load_any(kIn ? e.w_user : e.w_pad, e.w_bf16, kIn ? u : q, n, lane, w);
        if (kIn) load_any(e.g_user, e.g_bf16, u, n, lane, g);
        load_any(kIn ? e.m_user : e.m_pad, false, kIn ? u : q, n, lane, m);
        store_any(kIn ? e.w_pad : e.w_user, e.w_bf16, kIn ? q : u, n, lane, w);
        if (kIn) store_any(e.g_pad, e.g_bf16, q, n, lane, g);
        store_any(kIn ? e.m_pad : e.m_user, false, kIn ? q : u, n, lane, m);
        if (!kIn && !e.w_bf16 && e.wcopy_user != nullptr) {
            __nv_bfloat16* c = static_cast<__nv_bfloat16*>(e.wcopy_user) + u;
#pragma unroll
            for (int i = 0; i < kPadCols / 32; ++i)
                if (lane + 32 * i < n) c[lane + 32 * i] = __float2bfloat16_rn(__uint_as_float(w[i]));
        }
    }
    if (band == 0) {
        const int stride = segs * blockDim.x, first = (local % segs) * blockDim.x + threadIdx.x;
        for (int i = first; i < e.m; i += stride) {
            if (kIn) e.l_pad[i] = e.l_user[i]; else e.l_user[i] = e.l_pad[i];
        }
        for (int j = first; j < e.n; j += stride) {
            if (kIn) e.r_pad[j] = e.r_user[j]; else e.r_user[j] = e.r_pad[j];
        }
    }
}

// ------------------------------------------------------------------ stats
// The streaming kernels' minimum resident blocks per SM (statistics 3,
// prescale 5 for wide matrices and 4 for tall ones, apply 8) trade registers
// for resident warps: more warps per SM kept more of HBM busy than more loads
// in flight per thread did.  MALTER's prescale also reads G: with G's loads issued
// beside M's at one block per SM less, GPT-2 Medium's takes 478 us (6.3 TB/s)
// where loading G after M's arithmetic took 510, and at 5 blocks 518.
template <bool kStats>
__global__ void __launch_bounds__(256, 3)
stats_kernel(const MatDesc* __restrict__ mats, const UserPtrs* __restrict__ ptrs,
             const int32_t* __restrict__ pref, int nmat, float mu1) {
    __shared__ __align__(16) float colsh[8 * kStatCols];
    chain_wait();
    const int g = after_wait(find_mat(pref, nmat, blockIdx.x));
    blk::stats_block<kStats>(mats[g], ptrs[g], blockIdx.x - __ldg(pref + g), mu1, threadIdx.x,
                             colsh);
}

// --------------------------------------------------------------- finalize
__global__ void __launch_bounds__(256)
finalize_kernel(const MatDesc* __restrict__ mats, const UserPtrs* __restrict__ ptrs,
                const int32_t* __restrict__ pref, int nmat, int32_t total,
                StepHyper hp, StepClock* clock, int identity) {
    chain_wait();
    const int32_t x = blockIdx.x * blockDim.x + threadIdx.x;
    // (the last thread: the launch has one thread more than entries at least)
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == blockDim.x - 1)
        blk::advance_clock(clock, hp.mu1, hp.mu2, hp.eps, hp.malter);
    if (x >= total) return;
    const int g = after_wait(find_mat(pref, nmat, x));
    blk::finalize_entry(mats[g], ptrs[g], x - __ldg(pref + g), hp.mu2, hp.eps, identity);
}

// --------------------------------------------------------------- prescale
// One launch for the wide matrices, one for the tall ones (their NS frame is
// Mt^T, written through shared-memory transposes): ids lists the launch's
// matrices and pref its block prefix.
template <bool kMalter>
__global__ void __launch_bounds__(256, kMalter ? 4 : 5)
prescale_wide_kernel(const MatDesc* __restrict__ mats, const UserPtrs* __restrict__ ptrs,
                     const int32_t* __restrict__ ids, const int32_t* __restrict__ pref, int count) {
    __shared__ float2 red[8];
    chain_wait();
    const int32_t x = blockIdx.x;
    const int k = find_mat(pref, count, x);
    const int g = after_wait(__ldg(ids + k));
    blk::prescale_block<false, kMalter>(mats[g], ptrs[g], x - __ldg(pref + k), threadIdx.x, nullptr, red);
}

template <bool kMalter>
__global__ void __launch_bounds__(256, kMalter ? 3 : 4)
prescale_tall_kernel(const MatDesc* __restrict__ mats, const UserPtrs* __restrict__ ptrs,
                     const int32_t* __restrict__ ids, const int32_t* __restrict__ pref, int count,
                     int32_t base) {
    __shared__ __align__(16) float tile[blk::kPreTileFloats];
    __shared__ float2 red[8];
    chain_wait();
    const int32_t x = base + static_cast<int32_t>(blockIdx.x);   // pref continues the wide launch's
    const int k = find_mat(pref, count, x);
    const int g = after_wait(__ldg(ids + k));
    blk::prescale_block<true, kMalter>(mats[g], ptrs[g], x - __ldg(pref + k), threadIdx.x, tile, red);
}

// ------------------------------------------------------------------ norms
__global__ void __launch_bounds__(256)
norms_kernel(const MatDesc* __restrict__ mats, MatScalars* __restrict__ scal, float ns_eps,
             int malter, SchedCounters sched) {
    __shared__ float red[32];
    chain_wait();
    const int g = after_wait(static_cast<int>(blockIdx.x));
    // The persistent Newton-Schulz launches that follow count from zero.
    for (int s = threadIdx.x; s < sched.stages; s += blockDim.x)
        sched.done[static_cast<size_t>(s) * gridDim.x + g] = 0;
    for (int i = threadIdx.x; g == 0 && i < sched.queues; i += blockDim.x) sched.queue[i] = 0;
    blk::norms_matrix(mats[g], scal + g, ns_eps, malter, threadIdx.x, red);
}

// ---------------------------------------------------------------- scalars
__global__ void __launch_bounds__(blk::kScalarThreads)
scalars_kernel(const MatDesc* __restrict__ mats, MatScalars* __restrict__ scal,
               const StepClock* __restrict__ clock, StepHyper hp) {
    __shared__ float red[32];
    chain_wait();
    const int g = after_wait(static_cast<int>(blockIdx.x));
    blk::scalars_matrix(mats[g], scal + g, after_wait(clock), hp, threadIdx.x, red);
}

// ------------------------------------------------------------------ apply
__global__ void __launch_bounds__(256, 8)
apply_kernel(const MatDesc* __restrict__ mats, const UserPtrs* __restrict__ ptrs,
             const MatScalars* __restrict__ scal, const int32_t* __restrict__ pref, int nmat,
             float decay) {
    chain_wait();
    const int g = after_wait(find_mat(pref, nmat, blockIdx.x));
    blk::apply_block(mats[g], ptrs[g], blockIdx.x - __ldg(pref + g), scal[g].scale, decay,
                     threadIdx.x);
}

// ------------------------------------------------------------- wait probe
// One thread waits on an mbarrier that nothing ever arrives on, for at most
// budget_ns, and records whether the wait gave up.
__global__ void wait_probe_kernel(int32_t* status, uint64_t budget_ns) {
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        fence_barrier_init();
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const bool ok = mbar_wait_bounded(&bar, 0, budget_ns, nullptr);
        *status = ok ? 0 : kStatusTimeout;
    }
}

// ----------------------------------------------------------------- guards
constexpr uint32_t kGuardWord = 0xA5C3E10Fu;

// One block per guard region, one thread per 32-bit word.
__global__ void guard_kernel(uint8_t* base, const uint64_t* __restrict__ offsets, bool check,
                             unsigned long long* bad) {
    uint32_t* g = reinterpret_cast<uint32_t*>(base + offsets[blockIdx.x]);
    const int i = threadIdx.x;
    if (!check) {
        g[i] = kGuardWord;
        return;
    }
    const uint32_t diff = g[i] ^ kGuardWord;
    int nbytes = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) nbytes += ((diff >> (8 * k)) & 0xffu) != 0;
    if (nbytes != 0) atomicAdd(bad, static_cast<unsigned long long>(nbytes));
}

// ------------------------------------------------------------------ launch
cudaError_t launch_bind(const BindParams& P, UserPtrs* table, cudaStream_t s) {
    return launch_chained(bind_kernel, 1, kBindChunk, 0, s, P, table);
}

cudaError_t launch_pad(const PadParams& P, int32_t blocks, bool in, cudaStream_t s) {
    return launch_chained(in ? pad_kernel<true> : pad_kernel<false>, blocks, 32 * kPadRows, 0, s, P);
}

cudaError_t launch_stats(const MatDesc* mats, const UserPtrs* ptrs, const int32_t* pref,
                         int nmat, int32_t blocks, float mu1, int with_stats, cudaStream_t s) {
    return launch_chained(with_stats ? stats_kernel<true> : stats_kernel<false>, blocks, 256, 0, s,
                          mats, ptrs, pref, nmat, mu1);
}

cudaError_t launch_finalize(const MatDesc* mats, const UserPtrs* ptrs, const int32_t* pref,
                            int nmat, int32_t total, const StepHyper& hp, StepClock* clock,
                            int identity, cudaStream_t s) {
    return launch_chained(finalize_kernel, total / 256 + 1, 256, 0, s, mats, ptrs, pref, nmat, total, hp, clock,
                          identity);
}

cudaError_t launch_prescale(const MatDesc* mats, const UserPtrs* ptrs, const int32_t* ids,
                            const int32_t* pref, int wide, int32_t wide_blocks, int tall,
                            int32_t tall_blocks, int malter, cudaStream_t s) {
    if (wide > 0 && wide_blocks > 0) {
        const cudaError_t e = launch_chained(malter ? prescale_wide_kernel<true> : prescale_wide_kernel<false>,
                                             wide_blocks, 256, 0, s, mats, ptrs, ids, pref, wide);
        if (e != cudaSuccess) return e;
    }
    if (tall > 0 && tall_blocks > 0)
        return launch_chained(malter ? prescale_tall_kernel<true> : prescale_tall_kernel<false>, tall_blocks, 256,
                              0, s, mats, ptrs, ids + wide, pref + wide, tall, wide_blocks);
    return cudaSuccess;
}

cudaError_t launch_norms(const MatDesc* mats, MatScalars* scal, int nmat, float ns_eps,
                         int malter, const SchedCounters& sched, cudaStream_t s) {
    return launch_chained(norms_kernel, nmat, 256, 0, s, mats, scal, ns_eps, malter, sched);
}

cudaError_t launch_scalars(const MatDesc* mats, MatScalars* scal, const StepClock* clock,
                           int nmat, const StepHyper& hp, cudaStream_t s) {
    return launch_chained(scalars_kernel, nmat, blk::kScalarThreads, 0, s, mats, scal, clock, hp);
}

cudaError_t launch_apply(const MatDesc* mats, const UserPtrs* ptrs, const MatScalars* scal,
                         const int32_t* pref, int nmat, int32_t blocks, float decay,
                         cudaStream_t s) {
    return launch_chained(apply_kernel, blocks, 256, 0, s, mats, ptrs, scal, pref, nmat, decay);
}

cudaError_t launch_guards(void* base, const uint64_t* offsets, int32_t n, bool check,
                          unsigned long long* bad, cudaStream_t s) {
    guard_kernel<<<n, static_cast<int>(kGuardBytes / 4), 0, s>>>(static_cast<uint8_t*>(base), offsets,
                                                                 check, bad);
    return cudaGetLastError();
}

cudaError_t launch_wait_probe(int32_t* status, uint64_t budget_ns, cudaStream_t s) {
    wait_probe_kernel<<<1, 32, 0, s>>>(status, budget_ns);
    return cudaGetLastError();
}

}  // namespace malt
