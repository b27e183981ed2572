// ns_gemm.cu -- the Newton-Schulz engine: batched same-shape 16-bit GEMMs on the
// sm_103a tensor cores, two SMs per tile (tcgen05.mma.cta_group::2, fp32
// accumulators in TMEM, operands staged into shared memory by TMA with
// 128-byte swizzle).
//
// A Newton-Schulz run (the Orth step of Algorithm 1, run on the wide
// orientation X of Mt, p x q) is a list of products (ns_plan.h): the iterated
// form for nearly square and small frames, the grouped form for the others.  An
// iteration of the iterated form is three of them:
//   kGram  A  = X X^T               (M = N = p, K = q)    operands: rows of X, rows of X
//   kPoly  B' = a I + b A + c A A   (M = N = p, K = p)    operands: rows of A, rows of A (A = A^T)
// A and B' are symmetric, so those two phases compute and store only the tiles
// on and above the diagonal.  Readers take what lies below it from the tile
// above, transposed: the slice is loaded as an MN-major operand (slices_below).
//   kBX    X' = B' X                (M = p, N = q, K = p) operands: rows of B', X read MN-major
// so a X + (b A + c A A) X = B' X with the a X term folded into B' (its error
// is that of the bf16 B it rides on).  The kBX B operand is X itself, read as
// an MN-major [K][N] matrix, so no transposed copy of X is ever written.  The
// grouped form's further p x p products (H A, H A H, the running product of the
// H) are kPoly operations on other buffers, in fp16; they commute with A, so
// they are symmetric too and take the same path.  GPT-2 Large (36 layers, k = 5):
// 17 products in 8.24 ms where the iterated form's 15 take 10.12; one 16384 x 4096
// matrix at k = 8 2.81 where it takes 4.12 ms.  The
// 1/(||Mt||_F + ns_eps) normalisation is folded into the first iteration's
// epilogues (A scaled by k^2, X' by k).  The last product's epilogue writes O
// in W's orientation and per-warp partial sums of O^2 and of D^2 with
// D = L O R (Algorithm 1, D_t line) for the graft.  O is stored in W's layout:
// a tall matrix's tiles go out transposed, so the apply pass streams every
// matrix the same way.
//
// Work split.  A cluster of two CTAs (a CTA pair on two SMs) computes one
// 256 x 256 output tile per turn (256 x 128 in sets of few tiles, build_classes): CTA r owns rows [128 r, 128 r + 128) of the
// tile in its own TMEM.  Per 64-wide reduction slice each CTA loads its 128
// rows of A and its half (128 N-rows or N-columns) of B, 32 KB, into one of
// kStages slice slots; the MMA, issued by one thread of the even CTA, reads
// both CTAs' shared memory.  Each SM therefore pulls 32 KB from L2 per
// 128 x 256 x 64 of MMA work instead of 48 KB (16 KB on a diagonal tile of
// a symmetric product, whose B half is the CTA's own A rows).  The slots are filled,
// awaited and released in groups of kGroup slices (a 3-stage ring of 128-wide
// reductions): every barrier wait and commit on the MMA thread's path stalls
// the tensor pipe a little, and one per 8 MMAs measured 4 % faster on B*X
// than one per 4.
//
// Roles per CTA: warp 0 issues TMA loads (the peer's loads complete on the
// even CTA's full barrier, and both producers arrive on it), warp 1 owns
// TMEM (allocated for the pair) and, in the even CTA, issues tcgen05.mma into
// one of two TMEM accumulators; warps 2-9 drain the other accumulator
// (tcgen05.ld, pipelined per 32-column chunk) and run the epilogue, so the
// epilogue of tile i overlaps the MMAs of tile i+1.  Each epilogue warp
// converts its 32 x 32 chunk to 16 bits in a double-buffered shared-memory box
// (64-byte swizzle, bank-conflict free) and writes it with one TMA bulk
// tensor store.  MMA completion is multicast to both CTAs' barriers; both
// CTAs' epilogue warps release an accumulator on the even CTA's barrier.
// Every wait is bounded; a timeout sets the status word (and records where,
// for malt_debug_timeout_site) and the CTA winds down.
//
// Schedules.  A launch runs a range of the work list (NsParams): every tile
// of every product of every NS iteration, product by product.
//  * Phased: one launch per stage (a product of every class); pair j takes
//    items j, j + npairs, ...  The stream orders the stages.
//  * Persistent: one launch for the whole run.  A scheduler thread per pair (the
//    odd CTA's otherwise idle MMA-warp thread) claims items with an atomic on a
//    global counter and publishes them to a 3-slot ring in both CTAs' shared
//    memory (st.async messages on mbarriers).  Before it reads a tile's
//    operands, each producer waits (bounded, acquire) until the previous stage
//    of the tile's matrix is complete -- every epilogue warp of every tile of
//    that stage has signalled done[] after its TMA stores completed.  Each
//    product of a matrix depends only on the previous products of the same
//    matrix, so tiles of the next product of one matrix start while the current
//    product of another matrix is still running: no grid-wide barrier
//    between products, no launch gaps, no wave tails except the last.
//    Items are claimed in list order by running CTAs only and each pair runs its
//    items in order, so every item a tile waits for is held by a CTA that is
//    running and whose own dependencies come earlier still: the schedule cannot
//    deadlock, whatever number of CTA pairs is resident.
//  Both schedules run the same per-tile arithmetic, so their results are
//  bitwise identical.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <algorithm>
#include <cstdint>
#include <cstdio>
#include <mutex>
#include <type_traits>

#include "chain.cuh"
#include "common.cuh"
#include "kernels.h"
#include "ptx.cuh"

namespace malt {

namespace {

constexpr int kEpiWarps = kEpiWarpsPerCta;
// A persistent launch has one more warp, which signals finished tiles.
constexpr int ns_threads(int mode) { return 64 + 32 * kEpiWarps + (mode == kNsPersistent ? 32 : 0); }
constexpr uint32_t kABytes = kBM * kBK * 2;            // 16 KB
constexpr uint32_t kMnBoxBytes = kBMN * kBK * 2;       // one 64 x 64 MN-major box
constexpr uint32_t kMnLbo = kMnBoxBytes;               // next 64 MN-elements

// What follows from the width kN of an output tile.
template <int kN>
struct Tile {
    static constexpr int kEpiCols = kN / (kEpiWarps / 4);   // accumulator columns per warp
    static constexpr int kEpiChunks = kEpiCols / 32;
    static constexpr int kHalfN = kN / 2;                   // B rows (or columns) per CTA
    static constexpr uint32_t kBBytes = kHalfN * kBK * 2;   // 16 KB (wide), 8 KB (narrow)
    static constexpr uint32_t kStageBytes = kABytes + kBBytes;   // one 64-wide reduction slice
    static constexpr uint32_t kTmemCols = 2 * kN;
    static_assert(kTmemCols <= 512, "two accumulators must fit in TMEM");
    static_assert(kHalfN % kBMN == 0, "B half must be whole MN-major boxes");
    static_assert(kTileM % kN == 0, "a row of tiles starts on the diagonal");
};
// Ring granularity: the producer fills, and the MMA thread waits for and
// releases, kGroup slices at a time.  A barrier wait and a commit sit on the
// MMA issue path once per kGroup slices (8 MMAs) instead of once per 4 MMAs.
constexpr int kGroup = 2;
constexpr int kRing = kStages / kGroup;
static_assert(kStages % kGroup == 0, "the slice slots form whole ring stages");
constexpr uint32_t kStoreBoxBytes = 32 * 32 * 2;      // one 32 x 32 bf16 output box
constexpr uint32_t kStageOutBytes = 2 * kStoreBoxBytes * kEpiWarps;  // double-buffered per warp
constexpr size_t kSmemBytes =
    static_cast<size_t>(kStages) * Tile<kWideN>::kStageBytes + kStageOutBytes + 1024;
constexpr uint16_t kPairMask = 0x3;
// Persistent schedule: slots of the item ring, and the readers of each slot: both
// producers, the even CTA's MMA thread, every epilogue warp and the signal warp of
// both CTAs.  A slot is free again once its tile has been reported, so a pair holds
// at most this many published tiles (one in the epilogue, one in the MMAs, one in the
// loads) and one more that its scheduler has claimed and cannot publish yet.  With more
// slots pairs claim tiles that they cannot start yet while others idle:
// GPT-2 Small's step takes 1120 us with 3, 1132 with 4 and 1170 with 6, but 1151
// with 2; GPT-2 Medium and larger sets differ by less than 0.3 % between 3 and 6.
constexpr int kItemSlots = 3;
constexpr int kNoItem = -0x7fffffff;   // never stored in the ring
constexpr uint32_t kItemReaders = 5 + 2 * kEpiWarps;
static_assert(2 * kEpiWarps == static_cast<int>(kNsSignalsPerTile),
              "a finished tile counts one signal per epilogue warp of the pair");
// Phases of sig_bar in flight.  A slot is used again by the tile kSigSlots
// reported tiles later, at the earliest by the item kSigSlots later, which is
// published only after the signal warp has seen this one's phase complete (it
// frees the item's ring slot then) and processed only after every epilogue warp has
// arrived on it (each releases the accumulators of the tiles between after that).
constexpr int kSigSlots = 4;
static_assert(kSigSlots >= kItemSlots, "a phase of sig_bar is seen before the slot is used again");

static_assert(kBK * 2 == 128, "one K slice must be one 128-byte swizzle row");
static_assert(kEpiWarps == 8, "epilogue layout assumes two warps per lane quarter");

// Operands and output of one work item.
struct Ops {
    const CUtensorMap* a;
    const CUtensorMap* b;
    const CUtensorMap* a_mn;    // the same buffers as MN-major operands
    const CUtensorMap* b_mn;
    const CUtensorMap* out;
    int M, N, K;
};

__device__ __forceinline__ Ops item_operands(const NsParams& P, const NsWork& w) {
    const NsClass& C = P.cls[w.cls];
    const NsOp& o = w.op;
    const bool bx = o.kind == kBX;
    return Ops{&C.tmK[o.a], &C.tmK[o.b], &C.tmMn[o.a], &C.tmMn[o.b],
               o.out == kBufO ? &C.stO : &C.stK[o.out],
               C.p, bx ? C.q : C.p, o.kind == kGram ? C.q : C.p};
}

// A symmetric p x p buffer holds its 256 x 256 tiles on and above the diagonal.
// The reduction slices of operand rows in tile row `row` that lie below it are the
// first ones; their elements [r][k] are read as [k][r], MN-major instead of
// K-major.  Storing every such tile a second time, transposed, cost the epilogue
// (shuffles, a second staged box and store per chunk) more than these reads cost the
// loads and the MMAs, at every size: Newton-Schulz of GPT-2 Small 742 -> 711 us, of
// GPT-2 Medium 3050 -> 2932, one 4096 x 4096 matrix 894 -> 863, one 512 x 512 102 -> 96.
__device__ __forceinline__ int slices_below(int row) { return row * (kTileM / kBK); }
static_assert(kTileM / kBK % kGroup == 0, "the slices of a ring stage are read alike");

// Bytes CTA `rank` loads for one reduction slice of a tile.  Boxes that lie
// wholly past M or N are skipped: they only feed accumulator rows / columns
// that are never stored.
template <int kN>
__device__ __forceinline__ uint32_t slice_bytes(const Ops& op, const NsWork& w, int rank,
                                                bool b_mn, int* nbox_b) {
    uint32_t bytes = 0;
    if (w.mt * kTileM + rank * kBM < op.M) bytes += kABytes;
    constexpr int kHalfN = Tile<kN>::kHalfN;
    const int n0 = w.nt * kN + rank * kHalfN;
    int nb = 0;
    if (b_mn) {
        for (int j = 0; j < kHalfN / kBMN; ++j)
            if (n0 + j * kBMN < op.N) ++nb;
        bytes += nb * kMnBoxBytes;
    } else if (n0 < op.N) {
        nb = 1;
        bytes += Tile<kN>::kBBytes;
    }
    *nbox_b = nb;
    return bytes;
}

// Layout of an operand in its slot.
using Mn = std::integral_constant<bool, true>;
using Kn = std::integral_constant<bool, false>;

// The MMAs of one reduction slice (kb-th of its tile), each operand K-major or
// MN-major; idesc is that of two K-major operands.
template <bool kAMn, bool kBMn>
__device__ __forceinline__ void issue_slice(uint32_t d_tmem, uint32_t sa, bool same_ab, uint32_t idesc, int kb) {
    const uint32_t sb = same_ab ? sa : sa + kABytes;
    const uint64_t da = kAMn ? smem_desc_mn_sw128(sa, kMnLbo) : smem_desc_k_sw128(sa);
    const uint64_t db = kBMn ? smem_desc_mn_sw128(sb, kMnLbo) : smem_desc_k_sw128(sb);
    // Per 16-element MMA slice (addresses encoded >> 4): +32 bytes along K, or
    // +16 K-rows = two 1024-byte atoms.
    constexpr uint32_t kStepA = kAMn ? 2048u >> 4 : 2u, kStepB = kBMn ? 2048u >> 4 : 2u;
#pragma unroll
    for (int kk = 0; kk < kBK / 16; ++kk)
        tc_mma_16bit_pair(d_tmem, da + kStepA * kk, db + kStepB * kk, idesc | idesc_majors(kAMn, kBMn),
                          (kb | kk) != 0 ? 1u : 0u);
}

// Two floats <-> two 16-bit values (fp16 or bf16, round to nearest even).
template <bool kF16>
__device__ __forceinline__ float2 unpack2(uint32_t u) {
    if constexpr (kF16) return __half22float2(*reinterpret_cast<const __half2*>(&u));
    return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u));
}

template <bool kF16>
__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
    uint32_t u;
    if constexpr (kF16)
        *reinterpret_cast<__half2*>(&u) = __floats2half2_rn(lo, hi);
    else
        *reinterpret_cast<__nv_bfloat162*>(&u) = __floats2bfloat162_rn(lo, hi);
    return u;
}

// v <- sc v + beta x, x 16 words of two 16-bit values.
template <bool kF16>
__device__ __forceinline__ void add_ein(float (&v)[32], const uint32_t* x, float sc, float beta) {
#pragma unroll
    for (int j = 0; j < 32; j += 2) {
        const float2 e = unpack2<kF16>(x[j >> 1]);
        v[j] = fmaf(beta, e.x, sc * v[j]);
        v[j + 1] = fmaf(beta, e.y, sc * v[j + 1]);
    }
}

template <bool kF16>
__device__ __forceinline__ void pack32(const float (&v)[32], uint32_t (&w)[16]) {
#pragma unroll
    for (int j = 0; j < 16; ++j) w[j] = pack2<kF16>(v[2 * j], v[2 * j + 1]);
}

// Where a wait gave up (recorded once per status word, for malt_debug_timeout_site).
enum WaitSite : int32_t {
    kSiteClaim = 1,      // scheduler: a ring slot to become free
    kSiteDepLoad = 2,    // the previous stage of the matrix (producer; + 16 scheduler; + 32 epilogue)
    kSiteStage = 3,      // producer: a free operand stage
    kSiteItem = 4,       // ring reader: the next item (+ 16 * role)
    kSiteAccFree = 5,    // MMA: a free accumulator
    kSiteStageFull = 6,  // MMA: operands of a stage
    kSiteAccFull = 7,    // epilogue: a finished accumulator
    kSiteSignal = 8,     // signal warp: the epilogue warps' stores of a tile
    kSiteDrain = 9,      // MMA: the last MMAs before TMEM is freed
};

__device__ __forceinline__ void raise_timeout(const NsParams& P, volatile int* abort_flag,
                                              int site = 0, int item = -1, int seq = -1) {
    if (atomicCAS(P.status + 1, 0, site == 0 ? -1 : site) == 0) {
        P.status[2] = item;
        P.status[3] = seq;
        P.status[4] = static_cast<int32_t>(blockIdx.x);
        P.status[5] = static_cast<int32_t>(threadIdx.x);
    }
    atomicOr(P.status, kStatusTimeout);
    *abort_flag = 1;
}

// One unit of work as a role of the pair sees it.
enum JobState : int32_t { kJobWork = 0, kJobEnd = -1, kJobTimeout = -2 };
struct Job {
    int32_t state;
    int32_t stage;    // stage of the work table (persistent) or product index (phased)
    int32_t g;        // matrix (-1 when not known yet: phased)
    int32_t local;
    uint32_t target;  // signals that the matrix's previous stage must have (0: none)
    NsWork w;
};

template <int kN>
__device__ __forceinline__ Job job_of_entry(const NsParams& P, const NsEntry& e) {
    Job j;
    if (e.g < 0) {
        j.state = kJobEnd;
        return j;
    }
    j.state = kJobWork;
    j.stage = entry_stage(e);
    j.g = e.g;
    j.local = e.local;
    j.target = e.target;
    j.w.cls = entry_cls(e);
    j.w.op = ns_op(P, P.cls[j.w.cls], j.stage);
    j.w.b = entry_b(e);
    j.w.local = e.local;
    ns_tile_coords(P.cls[j.w.cls], kN, j.w.op.kind, e.local, &j.w.mt, &j.w.nt);
    return j;
}

}  // namespace

template <int kMode, int kN>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(ns_threads(kMode), 1)
ns_gemm_kernel(const __grid_constant__ NsParams P) {
    constexpr bool kPersistent = kMode == kNsPersistent;   // table-driven, claimed dynamically
    constexpr int kHalfN = Tile<kN>::kHalfN, kEpiCols = Tile<kN>::kEpiCols, kEpiChunks = Tile<kN>::kEpiChunks;
    constexpr uint32_t kStageBytes = Tile<kN>::kStageBytes, kTmemCols = Tile<kN>::kTmemCols;
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[kRing];
    __shared__ __align__(8) uint64_t empty_bar[kRing];
    __shared__ __align__(8) uint64_t tfull_bar[2];
    __shared__ __align__(8) uint64_t tempty_bar[2];
    __shared__ __align__(8) uint64_t drain_bar;
    __shared__ __align__(8) uint64_t item_full[kItemSlots];
    __shared__ __align__(8) uint64_t item_empty[kItemSlots];
    __shared__ NsEntry item_ring[kItemSlots];
    __shared__ __align__(8) uint64_t sig_bar[kSigSlots];
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_sh;
    volatile int* abort_flag = &abort_sh;

    // Same offset in both CTAs: the MMA addresses the peer's tiles through
    // the even CTA's descriptors.
    uint8_t* smem = reinterpret_cast<uint8_t*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint64_t budget = P.budget_ns;
    const int rank = static_cast<int>(cluster_ctarank());
    const bool leader = (rank == 0);
    const int pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kRing; ++s) {
            // Both producers arrive on the even CTA's full barrier for every
            // ring stage (the even one with the pair's transaction bytes), so the
            // MMA never consumes a slice the odd producer has not reached --
            // even when the odd CTA loads nothing (M or N within its partner's
            // half) -- and the odd producer can never fall a whole parity
            // cycle behind the empty barriers it waits on.
            mbar_init(&full_bar[s], 2);
            mbar_init(&empty_bar[s], 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(&tfull_bar[a], 1);
            mbar_init(&tempty_bar[a], 2 * kEpiWarps);
        }
        mbar_init(&drain_bar, 1);
        if (kPersistent) {
            for (int s = 0; s < kItemSlots; ++s) {
                mbar_init(&item_full[s], 1);
                mbar_init(&item_empty[s], kItemReaders);
            }
            for (int s = 0; s < kSigSlots; ++s) mbar_init(&sig_bar[s], kEpiWarps);
        }
        abort_sh = 0;
        fence_barrier_init();
        fence_proxy_async_smem();
    }
    if (warp == 0 && lane == 0) {
        for (int c = 0; c < P.nclasses; ++c) {
            const NsClass& C = P.cls[c];
            for (int j = 0; j < 2; ++j) {
                tma_prefetch_desc(&C.tmK[kBufX + j]);
                tma_prefetch_desc(&C.tmMn[kBufX + j]);
            }
            for (int j = 0; j < (C.grouped ? 4 : 2); ++j) tma_prefetch_desc(&C.tmK[j]);
        }
    }
    if (warp == 1) {
        tmem_alloc_pair(&tmem_slot, kTmemCols);
        tmem_relinquish_pair();
    }
    // What precedes touches no global memory that an earlier launch writes.
    chain_wait();
    tc_fence_before();
    cluster_sync();          // both CTAs' barriers initialised, TMEM allocated
    tc_fence_after();
    const uint32_t tmem_base = tmem_slot;

    // Work number `seq` of this pair.  Phased: static round-robin over the
    // product's item range.  Persistent: the next entry of the ring, which
    // the scheduler thread of the odd CTA fills from the work table.
    auto static_job = [&](int seq) -> Job {
        Job j;
        const long long it = pair + static_cast<long long>(seq) * npairs;
        if (it >= P.item_end) {
            j.state = kJobEnd;
            return j;
        }
        j.state = kJobWork;
        j.w = ns_decode(P, kN, static_cast<int>(it));
        j.stage = P.stage;
        j.g = -1;
        j.local = j.w.local;
        j.target = 0;
        return j;
    };
    // The ring entry of sequence number seq (false when the wait gave up); its
    // reader then frees the slot with ring_free.
    auto ring_free = [&](int seq) {
        // The slot's barrier lives in the odd CTA, with the scheduler.  The arrive
        // carries no data, so it is relaxed.
        mbar_arrive_cluster_relaxed(mapa_shared(smem_u32(&item_empty[seq % kItemSlots]), 1));
    };
    auto ring_peek = [&](int seq, NsEntry& e) -> bool {
        const int slot = seq % kItemSlots;
        const uint32_t par = static_cast<uint32_t>(seq / kItemSlots) & 1u;
        if (!mbar_wait_cluster_bounded(&item_full[slot], par, budget, abort_flag)) return false;
        const int4 v = ld_shared_v4(&item_ring[slot]);
        e.code = v.x;
        e.g = v.y;
        e.local = v.z;
        e.target = static_cast<uint32_t>(v.w);
        return true;
    };
    auto ring_entry = [&](int seq, NsEntry& e) -> bool {
        if (!ring_peek(seq, e)) return false;
        // Issued only once the slot's value is in hand (one load, and the branch
        // depends on it), so the scheduler cannot overwrite the slot before this read.
        if (e.code != kNoItem) ring_free(seq);
        return true;
    };
    auto ring_job = [&](int seq) -> Job {
        NsEntry e;
        if (!ring_entry(seq, e)) {
            Job j;
            j.state = kJobTimeout;
            return j;
        }
        return job_of_entry<kN>(P, e);
    };
    auto next_job = [&](int seq) -> Job { return kPersistent ? ring_job(seq) : static_job(seq); };
    // Scheduler (odd CTA): the table entry of the next claimed item (an end
    // marker past the end), and its publication to the ring slot of sequence
    // number seq in both CTAs (false when the slot did not come free in time).
    auto claim_next = [&]() -> NsEntry {
        const uint32_t claimed = atomicAdd(P.queue, 1u);
        if (claimed >= static_cast<uint32_t>(P.item_end)) {
            NsEntry e;
            e.code = 0;
            e.g = -1;
            e.local = 0;
            e.target = 0;
            return e;
        }
        const int4 v = __ldg(reinterpret_cast<const int4*>(P.table + claimed));
        NsEntry e;
        e.code = v.x;
        e.g = v.y;
        e.local = v.z;
        e.target = static_cast<uint32_t>(v.w);
        return e;
    };
    auto publish_item = [&](int seq, const NsEntry& e) -> bool {
        const int slot = seq % kItemSlots;
        const uint32_t par = static_cast<uint32_t>(seq / kItemSlots) & 1u;
        if (!mbar_wait_cluster_bounded(&item_empty[slot], par ^ 1u, budget, abort_flag)) return false;
        // The entry travels as an asynchronous store that completes on the
        // slot's full barrier in each CTA.  The arrive releases at cluster
        // scope what this thread may have acquired from the dependency counter,
        // so a reader of an item without a target sees the data the item reads.
        for (uint32_t r = 0; r < 2; ++r) {
            const uint32_t bar = mapa_shared(smem_u32(&item_full[slot]), r);
            mbar_arrive_expect_tx_cluster(bar, 16u);
            st_async_v4(mapa_shared(smem_u32(&item_ring[slot]), r), e.code, e.g, e.local,
                        static_cast<int32_t>(e.target), bar);
        }
        return true;
    };

    // Wait (bounded, acquire) until the previous stage of the job's matrix is
    // stored.  Each reader of another CTA's results waits for itself, with the
    // item already decoded: handed on by the scheduler only once the stage was
    // complete, an item reached the producers 1.2 us later (one 256 x 512 matrix
    // has 15 such waits in a row).
    auto stage_done = [&](int stage, int g, uint32_t target) -> bool {
        return target == 0 || counter_wait_bounded(P.done + (stage - 1) * P.nmat + g, target, budget, P.status,
                                                   kStatusTimeout, abort_flag);
    };

    if (warp == 0) {
        // ---------------------------------------------------- TMA producer
        if (lane == 0) {
            uint32_t stage = 0, phase = 0;
            for (int seq = 0;; ++seq) {
                const Job job = next_job(seq);
                if (job.state == kJobTimeout) {
                    raise_timeout(P, abort_flag, kSiteItem, -2, seq);
                    break;
                }
                if (job.state == kJobEnd) break;
                const int item = job.local;
                // The loads below read what other CTAs stored in this launch: wait
                // for the previous stage of this matrix.
                if (kPersistent) {
                    if (!stage_done(job.stage, job.g, job.target)) {
                        raise_timeout(P, abort_flag, kSiteDepLoad, item, seq);
                        break;
                    }
                    fence_proxy_async_global();
                }
                const NsWork& w = job.w;
                const Ops op = item_operands(P, w);
                const bool b_mn = w.op.kind == kBX;
                // A diagonal tile of a product of a matrix with itself: each CTA's
                // half of B is its own rows of A, so B is not loaded and the MMA
                // reads A twice.
                const bool same_ab = kN == kTileM && w.op.a == w.op.b && w.mt == w.nt;
                const int nkb = (op.K + kBK - 1) / kBK;
                int nb_self = 0, nb_peer = 0;
                uint32_t bytes_pair = slice_bytes<kN>(op, w, rank, b_mn, &nb_self) +
                                      slice_bytes<kN>(op, w, rank ^ 1, b_mn, &nb_peer);
                if (same_ab) {
                    nb_self = 0;
                    bytes_pair = (w.mt * kTileM < op.M ? kABytes : 0u) +
                                 (w.mt * kTileM + kBM < op.M ? kABytes : 0u);
                }
                const bool load_a = w.mt * kTileM + rank * kBM < op.M;
                const int a_row = w.mt * kTileM + rank * kBM;
                const int n0 = w.nt * kN + rank * kHalfN;
                const int a_below = w.op.kind != kGram ? slices_below(w.mt) : 0;
                const int b_below = b_mn ? nkb : w.op.kind == kPoly ? slices_below(w.nt * kN / kTileM) : 0;
                // MN-major boxes of a slice of B (a half is counted whole where it is
                // read from above the diagonal: boxes past N arrive as zeros)
                const int nb_mn = b_mn ? nb_self : nb_self > 0 ? kHalfN / kBMN : 0;
                // Slices [from, to), each operand K-major or MN-major.
                auto load_slices = [&](auto a_mn, auto b_mn_, int from, int to) -> bool {
                    for (int k0 = from; k0 < to; k0 += kGroup) {
                        if (!mbar_wait_cluster_bounded(&empty_bar[stage], phase ^ 1u, budget, abort_flag)) {
                            raise_timeout(P, abort_flag, kSiteStage, item, k0);
                            return false;
                        }
                        const int nsub = min(kGroup, to - k0);
                        const uint32_t fb = mapa_shared(smem_u32(&full_bar[stage]), 0);
                        if (leader) mbar_arrive_expect_tx(&full_bar[stage], nsub * bytes_pair);
                        for (int j = 0; j < nsub; ++j) {
                            const int kx = (k0 + j) * kBK;
                            uint8_t* sa = smem + (stage * kGroup + j) * kStageBytes;
                            if (load_a) {
                                if constexpr (decltype(a_mn)::value) {
#pragma unroll
                                    for (int h = 0; h < kBM; h += kBMN)
                                        tma_load_3d_pair(sa + h * (kBK * 2), op.a_mn, a_row + h, kx, w.b, fb);
                                } else {
#pragma unroll
                                    for (int h = 0; h < kBM; h += kHalfN)
                                        tma_load_3d_pair(sa + h * (kBK * 2), op.a, kx, a_row + h, w.b, fb);
                                }
                            }
                            if constexpr (decltype(b_mn_)::value) {
                                for (int jb = 0; jb < nb_mn; ++jb)
                                    tma_load_3d_pair(sa + kABytes + jb * kMnBoxBytes, op.b_mn, n0 + jb * kBMN, kx,
                                                     w.b, fb);
                            } else if (nb_self > 0) {
                                tma_load_3d_pair(sa + kABytes, op.b, kx, n0, w.b, fb);
                            }
                        }
                        if (!leader) mbar_arrive_cluster_relaxed(fb);
                        if (++stage == kRing) { stage = 0; phase ^= 1u; }
                    }
                    return true;
                };
                const bool ok = load_slices(Mn{}, Mn{}, 0, a_below) && load_slices(Kn{}, Mn{}, a_below, b_below) &&
                                load_slices(Kn{}, Kn{}, b_below, nkb);
                if (!ok) break;
            }
        }
    } else if (warp == 1) {
        if (kPersistent && lane == 0 && !leader) {
            // ------------------------------------------ scheduler (odd CTA)
            // Claim items in table order and publish them up to kItemSlots ahead
            // of the slowest reader.  The next item is claimed only once the
            // last one can run: claimed at once, five items a pair (with a ring of
            // four slots) left a stage of 136 tiles to 28 of the 76 pairs (one
            // 4096 x 4096 matrix 916 us -> 1245).
            for (int seq = 0;; ++seq) {
                NsEntry e = claim_next();
                const uint32_t target = e.target;
                // (complete already: the readers need not look again)
                if (e.g >= 0 && target > 0 &&
                    ld_acquire_gpu(P.done + (entry_stage(e) - 1) * P.nmat + e.g) >= target)
                    e.target = 0;
                if (!publish_item(seq, e)) {
                    raise_timeout(P, abort_flag, kSiteClaim, e.local, seq);
                    break;
                }
                if (e.g < 0) break;
                if (e.target > 0 && !stage_done(entry_stage(e), e.g, target)) {
                    raise_timeout(P, abort_flag, kSiteDepLoad + 16, e.local, seq);
                    break;
                }
            }
        }
        // ------------------------------------------- MMA issuer (even CTA)
        if (lane == 0 && leader) {
            uint32_t stage = 0, phase = 0;
            int gi = 0;                                  // product tiles so far (accumulator)
            for (int seq = 0;; ++seq) {
                const Job job = next_job(seq);
                if (job.state == kJobTimeout) {
                    raise_timeout(P, abort_flag, kSiteItem + 16, -2, seq);
                    break;
                }
                if (job.state == kJobEnd) break;
                const int item = job.local;
                const NsWork& w = job.w;
                const bool b_mn = w.op.kind == kBX;
                const bool same_ab = kN == kTileM && w.op.a == w.op.b && w.mt == w.nt;
                const int K = w.op.kind == kGram ? P.cls[w.cls].q : P.cls[w.cls].p;
                const int nkb = (K + kBK - 1) / kBK;
                const int a_below = w.op.kind != kGram ? slices_below(w.mt) : 0;
                const int b_below = b_mn ? nkb : w.op.kind == kPoly ? slices_below(w.nt * kN / kTileM) : 0;
                const uint32_t idesc = w.op.f16 ? idesc_16bit_f32(kTileM, kN, true)
                                                : idesc_16bit_f32(kTileM, kN, false);
                const uint32_t acc = gi & 1, acc_phase = (gi >> 1) & 1;
                ++gi;
                if (!mbar_wait_cluster_bounded(&tempty_bar[acc], acc_phase ^ 1u, budget, abort_flag)) {
                    raise_timeout(P, abort_flag, kSiteAccFree, item, seq);
                    break;
                }
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + acc * kN;
                // Slices [from, to): with each form a loop of its own, the descriptors'
                // steps and the instruction descriptor are constants (one loop that
                // picks the form per ring stage was 3 - 6 % slower on 4096 x 4096).
                auto issue_slices = [&](auto a_mn, auto b_mn_, int from, int to) -> bool {
                    for (int k0 = from; k0 < to; k0 += kGroup) {
                        if (!mbar_wait_cluster_bounded(&full_bar[stage], phase, budget, abort_flag)) {
                            raise_timeout(P, abort_flag, kSiteStageFull, item, k0);
                            return false;
                        }
                        tc_fence_after();
                        const int nsub = min(kGroup, to - k0);
                        for (int j = 0; j < nsub; ++j)
                            issue_slice<decltype(a_mn)::value, decltype(b_mn_)::value>(
                                d_tmem, smem_u32(smem + (stage * kGroup + j) * kStageBytes), same_ab, idesc, k0 + j);
                        tc_commit_pair_multicast(&empty_bar[stage], kPairMask);
                        if (++stage == kRing) { stage = 0; phase ^= 1u; }
                    }
                    return true;
                };
                const bool ok = issue_slices(Mn{}, Mn{}, 0, a_below) && issue_slices(Kn{}, Mn{}, a_below, b_below) &&
                                issue_slices(Kn{}, Kn{}, b_below, nkb);
                if (!ok) break;
                tc_commit_pair_multicast(&tfull_bar[acc], kPairMask);
            }
            // Do not release TMEM while MMAs may still be in flight.
            tc_commit_pair_multicast(&drain_bar, 0x1);
            if (!mbar_wait_cluster_bounded(&drain_bar, 0, budget, nullptr)) raise_timeout(P, abort_flag, kSiteDrain);
        }
    } else if (kPersistent && warp == 2 + kEpiWarps) {
        // ---------------------------------------------------------- signals
        // Every epilogue warp reports its finished part of a tile on sig_bar;
        // this thread adds the CTA's signals to the matrix's counter.  The
        // release at GPU scope takes 1.6 - 2.4K cycles, a sixth of the epilogue
        // warps' time per tile on GPT-2 Small, whose tile rate they bound.
        if (lane == 0) {
            int si = 0;
            for (int seq = 0;; ++seq) {
                NsEntry e;
                if (!ring_peek(seq, e)) {
                    raise_timeout(P, abort_flag, kSiteItem + 48, -2, seq);
                    break;
                }
                if (e.g < 0) break;
                const int stage = entry_stage(e);
                const bool report = stage + 1 < ns_num_stages(P, P.cls[entry_cls(e)]);
                if (report) {
                    if (!mbar_wait_bounded(&sig_bar[si % kSigSlots], (si / kSigSlots) & 1, budget, abort_flag)) {
                        raise_timeout(P, abort_flag, kSiteSignal, e.local, seq);
                        break;
                    }
                    ++si;
                }
                // Only now may the slot be published again: item seq + kItemSlots,
                // whose reports would complete this phase of sig_bar a second
                // time, cannot reach the epilogue before.
                ring_free(seq);
                if (report) red_release_gpu_add(P.done + stage * P.nmat + e.g, kEpiWarps);
            }
        }
    } else {
        // -------------------------------------------------------- epilogue
        uint8_t* stage_out = smem + kStages * kStageBytes;   // 1024-byte aligned
        int obuf = 0;
        const int ew = warp - 2;                  // epilogue warp 0..kEpiWarps-1
        const int quarter = warp & 3;             // TMEM lanes this warp may read
        const int colw = (ew >> 2) * kEpiCols;    // first accumulator column of this warp
        const uint32_t tempty_leader0 = mapa_shared(smem_u32(&tempty_bar[0]), 0);
        const uint32_t tempty_leader1 = mapa_shared(smem_u32(&tempty_bar[1]), 0);
        int gi = 0;                               // product tiles so far (accumulator)
        int si = 0;                               // reported tiles so far
        for (int seq = 0;; ++seq) {
            Job job;
            if (kPersistent) {
                // One lane waits on the ring; the warp shares the entry.
                NsEntry e;
                e.code = 0;
                e.g = -1;
                e.local = 0;
                e.target = 0;
                int ok = 1;
                if (lane == 0) ok = ring_entry(seq, e) ? 1 : 0;
                ok = __shfl_sync(0xffffffffu, ok, 0);
                e.code = __shfl_sync(0xffffffffu, e.code, 0);
                e.g = __shfl_sync(0xffffffffu, e.g, 0);
                e.local = __shfl_sync(0xffffffffu, e.local, 0);
                e.target = __shfl_sync(0xffffffffu, e.target, 0);
                if (!ok) {
                    job.state = kJobTimeout;
                } else {
                    job = job_of_entry<kN>(P, e);
                }
            } else {
                job = static_job(seq);
            }
            if (job.state == kJobTimeout) {
                if (lane == 0) raise_timeout(P, abort_flag, kSiteItem + 32, -2, seq);
                break;
            }
            if (job.state == kJobEnd) break;
            const int item = job.local;
            const NsWork& w = job.w;
            const NsClass& C = P.cls[w.cls];
            const uint32_t acc = gi & 1, acc_phase = (gi >> 1) & 1;
            ++gi;
            const NsOp& op = w.op;
            const bool in16 = op.f16 != 0, out16 = op.out16 != 0;
            const int M = C.p, N = op.kind == kBX ? C.q : C.p;
            const CUtensorMap* out_map0 = item_operands(P, w).out;
            const int row = w.mt * kTileM + rank * kBM + quarter * 32 + lane;
            const bool rok = row < M;
            const int g = job.g >= 0 ? job.g : C.mat_of[w.b];
            const MatDesc& md = P.mats[g];
            // (1/||Mt||, L and R come from launches before this one, complete since
            // chain_wait; the persistent instantiation reads them past L1, where a
            // tile would find nothing of the last one)
            float sc = op.gamma;
            if (op.kx != 0) {
                const float k = kPersistent ? __ldcg(&P.scal[g].k) : P.scal[g].k;
                sc = (op.kx == 2 ? k * k : k) * sc;
            }
            const bool need_ein = op.e != kBufNone;
            const uint16_t* ein = need_ein ? C.A + static_cast<size_t>(w.b) * C.p * ns_ld(C.p) : nullptr;
            const bool last_bx = op.out == kBufO;
            // O of a tall W (NS frame = W^T) goes out transposed, in W's layout.
            const bool store_t = last_bx && md.trans;
            const CUtensorMap* out_map = store_t ? &C.stOt : out_map0;
            // NS frame row / column scalings of D = L O R (swapped when transposed).
            const float* uvec = md.trans ? md.R : md.L;
            const float* vvec = md.trans ? md.L : md.R;
            const float urow = (last_bx && rok) ? (kPersistent ? __ldcg(uvec + row) : uvec[row]) : 0.f;
            float sum_o = 0.f, sum_d = 0.f;

            const int col_base = w.nt * kN + colw;     // first output column of this warp
            const int nch = max(0, min(kEpiChunks, (N - col_base + 31) / 32));
            const uint32_t tbase = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16) +
                                   acc * kN + colw;
            auto load_ein = [&](int ch, uint4 (&dst)[4]) {
                const int col0 = col_base + ch * 32;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    // Whole 32-byte sectors: each lane reads its own row, and with
                    // 16-byte loads half of every sector fetched was read again
                    // (Newton-Schulz of GPT-2 Small 719 -> 705 us, one 1280 x 5120
                    // and one 5120 x 1280 matrix 327 -> 320).  (Columns past N are
                    // never stored.)
                    // Through L2 only: A is rewritten within this launch (persistent,
                    // ordered by the acquire of the dependency's counter) or by a
                    // launch that this one overlaps (phased, ordered by chain_wait),
                    // so it is not read-only for the kernel's lifetime.
                    if (rok && col0 + h * 16 < N)
                        ld_global_32b(ein + static_cast<size_t>(row) * ns_ld(N) + col0 + h * 16, dst[2 * h],
                                      dst[2 * h + 1]);
                    else
                        dst[2 * h] = dst[2 * h + 1] = make_uint4(0u, 0u, 0u, 0u);
                }
            };
            uint4 xin[4];
            uint32_t rv[32];
            const int row0 = w.mt * kTileM + rank * kBM + quarter * 32;   // warp's first row
            // The back-map scalings of this warp's columns (lane j of chunk ch holds
            // column 32 ch + j; 0 past N).
            float vl[kEpiChunks];
            if (last_bx) {
#pragma unroll
                for (int ch = 0; ch < kEpiChunks; ++ch) {
                    const int col = col_base + ch * 32 + lane;
                    vl[ch] = col < N ? (kPersistent ? __ldcg(vvec + col) : vvec[col]) : 0.f;
                }
            }
            // The first chunk's A values (and the scalars above) are in flight
            // while the accumulator is still being computed.
            if (need_ein) {
                if (kPersistent) {
                    int ok = 1;
                    if (lane == 0) ok = stage_done(job.stage, job.g, job.target) ? 1 : 0;
                    if (!__shfl_sync(0xffffffffu, ok, 0)) {
                        if (lane == 0) raise_timeout(P, abort_flag, kSiteDepLoad + 32, item, seq);
                        break;
                    }
                    __syncwarp();   // lane 0's acquire holds for the warp's loads
                }
                if (nch > 0) load_ein(0, xin);
            }
            // The epilogue warps poll with a short sleep: sixteen warps spinning
            // on this barrier cost issue slots and power the MMA and load
            // warps need (measured 0.5-1 % on every product).
            if (!mbar_wait_cluster_bounded_sleep(&tfull_bar[acc], acc_phase, budget, abort_flag, 128)) {
                raise_timeout(P, abort_flag, kSiteAccFull, item, seq);
                break;
            }
            tc_fence_after();
            if (nch > 0) {
                tmem_ld_issue(tbase, rv);
                tmem_ld_wait(rv);
            }
#pragma unroll
            for (int ch = 0; ch < kEpiChunks; ++ch) {
                if (ch >= nch) break;
                uint4 xcur[4];
#pragma unroll
                for (int q8 = 0; q8 < 4; ++q8) xcur[q8] = xin[q8];
                if (need_ein && ch + 1 < nch) load_ein(ch + 1, xin);   // next chunk's A, one ahead

                const int col0 = col_base + ch * 32;
                float v[32];
#pragma unroll
                for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(rv[j]);
                // The next chunk's TMEM load is in flight during this chunk's work.
                if (ch + 1 < nch) tmem_ld_issue(tbase + (ch + 1) * 32, rv);
                if (need_ein) {
                    const uint32_t* xw = reinterpret_cast<const uint32_t*>(xcur);
                    if (in16)
                        add_ein<true>(v, xw, sc, op.beta);
                    else
                        add_ein<false>(v, xw, sc, op.beta);
                    // Rows and columns of a chunk start at multiples of 32, so
                    // only a chunk on the diagonal holds any of it, in lane = j.
                    if (row0 == col0) {
#pragma unroll
                        for (int j = 0; j < 32; ++j) v[j] += lane == j ? op.alpha : 0.f;
                    }
                } else {
#pragma unroll
                    for (int j = 0; j < 32; ++j) v[j] *= sc;
                }
                // This row's 32 results as they are stored.
                uint32_t wv[16];
                if (out16)
                    pack32<true>(v, wv);
                else
                    pack32<false>(v, wv);
                if (!store_t) {
                    // Stage the 32 x 32 chunk (row = lane, 64 bytes) with the 64-byte
                    // swizzle the store map expects, then one TMA store writes it
                    // (A, B', the next X, or a wide matrix's O on the last iteration).
                    uint8_t* box = stage_out + (ew * 2 + obuf) * kStoreBoxBytes;
                    if (lane == 0) bulk_wait_group_read<1>();   // this buffer's last store read it
                    __syncwarp();
#pragma unroll
                    for (int c = 0; c < 4; ++c)
                        *reinterpret_cast<uint4*>(box + lane * 64 + ((c ^ ((lane >> 1) & 3)) << 4)) =
                            make_uint4(wv[4 * c], wv[4 * c + 1], wv[4 * c + 2], wv[4 * c + 3]);
                    fence_proxy_async_smem();
                    __syncwarp();
                    if (lane == 0) {
                        tma_store_3d(out_map, box, col0, row0, w.b);
                        bulk_commit_group();
                    }
                    obuf ^= 1;
                }
                if (store_t) {
                    // A tall matrix's O goes out in W's layout: the transposed chunk
                    // (box row = column j, 32 rows of this warp) goes to rows
                    // [col0, col0+32) x columns [row0, row0+32) of the map.
                    // Lane pairs swap the packed word of each column pair, and
                    // each keeps one column of the two rows.
                    uint8_t* box = stage_out + (ew * 2 + obuf) * kStoreBoxBytes;
                    if (lane == 0) bulk_wait_group_read<1>();
                    __syncwarp();
                    const bool odd = lane & 1;
                    const int r2 = lane & ~1;                 // first of the two rows
#pragma unroll
                    for (int j = 0; j < 32; j += 2) {
                        // even lane keeps column j, odd lane keeps column j + 1
                        const uint32_t recv = __shfl_xor_sync(0xffffffffu, wv[j >> 1], 1);
                        const uint32_t pair = odd ? __byte_perm(recv, wv[j >> 1], 0x7632)
                                                  : __byte_perm(wv[j >> 1], recv, 0x5410);
                        const int jc = j + (odd ? 1 : 0);          // box row
                        const int off = jc * 64 + (((r2 >> 3) ^ ((jc >> 1) & 3)) << 4) + (r2 & 7) * 2;
                        *reinterpret_cast<uint32_t*>(box + off) = pair;
                    }
                    fence_proxy_async_smem();
                    __syncwarp();
                    if (lane == 0) {
                        tma_store_3d(out_map, box, row0, col0, w.b);
                        bulk_commit_group();
                    }
                    obuf ^= 1;
                }
                if (last_bx) {
                    // Partial sums of O^2 and (O v)^2 over the stored (bf16) O of this
                    // row; D^2 = u_row^2 (O v)^2 is formed once per tile.  Lane j holds
                    // v[col0 + j] and broadcasts it.  Columns past N (ragged frames
                    // only) hold what their accumulators held and do not count.
                    const bool full = col0 + 32 <= N;
#pragma unroll
                    for (int j = 0; j < 32; ++j) {
                        const float vj = __shfl_sync(0xffffffffu, vl[ch], j);
                        const float2 o2 = unpack2<false>(wv[j >> 1]);
                        const float o = j & 1 ? o2.y : o2.x;
                        const float ov = o * vj;
                        sum_o = fmaf(o, full || col0 + j < N ? o : 0.f, sum_o);
                        sum_d = fmaf(ov, ov, sum_d);
                    }
                }
                if (ch + 1 < nch) tmem_ld_wait(rv);
            }
            tc_fence_before();
            __syncwarp();
            // The accumulator has been read (the loads have completed and are
            // ordered by the fence above); no memory contents are handed over.
            if (lane == 0) mbar_arrive_remote(acc ? tempty_leader1 : tempty_leader0);
            if (last_bx) {
                if (!rok) sum_o = 0.f;
                sum_d = rok ? urow * urow * sum_d : 0.f;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    sum_o += __shfl_xor_sync(0xffffffffu, sum_o, o);
                    sum_d += __shfl_xor_sync(0xffffffffu, sum_d, o);
                }
                if (lane == 0) {
                    float* dst = md.nspart + (static_cast<size_t>(w.local) * kNsPartsPerTile +
                                              rank * kEpiWarps + ew) * 2;
                    dst[0] = sum_o;
                    dst[1] = sum_d;
                }
            }
            if (kPersistent && job.stage + 1 < ns_num_stages(P, C)) {
                // This warp's part of the tile is in global memory: report it
                // to the signal warp (the last stage has no reader inside the
                // launch).
                if (lane == 0) {
                    bulk_wait_group_all();
                    fence_proxy_async_global();
                    mbar_arrive(&sig_bar[si % kSigSlots]);
                }
                ++si;
            }
        }
        if (lane == 0) bulk_wait_group_all();     // every output store has landed
    }

    // Neither CTA may leave (or free TMEM) while its pair partner can still
    // signal its barriers or read its shared memory.
    tc_fence_before();
    cluster_sync();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc_pair(tmem_base, kTmemCols);
    }
}

namespace {

using NsKernel = void (*)(const NsParams);

NsKernel ns_kernel(int mode, int tile_n) {
    if (mode == kNsPersistent)
        return tile_n == kNarrowN ? ns_gemm_kernel<kNsPersistent, kNarrowN> : ns_gemm_kernel<kNsPersistent, kWideN>;
    return tile_n == kNarrowN ? ns_gemm_kernel<kNsPhased, kNarrowN> : ns_gemm_kernel<kNsPhased, kWideN>;
}

cudaError_t set_all_smem_attrs() {
    for (int mode : {kNsPhased, kNsPersistent})
        for (int n : {kWideN, kNarrowN}) {
            const cudaError_t e = cudaFuncSetAttribute(ns_kernel(mode, n), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                       static_cast<int>(kSmemBytes));
            if (e != cudaSuccess) return e;
        }
    return cudaSuccess;
}

// Per-device one-time set-up: the shared-memory opt-in of every
// instantiation (a function attribute holds for the device that was current
// when it was set) and the number of CTA pairs resident at once.  0 = not
// yet done on that device.
constexpr int kMaxDevices = 64;
std::mutex g_cfg_mu;
int g_pairs[kMaxDevices] = {};

cudaError_t configure_current_device(int* pairs) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_cfg_mu);
    if (g_pairs[dev] == 0) {
        e = set_all_smem_attrs();
        if (e != cudaSuccess) return e;
        // One CTA per SM either way (shared memory); the persistent
        // instantiation has the larger block.
        int n = 0;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(2, 1, 1);
        cfg.blockDim = dim3(ns_threads(kNsPersistent), 1, 1);
        cfg.dynamicSmemBytes = kSmemBytes;
        if (cudaOccupancyMaxActiveClusters(&n, ns_kernel(kNsPersistent, kWideN), &cfg) != cudaSuccess ||
            n <= 0) {
            cudaGetLastError();
            int sms = 0;
            e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
            if (e != cudaSuccess) return e;
            n = std::max(1, sms / 2);
        }
        g_pairs[dev] = n;
    }
    *pairs = g_pairs[dev];
    return cudaSuccess;
}

}  // namespace

// Number of CTA pairs that can be resident at once on the current device (the
// persistent grid); 1 if the device cannot be configured (the next launch
// then reports the error).
int ns_gemm_max_pairs() {
    int pairs = 0;
    if (configure_current_device(&pairs) != cudaSuccess) {
        cudaGetLastError();
        return 1;
    }
    return pairs;
}

cudaError_t ns_gemm_configure() {
    int pairs = 0;
    return configure_current_device(&pairs);
}

cudaError_t launch_ns_gemm(const NsParams& P, int mode, int grid_pairs, cudaStream_t s) {
    const cudaError_t ce = ns_gemm_configure();
    if (ce != cudaSuccess) return ce;
    const NsKernel kernel = ns_kernel(mode, P.cls[0].tile_n);
    const cudaError_t e = launch_chained(kernel, 2 * grid_pairs, ns_threads(mode), kSmemBytes, s, P);
    if (e != cudaSuccess) {
        cudaFuncAttributes fa{};
        cudaFuncGetAttributes(&fa, kernel);
        std::fprintf(stderr,
                     "malt: ns_gemm_kernel<%d> launch (%d CTAs x %d threads, %zu B dynamic smem, "
                     "%zu B parameters) refused: %s; kernel uses %d registers, %zu B static "
                     "smem, allows %d threads and %d B dynamic smem per block\n",
                     mode, 2 * grid_pairs, ns_threads(mode), kSmemBytes, sizeof(NsParams),
                     cudaGetErrorString(e), fa.numRegs, fa.sharedSizeBytes,
                     fa.maxThreadsPerBlock, fa.maxDynamicSharedSizeBytes);
    }
    return e;
}

}  // namespace malt
