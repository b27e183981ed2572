// common.cuh -- data structures shared by the host runtime and the kernels.
//
// Naming follows the paper: W weights, G gradient, M momentum, l / r row and
// column statistics, L / R their diagonal preconditioners, Mt = L M R, O the
// orthogonalised direction, D = L O R the back-mapped direction, nu the MALTER
// scalar.  "NS frame": Newton-Schulz runs on the wide orientation of Mt,
// p x q with p = min(m, n), q = max(m, n); a matrix with m > n is transposed.
#pragma once
#include <cstdint>
#include <cuda.h>
#include <cuda_bf16.h>

namespace malt {

// Statistics kernel tile (rows x cols of W per block).
constexpr int kStatRows = 64;
constexpr int kStatCols = 256;
// Prescale block (rows x cols of Mt).
constexpr int kPreRows = 64;
constexpr int kPreCols = 256;
// Apply kernel: contiguous elements per block (O is stored in W's layout, so
// wide and tall matrices stream alike).
constexpr int kApplyElems = 16384;
// Newton-Schulz GEMM: a CTA pair computes a kTileM x n output tile, n the set's
// tile width; each CTA owns kBM rows of it, loads kBM rows of A and n/2 rows (N)
// of B per kBK reduction slice (one 128-byte swizzle row of 16-bit elements).
constexpr int kBM = 128;
constexpr int kTileM = 2 * kBM;
constexpr int kWideN = 256;
constexpr int kNarrowN = 128;
constexpr int kBK = 64;
constexpr int kStages = 6;
constexpr int kBMN = 64;            // MN extent of one 128-byte swizzle atom (bf16)
constexpr int kEpiWarpsPerCta = 8;  // two per TMEM lane quarter
constexpr int kNsPartsPerTile = 2 * kEpiWarpsPerCta;  // graft partial pairs per tile
constexpr int kMaxClasses = 8;     // shape classes per GEMM launch
constexpr int kBindChunk = 128;    // parameters per pointer-binding launch
constexpr int kScalarsPerMat = 8;  // debug scalars per matrix

// Status bits set by kernels (OR-ed into the device status word).
constexpr int kStatusTimeout = 1;

// Caller pointers of one parameter for the current step (bound each step).
struct UserPtrs {
    void* w;
    const void* g;
    float* m;
    float* l;
    float* r;
    void* wcopy;    // bf16 copy of an fp32 W written by the apply pass, or null
};

// Static per-matrix description, built at init and kept on the device.
struct MatDesc {
    int32_t m, n;            // W is m x n
    int32_t trans;           // 1 when the NS frame is the transpose (m > n)
    int32_t p, q;            // NS frame shape
    int32_t w_bf16, g_bf16;  // element types of W and G
    int32_t cls, bidx;       // shape class and index within its batch
    int32_t stat_rb, stat_cb;       // statistics row bands / column chunks
    int32_t pre_tr, pre_tc;         // prescale blocks (kPreRows x kPreCols), rows and cols
    int32_t ns_tiles;               // GEMM tiles of one p x q product
    int32_t pad_;
    float* rowpart;          // [stat_cb][m] partial row sums of G^2
    float* colpart;          // [stat_rb][n] partial column sums of G^2
    float* L;                // [m]  (l + eps)^(-1/8)
    float* R;                // [n]  (r + eps)^(-1/8)
    float* prepart;          // [pre_tiles][2]  sum Mt^2, sum (L G R)^2
    float* nspart;           // [ns_tiles][kNsPartsPerTile][2]: sum O^2, sum D^2
    __nv_bfloat16* X0;       // NS-frame Mt (p x q, bf16): Mt, or Mt^T when trans
    __nv_bfloat16* O;        // orthogonalised direction in W's layout (m x n)
};

// Per-matrix scalars kept on the device (index = matrix).
struct MatScalars {
    float k;        // 1 / (||Mt||_F + ns_eps)
    float norm_mt;  // ||Mt||_F
    float lgr_sq;   // ||L G R||_F^2 (MALTER)
    float scale;    // lr * alpha * ||O|| / (||D|| + eps)
    float norm_o, norm_d, alpha, nu;
};

// The step count of a state and what follows from it alone.
struct StepClock {
    long long t;    // steps taken (1-based within a step)
    double bias;    // MALTER: sqrt(1 - mu2^t) / (1 - mu1^t + eps) of this step
};

struct StepHyper {
    float lr, mu1, mu2, eps, weight_decay;
    float ns_a, ns_b, ns_c, ns_eps;
    int32_t malter;
};

// ------------------------------------------------------ Newton-Schulz engine
enum GemmPhase : int32_t { kGram = 0, kPoly = 1, kBX = 2 };

// Launch modes of the Newton-Schulz kernel: one product with a static tile
// split, or a persistent work table of all products of the k iterations.
enum NsMode : int32_t { kNsPhased = 0, kNsPersistent = 1 };

// Epilogue warps of a CTA pair; each one signals a finished item once.
constexpr uint32_t kNsSignalsPerTile = 2 * kEpiWarpsPerCta;

// Stages of a persistent work table: operation s of a matrix's form.  In the
// iterated form the products of iteration i are stages 3 i + {kGram, kPoly,
// kBX}, and the table of k iterations is the first k iterations' entries of any
// longer one.
constexpr int kMaxNsSteps = 64;

// Buffers of a class that an operation reads or writes: the p x p matrices
// 0 .. 3 (0 holds A, 1 holds B' in the iterated form), the two iterates X, and
// the last iterate O.
constexpr int8_t kBufX = 4, kBufO = 6, kBufNone = -1;

// One product of a Newton-Schulz run:
//   out = gamma k^kx (a b) + beta e + alpha I
// with a read as K-major rows, b as K-major rows (Gram and p x p products; the
// p x p matrices are symmetric) or MN-major (kBX), and k = 1 / (||Mt|| + ns_eps).
struct NsOp {
    int8_t kind;            // GemmPhase: kGram X X^T (K = q), kPoly a p x p product (K = p), kBX
    int8_t f16, out16;      // operands (and e) fp16 instead of bf16; the output
    int8_t a, b, e, out;    // buffers
    int8_t kx;              // power of k that scales the product
    float alpha, beta, gamma;
};

// Operations of the longest grouped run (8 iterations in groups 1, 2, 2, 3).
constexpr int kMaxGroupedOps = 32;

// Product `kind` of iteration `iter` of the iterated form (X <- B' X).
__host__ __device__ __forceinline__ NsOp ns_iterated_op(int32_t iter, int32_t kind, bool last, float a,
                                                        float b, float c) {
    const int8_t cur = static_cast<int8_t>(kBufX + (iter & 1));
    NsOp o;
    o.kind = static_cast<int8_t>(kind);
    o.f16 = o.out16 = 0;
    o.kx = iter > 0 ? 0 : kind == kGram ? 2 : kind == kBX ? 1 : 0;
    o.a = kind == kGram ? cur : kind == kPoly ? 0 : 1;
    o.b = kind == kPoly ? 0 : cur;
    o.e = kind == kPoly ? 0 : kBufNone;
    o.out = kind == kGram ? 0 : kind == kPoly ? 1 : last ? kBufO : static_cast<int8_t>(kBufX + ((iter & 1) ^ 1));
    o.alpha = kind == kPoly ? a : 0.f;
    o.beta = kind == kPoly ? b : 0.f;
    o.gamma = kind == kPoly ? c : 1.f;
    return o;
}

// One item of a persistent work table.
struct __align__(16) NsEntry {
    int32_t code;     // stage (bits 0-11) | class slot (bits 12-15) | batch slot (bits 16-31)
    int32_t g;        // matrix; -1 marks the end of the table
    int32_t local;    // tile of the product
    uint32_t target;  // signals the previous stage of matrix g must reach (0: none)
};

__host__ __device__ __forceinline__ int32_t entry_stage(const NsEntry& e) { return e.code & 0xfff; }
__host__ __device__ __forceinline__ int32_t entry_cls(const NsEntry& e) { return (e.code >> 12) & 0xf; }
__host__ __device__ __forceinline__ int32_t entry_b(const NsEntry& e) {
    return static_cast<int32_t>(static_cast<uint32_t>(e.code) >> 16);
}

// Row stride of a p x p buffer: whole 32-byte sectors, which the epilogue loads at once.
__host__ __device__ __forceinline__ int32_t ns_ld(int32_t p) { return (p + 15) / 16 * 16; }

// One shape class (every matrix whose NS frame is p x q, stored batched) with
// the tensor maps of all its buffers.
struct NsClass {  // 64-byte aligned through its CUtensorMap members
    CUtensorMap tmK[6];           // p x p buffers 0 .. 3 and the iterates X as K-major rows (box kBK x tile_n / 2)
    CUtensorMap tmMn[6];          // the same buffers as an MN-major operand (box kBMN x kBK)
    CUtensorMap stK[6], stO;      // epilogue stores of the same buffers and of O: box 32 x 32, 64-byte swizzle
    CUtensorMap stOt;             // the O buffer as [q][p]: a tall W's O, stored in W's layout
    int32_t p, q, batch;
    int32_t tile_n;               // width of an output tile
    int32_t tiles_p, tiles_q;     // kTileM-high tiles along p, tile_n-wide ones along q
    int32_t sym_tiles;            // tiles of one matrix in a symmetric product
    int32_t item_begin;           // first item of this class in a phased launch
    int32_t can_group;            // the shape takes the grouped form when the run may
    int32_t grouped;              // this run's form
    int32_t bx_col_major;         // list B*X tiles column by column (X larger than kBxColBytes)
    const int32_t* mat_of;        // [batch] -> matrix index
    const uint16_t* A;            // p x p buffer 0 [batch][p][ns_ld(p)], 16-bit (read by the H epilogue)
};

// Work list of one launch.  Each class runs its form's operations in order
// (stage s = operation s); within a stage the items are the tiles of every
// class, batch slot by batch slot.  A phased launch runs one stage (items
// [0, item_end), static round-robin, class c's from cls[c].item_begin); a
// persistent launch runs all of them from a work table (claimed through
// *queue, each tile waiting for its matrix's previous stage in done[]).
struct NsParams {
    NsClass cls[kMaxClasses];
    NsOp ops[kMaxGroupedOps];     // the grouped form's operations
    int32_t nops;                 // their number (0: no class runs grouped)
    int32_t nclasses;
    int32_t nmat;                 // size of one row of done[]
    int32_t ns_steps;
    int32_t stage;                // phased launch: the stage it runs
    int32_t item_end;             // items of the launch
    int32_t sym_items, full_items;   // tiles of a symmetric product, of B*X, over all classes
    float a, b, c;
    const MatDesc* mats;
    MatScalars* scal;
    int32_t* status;
    uint32_t* queue;              // next unclaimed item (persistent schedule)
    uint32_t* done;               // [stages][nmat] finished-item signals (persistent)
    uint64_t budget_ns;
    const NsEntry* table;         // persistent launches: the work table (item_end entries)
};
static_assert(sizeof(NsParams) <= 32764, "NsParams is passed by value as the kernel parameter");

// Number of operations of a class in this launch's run, and operation s.
__host__ __device__ __forceinline__ int32_t ns_num_stages(const NsParams& P, const NsClass& C) {
    return C.grouped ? P.nops : 3 * P.ns_steps;
}
__host__ __device__ __forceinline__ NsOp ns_op(const NsParams& P, const NsClass& C, int32_t s) {
    if (C.grouped) return P.ops[s];
    const int32_t iter = s / 3;
    return ns_iterated_op(iter, s - 3 * iter, iter == P.ns_steps - 1, P.a, P.b, P.c);
}

// One decoded work item: an output tile of one product.
struct NsWork {
    NsOp op;
    int32_t cls, b;               // class and batch slot (matrix = cls.mat_of[b])
    int32_t mt, nt;               // tile row / column
    int32_t local;                // tile index within the matrix's product
};

// Tiles of one matrix in a product of this kind: all of them for B X, those that
// reach the diagonal or lie above it for the symmetric Gram and p x p products.
// Row r of tiles has those from column r * kTileM on.
// (tile_n is the class's, a constant of the kernel)
__host__ __device__ __forceinline__ int32_t ns_sym_row_tiles(int32_t p, int32_t tile_n, int32_t r) {
    return (p + tile_n - 1) / tile_n - r * (kTileM / tile_n);
}
__host__ __device__ __forceinline__ int32_t ns_phase_tiles(const NsClass& C, int32_t kind) {
    if (kind == kBX) return C.tiles_p * C.tiles_q;
    int32_t n = 0;
    for (int32_t r = 0; r < C.tiles_p; ++r) n += ns_sym_row_tiles(C.p, C.tile_n, r);
    return n;
}

// B*X tile order.  Row by row, the tiles that run at once read every column
// block of X; column by column, they read a few column blocks and all of B'
// (p x p).  Once one matrix's X is large against L2 (a 4096 x 16384 frame is
// 134 MB), row order reads X from DRAM once per wave of tiles: column order
// then cuts its DRAM reads five-fold and its time by 13 %.  Where X fits in
// L2 row order measured about 1.5 % faster (GPT-2 Large), so it stays there.
constexpr int64_t kBxColBytes = 32ll << 20;

// Tile row / column of the rem-th tile of one matrix's product of this kind:
// B*X row by row or column by column (bx_col_major), the upper triangle of
// the symmetric products row by row.
__host__ __device__ __forceinline__ void ns_tile_coords(const NsClass& C, int32_t tile_n, int32_t kind,
                                                        int32_t rem, int32_t* mt, int32_t* nt) {
    if (kind == kBX) {
        if (C.bx_col_major) {
            *nt = rem / C.tiles_p;
            *mt = rem - *nt * C.tiles_p;
        } else {
            *mt = rem / C.tiles_q;
            *nt = rem - *mt * C.tiles_q;
        }
        return;
    }
    const int32_t step = kTileM / tile_n;
    int32_t r = 0, u = rem, row = ns_sym_row_tiles(C.p, tile_n, 0);
    while (u >= row) {
        u -= row;
        row -= step;
        ++r;
    }
    *mt = r;
    *nt = r * step + u;
}

// Blocks of the apply pass of one matrix: kApplyElems contiguous elements
// (O is stored in W's layout for every matrix).
__host__ __device__ __forceinline__ int32_t mat_apply_blocks(const MatDesc& d) {
    return static_cast<int32_t>((static_cast<int64_t>(d.m) * d.n + kApplyElems - 1) / kApplyElems);
}

// Item `item` of a phased launch (stage P.stage of every class that has it).
__host__ __device__ __forceinline__ NsWork ns_decode(const NsParams& P, int32_t tile_n, int32_t item) {
    NsWork w;
    int32_t c = 0;
    while (c + 1 < P.nclasses && item >= P.cls[c + 1].item_begin) ++c;
    const NsClass& C = P.cls[c];
    w.op = ns_op(P, C, P.stage);
    const int32_t local = item - C.item_begin;
    const int32_t per = w.op.kind == kBX ? C.tiles_p * C.tiles_q : C.sym_tiles;
    w.cls = c;
    w.b = local / per;
    const int32_t rem = local - w.b * per;
    w.local = rem;
    ns_tile_coords(C, tile_n, w.op.kind, rem, &w.mt, &w.nt);
    return w;
}

}  // namespace malt
