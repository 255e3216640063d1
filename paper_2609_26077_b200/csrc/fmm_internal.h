// Internal declarations shared by the translation units of the library (not part of the C ABI).
#pragma once
#include <cuda_runtime.h>
#include <cuda.h>
#include <stdint.h>
#include <atomic>
#include "../../include/fmm.h"
#include "fmm_walk.h"

#define FMM_MAX_LEVELS 3

// One destination of a product in C: block origin, weight, and whether this is the first product written there (store) or a
// later one (accumulate, behind the one before).  FP32 scales.
struct FmmOutEntry {
    int row_off;   // element row of the destination block origin in C
    int col_off;   // element column
    float w;       // product of the W coefficients along the recursion path
    int gap;       // 0: overwrite; else add, and the previous update of this block is so many updates ago
};

// One step of the fp32-scale product kernel's walk over the leaf products: which term it multiplies, the factor of the
// previous step's sum that its accumulators start from, and where the sum goes (see fmm_walk.h).
struct FmmWalkEntry {
    int term;
    float carry;              // 0 at the first product of a parent
    int out0, out1;           // entries [out0, out1) of the FmmOutEntry table
};

// Store guard of the FMM_DEBUG build (the stand-in for a memory checker, which this library cannot count on
// having): the address ranges a launch may write, and where to report a store that falls outside them.  Every
// launch fills it in; the kernels test it only when compiled with -DFMM_DEBUG - a bad store is then skipped and its
// location code goes to *status (first one wins, nothing traps).
struct FmmGuard {
    const char* lo[2];
    const char* hi[2];
    int* status;
};
#if defined(FMM_DEBUG) && defined(__CUDACC__)
__device__ __forceinline__ bool fmm_guard_ok(const FmmGuard& g, const void* ptr, size_t bytes, int code)
{
    const char* c = static_cast<const char*>(ptr);
    if ((c >= g.lo[0] && c + bytes <= g.hi[0]) || (c >= g.lo[1] && c + bytes <= g.hi[1])) return true;
    if (g.status) atomicCAS(g.status, 0, code);
    return false;
}
#define FMM_GUARD(g, ptr, bytes, code) fmm_guard_ok(g, ptr, bytes, code)
#else
#define FMM_GUARD(g, ptr, bytes, code) true
#endif
static inline FmmGuard fmm_make_guard(const void* a, size_t na, const void* b, size_t nb, int* status)
{
    FmmGuard g;
    g.lo[0] = static_cast<const char*>(a); g.hi[0] = g.lo[0] + na;
    g.lo[1] = static_cast<const char*>(b); g.hi[1] = g.lo[1] + nb;
    g.status = status;
    return g;
}
// status word that receives guard violations: plan->d_status[FMM_GUARD_WORD]
#define FMM_GUARD_WORD 2

// Pair-fused decoder (UE8M0 product kernel): the R products of a parent are walked in an order in which consecutive
// products (2s, 2s+1) form a step; the epilogue keeps product A on chip until product B is done and sends ONE weighted
// update wA * M_A + wB * M_B to every output block either of them feeds, which cuts the number of block updates that
// go through L2 (18 -> 11 for the Phi-optimal realization, 12 -> 9 for Strassen).  An unpaired last product is a step
// with wA = 0.
struct FmmPairEntry {
    int row_off, col_off;     // destination block, in units of leaf blocks
    float wA, wB;             // weights of the step's first and second product (wA = 0: first product absent / not used)
    int first;                // 1: overwrite, 0: add
};

struct FmmLayout {            // byte offsets into the workspace
    int64_t m, n, k;          // leaf dimensions
    int64_t terms;            // R^levels (1 for levels == 0)
    size_t qa, qb;            // e4m3 codes, terms x m x k and terms x n x k
    size_t sa, sb;            // scales
    size_t sa_term, sb_term;  // bytes of scales per term
    size_t sb_down;           // fp32 scales per column: the B-side scales times fmm_scale_down, as the product kernels read them
    size_t inter_a[FMM_MAX_LEVELS], inter_b[FMM_MAX_LEVELS];  // fp32 combinations of outer levels
    size_t dec[FMM_MAX_LEVELS];   // dec[l]: R^l partially decoded products of (M/2^l) x (N/2^l) fp32, l = 1 .. levels-1
    size_t total;
};

// The product kernels promote a K block's partial product P as (P * sB) * sA: P * (sA * sB) makes the block-32 kernel 5 to 7 %
// slower.  |P| reaches 32 * 448^2 < 2^22.7 and sB 2^119.2, so P * sB could overflow (operands of B above 2e34) where the result
// does not.  The B-side encoder therefore writes its scales a second time, times this power of two, for the product kernels
// (n = 8192: 15 of 390 MB), and their sums are multiplied back up when they go out: the same bits for results above 1e-33.
// With a clamp (amax_floor) so low that the smallest product would leave the normal range, 1.
static inline bool fmm_scale_per_column(const fmm_quant_params_t& qp) { return qp.scale_mode == FMM_SCALE_FP32_AMAX_DIV_448 && qp.b_tile_n == 0; }
static inline float fmm_scale_down(const fmm_quant_params_t& qp) { return qp.amax_floor >= 3e-26f ? 0x1p-14f : 1.0f; }
// the factor that the sums, or their weights, carry in return
static inline float fmm_scale_up(const fmm_quant_params_t& qp) { return fmm_scale_per_column(qp) ? 1.0f / fmm_scale_down(qp) : 1.0f; }

struct fmm_plan {
    int rank, levels;
    fmm_quant_params_t qp;
    float U[FMM_MAX_RANK][4], V[FMM_MAX_RANK][4], W[FMM_MAX_RANK][4];
    int terms;
    int device, sms;
    fmm_product_shape_t forced;   // fmm_force_product_shape; kernel 0: none
    struct FmmHostLanes* lanes;   // streams and events of fmm_matmul_host
    // device tables
    int* d_status;            // [64] status words (word 0: first bounded wait that gave up)
    FmmWalkEntry* d_walk;     // [2 * terms]: with carried sums, and without
    unsigned small_weights;   // carried sums: bit s = a weight of step s of a parent is below 1 in magnitude
    FmmOutEntry* d_out;       // [total entries], block offsets in units of leaf blocks (scaled at launch)
    int order[FMM_MAX_RANK];  // pair-fused decoder: walk order of the R products of a parent
    int steps;                // pair-fused decoder: steps per parent, ceil(R / 2)
    int updates;              // of a parent's output blocks, by the walk with carried sums or by the pair-fused decoder
    int* d_pair_start;        // [parents * steps + 1]
    FmmPairEntry* d_pair;     // entries of all steps
    // kernels launched by the most recent call on this plan; written once, at the end of a call (calls take the
    // plan as const, and two host threads may share one)
    mutable std::atomic<int> last_launches;
};

struct EncodeParams {
    const float* in;          // batch of matrices, each 2*rows x 2*cols (or rows x cols when nq == 1)
    int64_t in_batch_stride;  // elements between consecutive input matrices
    int64_t ld;               // leading dimension of the input matrices
    int batch;                // number of input matrices
    int rows, cols;           // leaf (output) dimensions per combination
    int64_t qoff[4];          // element offsets of the four input blocks that are combined
    int64_t qoff_outer[4];    // two-level kernels: offsets of the four blocks of the outer level
    int nq;                   // number of input blocks read (4, or 1 for a plain pass over one matrix)
    int R;                    // combinations per input matrix
    float coef[FMM_MAX_RANK][4];
    uint8_t* q_out;           // codes, term t = b * R + r at q_out + t * q_term
    int64_t q_term;           // rows * cols, or more when the launch covers a strip of the rows (A) / columns (B) of every term
    void* s_out;              // scales
    int64_t s_term_stride;    // bytes between the scale arrays of consecutive terms
    int64_t s_down;           // B side, one fp32 scale per column: bytes from a scale to its copy times `down` (fmm_scale_down)
    float down;
    int s_step;               // rows (A side) / columns (B side) by which combination r is shifted inside a shared scale array
    int s_ld;                 // fp32 scales: columns of B / rows of A that the shared scale array covers
    int sf_blocks;            // UE8M0: number of 128-row blocks of the scale-tile array
    int cpt;                  // A side: 128-k chunks per task; B side: blocks that it prefetches ahead, 0: none (set by the launcher)
    float amax_floor;
    short b_tile;             // B side: 128 = one fp32 scale per 128 x 128 tile (blk 128 only), 0 = per column
    short preround_bf16;      // B side: round each combination to bfloat16 before the maximum and the cast
    int overlap_prev;         // B side: the kernel launched just before on the stream is the A-side encoder of the same
                              // call (nothing this kernel reads): it may start while that one drains.  A side: that kernel is
                              // combinations of the same call: it may be set up while that one drains
    FmmGuard guard;           // codes and scales of this side
};
// a launch with more parameter bytes takes the host 0.35 us longer (n = 256: 10.2 -> 10.5 us a call)
static_assert(sizeof(EncodeParams) <= 352, "encoder parameters");

struct CombParams {
    const float* in;
    int64_t in_batch_stride, ld;
    int batch, rows, cols, R;
    float coef[FMM_MAX_RANK][4];
    float* out;               // dense rows x cols per (b, r)
    FmmGuard guard;
};

// One outward step of the decoder: out[b] (2*rows x 2*cols, block q at (q>>1, q&1)) = sum_r W[r][q] * in[b*R + r]
struct DecodeParams {
    const float* in;          // batch * R matrices, rows x cols each, dense
    float* out;               // batch matrices, 2*rows x 2*cols each, dense
    int batch, rows, cols, R;
    float W[FMM_MAX_RANK][4];
    FmmGuard guard;
};
// steps: 1, or 2 outward steps at once (batch 1; rows x cols and W as for the inner step)
fmm_status_t fmm_launch_decode(const DecodeParams& p, int steps, cudaStream_t st);
// one level of combinations of the two sides (a side with rows == 0 has none); overlap: behind another such launch
fmm_status_t fmm_launch_comb(const CombParams& a, const CombParams& b, bool overlap, cudaStream_t st);
fmm_status_t fmm_launch_encode_a(EncodeParams p, int blk, int mode, cudaStream_t st);
// both sides of a small call in one launch: false if it is not one, or has coefficients without kernels of their own
bool fmm_launch_encode_both(EncodeParams a, const EncodeParams& b, int blk, int mode, cudaStream_t st, fmm_status_t* status);
fmm_status_t fmm_launch_encode_b(EncodeParams p, int blk, int mode, cudaStream_t st);
// last two recursion levels in one pass (p.rows x p.cols = leaf dimensions, inputs 4*rows x 4*cols)
bool fmm_encode2_supported(bool b_side, int blk, int b_tile, int preround_bf16);
fmm_status_t fmm_launch_encode2_a(const EncodeParams& p, int blk, int mode, cudaStream_t st);
fmm_status_t fmm_launch_encode2_b(const EncodeParams& p, int mode, cudaStream_t st);

struct GemmParams {
    const uint8_t* qa; const uint8_t* qb;   // terms x m x k, terms x n x k
    const void* sa; const void* sb;         // sb, one fp32 scale per column: times fmm_scale_down
    int64_t sa_term, sb_term;               // bytes per term
    float up;                               // fmm_scale_up
    unsigned small_weights;                 // fmm_plan::small_weights
    float* C; int64_t ldc;                  // full output
    int64_t Mfull, Nfull;
    int m, n, k, terms;
    int msub, nsub;                         // output rows / columns of every leaf block this launch covers (m, n: all of them); the
                                            // pointers above then point at the strip's first row and column
    const FmmWalkEntry* walk; const FmmOutEntry* out;  // walks (with carried sums, and from `terms` on without) and decoder of the fp32-scale kernel
    const int* pair_start; const FmmPairEntry* pair;   // pair-fused decoder tables (UE8M0 kernel)
    int order[FMM_MAX_RANK]; int steps;
    int device, sms;                        // the plan's device and its SM count
    int R, nq;                              // products per parent; blocks of a parent's matrix (4, or 1 for the cubic product)
    int updates;                            // fmm_plan::updates
    const float (*W)[4];                    // innermost decoder, R x 4 (host pointer; unused when nq == 1)
    int* status;
    int terms_per_group;                    // consecutive terms that feed the same output blocks (R at levels >= 2, else all)
    int sb_tile;                            // fp32 scales, blk 128: the B-side scale is constant over each 128-column tile
    fmm_product_shape_t forced;             // kernel 0: the launcher chooses
    int overlap_prev;                       // the kernel launched just before on the stream is the B-side encoder of the same call:
                                            // the product kernel may be set up while that one drains (its loads wait for it)
    FmmGuard guard;                         // the output matrix (C, or the stack of parent matrices)
};
// guard word of the statistics kernels, which have no plan (FMM_DEBUG build; always 0 otherwise)
fmm_status_t fmm_stats_guard_read(int* code);
fmm_status_t fmm_launch_bounded_wait_selftest(int* status, unsigned long long limit_ns, cudaStream_t st);
fmm_status_t fmm_launch_guard_selftest(int* status, cudaStream_t st);
// Tile shape (CTAs per tile, columns) with which the persistent kernel takes a leaf of m x n, its time in microseconds by the
// model the choice is made with, and the terms that its busiest CTA (pair) walks
struct GemmShape { int ncta, bn; float time; long long longest; };
GemmShape fmm_gemm_shape(const GemmParams& p, int blk, int mode, int m, int n);
// How the cluster kernel (fmm_split.cu) takes this product: K shares per term and columns per tile; 0 shares: the persistent
// kernel is faster
struct SplitChoice { int ksplit, bn, terms, places; };        // terms: of a CTA; places: clusters that the device holds at once
SplitChoice fmm_split_choice(const GemmParams& p, int blk, int mode);
// The forced shape, or the one that is expected to be fastest.  The kernel is chosen for the whole problem (m, n), also when
// a launch covers a strip of it (msub, nsub): the strips' results do not depend on the cut
fmm_product_shape_t fmm_choose_product(const GemmParams& p, int blk, int mode);
bool fmm_product_shape_exists(const fmm_product_shape_t& s, int blk, int mode, int sb_tile, int R);
fmm_status_t fmm_launch_split(const GemmParams& p, int blk, int mode, SplitChoice c, cudaStream_t st);
// The kernel that keeps a parent's output blocks on chip (fmm_keep.cu), for R > 1, and whether it is expected to take the problem in
// less time than the cluster kernel (`split`, where that has K shares) or else the persistent kernel with the tile shape `tile`, whose
// busiest CTA (pair) walks `longest` terms
bool fmm_keep_faster(const GemmParams& p, int blk, int mode, const SplitChoice& split, const GemmShape& tile);
fmm_status_t fmm_launch_keep(const GemmParams& p, int blk, int mode, cudaStream_t st);
fmm_status_t fmm_launch_gemm(const GemmParams& p, int blk, int mode, cudaStream_t st, int* launches);

// SMs of the current device (a cached host-side attribute: cheap); 1 where it cannot be read
static inline int fmm_sm_count()
{
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) cudaGetLastError();
    return n > 0 ? n : 1;
}

static inline int64_t fmm_ipow(int64_t b, int e) { int64_t r = 1; while (e-- > 0) r *= b; return r; }
