// The R^levels block-scaled fp8 sub-products and the fused post-addition (paper Sec. 2.1:
// c = sum_r <U_r,a><V_r,b> W_r; the products M_r = S_r^ * T_r^ of the quantized combinations are
// accumulated in fp32 and carried into the output blocks by the decoder W_r).
//
// A persistent CTA (NCTA == 1) or CTA pair on two adjacent SMs (NCTA == 2, tcgen05 cta_group::2)
// owns an output tile POSITION - the same (NCTA*128) x BN tile in every output block of C - and
// walks all terms for it, so the W-weighted accumulation into C is race-free and deterministic.
//
//   warp 0      TMA producer: K-major e4m3 tiles of S_r and T_r (128-byte swizzle), and where warp 2 does not their scales.
//               In a pair each CTA loads its own 128 rows of S_r and its own half of the T_r tile.
//   warp 1      tcgen05.mma issuer (the even CTA of a pair issues for both), fp32 accumulators in TMEM
//   warps 2, 3  FP32 scales: scale producer, or (block 32) the two output warps, see MODE_FP32_OUT_WARP
//   warps 4..11 epilogue (two warpgroups, given most of the register file with setmaxnreg): TMEM -> registers -> (x W[r][q]) -> swizzled smem -> TMA store / TMA
//               add-reduce into the C blocks (the read-modify-write happens in L2, not in the SM)
//
// Scale handling:
//   UE8M0 mode  kind::mxf8f6f4.block_scale: the power-of-two block scales are copied to TMEM with
//               tcgen05.cp and applied by the tensor core; one accumulation over the whole K.
//   FP32 mode   (the paper's scale = amax/448 in fp32 on BOTH sides, per 1 x blk block): no
//               tensor-core path can apply a per-row x per-column fp32 factor per K block, so
//               each K block's partial product is accumulated on its own in TMEM
//               (kind::f8f6f4) and promoted on the CUDA cores: acc += (P * sB[col]) * sA[row],
//               sB scaled down by a power of two against overflow (fmm_scale_down), two columns per instruction (fp32x2), overlapped with the next TMEM load.
//
// Every wait is bounded: on time-out a status word is set and all roles leave the kernel.
#include <algorithm>
#include "fmm_gemm_common.cuh"

namespace {

// Internal fourth mode: FP32 scales (per column, as mode 0) with two output warps.  The promoting warps hand a finished
// product to them through a shared-memory copy of the (unweighted) accumulators, half of the rows to each, and go straight on
// with the next term; the W-weighted stores / add-reductions then overlap the next term's promotion instead of stalling it.
// One output warp was the bound of all but the longest terms: n = 4096, T* (16 stages a term) 265 -> 249 us, 4096 x 2048 x 4096
// 153 -> 139; cubic and n = 8192 as before.  To make room one warp produces operands and scales.  Four output warps in a
// block of 512 threads: short terms 5 % faster still, cubic 8 % slower (the promotion loop compiled for fewer registers).
constexpr int MODE_FP32_OUT_WARP = 3;
constexpr int SEPARATE_STAGES = 16;        // block 32: K stages of a term from which on every product is summed on its own, see launch()

constexpr int EPI_WARPS = 8;               // two per TMEM lane quadrant, each half of the tile's columns
constexpr int EPI_WARP0 = 4;               // warps 0..3: operand producer, MMA issuer, and two that produce scales or write the output
constexpr int NUM_THREADS = (EPI_WARP0 + EPI_WARPS) * 32;
// setmaxnreg budget: the CTA's register pool is NUM_THREADS x (registers at launch); an increase
// beyond what the decrease freed would block forever, so every split is checked (see Cfg).
constexpr int REGS_AT_LAUNCH = 168;
static_assert(NUM_THREADS * (REGS_AT_LAUNCH + 8) > 65536, "REGS_AT_LAUNCH must be the launch-bound maximum");

template <int BN, int MODE, int BLK, int NCTA>
struct Cfg {
    static constexpr bool MX = (MODE == FMM_SCALE_UE8M0_CEIL);
    // FP32 scales per column: the promoting warps read the accumulators with the 16-lane load shape, four rows x
    // CW/4 columns per thread (see the promotion loop).  The weight-tile mode has no per-column scale loads to
    // save and is faster with one row per thread.
    static constexpr bool ROWS4 = !MX && MODE != MODE_FP32_SB_TILE;
    static constexpr bool DUMP = (MODE == MODE_FP32_OUT_WARP);
    // Register split between the four control warps and the eight epilogue warps.  Block 128 gives the promoting warps all
    // they can (accumulators, two TMEM chunks, scales).  Block 32 with output warps needs less: with 176 to 200 registers
    // ptxas finds a promotion loop that is 3 % faster than with 208 or more, with 168 it is 3 % slower (cubic n = 4096 233.4,
    // 240.9, 247.5 us; block 128 is 2 to 7 % slower with fewer than 224).  Every split is one that ptxas spills nothing with.
    // The weight-tile kernel needs 216 for two TMEM loads in flight beside 128 sums a thread.
    static constexpr bool TILE = MODE == MODE_FP32_SB_TILE;
    static constexpr int REGS_CTRL = MX || DUMP ? 88 : TILE || BLK == 32 ? 72 : 56, REGS_EPI = MX ? 208 : DUMP ? 192 : TILE || BLK == 32 ? 216 : 224;
    static_assert(EPI_WARP0 * 32 * REGS_CTRL + EPI_WARPS * 32 * REGS_EPI <= NUM_THREADS * REGS_AT_LAUNCH, "register pool");
    // Warp index, CTA rank and TMEM base as values the compiler knows to be warp-uniform (see warp_uniform): 3 % of the
    // block-32 kernel at n = 8192 and 4096, 7 % of the single-CTA UE8M0 kernel at 1280 x 2816 x 3328.  Not for the UE8M0
    // pair kernel, whose 256-column instructions hide their issue (2 % slower), nor for the weight-tile pair kernel, which
    // then spills in the promotion loop (10 % slower at n = 4096); the weight-tile kernel of single CTAs, whose 128-column
    // instructions do not hide it, gains 19 % (n = 4096 Winograd 105 -> 84.5 us, Phi-optimal 117 -> 99, cubic 98 -> 76).
    static constexpr bool UNIFORM = !(MX && NCTA == 2) && !(TILE && BN == 256);
    static constexpr int BROWS = BN / NCTA;                  // T_r rows this CTA loads per stage
    static constexpr int A_BYTES = BM * BK;
    static constexpr int B_BYTES = BROWS * BK;
    // The UE8M0 pair kernel keeps one staging chunk per epilogue warp: its shared memory goes to the operand stages,
    // and a second chunk in flight per warp was measured slower (more output traffic competing with the loads).
    static constexpr int STAGING_BUFS = (MX && NCTA == 2) ? 1 : 2;
    static_assert(!DUMP || (BN == 128 && BK / BLK == 4), "output-warp mode: 128-column tiles, block 32");
    static constexpr int STAGES = (MX && NCTA == 2) ? 5 : ((A_BYTES + B_BYTES) > 40000 || DUMP ? 3 : 4);
    // DUMP (output-warp mode): shared-memory copy of a finished product, BM x BN fp32
    static constexpr int DUMP_BYTES = DUMP ? BM * BN * 4 : 0;
    // output chunk of one epilogue warp: 32 rows x CH fp32, staged in shared memory for one TMA store.  Rows of 128
    // bytes everywhere: a TMA add-reduction of 64-byte rows runs at half the bytes per clock (11 against 21 per SM,
    // measured; plain stores 25 either way), which costs the UE8M0 pair kernel more than its sixth operand stage,
    // bought with 16-column chunks, gave (two levels at n = 8192: 0.579 -> 0.556 ms; one level 0.451 -> 0.447 ms).
    static constexpr int CH = 32;
    static constexpr int STAGING_BYTES = 32 * CH * 4;
    static constexpr int SFB_ATOMS = BN / 128;
    static constexpr int SF_STAGE_BYTES = MX ? (512 + SFB_ATOMS * 512) : 0;
    static constexpr int KB_PER_STAGE = BK / BLK;
    // depth of the scale ring: scales are small, so in the block-32 kernel with output warps, which has the room,
    // they run several stages ahead of the operand tiles (2.5 % for the cubic product at n = 8192, neutral for rank 7)
    static constexpr int SB_STAGES = STAGES + (DUMP ? 5 : 1);
    // FP32 modes: one stage of the scale ring = the B-side scales of the stage's K blocks (KB x BN fp32, stored
    // K-block-major) followed by the A-side scales of this CTA's 128 rows (128 x KB fp32: the A side stores the KB
    // scales of a 128-k chunk next to each other per row, one contiguous piece per stage)
    static constexpr int SB_PART_BYTES = MX ? 0 : KB_PER_STAGE * BN * 4;
    static constexpr int SB_STAGE_BYTES = MX ? 0 : KB_PER_STAGE * (BN + BM) * 4;
    static constexpr int TX_BYTES = NCTA * (A_BYTES + B_BYTES + SF_STAGE_BYTES);
    static constexpr int OFF_A = 0;
    static constexpr int OFF_B = OFF_A + STAGES * A_BYTES;
    static constexpr int OFF_STG = OFF_B + STAGES * B_BYTES;
    static constexpr int OUT_BUFS = 8;          // DUMP: staging chunks of the two output warps
    static constexpr int OFF_DUMP = OFF_STG + (DUMP ? OUT_BUFS * 4096 : EPI_WARPS * STAGING_BUFS * STAGING_BYTES);
    static constexpr int OFF_SF = OFF_DUMP + DUMP_BYTES;
    static constexpr int OFF_SB = OFF_SF + STAGES * SF_STAGE_BYTES;
    static constexpr int OFF_BAR = OFF_SB + SB_STAGES * SB_STAGE_BYTES;
    // FP32: the signals "K blocks multiplied" are a ring of their own, GROUPS per stage of the scale ring
    static constexpr int GPB = MX ? 1 : ((KB_PER_STAGE >= 2 && 512 / BN >= 4) ? 2 : 1);
    static constexpr int GROUPS = KB_PER_STAGE / GPB;
    static constexpr int FULL_SLOTS = MX ? 1 : SB_STAGES * GROUPS;
    static constexpr int NUM_BARS = 2 * STAGES + SB_STAGES + FULL_SLOTS + 4 + 4;
    static constexpr int SMEM_BYTES = OFF_BAR + NUM_BARS * 8 + 16 + 1024;   // + alignment slack
    // TMEM: MX: one BN-column accumulator, then per stage 4 SFA + 4*(BN/128) SFB columns.
    //       FP32: ring of 512/BN accumulators, one per K block in flight.
    // FP32: GPB consecutive K blocks ("granules") share one completion signal: their MMAs are issued back to
    // back into adjacent TMEM buffers and committed once, so the tensor pipe is not drained per K block.
    static constexpr int ACC_BUFS = MX ? 1 : (512 / BN) / GPB;        // ring of (GPB x BN)-column super-buffers
    static constexpr int SF_COLS = 4 + 4 * SFB_ATOMS;
    // UE8M0: TMEM columns [0, BN) accumulator, [BN, BN + SF_COLS) the scale factors of the stage being multiplied (one
    // slot: tcgen05.cp and tcgen05.mma execute in issue order), then the HOLD area of the pair-fused decoder: every
    // epilogue warp parks CW - 16 columns of a finished product there (the other 16 stay in registers) until the
    // product it is paired with is done.
    static constexpr int HOLD_T = MX ? (BN / 2 - 16) : 0;          // parked columns per warp
    static constexpr int OFF_HOLD = BN + 16;
    static constexpr int CW = BN / 2;      // columns per epilogue warp
    static_assert(SMEM_BYTES <= 232448, "shared memory budget");
    static_assert(!MX || (SF_COLS <= 16 && OFF_HOLD + 2 * HOLD_T <= 512), "TMEM budget");
    static_assert(!MX || HOLD_T == 112 || HOLD_T == 48, "hold area is parked with 32- and 16-column stores");
};

// Self-test of the bounded wait: one warp waits on a barrier that nothing ever signals; the wait must
// give up after limit_ns, record `where` in the status word and let the kernel end normally.
__global__ void bounded_wait_selftest_kernel(int* status, unsigned long long limit_ns, int where)
{
    __shared__ __align__(8) unsigned long long bar;
    __shared__ int abort_flag;
    if (threadIdx.x == 0) { mbar_init(smem_u32(&bar), 1); abort_flag = 0; fence_barrier_init(); }
    __syncthreads();
    Ctl ctl{&abort_flag, status, limit_ns};
    const bool ok = mbar_wait_warp(smem_u32(&bar), 0, ctl, where);
    if (threadIdx.x == 0 && ok) atomicExch(status + 1, 1);      // must not happen: nothing arrives on the barrier
}

struct KParams {
    const uint8_t* sa; const uint8_t* sb;   // scale arrays (bytes); fp32 mode only
    long long sa_term, sb_term;
    int m, n, k, terms;
    int msub, nsub;                          // rows and columns of a leaf that this launch multiplies (m and n, or a strip)
    // Work items.  A slot is (term group, tile position): the terms of one group (the R products of one parent
    // at the innermost level; all terms at one level) feed one set of output blocks and are walked by one CTA
    // (pair) in order.  (Cutting the slots of a short last wave into narrower items does not pay: a tcgen05.mma of
    // half the width takes as long to issue, measured 4 % slower at n = 8192.)
    int positions, tiles_n, terms_per_group, items;      // tiles_n: tile positions per row of positions
    const FmmWalkEntry* walk; const FmmOutEntry* out;  // FP32 scales
    const int* pair_start; const FmmPairEntry* pair;   // pair-fused decoder (UE8M0): steps of two products, see FmmPairEntry
    int order[FMM_MAX_RANK]; short steps;     // walk order of the R products of a parent; steps = ceil(R / 2)
    unsigned char R, small_weights;           // output warps, bit s: step s of a parent has weights below 1
    float up;                                 // factor of the sums (GemmParams)
    int* status;
    const float* c_base; long long ldc;       // the output matrix as plain memory: used by the FMM_DEBUG store guard only
    FmmGuard guard;
};
// no larger than it was: parameter bytes are host time per launch, see EncodeParams
static_assert(sizeof(KParams) <= 208, "product kernel parameters");

template <int BN, int MODE, int BLK, int NCTA>
__global__ void __launch_bounds__(NUM_THREADS, 1)
fmm_gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                const __grid_constant__ CUtensorMap tmC, const __grid_constant__ CUtensorMap tmSFA,
                const __grid_constant__ CUtensorMap tmSFB, const KParams p)
{
    using C = Cfg<BN, MODE, BLK, NCTA>;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw_addr = smem_u32(smem_raw);
    const uint32_t base = (raw_addr + 1023u) & ~1023u;
    uint8_t* base_ptr = smem_raw + (base - raw_addr);

    const uint32_t bar0 = base + C::OFF_BAR;
    auto bar_full = [&](int s) { return bar0 + 8u * s; };
    auto bar_empty = [&](int s) { return bar0 + 8u * (C::STAGES + s); };
    auto bar_sempty = [&](int s) { return bar0 + 8u * (2 * C::STAGES + s); };
    auto bar_tfull = [&](int b) { return bar0 + 8u * (2 * C::STAGES + C::SB_STAGES + b); };
    auto bar_tempty = [&](int b) { return bar0 + 8u * (2 * C::STAGES + C::SB_STAGES + C::FULL_SLOTS + b); };
    // DUMP: half of the rows of the accumulator copy is written, and consumed
    auto bar_dfull = [&](int i) { return bar0 + 8u * (2 * C::STAGES + C::SB_STAGES + C::FULL_SLOTS + 4 + i); };
    auto bar_dempty = [&](int i) { return bar_dfull(i) + 16u; };
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(base_ptr + C::OFF_BAR + C::NUM_BARS * 8);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    // DUMP: factor that a half of the accumulator copy is written with, for the step that it is free for
    volatile float* dump_up = reinterpret_cast<volatile float*>(tmem_slot + 2);
    const Ctl ctl{abort_flag, p.status};

    auto uniform = [](uint32_t v) { return C::UNIFORM ? warp_uniform(v) : v; };
    const int warp = uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
    const int cta_rank = (NCTA == 2) ? (int)uniform(cluster_ctarank()) : 0;
    const bool leader = (cta_rank == 0);
    const int unit = blockIdx.x / NCTA;            // CTA or CTA pair index
    const int units = gridDim.x / NCTA;

    if (threadIdx.x == 0) {
        for (int s = 0; s < C::STAGES; ++s) { mbar_init(bar_full(s), 1); mbar_init(bar_empty(s), 1); }
        for (int s = 0; s < C::SB_STAGES; ++s) mbar_init(bar_sempty(s), EPI_WARPS);
        // the first K blocks of a stage are signalled together with the stage's scales
        for (int b = 0; b < C::FULL_SLOTS; ++b) mbar_init(bar_tfull(b), !C::MX && b % C::GROUPS == 0 ? 2 : 1);
        for (int b = 0; b < 4; ++b) mbar_init(bar_tempty(b), NCTA * EPI_WARPS);
        for (int i = 0; i < 2; ++i) { mbar_init(bar_dfull(i), EPI_WARPS / 2); mbar_init(bar_dempty(i), 1); }
        *abort_flag = 0;
        if (C::DUMP) dump_up[0] = dump_up[1] = p.small_weights & 1 ? 1.0f : p.up;
        fence_barrier_init();
    }
    if (warp == 1) {
        tmem_alloc<NCTA>(smem_u32(tmem_slot), 512);
        tmem_relinquish<NCTA>();
    }
    tc_fence_before();
    __syncthreads();
    if (NCTA == 2) cluster_sync();                 // the peer's barriers are initialised before anyone signals them
    tc_fence_after();
    const uint32_t tmem_base = uniform(*tmem_slot);

    const int tiles_n = p.tiles_n;
    const int kstages = p.k / BK;
    const int nkb = p.k / BLK;
    // ti-th product a CTA (pair) walks in work-item group grp: the parents of the group one after the other, the R
    // products of a parent in the plan's walk order
    auto term_of = [&](int grp, int ti) {
        if constexpr (C::MX) return grp * p.terms_per_group + (ti / p.R) * p.R + p.order[ti % p.R];
        else return p.walk[grp * p.terms_per_group + ti].term;
    };
    const int row_blocks_a = p.m / 128, row_blocks_b = p.n / 128;

    // FP32 modes: the scales of the stages, in the order in which the promoting warps need them
    struct ScaleProducer {
        int w, ti, ks, ss;                          // the next stage's item, product and place in K, its place in the ring
        uint32_t phase;
        int sb_bytes; bool rows;
        const uint8_t* sa; const uint8_t* sb;       // of stage 0 of the product
        __device__ __forceinline__ void begin(int unit) { w = unit; ti = 0; ks = 0; ss = 0; phase = 0; }
    };
    constexpr int AHEAD = 2;
    auto produce_scales = [&](ScaleProducer& c) {
        if (c.w >= p.items) return true;
        if (c.ks == 0) {
            const int grp = c.w / p.positions, pos = c.w - grp * p.positions, tm = pos / tiles_n, tn = pos % tiles_n;
            const int t = term_of(grp, c.ti);
            c.sb = p.sb + (long long)t * p.sb_term + (long long)tn * BN * 4;
            c.sa = p.sa + (long long)t * p.sa_term + (long long)(tm * NCTA + cta_rank) * BM * (C::KB_PER_STAGE * 4);
            // a tile that hangs over the edge: only the scales that exist (those of its other rows or columns are whatever the
            // ring held, as their products are never stored)
            c.sb_bytes = min(BN, p.nsub - tn * BN) * 4;
            c.rows = (tm * NCTA + cta_rank) * BM < p.msub;
        }
        if (!mbar_wait_warp(bar_sempty(c.ss), c.phase ^ 1u, ctl, 102)) return false;
        if (elect_one()) {
            const uint32_t fb = bar_tfull(c.ss * C::GROUPS), dst = base + C::OFF_SB + c.ss * C::SB_STAGE_BYTES;
            mbar_expect_tx(fb, C::KB_PER_STAGE * (c.sb_bytes + (c.rows ? BM * 4 : 0)));
#pragma unroll
            for (int g = 0; g < C::KB_PER_STAGE; ++g)
                bulk_load(dst + g * BN * 4, c.sb + (long long)(c.ks * C::KB_PER_STAGE + g) * p.n * 4, c.sb_bytes, fb);
            if (c.rows) bulk_load(dst + C::SB_PART_BYTES, c.sa + (long long)c.ks * p.m * (C::KB_PER_STAGE * 4), BM * C::KB_PER_STAGE * 4, fb);
        }
        if (++c.ss == C::SB_STAGES) { c.ss = 0; c.phase ^= 1u; }
        if (++c.ks == kstages) {
            c.ks = 0;
            if (++c.ti == p.terms_per_group) { c.ti = 0; c.w += units; }
        }
        return true;
    };

    if (warp < EPI_WARP0) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(C::REGS_CTRL));
    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer
        // (all lanes walk the loops, one elected lane issues: see the note on warp-collective issue in fmm_ptx.cuh)
        {
            griddep_wait();        // the encoders' output is complete and visible (no-op unless launched to overlap them)
            int stage = 0; uint32_t phase = 0;
            bool ok = true;
            ScaleProducer scales;
            if constexpr (C::DUMP) {
                // the scales run AHEAD stages in front of the operands; their ring is longer by more than that, so that the
                // wait for a place in it is never longer than the one for the operands' place
                scales.begin(unit);
                for (int i = 0; i < AHEAD && ok; ++i) ok = produce_scales(scales);
            }
            for (int w = unit; w < p.items && ok; w += units) {
                const int slot = w;
                const int grp = slot / p.positions, pos = slot - grp * p.positions;
                const int tm = pos / tiles_n, tn = pos % tiles_n;
                const int row_blk = tm * NCTA + cta_rank;                 // 128-row block of S_r this CTA owns
                for (int ti = 0; ti < p.terms_per_group && ok; ++ti) {
                    const int t = term_of(grp, ti);
                    for (int ks = 0; ks < kstages; ++ks) {
                        if (!mbar_wait_warp(bar_empty(stage), phase ^ 1u, ctl, 101)) { ok = false; break; }
                        // completion is counted on the even CTA's barrier; only that CTA arms it
                        const uint32_t fb = (NCTA == 2) ? (bar_full(stage) & PEER_BIT_MASK) : bar_full(stage);
                        if (elect_one()) {
                            if (leader) mbar_expect_tx(bar_full(stage), C::TX_BYTES);
                            tma_load_2d<NCTA>(base + C::OFF_A + stage * C::A_BYTES, &tmA, ks * BK, t * p.m + row_blk * BM, fb);
                            tma_load_2d<NCTA>(base + C::OFF_B + stage * C::B_BYTES, &tmB, ks * BK,
                                              t * p.n + tn * BN + cta_rank * C::BROWS, fb);
                            if (C::MX) {
                                // scale tiles: 512-byte atoms, ordered [term][k quad][128-row block]
                                const uint32_t sf = base + C::OFF_SF + stage * C::SF_STAGE_BYTES;
                                tma_load_2d<NCTA>(sf, &tmSFA, 0, (t * (nkb >> 2) + ks) * row_blocks_a + row_blk, fb);
                                tma_load_2d<NCTA>(sf + 512, &tmSFB, 0, (t * (nkb >> 2) + ks) * row_blocks_b + tn * C::SFB_ATOMS, fb);
                            }
                        }
                        if (++stage == C::STAGES) { stage = 0; phase ^= 1u; }
                        if constexpr (C::DUMP) { if (!produce_scales(scales)) { ok = false; break; } }
                    }
                }
            }
        }
    } else if (warp == 2 && !C::MX && !C::DUMP) {
        // ------------------------------------------------------------------ FP32 modes: producer of the scales
        // (its own thread and ring: the operand producer above has no registers to spare, and the scale ring is
        // released by the promoting warps, not by the tensor pipe)
        griddep_wait();            // as the operand producer
        ScaleProducer scales;
        scales.begin(unit);
        while (scales.w < p.items && produce_scales(scales)) { }
    } else if (C::DUMP && warp >= 2) {
        // ------------------------------------------------------------------ FP32 scales, block 32: output warps
        const int half = warp - 2;                                           // rows 64 half .. 64 half + 63 of the tile
        constexpr int BUFS = C::OUT_BUFS / 2, CHS = 2 * (BN / 32);           // staging chunks; chunks of the copy
        const uint32_t dump = base + C::OFF_DUMP + half * CHS * 4096, stg = base + C::OFF_STG + half * BUFS * 4096;
        const uint64_t pol_c = policy_evict_last();                         // see the note on the C tiles' L2 policy below
        uint32_t dphase = 0, cnt = 0;
        // A sum above the range may have a weighted value in it: where a step has a weight below 1 its sum comes without the factor,
        // which goes with the weights, and its chunks of weight 1 through registers as well (one of T*'s twelve updates).
        int step = 0;                                                        // of the parent
        bool ok = true;
        for (int w = unit; w < p.items && ok; w += units) {
            const int grp = w / p.positions, pos = w - grp * p.positions;
            const int tm = pos / tiles_n, tn = pos % tiles_n;
            const bool rows = (tm * NCTA + cta_rank) * BM < p.msub;            // else this CTA's half hangs over the edge
            const int s_end = (grp + 1) * p.terms_per_group;
            for (int s = s_end - p.terms_per_group; s < s_end && ok; ++s) {
                const int o0 = p.walk[s].out0, o1 = rows ? p.walk[s].out1 : o0;
                if (!mbar_wait_warp(bar_dfull(half), dphase, ctl, 401)) { ok = false; break; }
                dphase ^= 1u;
                const bool small = p.small_weights >> step & 1;
                step = step + 1 == p.R ? 0 : step + 1;
                bool any_direct = false;
                for (int o = o0; o < o1; ++o) {
                    const FmmOutEntry ent = p.out[o];
                    const int row0 = ent.row_off * p.m + (tm * NCTA + cta_rank) * BM + half * 64, col0 = ent.col_off * p.n + tn * BN;
                    // A weight of exactly 1 needs no copy: the promoting warps stored the chunks in the swizzled layout the
                    // tensor map expects (and made them visible to the TMA engine), so they go out as they are.
                    const bool direct = !small && ent.w == 1.0f;
                    const float w = small ? ent.w * p.up : ent.w;
                    any_direct |= direct;
                    // this warp's previous update of the same block, `gap` updates of CHS bulk groups ago, has landed
                    if (lane == 0) {
                        if (ent.gap == 1) bulk_wait<0>();
                        else if (ent.gap == 2) bulk_wait<CHS>();
                        else if (ent.gap >= 3) bulk_wait<2 * CHS>();
                    }
#pragma unroll 1
                    for (int ch = 0; ch < CHS; ++ch) {
                        const uint32_t from = dump + ch * 4096, to = stg + (cnt % BUFS) * 4096;
                        if (!direct) {
                            if (lane == 0) bulk_wait_read<BUFS - 1>();
                            __syncwarp();
                            // same physical piece on both sides (the swizzle is kept); the lane-dependent order only
                            // spreads the 32 rows over the shared-memory banks.  All loads are issued before the first store.
                            float4 v[8];
#pragma unroll
                            for (int i4 = 0; i4 < 8; ++i4) v[i4] = lds128(from + lane * 128 + ((i4 ^ (lane & 7)) << 4));
#pragma unroll
                            for (int i4 = 0; i4 < 8; ++i4) {
                                v[i4].x *= w; v[i4].y *= w; v[i4].z *= w; v[i4].w *= w;
                                sts128(to + lane * 128 + ((i4 ^ (lane & 7)) << 4), v[i4]);
                            }
                            fence_proxy_async();
                            __syncwarp();
                            ++cnt;
                        }
                        if (lane == 0) {
                            const uint32_t src = direct ? from : to;
                            const int r = row0 + ch / (BN / 32) * 32, c = col0 + ch % (BN / 32) * 32;
                            if (FMM_GUARD(p.guard, p.c_base + (long long)r * p.ldc + c, (31 * p.ldc + 32) * 4, 1701)) {
                                if (ent.gap == 0) tma_store_2d_hint(&tmC, c, r, src, pol_c);
                                else tma_reduce_add_2d_hint(&tmC, c, r, src, pol_c);
                            }
                            bulk_commit();
                        }
                    }
                }
                // the TMA engine has read the copy for the last time (chunks sent as they are), and so has every lane
                if (lane == 0 && any_direct) bulk_wait_read<0>();
                __syncwarp();
                if (lane == 0) {
                    dump_up[half] = p.small_weights >> step & 1 ? 1.0f : p.up;
                    mbar_arrive(bar_dempty(half));
                }
            }
        }
        if (lane == 0) bulk_wait<0>();
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer (even CTA only in a pair)
        // The whole warp walks the loops (convergent, warp-uniform operands); each tcgen05 instruction is issued by
        // one elected lane inside its wrapper.
        if (leader) {
            int stage = 0; uint32_t phase = 0;
            int buf = 0, slot = 0; uint32_t bphase = 0;
            bool ok = true;
            constexpr uint32_t MDIM = (uint32_t)(BM * NCTA) >> 4;
            uint32_t idesc_full;
            if (C::MX) idesc_full = (1u << 23) | ((uint32_t)(BN >> 3) << 17) | (MDIM << 24);
            else idesc_full = (1u << 4) | ((uint32_t)(BN >> 3) << 17) | (MDIM << 24);
            for (int w = unit; w < p.items && ok; w += units) {
                const uint32_t idesc = idesc_full;
                for (int t = 0; t < p.terms_per_group && ok; ++t) {
                    if (C::MX) {
                        if (!mbar_wait_warp(bar_tempty(0), bphase ^ 1u, ctl, 201)) { ok = false; break; }
                        tc_fence_after();
                    }
                    for (int ks = 0; ks < kstages; ++ks) {
                        if (!mbar_wait_warp(bar_full(stage), phase, ctl, 202)) { ok = false; break; }
                        tc_fence_after();
                        const uint64_t adesc = make_kmajor_sw128_desc(base + C::OFF_A + stage * C::A_BYTES);
                        const uint64_t bdesc = make_kmajor_sw128_desc(base + C::OFF_B + stage * C::B_BYTES);
                        if (C::MX) {
                            const uint32_t sf = base + C::OFF_SF + stage * C::SF_STAGE_BYTES;
                            const uint32_t tsfa = tmem_base + BN;          // one slot: cp and mma execute in issue order
                            const uint32_t tsfb = tsfa + 4;
                            tc_cp_32x128b_warpx4<NCTA>(tsfa, make_sf_desc(sf));
#pragma unroll
                            for (int h = 0; h < C::SFB_ATOMS; ++h)
                                tc_cp_32x128b_warpx4<NCTA>(tsfb + 4 * h, make_sf_desc(sf + 512 + h * 512));
#pragma unroll
                            for (int j = 0; j < BK / 32; ++j) {
                                const uint32_t id = idesc | ((uint32_t)j << 29) | ((uint32_t)j << 4);
                                mma_mxf8<NCTA>(tmem_base, adesc + 2 * j, bdesc + 2 * j, id, (ks > 0 || j > 0) ? 1u : 0u, tsfa, tsfb);
                            }
                        } else {
#pragma unroll
                            for (int g0 = 0; g0 < C::KB_PER_STAGE; g0 += C::GPB) {
                                if (!mbar_wait_warp(bar_tempty(buf), bphase ^ 1u, ctl, 203)) { ok = false; break; }
                                tc_fence_after();
#pragma unroll
                                for (int gi = 0; gi < C::GPB; ++gi) {
#pragma unroll
                                    for (int j = 0; j < BLK / 32; ++j) {
                                        const int jj = (g0 + gi) * (BLK / 32) + j;
                                        mma_f8f6f4<NCTA>(tmem_base + (buf * C::GPB + gi) * BN, adesc + 2 * jj, bdesc + 2 * jj, idesc, j > 0 ? 1u : 0u);
                                    }
                                }
                                tc_commit<NCTA>(bar_tfull(slot));
                                if (++slot == C::FULL_SLOTS) slot = 0;
                                if (++buf == C::ACC_BUFS) { buf = 0; bphase ^= 1u; }
                            }
                            if (!ok) break;
                        }
                        tc_commit<NCTA>(bar_empty(stage));
                        if (++stage == C::STAGES) { stage = 0; phase ^= 1u; }
                    }
                    if (C::MX && ok) { tc_commit<NCTA>(bar_tfull(0)); bphase ^= 1u; }
                }
            }
        }
    }
    } else {
        // ------------------------------------------------------------------ epilogue warps
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(C::REGS_EPI));
        const int e = warp - EPI_WARP0;
        const int q = warp & 3;            // TMEM lane quadrant this warp may access
        const int h = e >> 2;              // column half
        const uint32_t stg = base + C::OFF_STG + e * C::STAGING_BUFS * C::STAGING_BYTES;
        // the accumulator-free signal goes to the MMA issuer, which lives in the even CTA
        auto release_acc = [&](int b) {
            if (NCTA == 2) mbar_arrive_cluster(bar_tempty(b) & PEER_BIT_MASK); else mbar_arrive(bar_tempty(b));
        };
        int buf = 0, ss = 0;
        uint32_t bphase = 0, sphase = 0;
        uint32_t store_cnt = 0;
        uint32_t dphase = 0;
        bool ok = true;
        uint32_t accu[C::MX ? C::CW : 1];               // UE8M0: raw fp32 bits drained from TMEM
        uint32_t kept[C::MX ? 16 : 1];                  // ... and the 16 columns of a parked product that stay in registers
        unsigned long long acc2[C::MX ? 1 : C::CW / 2]; // FP32: promoted accumulators, two columns per register pair

        // FP32 scales per column (ROWS4): the promotion, acc += (P * sB) * sA for every K block's partial product P, runs over
        // chunks of 16 rows x 32 columns of TMEM with two register sets, the next chunk's load - of the next K block, stage or
        // term as well - in flight while this one is added.  A stage's scales arrive on the barrier that says its first K
        // blocks are multiplied: every wait costs a warp some 40 cycles that nothing hides with two warps to a scheduler.
        // Block 32: 480 -> 440 cycles per 128 x 128 K block against 256 of arithmetic (cubic n = 4096 253 -> 240 us, n = 8192
        // 1685 -> 1550 in bursts); block 128, n = 4096: 141.5 -> 129 in bursts.  The arithmetic alone runs at 293, with the
        // TMEM loads and no barriers at 328, and the tensor cores' traffic costs another 40.  Measured around it: chunks of
        // 64 columns 5 % slower; 16 promoting warps of a quarter of the columns 3 to 10 %; the next barrier tested ahead of
        // the arithmetic 1.3 %, try_wait instead of test_wait 1 %; load shapes that are twice as fast need more scales a
        // thread (16x64b, 16x32bx2: 2 to 12 %) or each scale twice (16x128b: 20 %); one set of barriers, and one issuing
        // warp, per half of the columns gains nothing.
        constexpr bool ROWS4 = C::ROWS4;
        constexpr int KB = C::KB_PER_STAGE, CHUNKS = C::CW / 16;
        constexpr int JG = C::CW / 8;                               // column groups of eight per warp
        uint32_t set0[ROWS4 ? 16 : 1], set1[ROWS4 ? 16 : 1];
        unsigned long long sb2[4];                                  // B-side scales of the chunk's 32 columns
        float sa1[4];                                               // block 128: A-side scales of the thread's rows
        const uint32_t tq = tmem_base + ((uint32_t)(q * 32) << 16) + h * C::CW;
        // A-side scales of the thread's four rows (q*32 + lane/4 + 8k of this CTA's 128), per K block
        const uint32_t sa_lane = base + C::OFF_SB + C::SB_PART_BYTES + (q * 32 + (lane >> 2)) * (KB * 4);
        const uint32_t sb_lane = base + C::OFF_SB + (h * C::CW + 2 * (lane & 3)) * 4;
        auto wait_full = [&](int slot, uint32_t phase) {
            // test_wait: try_wait suspends the warp where the phase is not complete
            const bool ready = mbar_test_wait(bar_tfull(slot), phase);
            return __all_sync(0xffffffffu, ready) || mbar_wait_warp(bar_tfull(slot), phase, ctl, 303);
        };
        auto load_chunk = [&](uint32_t* r, int b, int gi, int i) {
            tmem_ld_16x256b_x4(tq + (b * C::GPB + gi) * BN + (i >> 1) * 32 + ((uint32_t)(16 * (i & 1)) << 16), r);
        };
        auto load_sb = [&](unsigned long long (&d)[4], int s, int g, int cg) {
#pragma unroll
            for (int j = 0; j < 4; ++j) d[j] = lds64(sb_lane + s * C::SB_STAGE_BYTES + (g * BN + cg * 32 + 8 * j) * 4);
        };
        auto load_sa1 = [&](float (&d)[4], int s) {
#pragma unroll
            for (int k = 0; k < 4; ++k) d[k] = lds32f(sa_lane + s * C::SB_STAGE_BYTES + 8 * k * 4);
        };
        if constexpr (ROWS4) {
            ok = wait_full(0, 0);
            tc_fence_after();
            load_chunk(set0, 0, 0, 0);
            load_sb(sb2, 0, 0, 0);
            if constexpr (KB == 1) load_sa1(sa1, 0);
            tmem_ld_wait16(set0);
        }
        for (int w = unit; w < p.items && ok; w += units) {
            const int slot = w;
            const int grp = slot / p.positions, pos = slot - grp * p.positions;
            const int tm = pos / tiles_n, tn = pos % tiles_n;
            const int row_in_leaf = (tm * NCTA + cta_rank) * BM + q * 32;
            // columns this warp owns, in 32-column chunks
            constexpr int cw = C::CW;
            const int nch = cw / 32;
            // rows and columns that hang over the leaf's edge are multiplied and staged like the others, but never stored (the
            // test stands where the store is issued: leaving the loops early instead makes the weight-tile kernel 5 % slower)
            auto live = [&]() { return row_in_leaf < p.msub && (BN == 128 || tn * BN + h * cw < p.nsub); };
            const uint32_t lane_taddr = tmem_base + ((uint32_t)(q * 32) << 16) + h * cw;
            for (int ti = 0, left = p.terms_per_group; left > 0 && ok; ++ti, --left) {
                const int t = C::MX ? term_of(grp, ti) : grp * p.terms_per_group + ti;      // FP32 scales: the step of the walk
                // FP32 scales: the sum starts from `carry` times the previous product's, still in the registers (the test of ti
                // says nothing that the table does not)
                const float carry = (C::MX || ti == 0) ? 0.0f : p.walk[t].carry;
                const unsigned long long carry2 = pack2(carry, carry);
                if (carry == 0.0f) {                    // not a product with zero: the sum before may not be finite
#pragma unroll
                    for (int i = 0; i < (C::MX ? 1 : C::CW / 2); ++i) acc2[i] = 0ull;
                }
                if constexpr (C::MX) {
                    if (!mbar_wait_warp(bar_tfull(0), bphase, ctl, 301)) { ok = false; break; }
                    tc_fence_after();
#pragma unroll
                    for (int c = 0; c < C::CW / 32; ++c)
                        if (c < nch) tmem_ld32(lane_taddr + c * 32, &accu[c * 32]);
                    tmem_ld_wait();
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) release_acc(0);
                    bphase ^= 1u;
                    // ---- pair-fused post-addition (see FmmPairEntry).  First product of a step: park it - CW - 16
                    // columns in this warp's part of the TMEM hold area, 16 in registers - and go on to the next product.
                    const int ri = ti % p.R;
                    const uint32_t hold_taddr = tmem_base + ((uint32_t)(q * 32) << 16) + C::OFF_HOLD + h * C::HOLD_T;
                    if ((ri & 1) == 0 && ri + 1 < p.R) {
#pragma unroll
                        for (int c = 0; c < C::HOLD_T / 32; ++c) tmem_st32(hold_taddr + c * 32, &accu[c * 32]);
                        tmem_st16(hold_taddr + (C::HOLD_T / 32) * 32, &accu[(C::HOLD_T / 32) * 32]);
#pragma unroll
                        for (int i = 0; i < 16; ++i) kept[i] = accu[C::HOLD_T + i];
                        tmem_st_wait();
                        continue;
                    }
                    // second product of a step, or an unpaired one: one weighted update per destination block
                    const uint64_t pol_c = policy_evict_last();
                    const int sidx = (t / p.R) * p.steps + (ri >> 1);
                    const int o0 = p.pair_start[sidx], o1 = p.pair_start[sidx + 1];
                    if (lane == 0) bulk_wait<0>();     // the previous step's writes to these tiles have landed
                    __syncwarp();
                    for (int o = o0; o < o1; ++o) {
                        const FmmPairEntry ent = p.pair[o];
                        const int row0 = ent.row_off * p.m + row_in_leaf;
                        const int col0 = ent.col_off * p.n + tn * BN + h * cw;
                        const bool useA = (ent.wA != 0.0f);
#pragma unroll
                        for (int c = 0; c < C::CW / C::CH; ++c) {
                            const uint32_t b = store_cnt & (C::STAGING_BUFS - 1);
                            if (lane == 0) bulk_wait_read<C::STAGING_BUFS - 1>();   // the buffer about to be rewritten has been read
                            __syncwarp();
                            const uint32_t dst = stg + b * C::STAGING_BYTES + lane * (C::CH * 4);
                            const int swz = (C::CH == 32) ? (lane & 7) : ((lane >> 1) & 3);
#pragma unroll
                            for (int s16 = 0; s16 < C::CH / 16; ++s16) {
                                const int col = c * C::CH + s16 * 16;          // first of 16 columns, within this warp's CW
                                uint32_t av[16];
                                if (useA) {
                                    if (col < C::HOLD_T) { tmem_ld16(hold_taddr + col, av); tmem_ld_wait(); }
                                    else {
#pragma unroll
                                        for (int i = 0; i < 16; ++i) av[i] = kept[i];
                                    }
                                }
#pragma unroll
                                for (int i4 = 0; i4 < 4; ++i4) {
                                    float4 v;
                                    v.x = __uint_as_float(accu[col + i4 * 4 + 0]) * ent.wB; v.y = __uint_as_float(accu[col + i4 * 4 + 1]) * ent.wB;
                                    v.z = __uint_as_float(accu[col + i4 * 4 + 2]) * ent.wB; v.w = __uint_as_float(accu[col + i4 * 4 + 3]) * ent.wB;
                                    if (useA) {
                                        v.x = fmaf(__uint_as_float(av[i4 * 4 + 0]), ent.wA, v.x); v.y = fmaf(__uint_as_float(av[i4 * 4 + 1]), ent.wA, v.y);
                                        v.z = fmaf(__uint_as_float(av[i4 * 4 + 2]), ent.wA, v.z); v.w = fmaf(__uint_as_float(av[i4 * 4 + 3]), ent.wA, v.w);
                                    }
                                    sts128(dst + (((s16 * 4 + i4) ^ swz) << 4), v);
                                }
                            }
                            fence_proxy_async();
                            __syncwarp();
                            if (lane == 0 && live()) {
                                if (FMM_GUARD(p.guard, p.c_base + (long long)row0 * p.ldc + col0 + c * C::CH, (31 * p.ldc + C::CH) * 4, 1703)) {
                                    if (ent.first) tma_store_2d_hint(&tmC, col0 + c * C::CH, row0, stg + b * C::STAGING_BYTES, pol_c);
                                    else tma_reduce_add_2d_hint(&tmC, col0 + c * C::CH, row0, stg + b * C::STAGING_BYTES, pol_c);
                                }
                                bulk_commit();
                            }
                            ++store_cnt;
                        }
                    }
                    continue;
                } else if constexpr (ROWS4) {
                    // ---- per-column fp32 scales.  The accumulators are read with the
                    // 16-lane load shape: a thread owns four rows (lane/4 + 8k) x CW/4 columns (8j + 2(lane%4), +1), so it
                    // needs CW/4 B-side scales per K block instead of CW (a broadcast 16-byte shared-memory load returns 512
                    // bytes to the register file; at one per four elements those loads were a quarter of the promotion) and
                    // four A-side scales instead of one.
                    static_assert(KB == 4 || KB == 1, "block 32 or 128");
                    static_assert(CHUNKS % 2 == 0, "a K block begins with the first register set");
                    // acc2[k * JG + j]: row slot k, column group j
#pragma unroll
                    for (int i = 0; i < C::CW / 2; ++i) acc2[i] = mul2(acc2[i], carry2);
                    const bool more = left > 1 || w + units < p.items;          // another product after this one
                    for (int ks = 0; ks < kstages && ok; ++ks) {
                        const bool wrap = ss + 1 == C::SB_STAGES;
                        const int sn = wrap ? 0 : ss + 1;
                        const uint32_t pn = wrap ? sphase ^ 1u : sphase;
                        // block 32: the stage's K blocks for the thread's four rows, from the scale ring (a global load here,
                        // even issued a stage early, stalled the promotion: 14 % of the kernel)
                        float sa4[KB == 4 ? 4 : 1][KB];
                        if constexpr (KB == 4) {
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                const float4 v4 = lds128(sa_lane + ss * C::SB_STAGE_BYTES + 8 * k * 16);
                                sa4[k][0] = v4.x; sa4[k][1] = v4.y; sa4[k][2] = v4.z; sa4[k][3] = v4.w;
                            }
                        }
#pragma unroll
                        for (int g = 0; g < KB; ++g) {
                            const int gi = g % C::GPB;
#pragma unroll
                            for (int i = 0; i < CHUNKS; ++i) {
                                uint32_t* cur = (i & 1) ? set1 : set0;
                                uint32_t* nxt = (i & 1) ? set0 : set1;
                                unsigned long long sbn[4];
                                float san[4];
                                int nb = buf;
                                if (i + 1 < CHUNKS) {
                                    load_chunk(nxt, buf, gi, i + 1);
                                    if (i & 1) load_sb(sbn, ss, g, (i + 1) >> 1);
                                } else {
                                    if (gi + 1 == C::GPB) {
                                        // the last chunk is in registers: hand the TMEM buffers back before the arithmetic
                                        tc_fence_before();
                                        __syncwarp();
                                        if (lane == 0) release_acc(buf);
                                        nb = buf + 1 == C::ACC_BUFS ? 0 : buf + 1;
                                        // (without another product the loads below fetch what nobody uses)
                                        if (g + 1 < KB) ok = ok && wait_full(ss * C::GROUPS + (g + 1) / C::GPB, sphase);
                                        else if (ks + 1 < kstages || more) ok = ok && wait_full(sn * C::GROUPS, pn);
                                        tc_fence_after();
                                    }
                                    load_chunk(nxt, nb, (gi + 1) % C::GPB, 0);
                                    load_sb(sbn, g + 1 < KB ? ss : sn, (g + 1) % KB, 0);
                                    if constexpr (KB == 1) load_sa1(san, sn);
                                }
                                // (P * sB) * sA rather than P * (sA * sB): see fmm_scale_down
#pragma unroll
                                for (int k2 = 0; k2 < 2; ++k2) {
                                    const int k = 2 * (i & 1) + k2;
                                    const float s = KB == 4 ? sa4[KB == 4 ? k : 0][g] : sa1[k];
                                    const unsigned long long sa2 = pack2(s, s);
#pragma unroll
                                    for (int j = 0; j < 4; ++j) {
                                        unsigned long long& acc = acc2[k * JG + (i >> 1) * 4 + j];
                                        acc = fma2(mul2(pack2u(cur[4 * j + 2 * k2], cur[4 * j + 2 * k2 + 1]), sb2[j]), sa2, acc);
                                    }
                                }
                                if (i & 1) {
#pragma unroll
                                    for (int j = 0; j < 4; ++j) sb2[j] = sbn[j];
                                }
                                tmem_ld_wait16(nxt);
                                if (KB == 1 && i + 1 == CHUNKS) {
#pragma unroll
                                    for (int k = 0; k < 4; ++k) sa1[k] = san[k];
                                }
                                if (i + 1 == CHUNKS) buf = nb;
                            }
                        }
                        __syncwarp();
                        if (lane == 0) mbar_arrive(bar_sempty(ss));
                        ss = sn; sphase = pn;
                    }
                    if (!ok) break;
                } else {
                    // ---- weight tiles: one scale per row and K block, sA * sB_tile; a thread owns one row
                    static_assert(C::GPB == 1 && KB == 1, "block 128");
#pragma unroll
                    for (int i = 0; i < C::CW / 2; ++i) acc2[i] = mul2(acc2[i], carry2);
                    const uint32_t sa_row = base + C::OFF_SB + C::SB_PART_BYTES + (q * 32 + lane) * 4;
                    for (int ks = 0; ks < kstages && ok; ++ks) {
                        if (!mbar_wait_warp(bar_tfull(ss), sphase, ctl, 303)) { ok = false; break; }
                        tc_fence_after();
                        const float s = lds32f(sa_row + ss * C::SB_STAGE_BYTES) * lds32f(base + C::OFF_SB + h * C::CW * 4 + ss * C::SB_STAGE_BYTES);
                        const unsigned long long s2 = pack2(s, s);
                        // 64 columns at a time, both loads in flight: an accumulator is handed back earlier and waited for less often
                        // than with 32 (pairs, n = 4096: Phi-optimal 91 -> 88 us, Winograd 77.3 -> 74.6, cubic 75.5 -> 72.4; 16 columns
                        // with the next load under the arithmetic 1 to 2 % slower)
#pragma unroll
                        for (int c = 0; c < C::CW / 64; ++c) {
                            uint32_t tmp[64];
                            const uint32_t taddr = lane_taddr + buf * BN + c * 64;
                            tmem_ld32(taddr, tmp);
                            tmem_ld32(taddr + 32, tmp + 32);
                            tmem_ld_wait();
                            if (c + 1 == C::CW / 64) {
                                // the last chunk is in registers: hand the TMEM buffer back before the arithmetic
                                tc_fence_before();
                                __syncwarp();
                                if (lane == 0) release_acc(buf);
                            }
#pragma unroll
                            for (int j = 0; j < 32; ++j) acc2[c * 32 + j] = fma2(pack2u(tmp[2 * j], tmp[2 * j + 1]), s2, acc2[c * 32 + j]);
                        }
                        if (++buf == C::ACC_BUFS) buf = 0;
                        __syncwarp();
                        if (lane == 0) mbar_arrive(bar_sempty(ss));
                        if (++ss == C::SB_STAGES) { ss = 0; sphase ^= 1u; }
                    }
                    if (!ok) break;
                }
                if (C::DUMP) {
                    // ---- hand the finished product to the output warps: rows q*32 + lane, columns h*CW .. of the tile,
                    // as 32 x 32 chunks in the 128-byte-swizzled layout of the output tensor map
                    if (!mbar_wait_warp(bar_dempty(q >> 1), dphase ^ 1u, ctl, 304)) { ok = false; break; }
                    dphase ^= 1u;
                    const float up = dump_up[q >> 1];
                    // thread: rows lane/4 + 8k of the warp's 32-row chunk, column pairs 8j + 2(lane%4) of its columns
                    const uint32_t dchunk = base + C::OFF_DUMP + (q * (BN / 32) + h * (C::CW / 32)) * 4096 + (lane & 1) * 8;
                    const unsigned long long up2 = pack2(up, up);
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const int rr = (lane >> 2) + 8 * k;
#pragma unroll
                        for (int j = 0; j < JG; ++j) {
                            const int pc = 2 * (j & 3) + ((lane & 3) >> 1);        // 16-byte piece of the 128-byte row
                            sts64(dchunk + (j >> 2) * 4096 + rr * 128 + ((pc ^ (rr & 7)) << 4), mul2(acc2[k * JG + j], up2));
                        }
                    }
                    fence_proxy_async();          // the output warps may hand these chunks to the TMA engine as they are
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar_dfull(q >> 1));
                    continue;
                }
                // ---- post-addition: W-weighted scatter of this product into its C blocks
                // Each C tile is updated once per term that feeds it, and between two updates a whole term's operands
                // stream through L2: the tiles are marked evict-last (at n = 8192: fewer write-backs of
                // half-accumulated tiles, product kernel 3 % faster; evict-first on the operand loads was slower).
                // The policy word is rebuilt here so that it is not live across the promotion loop.
                const uint64_t pol_c = policy_evict_last();
                const int o0 = p.walk[t].out0, o1 = p.walk[t].out1;
                if (lane == 0) bulk_wait<0>();     // the previous term's writes to these tiles have landed
                __syncwarp();
                for (int o = o0; o < o1; ++o) {
                    const FmmOutEntry ent = p.out[o];
                    const int row0 = ent.row_off * p.m + row_in_leaf;
                    const int col0 = ent.col_off * p.n + tn * BN + h * cw;
#pragma unroll
                    for (int c = 0; c < C::CW / C::CH; ++c) {
                        if (c * C::CH >= cw) break;
                        const uint32_t b = store_cnt & (C::STAGING_BUFS - 1);
                        if (lane == 0) bulk_wait_read<C::STAGING_BUFS - 1>();   // the buffer about to be rewritten has been read
                        __syncwarp();
                        // one row of the chunk per lane; 16-byte pieces permuted as the tensor map's swizzle expects
                        const uint32_t dst = stg + b * C::STAGING_BYTES + lane * (C::CH * 4);
                        const int swz = (C::CH == 32) ? (lane & 7) : ((lane >> 1) & 3);
                        if (C::ROWS4) {
                            // four-row layout: rows lane/4 + 8k, column pairs 8j + 2(lane%4) of this 32-column chunk
                            const uint32_t sdst = stg + b * C::STAGING_BYTES + (lane & 1) * 8;
                            const unsigned long long w2 = pack2(ent.w * p.up, ent.w * p.up);
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                const int rr = (lane >> 2) + 8 * k;
#pragma unroll
                                for (int j = 0; j < 4; ++j) {
                                    const int pc = 2 * j + ((lane & 3) >> 1);
                                    sts64(sdst + rr * 128 + ((pc ^ (rr & 7)) << 4), mul2(acc2[k * (C::CW / 8) + c * 4 + j], w2));
                                }
                            }
                        } else
#pragma unroll
                        for (int i4 = 0; i4 < C::CH / 4; ++i4) {
                            float4 v;
                            if (C::MX) {
                                v.x = __uint_as_float(accu[c * C::CH + i4 * 4 + 0]); v.y = __uint_as_float(accu[c * C::CH + i4 * 4 + 1]);
                                v.z = __uint_as_float(accu[c * C::CH + i4 * 4 + 2]); v.w = __uint_as_float(accu[c * C::CH + i4 * 4 + 3]);
                            } else {
                                unpack2(acc2[c * (C::CH / 2) + i4 * 2], v.x, v.y);
                                unpack2(acc2[c * (C::CH / 2) + i4 * 2 + 1], v.z, v.w);
                            }
                            v.x *= ent.w; v.y *= ent.w; v.z *= ent.w; v.w *= ent.w;        // weight tiles: p.up is 1
                            sts128(dst + ((i4 ^ swz) << 4), v);
                        }
                        fence_proxy_async();
                        __syncwarp();
                        if (lane == 0 && live()) {
                            if (FMM_GUARD(p.guard, p.c_base + (long long)row0 * p.ldc + col0 + c * C::CH, (31 * p.ldc + C::CH) * 4, 1702)) {
                                if (ent.gap == 0) tma_store_2d_hint(&tmC, col0 + c * C::CH, row0, stg + b * C::STAGING_BYTES, pol_c);
                                else tma_reduce_add_2d_hint(&tmC, col0 + c * C::CH, row0, stg + b * C::STAGING_BYTES, pol_c);
                            }
                            bulk_commit();
                        }
                        ++store_cnt;
                    }
                }
            }
        }
        if (lane == 0) bulk_wait<0>();
    }

    // ---------------------------------------------------------------------- teardown
    if (*abort_flag) {
        // let copies that are still in flight towards this CTA's shared memory land
        const uint64_t t0 = global_timer();
        while (global_timer() - t0 < 200000ull) __nanosleep(1000);
    }
    tc_fence_before();
    __syncthreads();
    if (NCTA == 2) cluster_sync();      // the peer no longer reads this CTA's shared memory or signals its barriers
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc<NCTA>(tmem_base, 512);
    }
}

// --------------------------------------------------------------------------------- host side
// Tile positions of a leaf of m x n, the ones that hang over its edges included.
int tile_positions(int m, int n, int ncta, int bn) { return (m + BM * ncta - 1) / (BM * ncta) * ((n + bn - 1) / bn); }

// Term groups as separate work items only where that shortens the longest CTA's list of terms (many terms on few tile
// positions); otherwise one CTA (pair) walks all terms of its position.
int terms_per_item(const GemmParams& g, int positions, int units)
{
    const int tpg = (g.terms_per_group > 0 && g.terms % g.terms_per_group == 0) ? g.terms_per_group : g.terms;
    const long long one = (long long)((positions + units - 1) / units) * g.terms;
    const long long many = ((long long)positions * (g.terms / tpg) + units - 1) / units * tpg;
    return many >= one ? g.terms : tpg;
}

template <int BN, int MODE, int BLK, int NCTA>
fmm_status_t launch(const GemmParams& g, cudaStream_t st, bool separate = false)
{
    using C = Cfg<BN, MODE, BLK, NCTA>;
    CUtensorMap tmA, tmB, tmC, tmSFA, tmSFB;
    const CUtensorMapSwizzle SW = CU_TENSOR_MAP_SWIZZLE_128B;
    if (!make_map_2d(&tmA, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, g.qa, (uint64_t)g.k, (uint64_t)(g.terms - 1) * g.m + g.msub, BK, BM, SW)) return FMM_ERR_CUDA;
    if (!make_map_2d(&tmB, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, g.qb, (uint64_t)g.k, (uint64_t)(g.terms - 1) * g.n + g.nsub, BK, C::BROWS, SW)) return FMM_ERR_CUDA;
    if (!make_map_2d(&tmC, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, g.C, (uint64_t)(g.Nfull - g.n + g.nsub), (uint64_t)(g.Mfull - g.m + g.msub), C::CH, 32,
                     C::CH == 32 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B, (uint64_t)g.Nfull)) return FMM_ERR_CUDA;
    if (C::MX) {
        // scale tiles as rows of 128 uint32 (one 512-byte atom per row)
        const uint64_t chunks = (uint64_t)g.terms * (g.k / 128);
        const uint64_t atoms_a = (chunks - 1) * (g.m / 128) + g.msub / 128, atoms_b = (chunks - 1) * (g.n / 128) + g.nsub / 128;
        if (!make_map_2d(&tmSFA, CU_TENSOR_MAP_DATA_TYPE_UINT32, 4, g.sa, 128, atoms_a, 128, 1, CU_TENSOR_MAP_SWIZZLE_NONE)) return FMM_ERR_CUDA;
        if (!make_map_2d(&tmSFB, CU_TENSOR_MAP_DATA_TYPE_UINT32, 4, g.sb, 128, atoms_b, 128, C::SFB_ATOMS, CU_TENSOR_MAP_SWIZZLE_NONE)) return FMM_ERR_CUDA;
    } else {
        tmSFA = tmA; tmSFB = tmB;       // unused in this mode
    }
    const int dev = g.device, sms = g.sms;
    // the dynamic shared memory limit is a per-device attribute of the function: set once per device
    static std::atomic<bool> attr_set[64];
    if (dev < 0 || dev >= 64 || !attr_set[dev].load(std::memory_order_acquire)) {
        if (cudaFuncSetAttribute(fmm_gemm_kernel<BN, MODE, BLK, NCTA>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM_BYTES) != cudaSuccess) {
            cudaGetLastError();
            return FMM_ERR_CUDA;
        }
        if (dev >= 0 && dev < 64) attr_set[dev].store(true, std::memory_order_release);
    }
    const int tiles_n = (g.nsub + BN - 1) / BN, positions = tile_positions(g.msub, g.nsub, NCTA, BN);
    const int max_units = sms / NCTA;
    const int tpg = terms_per_item(g, positions, max_units);
    const int slots = positions * (g.terms / tpg);
    // as few CTAs (pairs) as finish in the same number of waves: every unit then gets the same number of items, and
    // fewer units contend for L2 (256 positions: 64 pairs in 4 waves instead of 74 pairs with a ragged fourth wave)
    const int waves = (slots + max_units - 1) / max_units;
    const int units = (slots + waves - 1) / waves;
    KParams kp;
    kp.sa = static_cast<const uint8_t*>(g.sa); kp.sb = static_cast<const uint8_t*>(g.sb);
    kp.sa_term = g.sa_term; kp.sb_term = g.sb_term;
    kp.m = g.m; kp.n = g.n; kp.k = g.k; kp.msub = g.msub; kp.nsub = g.nsub; kp.terms = g.terms;
    kp.positions = positions; kp.tiles_n = tiles_n; kp.terms_per_group = tpg;
    kp.items = slots;
    // In the second half of the table every product is summed on its own: from SEPARATE_STAGES on the updates that carried sums
    // save are hidden behind the next product (product kernel, us, carried and separate: Phi-optimal n = 8192 1372, 1374, two levels
    // 1425, 1445; n = 4096 215.0, 215.8, Winograd 206.1, 208.3, Strassen 211.6, 210.8; with 12 stages a term 173.3, 176.9 / 160.8, 162.1 /
    // 163.4, 163.5, with 8 121.8, 135.7 / 113.4, 115.4 / 115.0, 114.1), and they cost the most accuracy: 1.19 times the error for
    // Winograd, 1.20 for Phi-optimal (n = 4096)
    kp.walk = separate ? g.walk + g.terms : g.walk;
    kp.out = g.out; kp.status = g.status;
    kp.pair_start = g.pair_start; kp.pair = g.pair; kp.steps = (short)g.steps;
    for (int r = 0; r < FMM_MAX_RANK; ++r) kp.order[r] = g.order[r];
    kp.R = (unsigned char)(g.terms_per_group > 0 ? g.terms_per_group : 1);       // products per parent (1 for the cubic product)
    kp.up = g.up; kp.small_weights = (unsigned char)(separate ? 0 : g.small_weights);
    kp.c_base = g.C; kp.ldc = g.Nfull; kp.guard = g.guard;

    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)(units * NCTA), 1, 1);
    cfg.blockDim = dim3(NUM_THREADS, 1, 1);
    cfg.dynamicSmemBytes = C::SMEM_BYTES;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = NCTA; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    // right behind the encoders of the same call: the CTAs may be set up (barriers, TMEM, tensor maps) while the B-side
    // encoder drains; the producer warps wait for it before their first load
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = g.overlap_prev ? 2 : 1;
    cudaError_t ce = cudaLaunchKernelEx(&cfg, fmm_gemm_kernel<BN, MODE, BLK, NCTA>, tmA, tmB, tmC, tmSFA, tmSFB, kp);
    if (ce != cudaSuccess) { cudaGetLastError(); return FMM_ERR_CUDA; }
    return FMM_OK;
}

// The tile shapes each kind of product can be launched with, and the time of one: base + L * (kst * c + o) in microseconds,
// L being the terms that the busiest CTA (pair) walks, kst the stages of 128 k, o a term's chain from the first load to its
// output (o_cubic: of the cubic product, which writes every tile once).  A leaf need not be a multiple of the tile: what
// hangs over the edge is multiplied and not stored, so a leaf of an odd number of 128-row or 128-column blocks may take the
// wide tiles as well, at the price of a part of its last row or column of tiles.  Fitted, together with the cluster kernel's
// model (fmm_split.cu), to the times of every shape over leaves of 128 to 8192 in every direction and zero to three levels.
// Over 60 random problems per kind (leaves of 128 to 5000) the choice among all product kernels is the fastest shape for 43 to 54 of them
// and costs, in the mean, 3.4 % (block 32), 1.4 % (UE8M0), 2.2 % (block 128) and 0.1 % (weight tiles) more than the fastest; those above
// 12 us 2.7 %, 1.9 %, 2.0 % and 0.2 %.  The worst are single products of about 8 us, at up to 1.32 times, and at block 32, whose constants and the
// cluster kernel's stand as fitted to a slower promotion, products of 39 to 66 us that the persistent kernel would take in 0.80 times
// the cluster kernel's time (3328 x 2304 x 1536, 9728 x 1024 x 512; with carried sums instead of separate ones).  Product kernel
// against the rule before, which gave wide tiles only to leaves that are multiples of them: UE8M0 8192 x 8192 x 8448 one
// level 674 -> 492 us, cubic 4096 x 1024 x 4224 47.6 -> 26.4; block 128 8192 x 8192 x 8448 956 -> 787; weight tiles
// 888 -> 664.
// Block 128: with the faster promotion the single CTAs have gained more than the pairs, whose constants are fitted again, to 666
// problems (5 % faster on the 7 % of them that change; cubic n = 4096 122.3 -> 115.7 us a call, two levels 270 -> 257; the pairs stay at
// n = 8192, 739 against 781, cubic 718 against 893).
// Weight tiles: the same once more since the single CTAs' issuing warp knows its values to be uniform (of 330 problems the choice between the
// two is 0.1 % off the faster one in the mean, 0.6 % with the constants before).  The pairs' constants are higher than before in that ratio, but nothing
// has become slower, so both are scaled by 0.87 for the comparison with the cluster kernel: of 160 problems (cubic, rank 7) the choice is 1.9 % off
// the fastest of these kernels in the mean and without that 3.6 %, at worst 1.66 times (cubic 4480 x 4608 x 640 22.8, 34.5 us; 2816 x 5760 x 1024 51 and
// 64 a call); 0.8 to 0.9 are within 0.5 %.
struct ShapeModel { int ncta, bn; float c, o, o_cubic; };
constexpr ShapeModel MODEL_MX[] = {{2, 256, 0.26f, 3.9f, 3.6f}, {1, 256, 0.35f, 3.4f, 2.7f}, {1, 128, 0.22f, 1.7f, 1.2f}};
constexpr ShapeModel MODEL_B32[] = {{2, 128, 0.71f, 3.6f, 2.2f}, {1, 128, 0.67f, 3.55f, 1.85f}};
constexpr ShapeModel MODEL_B128[] = {{2, 256, 0.43f, 6.0f, 5.1f}, {1, 128, 0.28f, 2.5f, 1.8f}};
constexpr ShapeModel MODEL_TILE[] = {{2, 256, 0.322f, 4.7f, 2.96f}, {1, 128, 0.226f, 2.09f, 1.0f}};
constexpr float BASE_MX = 3.3f, BASE_B32 = 2.4f, BASE_B128 = 3.85f, BASE_TILE = 3.65f;

template <int N>
GemmShape best_shape(const GemmParams& g, int m, int n, const ShapeModel (&models)[N], float base)
{
    GemmShape best = {0, 0, 0.0f, 0};
    for (const ShapeModel& s : models) {
        const int positions = tile_positions(m, n, s.ncta, s.bn), units = g.sms / s.ncta, tpg = terms_per_item(g, positions, units);
        const long long longest = ((long long)positions * (g.terms / tpg) + units - 1) / units * tpg;
        const float time = base + (float)longest * ((float)(g.k / BK) * s.c + (g.R > 1 ? s.o : s.o_cubic));
        if (best.ncta == 0 || time < best.time) best = {s.ncta, s.bn, time, longest};
    }
    return best;
}

// Block 32: whether the products are written by the output warps.  They need a fixed time per term: with fewer K stages the
// promoting warps would wait for them (three levels n = 2048, two stages: 131 us with, 117 without; two levels 3072 x 2048 x 3072,
// four stages: 121.0 and 123.5; 4096 x 2048 x 4096, eight stages: 138.9 and 153.2).
bool output_warps(const GemmParams& g, const fmm_product_shape_t& s) { return s.output_warp || g.k / BK >= 4; }

template <int MODE, int BLK>
fmm_status_t launch_shape(const GemmParams& g, const fmm_product_shape_t& s, cudaStream_t st)
{
    if constexpr (MODE == FMM_SCALE_UE8M0_CEIL) {
        if (s.ctas == 2) return launch<256, MODE, 32, 2>(g, st);
        return s.columns == 256 ? launch<256, MODE, 32, 1>(g, st) : launch<128, MODE, 32, 1>(g, st);
    } else if constexpr (BLK == 128) {
        // one promotion per 128 k: 256-column tiles with two TMEM accumulators in a pair
        return s.ctas == 2 ? launch<256, MODE, BLK, 2>(g, st) : launch<128, MODE, BLK, 1>(g, st);
    } else {
        // bound by the promotion on the CUDA cores: 128-column tiles, whose four TMEM accumulators let the MMA issuer run
        // further ahead of the promoting warps.  Post-addition by the output warps.  (Block 128 does not gain
        // from them: with 128-column tiles and an output warp it runs as fast as with 256-column tiles and none, 0.81 ms at
        // n = 8192, and the cubic product, which has a single store per tile, is 20 % slower.)
        if (output_warps(g, s)) return s.ctas == 2 ? launch<128, MODE_FP32_OUT_WARP, BLK, 2>(g, st, s.output_warp) : launch<128, MODE_FP32_OUT_WARP, BLK, 1>(g, st, s.output_warp);
        return s.ctas == 2 ? launch<128, MODE, BLK, 2>(g, st) : launch<128, MODE, BLK, 1>(g, st);
    }
}

}  // namespace

GemmShape fmm_gemm_shape(const GemmParams& g, int blk, int mode, int m, int n)
{
    if (mode == FMM_SCALE_UE8M0_CEIL) return best_shape(g, m, n, MODEL_MX, BASE_MX);
    if (blk == 32) return best_shape(g, m, n, MODEL_B32, BASE_B32);
    return g.sb_tile ? best_shape(g, m, n, MODEL_TILE, BASE_TILE) : best_shape(g, m, n, MODEL_B128, BASE_B128);
}

fmm_product_shape_t fmm_choose_product(const GemmParams& g, int blk, int mode)
{
    if (g.forced.kernel) return g.forced;
    const SplitChoice split = fmm_split_choice(g, blk, mode);
    if (g.R > 1 && fmm_keep_faster(g, blk, mode, split, fmm_gemm_shape(g, blk, mode, g.m, g.n))) return {8, 1, 64, 1, 0};
    if (split.ksplit > 0) return {split.terms == 2 ? 4 : 2, 1, split.bn, split.ksplit, 0};
    const GemmShape s = fmm_gemm_shape(g, blk, mode, g.msub, g.nsub);
    return {1, s.ncta, s.bn, 1, mode != FMM_SCALE_UE8M0_CEIL && blk == 32 && g.k / BK >= SEPARATE_STAGES};
}

bool fmm_product_shape_exists(const fmm_product_shape_t& s, int blk, int mode, int sb_tile, int R)
{
    const bool mx = mode == FMM_SCALE_UE8M0_CEIL;
    if (s.kernel == 8) return R > 1 && s.ctas == 1 && s.columns == 64 && s.k_shares == 1 && !s.output_warp;
    if (s.kernel == 4) return mx && R > 1 && s.ctas == 1 && s.columns == 128 && s.k_shares == 1 && !s.output_warp;
    if (s.kernel == 2) {
        const bool width = s.columns == 128 || (!mx && (s.columns == 64 || s.columns == 32));
        const bool shares = s.k_shares == 1 || (R == 1 && (s.k_shares == 2 || s.k_shares == 4 || s.k_shares == 8));
        return width && shares && s.ctas == 1 && !s.output_warp;
    }
    auto known = [&](const auto& models) {
        for (const ShapeModel& m : models) if (m.ncta == s.ctas && m.bn == s.columns) return true;
        return false;
    };
    if (s.kernel != 1 || s.k_shares != 1 || s.output_warp < 0 || s.output_warp > (!mx && blk == 32 ? 1 : 0)) return false;
    return mx ? known(MODEL_MX) : blk == 32 ? known(MODEL_B32) : sb_tile ? known(MODEL_TILE) : known(MODEL_B128);
}

fmm_status_t fmm_launch_bounded_wait_selftest(int* status, unsigned long long limit_ns, cudaStream_t st)
{
    bounded_wait_selftest_kernel<<<1, 32, 0, st>>>(status, limit_ns, 901);
    return cudaGetLastError() == cudaSuccess ? FMM_OK : FMM_ERR_CUDA;
}

fmm_status_t fmm_launch_gemm(const GemmParams& g, int blk, int mode, cudaStream_t st, int* launches)
{
    fmm_status_t s;
    const fmm_product_shape_t shape = fmm_choose_product(g, blk, mode);
    if (shape.kernel == 8) s = fmm_launch_keep(g, blk, mode, st);
    else if (shape.kernel == 2 || shape.kernel == 4)
        s = shape.k_shares <= g.k / BK ? fmm_launch_split(g, blk, mode, {shape.k_shares, shape.columns, shape.kernel / 2, 0}, st) : FMM_ERR_SHAPE;
    else if (mode == FMM_SCALE_UE8M0_CEIL) s = launch_shape<FMM_SCALE_UE8M0_CEIL, 32>(g, shape, st);
    else if (blk == 128 && g.sb_tile) s = launch_shape<MODE_FP32_SB_TILE, 128>(g, shape, st);
    else if (blk == 32) s = launch_shape<FMM_SCALE_FP32_AMAX_DIV_448, 32>(g, shape, st);
    else s = launch_shape<FMM_SCALE_FP32_AMAX_DIV_448, 128>(g, shape, st);
    if (s == FMM_OK && launches) *launches += 1;
    return s;
}
