// Product kernel for problems with few output tiles (the operation is the one of fmm_gemm.cu).
//
// A cluster of CTAs owns one tile position (128 x 128; with FP32 scales also 128 x 64 or 128 x 32) of one parent: CTA j
// multiplies one of the parent's R terms (of the cubic product, which has one term: one share of K), so the terms that the
// persistent kernel of fmm_gemm.cu walks one after the other run side by side.  The partial products then meet in
// distributed shared memory: every CTA leaves its fp32 tile in its own shared memory (over the operand ring, which is
// drained by then), and after a cluster barrier CTA j forms the weighted sums of its share of the rows,
// out_q = sum_j W[j][q] * M_j in ascending j, and writes each output element once.  Nothing is read back from C, no
// partial result goes through L2, and the order of the sum is fixed.
//
// Bound: latency (launch, first operand load, the chain MMA -> promotion -> exchange), which is why the work is spread
// over as many SMs as the problem has (tile, term, K share) triples.  Two CTAs fit an SM, so that one exchanges or
// waits for its first operands while the other multiplies.  Promotion and exchange take time in proportion to the tile's
// columns, so where the narrower tiles still find room at once they are the faster ones (see the time models below).
//
// With UE8M0 scales a CTA may multiply two of the terms, one after the other: clusters of ceil(R / 2) fit the GPCs where clusters
// of 7 leave 86 of 296 places empty, and hold 66 tiles at once instead of 30.  The first product waits in registers until the
// operand ring is free; three halves of 64 columns fit over the ring, so the exchange goes in two passes.  (With FP32 scales the
// registers hold the running sums, and neither TMEM nor shared memory has room for another product beside a second CTA.)
//
//   warp 0  TMA producer of the operand tiles (UE8M0: and of the scale tiles)
//   warp 1  tcgen05.mma issuer
//   warp 2  FP32 scales: producer of both sides' scales
//   warps 4..7  promotion (FP32 scales) or drain (UE8M0), exchange, weighted sums: one TMEM lane quadrant each
#include <algorithm>
#include "fmm_gemm_common.cuh"

namespace {

constexpr int MODE_FP32_COLUMN = FMM_SCALE_FP32_AMAX_DIV_448;      // one B-side scale per column and K block

struct SplitParams {
    const uint8_t* sa; const uint8_t* sb;      // fp32 scale arrays (bytes)
    long long sa_term, sb_term;
    int m, n, k;
    int R, ksplit;                              // cluster size R * ksplit, one of the two being 1: CTA j = term j, or K share j
    int nq;                                     // output blocks per parent: 4, or 1 without recursion
    float W[FMM_MAX_RANK][4];                   // weight of CTA j's partial product in output block b (0 beyond the cluster)
    float* C; long long ldc;                    // the stack of parent matrices (C itself for one level)
    int* status;
    FmmGuard guard;
};

template <int MODE, int BLK, int BN_, int TPC = 1>
struct SplitCfg {
    static constexpr bool MX = (MODE == FMM_SCALE_UE8M0_CEIL);
    static_assert(TPC == 1 || (TPC == 2 && MX), "terms per CTA");
    static constexpr int BN = BN_;                           // columns of a tile
    static_assert(BN == 128 || (!MX && (BN == 64 || BN == 32)), "tile widths");
    static constexpr int EPI_WARPS = 4, EPI_WARP0 = 4, THREADS = (EPI_WARP0 + EPI_WARPS) * 32;
    static constexpr int REGS_AT_LAUNCH = 128;               // 65536 / (2 CTAs x 256 threads)
    static constexpr int REGS_CTRL = 56, REGS_EPI = 200;
    static_assert(EPI_WARP0 * 32 * REGS_CTRL + EPI_WARPS * 32 * REGS_EPI <= THREADS * REGS_AT_LAUNCH, "register pool");
    static constexpr int KB = BK / BLK;                      // K blocks per stage
    static constexpr int A_BYTES = BM * BK, B_BYTES = BN * BK, SF_BYTES = MX ? 1024 : 0;
    static constexpr int STAGES = 3;
    static constexpr int S_STAGES = MX ? 0 : (KB == 4 ? 3 : 4);
    static constexpr int SB_BYTES = KB * BN * 4, S_BYTES = KB * (BN + BM) * 4;
    static constexpr int TX_BYTES = A_BYTES + B_BYTES + SF_BYTES;
    static constexpr int OFF_A = 0;
    static constexpr int OFF_B = OFF_A + STAGES * A_BYTES;
    static constexpr int OFF_SF = OFF_B + STAGES * B_BYTES;
    static constexpr int OFF_S = OFF_SF + STAGES * SF_BYTES;
    static constexpr int OFF_BAR = OFF_S + S_STAGES * S_BYTES;
    static constexpr int OFF_TILE = 0;                       // the finished partial product, over the operand ring
    static constexpr int BUFS = MX ? 1 : 2;                  // TMEM accumulators
    static constexpr int TMEM_COLS = MX ? 256 : BUFS * BN;
    static constexpr int NUM_BARS = 2 * STAGES + 2 * S_STAGES + 2 * BUFS;
    static constexpr int SMEM_BYTES = OFF_BAR + NUM_BARS * 8 + 16 + 1024;   // + alignment slack
    static_assert(SMEM_BYTES + 1024 <= 233472 / 2, "two CTAs per SM");
    static constexpr int ROW_BYTES = BN * 4;                 // exchange tile: bytes and 16-byte pieces per row
    static_assert(BM * ROW_BYTES <= OFF_SF, "the exchange tile lies inside the operand ring");
    // two terms: halves of 64 columns, [first product's left | second product's, one half after the other | first's right]
    static constexpr int HALF_BYTES = BM * 64 * 4;
    static_assert(TPC == 1 || 3 * HALF_BYTES <= OFF_SF, "three halves lie inside the operand ring");
};

__device__ __forceinline__ uint32_t cluster_id_x()
{ uint32_t r; asm volatile("mov.u32 %0, %%clusterid.x;" : "=r"(r)); return r; }
__device__ __forceinline__ uint32_t map_to_cta(uint32_t saddr, uint32_t cta)
{ uint32_t r; asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(cta)); return r; }
__device__ __forceinline__ float4 ld_cluster128(uint32_t addr)
{
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
    return v;
}

template <int MODE, int BLK, int BN, int TPC>
__global__ void __launch_bounds__(SplitCfg<MODE, BLK, BN, TPC>::THREADS, 2)
fmm_split_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                 const __grid_constant__ CUtensorMap tmSFA, const __grid_constant__ CUtensorMap tmSFB, const SplitParams p)
{
    using C = SplitCfg<MODE, BLK, BN, TPC>;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw_addr = smem_u32(smem_raw);
    const uint32_t base = (raw_addr + 1023u) & ~1023u;       // the same offset in every CTA of the cluster
    uint8_t* base_ptr = smem_raw + (base - raw_addr);

    const uint32_t bar0 = base + C::OFF_BAR;
    auto bar_full = [&](int s) { return bar0 + 8u * s; };
    auto bar_empty = [&](int s) { return bar0 + 8u * (C::STAGES + s); };
    auto bar_sfull = [&](int s) { return bar0 + 8u * (2 * C::STAGES + s); };
    auto bar_sempty = [&](int s) { return bar0 + 8u * (2 * C::STAGES + C::S_STAGES + s); };
    auto bar_tfull = [&](int b) { return bar0 + 8u * (2 * C::STAGES + 2 * C::S_STAGES + b); };
    auto bar_tempty = [&](int b) { return bar0 + 8u * (2 * C::STAGES + 2 * C::S_STAGES + C::BUFS + b); };
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(base_ptr + C::OFF_BAR + C::NUM_BARS * 8);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    const Ctl ctl{abort_flag, p.status};

    const int warp = warp_uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < C::STAGES; ++s) { mbar_init(bar_full(s), 1); mbar_init(bar_empty(s), 1); }
        for (int s = 0; s < C::S_STAGES; ++s) { mbar_init(bar_sfull(s), 1); mbar_init(bar_sempty(s), C::EPI_WARPS); }
        for (int b = 0; b < C::BUFS; ++b) { mbar_init(bar_tfull(b), 1); mbar_init(bar_tempty(b), C::EPI_WARPS); }
        *abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 1) {
        tmem_alloc<1>(smem_u32(tmem_slot), C::TMEM_COLS);
        tmem_relinquish<1>();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = warp_uniform(*tmem_slot);

    // grid (S * tiles_n, tiles_m, parents), clusters of S along x: no index needs a division
    const int S = TPC == 2 ? (p.R + 1) / 2 : p.R * p.ksplit, rank = (int)warp_uniform(cluster_ctarank());
    const int parent = blockIdx.z, tm = blockIdx.y, tn = (int)warp_uniform(cluster_id_x());
    const int r = p.R == 1 ? 0 : TPC * rank, kpart = p.R == 1 ? rank : 0;
    const int t0 = parent * p.R + r, nt = TPC == 2 && r + 1 < p.R ? 2 : 1;       // this CTA's terms: t0 .. t0 + nt - 1
    const int kstages = p.k / BK;
    const int ks0 = kstages * kpart / p.ksplit, ks1 = kstages * (kpart + 1) / p.ksplit;
    const uint32_t tile = base + C::OFF_TILE;

    if (warp < C::EPI_WARP0) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(C::REGS_CTRL));
        if (warp == 0) {
            // ------------------------------------------------------------------ TMA producer
            griddep_wait();        // the encoders' output is complete and visible (no-op unless launched to overlap them)
            int stage = 0; uint32_t phase = 0;
            const int nq4 = p.k / BK, row_blocks_a = p.m / 128, row_blocks_b = p.n / 128;
            bool ok = true;
            for (int t = t0; t < t0 + nt && ok; ++t)
            for (int ks = ks0; ks < ks1; ++ks) {
                if (!mbar_wait_warp(bar_empty(stage), phase ^ 1u, ctl, 121)) { ok = false; break; }
                if (elect_one()) {
                    mbar_expect_tx(bar_full(stage), C::TX_BYTES);
                    tma_load_2d<1>(base + C::OFF_A + stage * C::A_BYTES, &tmA, ks * BK, t * p.m + tm * BM, bar_full(stage));
                    tma_load_2d<1>(base + C::OFF_B + stage * C::B_BYTES, &tmB, ks * BK, t * p.n + tn * BN, bar_full(stage));
                    if (C::MX) {
                        const uint32_t sf = base + C::OFF_SF + stage * C::SF_BYTES;
                        tma_load_2d<1>(sf, &tmSFA, 0, (t * nq4 + ks) * row_blocks_a + tm, bar_full(stage));
                        tma_load_2d<1>(sf + 512, &tmSFB, 0, (t * nq4 + ks) * row_blocks_b + tn, bar_full(stage));
                    }
                }
                if (++stage == C::STAGES) { stage = 0; phase ^= 1u; }
            }
        } else if (warp == 2 && !C::MX) {
            // ------------------------------------------------------------------ producer of both sides' fp32 scales
            griddep_wait();
            int ss = 0; uint32_t sphase = 0;
            const uint8_t* sb_t = p.sb + (long long)t0 * p.sb_term + (long long)tn * BN * 4;
            const uint8_t* sa_t = p.sa + (long long)t0 * p.sa_term + (long long)tm * BM * (C::KB * 4);
            for (int ks = ks0; ks < ks1; ++ks) {
                if (!mbar_wait_warp(bar_sempty(ss), sphase ^ 1u, ctl, 122)) break;
                if (elect_one()) {
                    mbar_expect_tx(bar_sfull(ss), C::S_BYTES);
#pragma unroll
                    for (int g = 0; g < C::KB; ++g)
                        bulk_load(base + C::OFF_S + ss * C::S_BYTES + g * BN * 4,
                                  sb_t + (long long)(ks * C::KB + g) * p.n * 4, BN * 4, bar_sfull(ss));
                    bulk_load(base + C::OFF_S + ss * C::S_BYTES + C::SB_BYTES,
                              sa_t + (long long)ks * p.m * (C::KB * 4), BM * C::KB * 4, bar_sfull(ss));
                }
                if (++ss == C::S_STAGES) { ss = 0; sphase ^= 1u; }
            }
        } else if (warp == 1) {
            // ------------------------------------------------------------------ MMA issuer
            int stage = 0; uint32_t phase = 0;
            int buf = 0; uint32_t bphase = 0;
            bool ok = true;
            constexpr uint32_t idesc = (C::MX ? (1u << 23) : (1u << 4)) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
            for (int tt = 0; tt < nt && ok; ++tt) {
            if (tt > 0) {                                    // the first product has left its accumulator
                if (!mbar_wait_warp(bar_tempty(0), 0, ctl, 223)) { ok = false; break; }
                tc_fence_after();
            }
            for (int ks = ks0; ks < ks1 && ok; ++ks) {
                if (!mbar_wait_warp(bar_full(stage), phase, ctl, 221)) { ok = false; break; }
                tc_fence_after();
                const uint64_t adesc = make_kmajor_sw128_desc(base + C::OFF_A + stage * C::A_BYTES);
                const uint64_t bdesc = make_kmajor_sw128_desc(base + C::OFF_B + stage * C::B_BYTES);
                if (C::MX) {
                    const uint32_t sf = base + C::OFF_SF + stage * C::SF_BYTES;
                    const uint32_t tsfa = tmem_base + BN, tsfb = tsfa + 4;     // one slot: cp and mma execute in issue order
                    tc_cp_32x128b_warpx4<1>(tsfa, make_sf_desc(sf));
                    tc_cp_32x128b_warpx4<1>(tsfb, make_sf_desc(sf + 512));
#pragma unroll
                    for (int j = 0; j < BK / 32; ++j) {
                        const uint32_t id = idesc | ((uint32_t)j << 29) | ((uint32_t)j << 4);
                        mma_mxf8<1>(tmem_base, adesc + 2 * j, bdesc + 2 * j, id, (ks > ks0 || j > 0) ? 1u : 0u, tsfa, tsfb);
                    }
                } else {
#pragma unroll
                    for (int g = 0; g < C::KB; ++g) {
                        if (!mbar_wait_warp(bar_tempty(buf), bphase ^ 1u, ctl, 222)) { ok = false; break; }
                        tc_fence_after();
#pragma unroll
                        for (int j = 0; j < BLK / 32; ++j) {
                            const int jj = g * (BLK / 32) + j;
                            mma_f8f6f4<1>(tmem_base + buf * BN, adesc + 2 * jj, bdesc + 2 * jj, idesc, j > 0 ? 1u : 0u);
                        }
                        tc_commit<1>(bar_tfull(buf));
                        if (++buf == C::BUFS) { buf = 0; bphase ^= 1u; }
                    }
                    if (!ok) break;
                }
                tc_commit<1>(bar_empty(stage));
                if (++stage == C::STAGES) { stage = 0; phase ^= 1u; }
            }
            if (C::MX && ok) tc_commit<1>(bar_tfull(0));
            }
        }
        cluster_sync();                                      // every CTA's partial product is in its shared memory
        if (TPC == 2) { cluster_sync(); cluster_sync(); }    // as below
    } else {
        // ---------------------------------------------------------------------- promotion / drain, exchange, output
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(C::REGS_EPI));
        const int q = warp & 3;            // TMEM lane quadrant this warp may access
        const uint32_t lane_taddr = tmem_base + ((uint32_t)(q * 32) << 16);
        bool ok = true;
        // The exchange tile: row-major fp32, the row's 16-byte pieces permuted by piece ^ (row & 7).
        if constexpr (TPC == 2) {
            uint32_t v[64];
            auto put_half = [&](uint32_t region) {
                const int row = q * 32 + lane;
#pragma unroll
                for (int i = 0; i < 16; ++i)
                    sts128(tile + region * C::HALF_BYTES + row * 256 + ((i ^ (row & 7)) << 4),
                           make_float4(__uint_as_float(v[4 * i]), __uint_as_float(v[4 * i + 1]), __uint_as_float(v[4 * i + 2]), __uint_as_float(v[4 * i + 3])));
            };
            auto load_half = [&](int h) {
                tmem_ld32(lane_taddr + h * 64, v); tmem_ld32(lane_taddr + h * 64 + 32, v + 32);
                tmem_ld_wait();
            };
            // the first product waits in registers for the operand ring to be free
            uint32_t first[128];
            ok = mbar_wait_warp(bar_tfull(0), 0, ctl, 321);
            tc_fence_after();
#pragma unroll
            for (int c = 0; c < 4; ++c) tmem_ld32(lane_taddr + c * 32, first + c * 32);
            tmem_ld_wait();
            if (nt == 2) {
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_tempty(0));
                ok = ok && mbar_wait_warp(bar_tfull(0), 1, ctl, 324);
                tc_fence_after();
                load_half(0);
                put_half(1);
            }
#pragma unroll
            for (int i = 0; i < 64; ++i) v[i] = first[i];
            put_half(0);
#pragma unroll
            for (int i = 0; i < 64; ++i) v[i] = first[64 + i];
            put_half(2);
            cluster_sync();                                  // the left halves of every product, and the firsts' right ones
            const int r0 = BM * rank / S, r1 = BM * (rank + 1) / S, piece = lane & 15;
            uint32_t peer[FMM_MAX_RANK / 2];
#pragma unroll
            for (int j = 0; j < FMM_MAX_RANK / 2; ++j) peer[j] = map_to_cta(tile, j < S ? j : 0);
            float* c_tile = p.C + ((long long)parent * 2 * p.m + tm * BM) * p.ldc + tn * BN + piece * 4;
#pragma unroll 1
            for (int h = 0; h < 2; ++h) {
                if (h == 1) {
                    cluster_sync();                          // the second products' left halves have been read
                    if (nt == 2) { load_half(1); put_half(1); }
                    cluster_sync();                          // their right halves are there
                }
                // two rows per warp and step, as below; product j is CTA j / 2's first or second
                auto fetch = [&](int row, float4 (&x)[FMM_MAX_RANK]) {
                    const uint32_t off = row * 256 + ((piece ^ (row & 7)) << 4);
#pragma unroll
                    for (int j = 0; j < FMM_MAX_RANK; ++j)
                        if (j < p.R) x[j] = ld_cluster128(peer[j >> 1] + off + (j & 1 ? 1 : 2 * h) * C::HALF_BYTES);
                };
                auto sum_and_store = [&](int row, const float4 (&x)[FMM_MAX_RANK]) {
#pragma unroll
                    for (int b = 0; b < 4; ++b) {
                        float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                        for (int j = 0; j < FMM_MAX_RANK; ++j) {
                            const float wj = p.W[j][b];      // zero for j >= R
                            if (wj != 0.0f) { o.x = fmaf(wj, x[j].x, o.x); o.y = fmaf(wj, x[j].y, o.y); o.z = fmaf(wj, x[j].z, o.z); o.w = fmaf(wj, x[j].w, o.w); }
                        }
                        float* dst = c_tile + ((long long)(b >> 1) * p.m + row) * p.ldc + (long long)(b & 1) * p.n + h * 64;
                        if (FMM_GUARD(p.guard, dst, 16, 1722)) *reinterpret_cast<float4*>(dst) = o;
                    }
                };
                float4 x0[FMM_MAX_RANK], x1[FMM_MAX_RANK];
                constexpr int STEP = C::EPI_WARPS * 2;
                int row = r0 + q * 2 + (lane >> 4);
                if (row < r1) fetch(row, x0);
#pragma unroll 1
                for (; row < r1; row += 2 * STEP) {
                    const bool more1 = row + STEP < r1, more2 = row + 2 * STEP < r1;
                    if (more1) fetch(row + STEP, x1);
                    sum_and_store(row, x0);
                    if (more2) fetch(row + 2 * STEP, x0);
                    if (more1) sum_and_store(row + STEP, x1);
                }
            }
        } else {
        if constexpr (C::MX) {
            ok = mbar_wait_warp(bar_tfull(0), 0, ctl, 321);
            tc_fence_after();
            const int row = q * 32 + lane;
#pragma unroll
            for (int c = 0; c < BN / 32; ++c) {
                uint32_t v[32];
                tmem_ld32(lane_taddr + c * 32, v);
                tmem_ld_wait();
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    sts128(tile + row * C::ROW_BYTES + (((c * 8 + i) ^ (row & 7)) << 4),
                           make_float4(__uint_as_float(v[4 * i]), __uint_as_float(v[4 * i + 1]), __uint_as_float(v[4 * i + 2]), __uint_as_float(v[4 * i + 3])));
            }
        } else {
            // The accumulators are read with the 16-lane load shape: a thread owns four rows (lane/4 + 8k) x 32 columns
            // (8j + 2(lane%4), +1), so that one B-side scale fetched from shared memory serves four rows.
            constexpr int JG = BN / 8;
            const uint32_t sa_lane = base + C::OFF_S + C::SB_BYTES + (q * 32 + (lane >> 2)) * (C::KB * 4);
            const uint32_t sb_lane = base + C::OFF_S + 2 * (lane & 3) * 4;
            int buf = 0; uint32_t bphase = 0;
            int ss = 0; uint32_t sphase = 0;
            unsigned long long acc2[4 * JG];   // [row slot k][column group j]
#pragma unroll
            for (int i = 0; i < 4 * JG; ++i) acc2[i] = 0ull;
            for (int ks = ks0; ks < ks1 && ok; ++ks) {
                if (!mbar_wait_warp(bar_sfull(ss), sphase, ctl, 322)) { ok = false; break; }
#pragma unroll 1
                for (int g = 0; g < C::KB; ++g) {
                    float sa4[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) sa4[k] = lds32f(sa_lane + ss * C::S_BYTES + 8 * k * (C::KB * 4) + g * 4);
                    if (MODE == MODE_FP32_SB_TILE) {
                        const float sbt = lds32f(base + C::OFF_S + ss * C::S_BYTES + g * BN * 4);
#pragma unroll
                        for (int k = 0; k < 4; ++k) sa4[k] *= sbt;
                    }
                    if (!mbar_wait_warp(bar_tfull(buf), bphase, ctl, 323)) { ok = false; break; }
                    tc_fence_after();
                    const uint32_t taddr = lane_taddr + buf * BN;
                    const uint32_t sbs = sb_lane + ss * C::S_BYTES + g * BN * 4;
#pragma unroll
                    for (int c = 0; c < BN / 32; ++c) {
                        uint32_t lo[16], hi[16];
                        tmem_ld_16x256b_x4(taddr + c * 32, lo);                       // rows lane/4, lane/4 + 8
                        tmem_ld_16x256b_x4(taddr + c * 32 + (16u << 16), hi);         // rows lane/4 + 16, lane/4 + 24
                        unsigned long long sb2[4];
                        if (MODE != MODE_FP32_SB_TILE) {
#pragma unroll
                            for (int j = 0; j < 4; ++j) sb2[j] = lds64(sbs + (c * 32 + 8 * j) * 4);
                        }
                        tmem_ld_wait();
                        if (c + 1 == BN / 32) {
                            // the last chunk is in registers: hand the TMEM buffer back before the arithmetic
                            tc_fence_before();
                            __syncwarp();
                            if (lane == 0) mbar_arrive(bar_tempty(buf));
                        }
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const unsigned long long sa2 = pack2(sa4[k], sa4[k]);
                            const uint32_t* src = (k < 2) ? lo : hi;
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                const uint32_t* tp = src + 4 * j + 2 * (k & 1);
                                const unsigned long long v = pack2u(tp[0], tp[1]);
                                acc2[k * JG + c * 4 + j] = fma2((MODE == MODE_FP32_SB_TILE) ? v : mul2(v, sb2[j]), sa2, acc2[k * JG + c * 4 + j]);
                            }
                        }
                    }
                    if (++buf == C::BUFS) { buf = 0; bphase ^= 1u; }
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_sempty(ss));
                if (++ss == C::S_STAGES) { ss = 0; sphase ^= 1u; }
            }
            // the last hand-off says that every MMA of this CTA has read its operands: the ring may be overwritten
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int rr = lane >> 2, row = q * 32 + rr + 8 * k;
#pragma unroll
                for (int j = 0; j < JG; ++j) {
                    const int piece = 2 * j + ((lane & 3) >> 1);
                    sts64(tile + row * C::ROW_BYTES + ((piece ^ rr) << 4) + (lane & 1) * 8, acc2[k * JG + j]);
                }
            }
        }
        cluster_sync();                                      // every CTA's partial product is in its shared memory

        // ---- weighted sums of this CTA's share of the rows, 128 / BN rows per warp and step; the remote loads
        // of the next step are in flight while this one is summed and stored (remote shared memory delivers 12 bytes per
        // clock and SM, 4.5k cycles for the 64 KB of a CTA with 128 columns, measured)
        constexpr int LANES = BN / 4, RPW = 32 / LANES;       // lanes per row, rows per warp and step
        const int r0 = BM * rank / S, r1 = BM * (rank + 1) / S, piece = lane % LANES;
        uint32_t peer[FMM_MAX_RANK];
#pragma unroll
        for (int j = 0; j < FMM_MAX_RANK; ++j) peer[j] = map_to_cta(tile, j < S ? j : 0);
        float* c_tile = p.C + ((long long)parent * (p.nq == 4 ? 2 : 1) * p.m + tm * BM) * p.ldc + tn * BN + piece * 4;
        auto fetch = [&](int row, float4 (&v)[FMM_MAX_RANK]) {
            const uint32_t off = row * C::ROW_BYTES + ((piece ^ (row & 7)) << 4);
#pragma unroll
            for (int j = 0; j < FMM_MAX_RANK; ++j) if (j < S) v[j] = ld_cluster128(peer[j] + off);
        };
        auto sum_and_store = [&](int row, const float4 (&v)[FMM_MAX_RANK]) {
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                if (b >= p.nq) break;
                float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int j = 0; j < FMM_MAX_RANK; ++j) {
                    const float wj = p.W[j][b];                // zero for j >= S
                    if (wj != 0.0f) { o.x = fmaf(wj, v[j].x, o.x); o.y = fmaf(wj, v[j].y, o.y); o.z = fmaf(wj, v[j].z, o.z); o.w = fmaf(wj, v[j].w, o.w); }
                }
                float* dst = c_tile + ((long long)(b >> 1) * p.m + row) * p.ldc + (long long)(b & 1) * p.n;
                if (FMM_GUARD(p.guard, dst, 16, 1721)) *reinterpret_cast<float4*>(dst) = o;
            }
        };
        float4 v0[FMM_MAX_RANK], v1[FMM_MAX_RANK];
        constexpr int STEP = C::EPI_WARPS * RPW;
        int row = r0 + q * RPW + lane / LANES;
        if (row < r1) fetch(row, v0);
#pragma unroll 1
        for (; row < r1; row += 2 * STEP) {
            const bool more1 = row + STEP < r1, more2 = row + 2 * STEP < r1;
            if (more1) fetch(row + STEP, v1);
            sum_and_store(row, v0);
            if (more2) fetch(row + 2 * STEP, v0);
            if (more1) sum_and_store(row + STEP, v1);
        }
        }
        (void)ok;
    }

    // ---------------------------------------------------------------------- teardown
    if (*abort_flag) {
        // let copies that are still in flight towards this CTA's shared memory land
        const uint64_t t0 = global_timer();
        while (global_timer() - t0 < 200000ull) __nanosleep(1000);
    }
    tc_fence_before();
    cluster_sync_relaxed();                // the peers no longer read this CTA's shared memory (their loads have returned)
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc<1>(tmem_base, C::TMEM_COLS);
    }
}

// The kernel's shared memory limit, raised once per device.
template <int MODE, int BLK, int BN, int TPC = 1>
bool prepare_split(int dev)
{
    static std::atomic<bool> attr_set[64];
    if (dev >= 0 && dev < 64 && attr_set[dev].load(std::memory_order_acquire)) return true;
    if (cudaFuncSetAttribute(fmm_split_kernel<MODE, BLK, BN, TPC>, cudaFuncAttributeMaxDynamicSharedMemorySize, SplitCfg<MODE, BLK, BN, TPC>::SMEM_BYTES) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    if (dev >= 0 && dev < 64) attr_set[dev].store(true, std::memory_order_release);
    return true;
}

template <int MODE, int BLK, int BN>
cudaLaunchConfig_t split_config(int S, unsigned tiles_n, unsigned tiles_m, unsigned parents, cudaStream_t st, cudaLaunchAttribute* attr)
{
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3(tiles_n * S, tiles_m, parents);
    cfg.blockDim = dim3(SplitCfg<MODE, BLK, BN>::THREADS, 1, 1);
    cfg.dynamicSmemBytes = SplitCfg<MODE, BLK, BN>::SMEM_BYTES;
    cfg.stream = st;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = S; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    return cfg;
}

// CTAs that an SM holds, by what they take of its registers, shared memory and TMEM, and as the runtime counts them: one per SM
// for a kernel that allocates TMEM, though two are resident (3.1 warps per scheduler, measured).
template <int MODE, int BLK, int BN>
bool ctas_per_sm(int dev, int* own, int* runtime)
{
    using C = SplitCfg<MODE, BLK, BN>;
    int regs = 0, smem = 0, reserved = 0;
    cudaFuncAttributes attr;
    if (cudaDeviceGetAttribute(&regs, cudaDevAttrMaxRegistersPerMultiprocessor, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&smem, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev) != cudaSuccess ||
        cudaFuncGetAttributes(&attr, fmm_split_kernel<MODE, BLK, BN, 1>) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(runtime, fmm_split_kernel<MODE, BLK, BN, 1>, C::THREADS, C::SMEM_BYTES) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    *own = std::min(std::min(regs / (attr.numRegs * C::THREADS), smem / (C::SMEM_BYTES + reserved)), 512 / C::TMEM_COLS);
    return *own > 0 && *runtime > 0;
}

// How many clusters of S CTAs the device holds at once: clusters stay inside a GPC, so this is less than SMs / S times the CTAs
// of an SM.  Asked for the widest tile: the narrower ones are resident as often, two to an SM by their registers.
template <int MODE, int BLK>
int resident_clusters(int dev, int S)
{
    static std::atomic<int> known[64][FMM_MAX_RANK + 1];
    if (dev >= 0 && dev < 64) { const int n = known[dev][S].load(std::memory_order_relaxed); if (n > 0) return n; }
    int n = 0, own = 0, runtime = 0;
    cudaLaunchAttribute attr[1];
    const cudaLaunchConfig_t cfg = split_config<MODE, BLK, 128>(S, 1, 1, 1, nullptr, attr);
    if (!prepare_split<MODE, BLK, 128>(dev) || cudaOccupancyMaxActiveClusters(&n, fmm_split_kernel<MODE, BLK, 128, 1>, &cfg) != cudaSuccess || n <= 0 ||
        !ctas_per_sm<MODE, BLK, 128>(dev, &own, &runtime)) {
        cudaGetLastError();
        return 0;
    }
    n = n * own / runtime;
    if (dev >= 0 && dev < 64) known[dev][S].store(n, std::memory_order_relaxed);
    return n;
}

template <int MODE, int BLK, int BN, int TPC = 1>
fmm_status_t launch_split(const GemmParams& g, int ksplit, cudaStream_t st)
{
    using C = SplitCfg<MODE, BLK, BN>;
    CUtensorMap tmA, tmB, tmSFA, tmSFB;
    const CUtensorMapSwizzle SW = CU_TENSOR_MAP_SWIZZLE_128B;
    if (!make_map_2d(&tmA, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, g.qa, (uint64_t)g.k, (uint64_t)(g.terms - 1) * g.m + g.msub, BK, BM, SW)) return FMM_ERR_CUDA;
    if (!make_map_2d(&tmB, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, g.qb, (uint64_t)g.k, (uint64_t)(g.terms - 1) * g.n + g.nsub, BK, C::BN, SW)) return FMM_ERR_CUDA;
    if (C::MX) {
        const uint64_t chunks = (uint64_t)g.terms * (g.k / 128);
        const uint64_t atoms_a = (chunks - 1) * (g.m / 128) + g.msub / 128, atoms_b = (chunks - 1) * (g.n / 128) + g.nsub / 128;
        if (!make_map_2d(&tmSFA, CU_TENSOR_MAP_DATA_TYPE_UINT32, 4, g.sa, 128, atoms_a, 128, 1, CU_TENSOR_MAP_SWIZZLE_NONE)) return FMM_ERR_CUDA;
        if (!make_map_2d(&tmSFB, CU_TENSOR_MAP_DATA_TYPE_UINT32, 4, g.sb, 128, atoms_b, 128, 1, CU_TENSOR_MAP_SWIZZLE_NONE)) return FMM_ERR_CUDA;
    } else {
        tmSFA = tmA; tmSFB = tmB;       // unused in this mode
    }
    if (!prepare_split<MODE, BLK, BN, TPC>(g.device)) return FMM_ERR_CUDA;
    SplitParams p;
    p.sa = static_cast<const uint8_t*>(g.sa); p.sb = static_cast<const uint8_t*>(g.sb);
    p.sa_term = g.sa_term; p.sb_term = g.sb_term;
    p.m = g.m; p.n = g.n; p.k = g.k;
    p.R = g.R; p.ksplit = ksplit; p.nq = g.nq;
    memset(p.W, 0, sizeof(p.W));
    // times the factor that the sums were kept small by, see fmm_scale_down
    if (g.nq == 4) for (int r = 0; r < g.R; ++r) for (int b = 0; b < 4; ++b) p.W[r][b] = g.W[r][b] * g.up;
    else for (int j = 0; j < ksplit; ++j) p.W[j][0] = g.up;
    p.C = g.C; p.ldc = g.Nfull; p.status = g.status; p.guard = g.guard;
    const int S = (g.R + TPC - 1) / TPC * ksplit;

    cudaLaunchAttribute attr[2];
    cudaLaunchConfig_t cfg = split_config<MODE, BLK, BN>(S, (unsigned)(g.nsub / C::BN), (unsigned)(g.msub / BM), (unsigned)(g.terms / g.R), st, attr);
    // right behind the encoders of the same call: set up while they drain, the producer warps wait before their first load
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.numAttrs = g.overlap_prev ? 2 : 1;
    if (cudaLaunchKernelEx(&cfg, fmm_split_kernel<MODE, BLK, BN, TPC>, tmA, tmB, tmSFA, tmSFB, p) != cudaSuccess) { cudaGetLastError(); return FMM_ERR_CUDA; }
    return FMM_OK;
}

// Time model of the cluster kernel in microseconds, fitted together with the one of the persistent kernel (fmm_gemm_shape): lat +
// waves * (f + k * c), k in stages of 128, f being set-up, exchange and output; f and c depend on the tile's width.  A
// cluster that ends makes room for the next at once, so waves is a fraction (of the places; without an exchange the CTAs of
// an SM get in each other's way, and `alone` of the places count).  So the cluster kernel takes the products of few tiles,
// whatever their K: leaves of 128 to 1024, and it takes tiles of 64 or 32 columns as long as about all of them are resident
// at once.  Rank 7, block 32, one level, 128 columns -> the width chosen: n = 256 8.6 -> 5.1 us, n = 512 10.7 -> 7.2,
// n = 1024 18.5 -> 14.0, 512 x 4096 x 1024 40.6 -> 19.7, 256 x 8192 x 256 74.7 -> 27.6.
struct SplitModel { float lat, alone; int widths; float f[3], c[3], f_two; };       // f, c: 128, 64, 32 columns; f_two: two terms per CTA
constexpr SplitModel SPLIT_MX = {0.65f, 0.67f, 1, {6.6f, 0.f, 0.f}, {0.33f, 0.f, 0.f}, 10.5f};
constexpr SplitModel SPLIT_B32 = {1.7f, 0.89f, 3, {7.15f, 5.55f, 3.75f}, {2.02f, 1.31f, 0.82f}, 0.0f};
constexpr SplitModel SPLIT_B128 = {1.55f, 0.85f, 3, {7.5f, 5.9f, 4.25f}, {0.61f, 0.34f, 0.34f}, 0.0f};
constexpr SplitModel SPLIT_TILE = {1.55f, 0.88f, 3, {6.9f, 4.85f, 3.55f}, {0.47f, 0.37f, 0.33f}, 0.0f};

template <int MODE, int BLK>
SplitChoice choose_split(const GemmParams& g, const SplitModel& m, float persistent_time)
{
    const int kst = g.k / BK;
    const long long parents = g.terms / g.R;
    float best_time = persistent_time;
    SplitChoice best = {0, 0, 1, 0};
    for (int ks = 1; g.R * ks <= FMM_MAX_RANK && ks <= kst; ks *= 2) {
        const int cap = resident_clusters<MODE, BLK>(g.device, g.R * ks);
        if (cap <= 0) break;
        const float places = g.R * ks > 1 ? (float)cap : cap * m.alone;
        for (int w = 0; w < m.widths; ++w) {
            const long long tiles = (long long)(g.m / BM) * (g.n / (128 >> w)) * parents;
            const float waves = std::max(1.0f, (float)tiles / places);
            const float time = m.lat + waves * (m.f[w] + ((kst + ks - 1) / ks) * m.c[w]);
            if (time < best_time) { best_time = time; best = {ks, 128 >> w, 1, cap}; }
        }
        if (g.R > 1) break;
    }
    // two terms per CTA (UE8M0): for the products that clusters of R do not hold at once and these do.  f: a longer exchange, as a
    // CTA sums twice the rows.  n = 2048 33.4 -> 30.9 us a call, 2048 x 512 x 2048 23.0 -> 20.6, 1280 x 3328 x 2816 42.3 -> 40.7, 512 x 4096
    // x 8192 76.0 -> 71.1, two levels n = 1536 35.4 -> 34.3; where one wave of clusters of R is enough it is slower (n = 1536 20.8, 26.6;
    // n = 1024 14.4, 17.9), and so it is in more than one wave of its own (n = 2560 54.4, the persistent kernel 47.3).
    if (m.f_two > 0.0f && g.R > 1) {
        const int cap = resident_clusters<MODE, BLK>(g.device, (g.R + 1) / 2);
        const long long tiles = (long long)(g.m / BM) * (g.n / 128) * parents;
        if (tiles <= cap && m.lat + m.f_two + 2 * kst * m.c[0] < best_time) best = {1, 128, 2, cap};
    }
    return best;
}

template <int BN>
fmm_status_t launch_fp32(const GemmParams& g, int blk, int ksplit, cudaStream_t st)
{
    if (blk == 32) return launch_split<MODE_FP32_COLUMN, 32, BN>(g, ksplit, st);
    if (g.sb_tile) return launch_split<MODE_FP32_SB_TILE, 128, BN>(g, ksplit, st);
    return launch_split<MODE_FP32_COLUMN, 128, BN>(g, ksplit, st);
}

}  // namespace

SplitChoice fmm_split_choice(const GemmParams& g, int blk, int mode)
{
    if (g.m / BM > 65535 || g.terms / g.R > 65535) return {0, 0, 1, 0};     // grid dimensions
    const float t = fmm_gemm_shape(g, blk, mode, g.m, g.n).time;
    if (mode == FMM_SCALE_UE8M0_CEIL) return choose_split<FMM_SCALE_UE8M0_CEIL, 32>(g, SPLIT_MX, t);
    if (blk == 32) return choose_split<MODE_FP32_COLUMN, 32>(g, SPLIT_B32, t);
    if (g.sb_tile) return choose_split<MODE_FP32_SB_TILE, 128>(g, SPLIT_TILE, t);
    return choose_split<MODE_FP32_COLUMN, 128>(g, SPLIT_B128, t);
}

fmm_status_t fmm_launch_split(const GemmParams& g, int blk, int mode, SplitChoice c, cudaStream_t st)
{
    if (mode == FMM_SCALE_UE8M0_CEIL) return c.terms == 2 ? launch_split<FMM_SCALE_UE8M0_CEIL, 32, 128, 2>(g, c.ksplit, st) : launch_split<FMM_SCALE_UE8M0_CEIL, 32, 128>(g, c.ksplit, st);
    if (c.bn == 32) return launch_fp32<32>(g, blk, c.ksplit, st);
    if (c.bn == 64) return launch_fp32<64>(g, blk, c.ksplit, st);
    return launch_fp32<128>(g, blk, c.ksplit, st);
}
