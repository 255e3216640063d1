// Product kernel for short terms (the operation is the one of fmm_gemm.cu): the parent's output blocks stay on chip.
//
// A persistent CTA owns a 128 x 64 tile position of one parent and walks its R terms; the four tiles of the position, one in each
// output block, stay in the registers of the promoting warps, and every finished product is added to those it feeds,
// C_q += W[r][q] * M_r in ascending r (the cluster kernel's sums, to the bit).  A tile of C is written once, after the last term,
// where the kernel of fmm_gemm.cu sends a weighted update per term and block through L2 (12 of 64 KB for the Phi-optimal
// realization, at about 25 bytes per clock and SM): with terms of a few K stages those updates take longer than the products.
// Against the cluster kernel, whose exchange goes through distributed shared memory at 15 bytes per clock and SM, it gains where the
// tiles are more than two thirds of the clusters' places.
//
// 64 columns are what the registers hold: four tiles of 128 x 64 are half of the register file.  The price is operand traffic,
// 24 KB per stage and 128 x 64 tile instead of 32 KB per 128 x 128: an SM receives about 59 bytes per clock from L2, so a
// stage cannot take less than 410 cycles, which the block-32 promotion (4 x 280 cycles) does not notice and UE8M0 and
// block 128 pay for with long terms.  Five operand stages for that reason (three: UE8M0 n = 4096 159 us instead of 108, 2048 x 1024 x 2048
// 14.7 instead of 13.0), paid for with two staging pieces a warp instead of one per block, which costs nothing.  Block 32: a stage's
// four K blocks share one completion signal (two signals, with the fourth block in TMEM: three levels n = 2048 57.7 us instead of 54.3).
//
//   warp 0  TMA producer of the operand tiles (UE8M0: and of the scale tiles)
//   warp 1  tcgen05.mma issuer
//   warp 2  FP32 scales: producer of both sides' scales
//   warps 4..11  promotion (FP32 scales) or drain (UE8M0), sums of the blocks, output
#include <algorithm>
#include "fmm_gemm_common.cuh"

namespace {

constexpr int MODE_FP32_COLUMN = FMM_SCALE_FP32_AMAX_DIV_448;      // one B-side scale per column and K block

struct KeepParams {
    const uint8_t* sa; const uint8_t* sb;      // fp32 scale arrays (bytes)
    long long sa_term, sb_term;
    int m, n, k, R;
    int tiles_m, tiles_n, items;                // tile positions of a parent (of a strip of it), of all parents
    float W[FMM_MAX_RANK][4];                   // weight of product r in output block q, times the factor of fmm_scale_up
    int* status;
    const float* c_base; long long ldc;         // the output matrix as plain memory: used by the FMM_DEBUG store guard only
    FmmGuard guard;
};

template <int MODE, int BLK>
struct KeepCfg {
    static constexpr bool MX = (MODE == FMM_SCALE_UE8M0_CEIL), ROWS4 = (MODE == MODE_FP32_COLUMN);
    static constexpr int BN = 64, CW = 32;                   // columns of a tile, of a promoting warp
    static constexpr int EPI_WARP0 = 4, EPI_WARPS = 8, THREADS = (EPI_WARP0 + EPI_WARPS) * 32;
    static constexpr int REGS_AT_LAUNCH = 168;
    // (224 or 232 registers with FP32 scales per column: the same within 1 %, no spills)
    static constexpr int REGS_CTRL = ROWS4 ? 56 : 72, REGS_EPI = ROWS4 ? 224 : 216;
    static_assert(EPI_WARP0 * 32 * REGS_CTRL + EPI_WARPS * 32 * REGS_EPI <= THREADS * REGS_AT_LAUNCH, "register pool");
    static constexpr int KB = MX ? 1 : BK / BLK;             // accumulations of a stage
    // K blocks that share a completion signal (those of a stage), and buffers of that many accumulators.  UE8M0: a product each
    static constexpr int GPB = KB, ACC_BUFS = KB == 4 ? 2 : 4;
    static constexpr int OFF_SFT = GPB * ACC_BUFS * BN;      // TMEM: the accumulators, UE8M0: the scales
    static_assert(OFF_SFT + (MX ? 16 : 0) <= 512, "TMEM budget");
    static constexpr int A_BYTES = BM * BK, B_BYTES = BN * BK, SF_BYTES = MX ? 1024 : 0;
    static constexpr int TX_BYTES = A_BYTES + B_BYTES + SF_BYTES;
    static constexpr int STAGES = 5;
    static constexpr int S_STAGES = MX ? 0 : STAGES + 1;
    static constexpr int SB_BYTES = KB * BN * 4, S_BYTES = MX ? 0 : KB * (BN + BM) * 4;
    static constexpr int FULL_SLOTS = MX ? ACC_BUFS : S_STAGES;
    // the issuer runs up to ACC_BUFS signals ahead of the promoting warps: their barriers must not come round before
    static_assert(FULL_SLOTS >= ACC_BUFS, "ring of signals");
    static constexpr int STG_BYTES = 4096;                   // a warp's 32 x 32 piece of a tile; two per warp
    static constexpr int OFF_A = 0;
    static constexpr int OFF_B = OFF_A + STAGES * A_BYTES;
    static constexpr int OFF_STG = OFF_B + STAGES * B_BYTES;
    static constexpr int OFF_SF = OFF_STG + EPI_WARPS * 2 * STG_BYTES;
    static constexpr int OFF_S = OFF_SF + STAGES * SF_BYTES;
    static constexpr int OFF_BAR = OFF_S + S_STAGES * S_BYTES;
    static constexpr int NUM_BARS = 2 * STAGES + S_STAGES + FULL_SLOTS + ACC_BUFS;
    static constexpr int SMEM_BYTES = OFF_BAR + NUM_BARS * 8 + 16 + 1024;   // + alignment slack
    static_assert(SMEM_BYTES <= 232448, "shared memory budget");
};

template <int MODE, int BLK>
__global__ void __launch_bounds__(KeepCfg<MODE, BLK>::THREADS, 1)
fmm_keep_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const __grid_constant__ CUtensorMap tmC,
                const __grid_constant__ CUtensorMap tmSFA, const __grid_constant__ CUtensorMap tmSFB, const KeepParams p)
{
    using C = KeepCfg<MODE, BLK>;
    constexpr int BN = C::BN, KB = C::KB;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw_addr = smem_u32(smem_raw);
    const uint32_t base = (raw_addr + 1023u) & ~1023u;
    uint8_t* base_ptr = smem_raw + (base - raw_addr);

    const uint32_t bar0 = base + C::OFF_BAR;
    auto bar_full = [&](int s) { return bar0 + 8u * s; };
    auto bar_empty = [&](int s) { return bar0 + 8u * (C::STAGES + s); };
    auto bar_sempty = [&](int s) { return bar0 + 8u * (2 * C::STAGES + s); };
    auto bar_tfull = [&](int b) { return bar0 + 8u * (2 * C::STAGES + C::S_STAGES + b); };
    auto bar_tempty = [&](int b) { return bar0 + 8u * (2 * C::STAGES + C::S_STAGES + C::FULL_SLOTS + b); };
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(base_ptr + C::OFF_BAR + C::NUM_BARS * 8);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    const Ctl ctl{abort_flag, p.status};

    const int warp = warp_uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < C::STAGES; ++s) { mbar_init(bar_full(s), 1); mbar_init(bar_empty(s), 1); }
        for (int s = 0; s < C::S_STAGES; ++s) mbar_init(bar_sempty(s), C::EPI_WARPS);
        // FP32 scales: a stage's K blocks are signalled together with its scales
        for (int b = 0; b < C::FULL_SLOTS; ++b) mbar_init(bar_tfull(b), C::MX ? 1 : 2);
        for (int b = 0; b < C::ACC_BUFS; ++b) mbar_init(bar_tempty(b), C::EPI_WARPS);
        *abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 1) {
        tmem_alloc<1>(smem_u32(tmem_slot), 512);
        tmem_relinquish<1>();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = warp_uniform(*tmem_slot);

    const int kstages = p.k / BK, per_parent = p.tiles_m * p.tiles_n;
    struct Item { int parent, tm, tn; };
    auto item = [&](int w) {
        Item i;
        i.parent = w / per_parent;
        const int pos = w - i.parent * per_parent;
        i.tm = pos / p.tiles_n; i.tn = pos - i.tm * p.tiles_n;
        return i;
    };

    if (warp < C::EPI_WARP0) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(C::REGS_CTRL));
        bool ok = true;
        if (warp == 0) {
            // ------------------------------------------------------------------ TMA producer
            griddep_wait();        // the encoders' output is complete and visible (no-op unless launched to overlap them)
            int stage = 0; uint32_t phase = 0;
            const int row_blocks_a = p.m / 128, row_blocks_b = p.n / 128;
            for (int w = blockIdx.x; w < p.items && ok; w += gridDim.x) {
                const Item it = item(w);
                for (int t = it.parent * p.R; t < (it.parent + 1) * p.R && ok; ++t)
                    for (int ks = 0; ks < kstages; ++ks) {
                        if (!mbar_wait_warp(bar_empty(stage), phase ^ 1u, ctl, 141)) { ok = false; break; }
                        if (elect_one()) {
                            mbar_expect_tx(bar_full(stage), C::TX_BYTES);
                            tma_load_2d<1>(base + C::OFF_A + stage * C::A_BYTES, &tmA, ks * BK, t * p.m + it.tm * BM, bar_full(stage));
                            tma_load_2d<1>(base + C::OFF_B + stage * C::B_BYTES, &tmB, ks * BK, t * p.n + it.tn * BN, bar_full(stage));
                            if (C::MX) {
                                const uint32_t sf = base + C::OFF_SF + stage * C::SF_BYTES;
                                tma_load_2d<1>(sf, &tmSFA, 0, (t * kstages + ks) * row_blocks_a + it.tm, bar_full(stage));
                                tma_load_2d<1>(sf + 512, &tmSFB, 0, (t * kstages + ks) * row_blocks_b + (it.tn >> 1), bar_full(stage));
                            }
                        }
                        if (++stage == C::STAGES) { stage = 0; phase ^= 1u; }
                    }
            }
        } else if (warp == 2 && !C::MX) {
            // ------------------------------------------------------------------ producer of both sides' fp32 scales
            griddep_wait();
            int ss = 0; uint32_t sphase = 0;
            for (int w = blockIdx.x; w < p.items && ok; w += gridDim.x) {
                const Item it = item(w);
                for (int t = it.parent * p.R; t < (it.parent + 1) * p.R && ok; ++t) {
                    const uint8_t* sb = p.sb + (long long)t * p.sb_term + (long long)it.tn * BN * 4;
                    const uint8_t* sa = p.sa + (long long)t * p.sa_term + (long long)it.tm * BM * (KB * 4);
                    for (int ks = 0; ks < kstages; ++ks) {
                        if (!mbar_wait_warp(bar_sempty(ss), sphase ^ 1u, ctl, 142)) { ok = false; break; }
                        if (elect_one()) {
                            const uint32_t fb = bar_tfull(ss), dst = base + C::OFF_S + ss * C::S_BYTES;
                            mbar_expect_tx(fb, C::S_BYTES);
#pragma unroll
                            for (int g = 0; g < KB; ++g)
                                bulk_load(dst + g * BN * 4, sb + (long long)(ks * KB + g) * p.n * 4, BN * 4, fb);
                            bulk_load(dst + C::SB_BYTES, sa + (long long)ks * p.m * (KB * 4), BM * KB * 4, fb);
                        }
                        if (++ss == C::S_STAGES) { ss = 0; sphase ^= 1u; }
                    }
                }
            }
        } else if (warp == 1) {
            // ------------------------------------------------------------------ MMA issuer
            int stage = 0; uint32_t phase = 0;
            int buf = 0, slot = 0; uint32_t bphase = 0;
            constexpr uint32_t idesc = (C::MX ? (1u << 23) : (1u << 4)) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
            for (int w = blockIdx.x; w < p.items && ok; w += gridDim.x) {
                // UE8M0: this tile's half of the 128 columns that a scale tile covers
                const uint32_t sf_half = C::MX ? 2u * (item(w).tn & 1) : 0u;
                for (int r = 0; r < p.R && ok; ++r) {
                    if (C::MX) {
                        if (!mbar_wait_warp(bar_tempty(buf), bphase ^ 1u, ctl, 241)) { ok = false; break; }
                        tc_fence_after();
                    }
                    for (int ks = 0; ks < kstages && ok; ++ks) {
                        if (!mbar_wait_warp(bar_full(stage), phase, ctl, 242)) { ok = false; break; }
                        tc_fence_after();
                        const uint64_t adesc = make_kmajor_sw128_desc(base + C::OFF_A + stage * C::A_BYTES);
                        const uint64_t bdesc = make_kmajor_sw128_desc(base + C::OFF_B + stage * C::B_BYTES);
                        if (C::MX) {
                            const uint32_t sf = base + C::OFF_SF + stage * C::SF_BYTES;
                            const uint32_t tsfa = tmem_base + C::OFF_SFT, tsfb = tsfa + 4;     // one slot: cp and mma execute in issue order
                            tc_cp_32x128b_warpx4<1>(tsfa, make_sf_desc(sf));
                            tc_cp_32x128b_warpx4<1>(tsfb, make_sf_desc(sf + 512));
#pragma unroll
                            for (int j = 0; j < BK / 32; ++j) {
                                const uint32_t id = idesc | ((uint32_t)j << 29) | ((uint32_t)j << 4);
                                mma_mxf8<1>(tmem_base + buf * BN, adesc + 2 * j, bdesc + 2 * j, id, (ks > 0 || j > 0) ? 1u : 0u, tsfa, tsfb + sf_half);
                            }
                        } else {
                            if (!mbar_wait_warp(bar_tempty(buf), bphase ^ 1u, ctl, 243)) { ok = false; break; }
                            tc_fence_after();
#pragma unroll
                            for (int j = 0; j < BK / 32; ++j)
                                mma_f8f6f4<1>(tmem_base + (buf * C::GPB + (KB == 4 ? j : 0)) * BN, adesc + 2 * j, bdesc + 2 * j, idesc, KB == 4 || j == 0 ? 0u : 1u);
                            tc_commit<1>(bar_tfull(slot));
                            if (++slot == C::FULL_SLOTS) slot = 0;
                            if (++buf == C::ACC_BUFS) { buf = 0; bphase ^= 1u; }
                        }
                        tc_commit<1>(bar_empty(stage));
                        if (++stage == C::STAGES) { stage = 0; phase ^= 1u; }
                    }
                    if (C::MX && ok) {
                        tc_commit<1>(bar_tfull(buf));
                        if (++buf == C::ACC_BUFS) { buf = 0; bphase ^= 1u; }
                    }
                }
            }
        }
    } else {
        // ---------------------------------------------------------------------- promotion / drain, sums of the blocks, output
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(C::REGS_EPI));
        const int e = warp - C::EPI_WARP0, q = warp & 3, h = e >> 2;       // TMEM lane quadrant, column half
        constexpr int CW = C::CW;
        const uint32_t tq = tmem_base + ((uint32_t)(q * 32) << 16) + h * CW;
        const uint32_t stg = base + C::OFF_STG + e * 2 * C::STG_BYTES;
        // A thread's 32 elements of the tile, as pairs.  ROWS4: rows lane/4 + 8k, columns 8j + 2(lane%4) and the next, at k * 4 + j;
        // otherwise row `lane`, columns 2i and the next.
        unsigned long long acc[CW / 2], blk[4][CW / 2];
        int buf = 0, ss = 0; uint32_t bphase = 0, sphase = 0;
        bool ok = true;
        auto release_acc = [&](int b) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_tempty(b));
        };
        // ROWS4: see the promotion loop of fmm_gemm.cu
        uint32_t set0[C::ROWS4 ? 16 : 1], set1[C::ROWS4 ? 16 : 1];
        unsigned long long sb2[4];
        float sa[KB == 4 ? 4 : 1][4];                               // A-side scales of the thread's rows: of a stage's K blocks [row][block], or [0][row]
        const uint32_t sa_lane = base + C::OFF_S + C::SB_BYTES + (q * 32 + (lane >> 2)) * (KB * 4);
        const uint32_t sb_lane = base + C::OFF_S + (h * CW + 2 * (lane & 3)) * 4;
        auto wait_full = [&](int slot, uint32_t phase) {
            const bool ready = mbar_test_wait(bar_tfull(slot), phase);
            return __all_sync(0xffffffffu, ready) || mbar_wait_warp(bar_tfull(slot), phase, ctl, 341);
        };
        auto load_chunk = [&](uint32_t* r, int b, int gi, int i) {
            tmem_ld_16x256b_x4(tq + (b * C::GPB + gi) * BN + ((uint32_t)(16 * i) << 16), r);
        };
        auto load_sb = [&](unsigned long long (&d)[4], int s, int g) {
#pragma unroll
            for (int j = 0; j < 4; ++j) d[j] = lds64(sb_lane + s * C::S_BYTES + (g * BN + 8 * j) * 4);
        };
        auto load_sa1 = [&](float (&d)[4], int s) {
#pragma unroll
            for (int k = 0; k < 4; ++k) d[k] = lds32f(sa_lane + s * C::S_BYTES + 8 * k * 4);
        };
        if constexpr (C::ROWS4) {
            ok = wait_full(0, 0);
            tc_fence_after();
            load_chunk(set0, 0, 0, 0);
            load_sb(sb2, 0, 0);
            if constexpr (KB == 1) load_sa1(sa[0], 0);
            tmem_ld_wait16(set0);
        }
        for (int w = blockIdx.x; w < p.items && ok; w += gridDim.x) {
            const Item it = item(w);
#pragma unroll
            for (int b = 0; b < 4; ++b)
#pragma unroll
                for (int i = 0; i < CW / 2; ++i) blk[b][i] = 0ull;
            for (int r = 0; r < p.R && ok; ++r) {
                if constexpr (C::MX) {
                    if (!mbar_wait_warp(bar_tfull(buf), bphase, ctl, 342)) { ok = false; break; }
                    tc_fence_after();
                    uint32_t v[CW];
                    tmem_ld32(tq + buf * BN, v);
                    tmem_ld_wait();
                    release_acc(buf);
                    if (++buf == C::ACC_BUFS) { buf = 0; bphase ^= 1u; }
#pragma unroll
                    for (int i = 0; i < CW / 2; ++i) acc[i] = pack2u(v[2 * i], v[2 * i + 1]);
                } else if constexpr (C::ROWS4) {
#pragma unroll
                    for (int i = 0; i < CW / 2; ++i) acc[i] = 0ull;
                    const bool more = r + 1 < p.R || w + (int)gridDim.x < p.items;       // another product after this one
                    for (int ks = 0; ks < kstages && ok; ++ks) {
                        const bool wrap = ss + 1 == C::S_STAGES;
                        const int sn = wrap ? 0 : ss + 1;
                        const uint32_t pn = wrap ? sphase ^ 1u : sphase;
                        if constexpr (KB == 4) {
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                const float4 v4 = lds128(sa_lane + ss * C::S_BYTES + 8 * k * 16);
                                sa[k][0] = v4.x; sa[k][1] = v4.y; sa[k][2] = v4.z; sa[k][3] = v4.w;
                            }
                        }
#pragma unroll
                        for (int g = 0; g < KB; ++g) {
                            // acc += (P * sB) * sA, 16 rows at a time
                            auto promote = [&](const uint32_t* cur, int k0) {
#pragma unroll
                                for (int k = k0; k < k0 + 2; ++k) {
                                    const float s = KB == 4 ? sa[KB == 4 ? k : 0][g] : sa[0][k];
                                    const unsigned long long s2 = pack2(s, s);
#pragma unroll
                                    for (int j = 0; j < 4; ++j)
                                        acc[k * 4 + j] = fma2(mul2(pack2u(cur[4 * j + 2 * (k - k0)], cur[4 * j + 2 * (k - k0) + 1]), sb2[j]), s2, acc[k * 4 + j]);
                                }
                            };
                            load_chunk(set1, buf, g, 1);
                            promote(set0, 0);
                            tmem_ld_wait16(set1);
                            int nb = buf;
                            if (g + 1 == KB) {
                                // the buffer's last chunk is in registers: hand it back before the arithmetic
                                release_acc(buf);
                                nb = buf + 1 == C::ACC_BUFS ? 0 : buf + 1;
                                // (without another product the loads below fetch what nobody uses)
                                if (ks + 1 < kstages || more) ok = ok && wait_full(sn, pn);
                                tc_fence_after();
                            }
                            unsigned long long sbn[4];
                            float san[4];
                            load_chunk(set0, nb, (g + 1) % KB, 0);
                            load_sb(sbn, g + 1 < KB ? ss : sn, (g + 1) % KB);
                            if constexpr (KB == 1) load_sa1(san, sn);
                            promote(set1, 2);
#pragma unroll
                            for (int j = 0; j < 4; ++j) { sb2[j] = sbn[j]; if (KB == 1) sa[0][j] = san[j]; }
                            tmem_ld_wait16(set0);
                            buf = nb;
                        }
                        __syncwarp();
                        if (lane == 0) mbar_arrive(bar_sempty(ss));
                        ss = sn; sphase = pn;
                    }
                    if (!ok) break;
                } else {
                    // weight tiles: one scale per row and K block, sA * sB_tile
#pragma unroll
                    for (int i = 0; i < CW / 2; ++i) acc[i] = 0ull;
                    const uint32_t sa_row = base + C::OFF_S + C::SB_BYTES + (q * 32 + lane) * 4;
                    for (int ks = 0; ks < kstages; ++ks) {
                        if (!wait_full(ss, sphase)) { ok = false; break; }
                        tc_fence_after();
                        uint32_t v[CW];
                        tmem_ld32(tq + buf * BN, v);
                        const float s = lds32f(sa_row + ss * C::S_BYTES) * lds32f(base + C::OFF_S + ss * C::S_BYTES);
                        const unsigned long long s2 = pack2(s, s);
                        tmem_ld_wait();
                        release_acc(buf);
                        if (++buf == C::ACC_BUFS) buf = 0;
#pragma unroll
                        for (int i = 0; i < CW / 2; ++i) acc[i] = fma2(pack2u(v[2 * i], v[2 * i + 1]), s2, acc[i]);
                        __syncwarp();
                        if (lane == 0) mbar_arrive(bar_sempty(ss));
                        if (++ss == C::S_STAGES) { ss = 0; sphase ^= 1u; }
                    }
                    if (!ok) break;
                }
                // ---- post-addition
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    const float wt = p.W[r][b];
                    if (wt != 0.0f) {
                        const unsigned long long w2 = pack2(wt, wt);
#pragma unroll
                        for (int i = 0; i < CW / 2; ++i) blk[b][i] = fma2(acc[i], w2, blk[b][i]);
                    }
                }
            }
            if (!ok) break;
            // ---- output: one 32 x 32 piece per block, rows of 128 bytes in the layout of the output tensor map
            if (lane == 0) bulk_wait_read<0>();          // the last pieces of the position before have been read
            __syncwarp();
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                if (b >= 2) {
                    if (lane == 0) bulk_wait_read<1>();
                    __syncwarp();
                }
                if constexpr (C::ROWS4) {
                    const uint32_t dst = stg + (b & 1) * C::STG_BYTES + (lane & 1) * 8;
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const int rr = (lane >> 2) + 8 * k;
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const int pc = 2 * j + ((lane & 3) >> 1);
                            sts64(dst + rr * 128 + ((pc ^ (rr & 7)) << 4), blk[b][k * 4 + j]);
                        }
                    }
                } else {
#pragma unroll
                    for (int i4 = 0; i4 < 8; ++i4) {
                        float4 v;
                        unpack2(blk[b][2 * i4], v.x, v.y); unpack2(blk[b][2 * i4 + 1], v.z, v.w);
                        sts128(stg + (b & 1) * C::STG_BYTES + lane * 128 + ((i4 ^ (lane & 7)) << 4), v);
                    }
                }
                fence_proxy_async();
                __syncwarp();
                if (lane == 0) {
                    const int row = (2 * it.parent + (b >> 1)) * p.m + it.tm * BM + q * 32, col = (b & 1) * p.n + it.tn * BN + h * CW;
                    if (FMM_GUARD(p.guard, p.c_base + (long long)row * p.ldc + col, (31 * p.ldc + 32) * 4, 1731))
                        tma_store_2d(&tmC, col, row, stg + (b & 1) * C::STG_BYTES);
                    bulk_commit();
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
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc<1>(tmem_base, 512);
    }
}

template <int MODE, int BLK>
fmm_status_t launch_keep(const GemmParams& g, cudaStream_t st)
{
    using C = KeepCfg<MODE, BLK>;
    CUtensorMap tmA, tmB, tmC, tmSFA, tmSFB;
    const CUtensorMapSwizzle SW = CU_TENSOR_MAP_SWIZZLE_128B;
    if (!make_map_2d(&tmA, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, g.qa, (uint64_t)g.k, (uint64_t)(g.terms - 1) * g.m + g.msub, BK, BM, SW)) return FMM_ERR_CUDA;
    if (!make_map_2d(&tmB, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, g.qb, (uint64_t)g.k, (uint64_t)(g.terms - 1) * g.n + g.nsub, BK, C::BN, SW)) return FMM_ERR_CUDA;
    if (!make_map_2d(&tmC, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, g.C, (uint64_t)(g.Nfull - g.n + g.nsub), (uint64_t)(g.Mfull - g.m + g.msub), 32, 32, SW, (uint64_t)g.Nfull)) return FMM_ERR_CUDA;
    if (C::MX) {
        const uint64_t chunks = (uint64_t)g.terms * (g.k / 128);
        const uint64_t atoms_a = (chunks - 1) * (g.m / 128) + g.msub / 128, atoms_b = (chunks - 1) * (g.n / 128) + g.nsub / 128;
        if (!make_map_2d(&tmSFA, CU_TENSOR_MAP_DATA_TYPE_UINT32, 4, g.sa, 128, atoms_a, 128, 1, CU_TENSOR_MAP_SWIZZLE_NONE)) return FMM_ERR_CUDA;
        if (!make_map_2d(&tmSFB, CU_TENSOR_MAP_DATA_TYPE_UINT32, 4, g.sb, 128, atoms_b, 128, 1, CU_TENSOR_MAP_SWIZZLE_NONE)) return FMM_ERR_CUDA;
    } else {
        tmSFA = tmA; tmSFB = tmB;       // unused in this mode
    }
    static std::atomic<bool> attr_set[64];       // the limit is a per-device attribute of the function
    if (g.device < 0 || g.device >= 64 || !attr_set[g.device].load(std::memory_order_acquire)) {
        if (cudaFuncSetAttribute(fmm_keep_kernel<MODE, BLK>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM_BYTES) != cudaSuccess) {
            cudaGetLastError();
            return FMM_ERR_CUDA;
        }
        if (g.device >= 0 && g.device < 64) attr_set[g.device].store(true, std::memory_order_release);
    }
    KeepParams p;
    p.sa = static_cast<const uint8_t*>(g.sa); p.sb = static_cast<const uint8_t*>(g.sb);
    p.sa_term = g.sa_term; p.sb_term = g.sb_term;
    p.m = g.m; p.n = g.n; p.k = g.k; p.R = g.R;
    p.tiles_m = g.msub / BM; p.tiles_n = g.nsub / C::BN;
    p.items = p.tiles_m * p.tiles_n * (g.terms / g.R);
    memset(p.W, 0, sizeof(p.W));
    for (int r = 0; r < g.R; ++r) for (int b = 0; b < 4; ++b) p.W[r][b] = g.W[r][b] * g.up;
    p.status = g.status; p.c_base = g.C; p.ldc = g.Nfull; p.guard = g.guard;
    // as few CTAs as finish in the same number of waves
    const int waves = (p.items + g.sms - 1) / g.sms, grid = (p.items + waves - 1) / waves;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)grid, 1, 1);
    cfg.blockDim = dim3(C::THREADS, 1, 1);
    cfg.dynamicSmemBytes = C::SMEM_BYTES;
    cfg.stream = st;
    // right behind the encoders of the same call: set up while they drain, the producer warps wait before their first load
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = g.overlap_prev ? 1 : 0;
    if (cudaLaunchKernelEx(&cfg, fmm_keep_kernel<MODE, BLK>, tmA, tmB, tmC, tmSFA, tmSFB, p) != cudaSuccess) { cudaGetLastError(); return FMM_ERR_CUDA; }
    return FMM_OK;
}

// Times of a product kernel's launch in microseconds, for the choice of this one.  kst: stages of 128 k of a term, u: updates of a
// parent's output blocks, items: 128 x 64 tiles of all parents' blocks; mem only where there are several parents, whose matrices
// lie in the workspace one behind the other and go through memory.
//   this kernel        base + waves * (o + R * kst * k) + mem * items                      waves of items over the SMs
//   persistent kernel  base + walks * (o + R * kst * k + u * out) + mem * items * u        parents that the busiest CTA (pair) walks
//   cluster kernel     base + waves * (o + kst * k) + mem * items                          waves of tiles over the clusters' places
// Fitted to 1500 problems of 40 to 5500 items (Strassen, Winograd, Phi-optimal, one to three levels, leaves of up to 2560 in K): 3 to 8 %
// off.  With the margin of 3 % the kernel is chosen for half of them, takes 0.80 times the time of the fastest other kernel there in
// the mean (all problems: 0.88 block 32, 0.85 UE8M0, 0.91 block 128, 0.87 weight tiles; the best choice would gain 0.5 % more)
// and at most 1.02 times.  (In another sample, timed in a graph, at most 1.05 times, of 1012 problems that take it; beyond the fit, at 6272 to 25088 items, it is
// chosen for 45 of 68 problems, in 0.77 times the other kernels' time in the mean and at most 0.98 times, and would be faster by up to 1.17 times
// for nine more.)  Phi-optimal, us, block 32 / UE8M0 / block 128 / weight tiles: 2048 x 512 x 2048 29.7 -> 17.1, 18.8 -> 11.5,
// 24.3 -> 14.7, 24.4 -> 12.7; three levels n = 2048 78.5 -> 55.6, 59.5 -> 41.2, 64.0 -> 46.6, 59.9 -> 41.1; not chosen: one level n = 4096
// (16 stages) 216 against 274, 70 against 110, 110 against 168, 97 against 126.
struct KeepTime { float base, o, k, mem; };
struct WalkTime { int ncta, bn; float base, o, k, out, mem; };
struct KeepModel { KeepTime keep, cluster, two_terms; WalkTime walk[3]; };
constexpr KeepModel KEEP_B32 = {{6.0f, 3.06f, 0.562f, 0.0315f}, {7.48f, 5.56f, 2.168f, 0.0322f}, {},
    {{1, 128, 6.01f, 5.3f, 0.758f, 0.863f, 0.00326f}, {2, 128, 6.82f, 5.23f, 0.848f, 0.909f, 0.00327f}, {}}};
constexpr KeepModel KEEP_MX = {{4.72f, 2.94f, 0.1965f, 0.0341f}, {4.91f, 5.86f, 0.432f, 0.0359f}, {1.11f, 12.93f, 0.88f, 0.0431f},
    {{1, 128, 5.06f, 10.15f, 0.208f, 0.3445f, 0.00377f}, {1, 256, 7.4f, 16.1f, 0.341f, 0.628f, 0.00403f}, {2, 256, 5.96f, 17.8f, 0.2586f, 0.968f, 0.00352f}}};
constexpr KeepModel KEEP_B128 = {{5.71f, 2.94f, 0.3177f, 0.0311f}, {5.9f, 6.16f, 0.677f, 0.034f}, {},
    {{1, 128, 5.73f, 2.43f, 0.309f, 0.992f, 0.00355f}, {2, 256, 7.17f, 3.2f, 0.59f, 2.088f, 0.00354f}, {}}};
constexpr KeepModel KEEP_TILE = {{5.68f, 2.655f, 0.2362f, 0.0316f}, {6.01f, 6.06f, 0.592f, 0.0335f}, {},
    {{1, 128, 5.1f, 1.92f, 0.272f, 0.985f, 0.00355f}, {2, 256, 7.0f, 0.66f, 0.449f, 2.153f, 0.00372f}, {}}};

}  // namespace

bool fmm_keep_faster(const GemmParams& g, int blk, int mode, const SplitChoice& split, const GemmShape& tile)
{
    const KeepModel& m = mode == FMM_SCALE_UE8M0_CEIL ? KEEP_MX : blk == 32 ? KEEP_B32 : g.sb_tile ? KEEP_TILE : KEEP_B128;
    const long long tiles = (long long)(g.m / BM) * (g.n / 128) * (g.terms / g.R), items = 2 * tiles;
    // below the fitted range the clusters, which put a tile's terms on as many SMs, are faster (0.5 to 0.95 times their time)
    if (items < 40 || items > 0x3FFFFFFF) return false;
    const float kst = (float)(g.k / BK), stacked = g.terms > g.R ? (float)items : 0.0f;
    const float time = m.keep.base + (float)((items + g.sms - 1) / g.sms) * (m.keep.o + g.R * kst * m.keep.k) + m.keep.mem * stacked;
    if (split.ksplit > 0) {
        // Clusters of two terms a CTA keep their terms of 8 and more stages: that choice is fixed (tests/test_gpu_cluster_two_terms.py),
        // though this kernel is faster there too (product kernel, n = 2048 23.2 -> 18.7 us, 1280 x 3328 x 2816 26.9 -> 24.9).
        if (split.bn != 128 || split.places <= 0 || (split.terms == 2 && kst >= 8.0f)) return false;
        const KeepTime& c = split.terms == 2 ? m.two_terms : m.cluster;
        return time < 0.97f * (c.base + std::max(1.0f, (float)tiles / split.places) * (c.o + kst * c.k) + c.mem * stacked);
    }
    for (const WalkTime& w : m.walk)
        if (w.ncta == tile.ncta && w.bn == tile.bn)
            return time < 0.97f * (w.base + (float)tile.longest / g.R * (w.o + g.R * kst * w.k + g.updates * w.out) + w.mem * stacked * g.updates);
    return false;
}

fmm_status_t fmm_launch_keep(const GemmParams& g, int blk, int mode, cudaStream_t st)
{
    if (mode == FMM_SCALE_UE8M0_CEIL) return launch_keep<FMM_SCALE_UE8M0_CEIL, 32>(g, st);
    if (blk == 32) return launch_keep<MODE_FP32_COLUMN, 32>(g, st);
    return g.sb_tile ? launch_keep<MODE_FP32_SB_TILE, 128>(g, st) : launch_keep<MODE_FP32_COLUMN, 128>(g, st);
}
