// Pre-addition + block quantization kernels (paper Sec. 2.2 / App. D.1: the encoded combinations
// S_r = sum_j U[r][j] A_j and T_r = sum_j V[r][j] B_j are formed in fp32 from the unquantized
// operand blocks and only then quantized; App. E.2: per block of `blk` elements along the
// contracted axis, scale = amax / 448 in fp32, round-to-nearest-even cast to e4m3).
//
// Arithmetic is pinned so that the bytes are reproducible: quadrant order 11,12,21,22, zero
// coefficients skipped, first term a rounded multiply, later terms single-rounded FMAs; the
// block is scaled by inv = 448 / max(amax, floor) (one IEEE division per block) and the stored
// scale is max(amax, floor) / 448.  In the power-of-two mode the scale is 2^ceil(log2(.)).
//
// Both kernels are HBM-bound streaming kernels: every input element is read once with
// full-line coalesced loads and every output byte is written once in whole 32-byte sectors.
#include <cuda_bf16.h>
#include <string.h>
#include "fmm_internal.h"
#include "fmm_ptx.cuh"

namespace {
using fmmptx::pack2; using fmmptx::unpack2; using fmmptx::mul2; using fmmptx::fma2;

__device__ __forceinline__ uint16_t cvt_e4m3x2(float hi, float lo)
{
    uint16_t r;
    asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(r) : "f"(hi), "f"(lo));
    return r;
}

__device__ __forceinline__ uint32_t pack4_e4m3(float a, float b, float c, float d)
{
    return (uint32_t)cvt_e4m3x2(b, a) | ((uint32_t)cvt_e4m3x2(d, c) << 16);
}

// four codes of v * inv (the multiplications two per instruction)
__device__ __forceinline__ uint32_t scaled_pack4(const float4& v, float inv)
{
    const unsigned long long i2 = pack2(inv, inv);
    float a, b, c, d;
    unpack2(mul2(pack2(v.x, v.y), i2), a, b); unpack2(mul2(pack2(v.z, v.w), i2), c, d);
    return pack4_e4m3(a, b, c, d);
}

// Scale of one block from its amax.  Returns the multiplier applied before the cast and writes
// the stored scale (fp32 mode) or the biased power-of-two exponent (UE8M0 mode).
template <int MODE>
__device__ __forceinline__ float block_scale(float amax, float floor_, float& s_out, uint32_t& e8_out)
{
    const float amax_c = fmaxf(amax, floor_);
    if (MODE == FMM_SCALE_FP32_AMAX_DIV_448) {
        s_out = __fdiv_rn(amax_c, 448.0f);
        e8_out = 0;
        return __fdiv_rn(448.0f, amax_c);
    } else {
        const float s0 = __fdiv_rn(amax_c, 448.0f);
        const uint32_t u = __float_as_uint(s0);
        const int ex = (int)(u >> 23);
        const uint32_t man = u & 0x7fffffu;
        int e;
        if (ex == 0) {
            const int hi = 31 - __clz((int)man);
            e = hi - 149 + ((man & (man - 1u)) ? 1 : 0);
        } else {
            e = ex - 127 + (man ? 1 : 0);
        }
        e = max(-127, min(127, e));
        e8_out = (uint32_t)(e + 127);
        s_out = 0.0f;
        // 2^-e, exact; -e == -127 is the subnormal 2^-127
        const int ne = -e;
        return ne >= -126 ? __uint_as_float((uint32_t)(ne + 127) << 23) : __uint_as_float(0x00400000u);
    }
}

// ---------------------------------------------------------------------------------------------
// A side.  One warp handles 128 consecutive k of one output row: 32 lanes x float4, a 512-byte
// coalesced read per quadrant.  A block of BLK elements is held by BLK/4 adjacent lanes.  All R
// combinations are formed first (two elements per fp32x2 instruction); their R block maxima are
// reduced with a transposing butterfly that leaves combination (lane & 7) in each lane, so the
// two IEEE divisions of a block are executed once per block instead of once per lane and
// combination; the multiplier is then broadcast back with one shuffle per combination.
//
// NZ is the zero pattern of the coefficients (bit 4r+j set when coef[r][j] != 0) when it is known at
// compile time - the named realizations are pre-instantiated so that the zero tests, the "first term"
// distinction and the rank guard cost nothing - or 0 for the generic run-time tests.
template <uint32_t NZ> __device__ __forceinline__ bool coef_used(int r, int j, float c)
{ return NZ ? ((NZ >> (4 * r + j)) & 1u) != 0 : (c != 0.0f); }
template <uint32_t NZ> __device__ __forceinline__ bool row_used(int r, int R)
{ return NZ ? ((NZ >> (4 * r)) & 15u) != 0 : (r < R); }

// The arithmetic of one chunk, shared by the one-level and two-level kernels.  x[j] holds four consecutive
// elements (along the contracted axis) of input block j; the GROUP lanes that share a quantization block are
// adjacent.  Forms the R combinations v[r], reduces their block maxima with a transposing butterfly over the
// 8 lanes (lane & 7) - afterwards each lane holds the maximum of combination (lane & 7) - and computes that
// combination's multiplier `inv` and stored scale (s or e8) once per block instead of once per lane.
//
// PACKED: two elements per fp32x2 instruction, the same IEEE operations in half the issue slots (two-level kernels, whose
// 49 combinations bind them to the issue rate: 217 -> 202 us for both sides at n = 8192; no gain in the one-level kernels,
// which wait for memory, and 1 % slower at block 128, where the pairs cost registers).
template <int GROUP, int MODE, uint32_t NZ, bool PACKED = true>
__device__ __forceinline__ void combine_chunk(const EncodeParams& p, const float4 (&x)[4], int lane,
                                              float4 (&v)[FMM_MAX_RANK], float& inv, float& s, uint32_t& e8)
{
    constexpr unsigned FULL = 0xffffffffu;
    const bool b2 = lane & 4, b1 = lane & 2, b0 = lane & 1;
    float am[FMM_MAX_RANK];
#pragma unroll
    for (int r = 0; r < FMM_MAX_RANK; ++r) {
        v[r] = make_float4(0.f, 0.f, 0.f, 0.f); am[r] = 0.0f;
        if (row_used<NZ>(r, p.R)) {
            bool set = false;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float cj = p.coef[r][j];
                if (coef_used<NZ>(r, j, cj)) {
                    const unsigned long long c2 = pack2(cj, cj);
                    if (PACKED && !set) {
                        unpack2(mul2(c2, pack2(x[j].x, x[j].y)), v[r].x, v[r].y); unpack2(mul2(c2, pack2(x[j].z, x[j].w)), v[r].z, v[r].w);
                    } else if (PACKED) {
                        unpack2(fma2(c2, pack2(x[j].x, x[j].y), pack2(v[r].x, v[r].y)), v[r].x, v[r].y);
                        unpack2(fma2(c2, pack2(x[j].z, x[j].w), pack2(v[r].z, v[r].w)), v[r].z, v[r].w);
                    } else if (!set) {
                        v[r].x = __fmul_rn(cj, x[j].x); v[r].y = __fmul_rn(cj, x[j].y);
                        v[r].z = __fmul_rn(cj, x[j].z); v[r].w = __fmul_rn(cj, x[j].w);
                    } else {
                        v[r].x = __fmaf_rn(cj, x[j].x, v[r].x); v[r].y = __fmaf_rn(cj, x[j].y, v[r].y);
                        v[r].z = __fmaf_rn(cj, x[j].z, v[r].z); v[r].w = __fmaf_rn(cj, x[j].w, v[r].w);
                    }
                    set = true;
                }
            }
            am[r] = fmaxf(fmaxf(fabsf(v[r].x), fabsf(v[r].y)), fmaxf(fabsf(v[r].z), fabsf(v[r].w)));
        }
    }
    float w[4], x2[2], mine;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float send = b2 ? am[j] : am[j + 4], keep = b2 ? am[j + 4] : am[j];
        w[j] = fmaxf(keep, __shfl_xor_sync(FULL, send, 4));
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const float send = b1 ? w[j] : w[j + 2], keep = b1 ? w[j + 2] : w[j];
        x2[j] = fmaxf(keep, __shfl_xor_sync(FULL, send, 2));
    }
    {
        const float send = b0 ? x2[0] : x2[1], keep = b0 ? x2[1] : x2[0];
        mine = fmaxf(keep, __shfl_xor_sync(FULL, send, 1));
    }
    if (GROUP == 32) {
        mine = fmaxf(mine, __shfl_xor_sync(FULL, mine, 8));
        mine = fmaxf(mine, __shfl_xor_sync(FULL, mine, 16));
    }
    inv = block_scale<MODE>(mine, p.amax_floor, s, e8);
}

// One combination of the outer level, in registers: the same rounded-multiply / FMA chain as above.
template <uint32_t NZ>
__device__ __forceinline__ float4 combine_outer(const EncodeParams& p, int r, const float4 (&raw)[4][4], int q2)
{
    float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
    bool set = false;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float cj = p.coef[r][j];
        if (coef_used<NZ>(r, j, cj)) {
            const float4 a = raw[j][q2];
            const unsigned long long c2 = pack2(cj, cj);
            if (!set) {
                unpack2(mul2(c2, pack2(a.x, a.y)), o.x, o.y); unpack2(mul2(c2, pack2(a.z, a.w)), o.z, o.w);
                set = true;
            } else {
                unpack2(fma2(c2, pack2(a.x, a.y), pack2(o.x, o.y)), o.x, o.y);
                unpack2(fma2(c2, pack2(a.z, a.w), pack2(o.z, o.w)), o.z, o.w);
            }
        }
    }
    return o;
}

// A-side stores of one chunk: four code bytes per lane and combination; the scale of combination (lane & 7).
// b = index of the input matrix (terms b*R .. b*R + R-1), i = leaf row, c = 128-k chunk.
template <int BLK, int MODE, uint32_t NZ>
__device__ __forceinline__ void store_chunk_a(const EncodeParams& p, const float4 (&v)[FMM_MAX_RANK], float inv, float s,
                                              uint32_t e8, int b, int i, int c, int lane)
{
    constexpr int GROUP = BLK / 4;
    constexpr unsigned FULL = 0xffffffffu;
    const int64_t term_codes = p.q_term;
    const int my_r = lane & 7;
    uint8_t* row = p.q_out + ((int64_t)b * p.R) * term_codes + (int64_t)i * p.cols + c * 128;      // warp-uniform
#pragma unroll
    for (int r = 0; r < FMM_MAX_RANK; ++r) {
        if (row_used<NZ>(r, p.R)) {
            const float inv_r = __shfl_sync(FULL, inv, (GROUP == 32) ? r : ((lane & 24) | r));
            uint8_t* qp = row + (uint32_t)(lane * 4);
            if (FMM_GUARD(p.guard, qp, 4, 1101))
            *reinterpret_cast<uint32_t*>(qp) = BLK == 32 ? scaled_pack4(v[r], inv_r) : pack4_e4m3(__fmul_rn(v[r].x, inv_r), __fmul_rn(v[r].y, inv_r),
                                                                                        __fmul_rn(v[r].z, inv_r), __fmul_rn(v[r].w, inv_r));
        }
        row += term_codes;
    }
    // scales: lane holds the scale of combination my_r, block (lane / GROUP) of this chunk
    if (MODE == FMM_SCALE_FP32_AMAX_DIV_448) {
        if (my_r < p.R && (GROUP == 8 || lane < 8)) {
            // chunk-major: [128-k chunk c][row i][K block of the chunk], so the scales one pipeline stage of the
            // product kernel needs for 128 rows are contiguous, and this warp's (up to four) scales are adjacent;
            // combination my_r is shifted by my_r * s_step rows when several combinations share one array
            // (row panels of a plain pass)
            float* so = reinterpret_cast<float*>(reinterpret_cast<char*>(p.s_out) + ((int64_t)b * p.R + my_r) * p.s_term_stride);
            float* sp = so + ((int64_t)c * p.s_ld + i + my_r * p.s_step) * (128 / BLK) + (GROUP == 8 ? (lane >> 3) : 0);
            if (FMM_GUARD(p.guard, sp, 4, 1102)) *sp = s;
        }
    } else {
        // four exponent bytes of this row (blocks 4c .. 4c+3) form one aligned word of the scale tile
        uint32_t wv = e8 << (8 * (lane >> 3));
        wv |= __shfl_xor_sync(FULL, wv, 8);
        wv |= __shfl_xor_sync(FULL, wv, 16);
        if (lane < 8 && lane < p.R) {
            char* so = reinterpret_cast<char*>(p.s_out) + ((int64_t)b * p.R + lane) * p.s_term_stride;
            const int ig = i + lane * p.s_step;            // row inside the scale-tile array
            const int64_t tile = (int64_t)c * p.sf_blocks + (ig >> 7);
            char* sp = so + tile * 512 + (ig & 31) * 16 + ((ig & 127) >> 5) * 4;
            if (FMM_GUARD(p.guard, sp, 4, 1103)) *reinterpret_cast<uint32_t*>(sp) = wv;
        }
    }
}

// Rows that a task of the A-side encoder walks together (its rows are multiples of 32: of 128, or 128 / 4 in row panels).
template <int BLK, int MODE> struct RowsPerTask { static constexpr int value = MODE == FMM_SCALE_FP32_AMAX_DIV_448 && BLK == 32 ? 2 : 1; };

template <int BLK, int MODE, uint32_t NZ>
__device__ __forceinline__ void encode_a_tasks(const EncodeParams& p, uint32_t warp_gid, uint32_t nwarps)
{
    constexpr int GROUP = BLK / 4;                 // lanes per block
    const int lane = threadIdx.x & 31;
    const int chunks = p.cols / 128;
    // a task is CPT consecutive 128-k chunks of one output row (two adjacent rows at block 32 with fp32 scales).  Tasks
    // are dealt to warps round-robin (32-bit index arithmetic only: one division per task, none per chunk; the warp index
    // is warp-uniform, and so are all addresses but the lane's offset).  The fp32
    // scales of a chunk are stored row after row (16 bytes per row at block 32, 4 at block 128), so partial sectors
    // are avoided this way: block 32 walks two rows per task, the two rows of a chunk back to back (one 32-byte sector
    // per pair of stores); block 128 makes the ROW the fastest task index, so that the eight warps of a block hold
    // eight consecutive rows of the same chunks.  Both choices are the measured better one for their block size
    // (n = 8192, both sides: 0.160 vs 0.165 ms, and 0.158 vs 0.162 ms).  The power-of-two mode writes its exponent
    // bytes in row-major tiles: one row per task, chunk group fastest.
    const int CPT = p.cpt;
    constexpr int RPT = RowsPerTask<BLK, MODE>::value;
    constexpr bool ROW_FASTEST = (MODE == FMM_SCALE_FP32_AMAX_DIV_448) && BLK == 128;
    const uint32_t tasks_per_row = (uint32_t)((chunks + CPT - 1) / CPT);
    const uint32_t row_groups = (uint32_t)(p.rows / RPT);
    const uint32_t rows_all = (uint32_t)p.batch * row_groups;
    const uint32_t tasks = rows_all * tasks_per_row;

    for (uint32_t task = warp_gid; task < tasks; task += nwarps) {
        const uint32_t cgrp = ROW_FASTEST ? task / rows_all : 0u;
        const uint32_t row_id = ROW_FASTEST ? task - cgrp * rows_all : task / tasks_per_row;
        const int c0 = (int)(ROW_FASTEST ? cgrp : task - row_id * tasks_per_row) * CPT;
        const int b = (int)(row_id / row_groups);
        const int i0 = (int)(row_id - (uint32_t)b * row_groups) * RPT;
        const int steps = min(CPT, chunks - c0) * RPT;     // step = (chunk, row)
        const float* row_base = p.in + (int64_t)b * p.in_batch_stride + (int64_t)i0 * p.ld + c0 * 128;
        auto load = [&](int st, float4 (&x)[4]) {
            const float* at = row_base + (int64_t)(st % RPT) * p.ld + (st / RPT) * 128;
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (NZ || j < p.nq) x[j] = __ldcs(reinterpret_cast<const float4*>(at + p.qoff[j]) + lane);
        };
        auto process = [&](int st, const float4 (&x)[4]) {
            float4 v[FMM_MAX_RANK];
            float inv, s; uint32_t e8;
            combine_chunk<GROUP, MODE, NZ, BLK == 32>(p, x, lane, v, inv, s, e8);
            store_chunk_a<BLK, MODE, NZ>(p, v, inv, s, e8, b, i0 + st % RPT, c0 + st / RPT, lane);
        };
        // the loads of step n+1 are issued before step n is processed (two steps in flight per warp)
        float4 xa[4], xb[4];
        load(0, xa);
        for (int st = 0; st < steps; st += 2) {
            if (st + 1 < steps) load(st + 1, xb);
            process(st, xa);
            if (st + 1 < steps) {
                if (st + 2 < steps) load(st + 2, xa);
                process(st + 1, xb);
            }
        }
    }
}

// Blocks per SM.  Block 128 with a known zero pattern: four, although 64 registers spill up to 48 bytes (both sides, n = 4096:
// Winograd 39.1 us against 40.9 with three blocks, n = 8192 146.2 against 147.6).  Without one the spills are nine times that
// and three blocks are faster (4096: 71.0 -> 67.5, 8192: 254 -> 234).  Block 32: three, and the 4 bytes that the power-of-two
// kernel without a zero pattern spills then cost less than two blocks would (n = 4096: 51.5 against 56.6).
template <int BLK, int MODE, uint32_t NZ>
__global__ void __launch_bounds__(256, BLK == 128 && NZ != 0 ? 4 : 3) encode_a_kernel(const EncodeParams p)
{
    // The combinations of this call, when this launch overlaps their tail.  Always ahead of the signal: the B-side encoder that it
    // releases reads nothing written here and does not wait at its start, so what this kernel is behind has to be complete by then.
    fmmptx::griddep_wait();
    fmmptx::griddep_launch_dependents();
    encode_a_tasks<BLK, MODE, NZ>(p, blockIdx.x * 8 + fmmptx::warp_uniform(threadIdx.x >> 5), gridDim.x * 8);
}

// ---------------------------------------------------------------------------------------------
// B side.  Blocks run along k, the strided axis of row-major B, and the output is K-major (the
// tensor-core operand layout).  A thread owns 16 consecutive k of one column n; lanes l and l+16
// hold the two halves of a 32-element (sub-)block, so one shuffle completes the amax.  Each load
// is two 64-byte row segments per warp; each thread writes 16 contiguous code bytes and the two
// lanes of a block fill one 32-byte sector.

// The same place of the block p.cpt blocks further on in the grid, into L2: ROWS rows of 16 columns, one row of every input
// block per thread.
template <int ROWS>
__device__ __forceinline__ void prefetch_block(const EncodeParams& p, int block_row)
{
    if (p.cpt == 0) return;
    const uint32_t next = (uint32_t)block_row * gridDim.x + blockIdx.x + (uint32_t)p.cpt;
    const uint32_t y = next / gridDim.x, x = next - y * gridDim.x;
    if (y >= (uint32_t)p.rows / ROWS) return;
    const float* at = p.in + (int64_t)blockIdx.z * p.in_batch_stride + (int64_t)(y * ROWS + threadIdx.x) * p.ld + x * 16;
#pragma unroll
    for (int jq = 0; jq < 4; ++jq)
        if (jq < p.nq) asm volatile("prefetch.global.L2 [%0];" ::"l"(at + p.qoff[jq]));
}

// B side, block 32, one 32-k block of 16 columns per warp (thread = 16 k of one column, lanes l and l+16 the two
// halves of a block), so every thread issues all its loads at once.  A thread block is a single warp: the warps
// share nothing, and one-warp blocks let the scheduler replace each finished warp on its own (2 % faster than four
// warps of one 128-k chunk per block; blocks of two to eight warps side by side, covering 128- to 512-byte row
// segments, are within 1 %).  Grid: (cols / 16, rows / 32, batch), 32 threads.
// `only` >= 0: nothing but that combination (a grid with one block for each, see encode_both_kernel).
template <int MODE, uint32_t NZ>
__device__ __forceinline__ void encode_b32_block(const EncodeParams& p, int b, int only = -1)
{
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x;
    const int col = lane & 15, khalf = lane >> 4;
    const int j = blockIdx.x * 16 + col;
    const int kb = blockIdx.y;                      // this warp's quantization block
    const int kc = kb >> 2;                         // its chunk of 128 k
    const int k0 = kb * 32 + khalf * 16;
    const float* base = p.in + (int64_t)b * p.in_batch_stride + j;
    const int64_t term_codes = p.q_term;

    float raw[4][16];
#pragma unroll
    for (int jq = 0; jq < 4; ++jq)
        if (jq < p.nq && (only < 0 || p.coef[only][jq] != 0.0f)) {
#pragma unroll
            for (int kk = 0; kk < 16; ++kk)
                raw[jq][kk] = __ldg(base + p.qoff[jq] + (int64_t)(k0 + kk) * p.ld);
        }
    prefetch_block<32>(p, kb);
#pragma unroll
    for (int r = 0; r < FMM_MAX_RANK; ++r) {
        if (row_used<NZ>(r, p.R) && (only < 0 || r == only)) {
            float v[16];
            bool set = false;
#pragma unroll
            for (int jq = 0; jq < 4; ++jq) {
                const float cj = p.coef[r][jq];
                if (coef_used<NZ>(r, jq, cj)) {
                    if (!set) {
#pragma unroll
                        for (int kk = 0; kk < 16; kk += 2) unpack2(mul2(pack2(cj, cj), pack2(raw[jq][kk], raw[jq][kk + 1])), v[kk], v[kk + 1]);
                        set = true;
                    } else {
#pragma unroll
                        for (int kk = 0; kk < 16; kk += 2) unpack2(fma2(pack2(cj, cj), pack2(raw[jq][kk], raw[jq][kk + 1]), pack2(v[kk], v[kk + 1])), v[kk], v[kk + 1]);
                    }
                }
            }
            if (!set) {
#pragma unroll
                for (int kk = 0; kk < 16; ++kk) v[kk] = 0.0f;
            }
            float amax = 0.0f;
#pragma unroll
            for (int kk = 0; kk < 16; ++kk) amax = fmaxf(amax, fabsf(v[kk]));
            amax = fmaxf(amax, __shfl_xor_sync(FULL, amax, 16));
            float sc; uint32_t e8;
            const float inv = block_scale<MODE>(amax, p.amax_floor, sc, e8);
            const int64_t t = (int64_t)b * p.R + r;
            if (MODE == FMM_SCALE_FP32_AMAX_DIV_448 || khalf == 0) {
                char* so = reinterpret_cast<char*>(p.s_out) + t * p.s_term_stride;
                const int jg = j + r * p.s_step;                   // column inside the scale array
                if (MODE == FMM_SCALE_FP32_AMAX_DIV_448) {
                    // the other half of the block's lanes writes the copy for the product kernels
                    float* sp = reinterpret_cast<float*>(so + khalf * p.s_down) + (int64_t)kb * p.s_ld + jg;
                    if (FMM_GUARD(p.guard, sp, 4, 1205)) *sp = khalf ? sc * p.down : sc;
                } else {
                    const int64_t tile = (int64_t)kc * p.sf_blocks + (jg >> 7);
                    char* sp = so + tile * 512 + (jg & 31) * 16 + ((jg & 127) >> 5) * 4 + (kb & 3);
                    if (FMM_GUARD(p.guard, sp, 1, 1206)) *reinterpret_cast<uint8_t*>(sp) = (uint8_t)e8;
                }
            }
            uint32_t wv[4];
#pragma unroll
            for (int g = 0; g < 4; ++g)
                wv[g] = scaled_pack4(make_float4(v[4 * g], v[4 * g + 1], v[4 * g + 2], v[4 * g + 3]), inv);
            uint8_t* qp = p.q_out + t * term_codes + (int64_t)j * p.rows + k0;
            if (FMM_GUARD(p.guard, qp, 16, 1207)) *reinterpret_cast<uint4*>(qp) = make_uint4(wv[0], wv[1], wv[2], wv[3]);
        }
    }
}

// End of a B-side encoder.
__device__ __forceinline__ void end_of_b_side()
{
    // the product kernel, launched behind this one by the same call, may be scheduled as soon as every block has got
    // here: its launch latency and set-up then fall under this grid's last blocks (signalling at the start instead lets
    // its CTAs take SMs from this grid's tail: 0.5 % slower back to back)
    fmmptx::griddep_launch_dependents();
    // a launch that overlapped the A-side encoder must not end before it (what follows on the stream needs both):
    // the last block of the grid waits for it, the others leave as they finish
    if (blockIdx.x + 1 == gridDim.x && blockIdx.y + 1 == gridDim.y && blockIdx.z + 1 == gridDim.z) fmmptx::griddep_wait();
}

template <int MODE, uint32_t NZ>
__global__ void __launch_bounds__(32, 16) encode_b32_kernel(const EncodeParams p)
{
    encode_b32_block<MODE, NZ>(p, blockIdx.z);
    end_of_b_side();
}

// B side, block 128, one pass.  The four warps of a block take the four 32-k sub-blocks of one
// 128-k block of the same 16 columns; every thread forms the combinations of its 16 k x 1 column, the sub-block
// maxima meet in shared memory, and each warp then quantizes its own sub-block from the raw values it still holds
// (the combinations are formed a second time in registers - the same rounded-multiply / FMA chain, so the same bits -
// instead of reading the operand a second time).  Grid: (cols / 16, rows / 128, batch), 128 threads.
//
// TILE (App. E.5, the deployment-matched weight grouping): one scale per tile of 128 k x 128 columns of each encoded
// combination.  The eight blocks of a tile are a cluster and read each other's maxima from distributed shared memory, so
// this takes one pass as well (two passes over the operand by one block per tile took 39 instead of 23 us for a 4096 x 4096
// operand); every column stores the tile's scale, so the scale array keeps its per-column shape.  PRE rounds each encoded
// combination to bfloat16 (nearest even) before the maximum and the cast, as the paper's real kernel does.
template <uint32_t NZ, bool TILE, bool PRE>
__device__ __forceinline__ void encode_b128_block(const EncodeParams& p, int b, int only = -1)
{
    constexpr unsigned FULL = 0xffffffffu;
    constexpr int MODE = FMM_SCALE_FP32_AMAX_DIV_448;
    __shared__ float sub_amax[4][FMM_MAX_RANK][16];      // TILE: [warp][r][0]
    __shared__ float blk_amax[FMM_MAX_RANK], tile_amax[FMM_MAX_RANK];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int col = lane & 15, khalf = lane >> 4;
    const int j = blockIdx.x * 16 + col;
    const int kc = blockIdx.y;                      // chunk of 128 k = one quantization block
    const int k0 = kc * 128 + warp * 32 + khalf * 16;
    const float* base = p.in + (int64_t)b * p.in_batch_stride + j;
    const int64_t term_codes = p.q_term;

    float raw[4][16];
#pragma unroll
    for (int jq = 0; jq < 4; ++jq)
        if (jq < p.nq && (only < 0 || p.coef[only][jq] != 0.0f)) {
#pragma unroll
            for (int kk = 0; kk < 16; ++kk)
                raw[jq][kk] = __ldg(base + p.qoff[jq] + (int64_t)(k0 + kk) * p.ld);
        }
    prefetch_block<128>(p, kc);
    auto combine = [&](int r, float (&v)[16]) {
        bool set = false;
#pragma unroll
        for (int jq = 0; jq < 4; ++jq) {
            const float cj = p.coef[r][jq];
            if (coef_used<NZ>(r, jq, cj)) {
                if (!set) {
#pragma unroll
                    for (int kk = 0; kk < 16; kk += 2) unpack2(mul2(pack2(cj, cj), pack2(raw[jq][kk], raw[jq][kk + 1])), v[kk], v[kk + 1]);
                    set = true;
                } else {
#pragma unroll
                    for (int kk = 0; kk < 16; kk += 2) unpack2(fma2(pack2(cj, cj), pack2(raw[jq][kk], raw[jq][kk + 1]), pack2(v[kk], v[kk + 1])), v[kk], v[kk + 1]);
                }
            }
        }
        if (!set) {
#pragma unroll
            for (int kk = 0; kk < 16; ++kk) v[kk] = 0.0f;
        }
        if (PRE) {
#pragma unroll
            for (int kk = 0; kk < 16; ++kk) v[kk] = __bfloat162float(__float2bfloat16_rn(v[kk]));
        }
    };
#pragma unroll
    for (int r = 0; r < FMM_MAX_RANK; ++r) {
        if (row_used<NZ>(r, p.R) && (only < 0 || r == only)) {
            float v[16];
            combine(r, v);
            float amax = 0.0f;
#pragma unroll
            for (int kk = 0; kk < 16; ++kk) amax = fmaxf(amax, fabsf(v[kk]));
            // non-negative floats order like their bits: one warp-wide integer maximum
            if (TILE) amax = __uint_as_float(__reduce_max_sync(FULL, __float_as_uint(amax)));
            else amax = fmaxf(amax, __shfl_xor_sync(FULL, amax, 16));
            if (TILE ? lane == 0 : khalf == 0) sub_amax[warp][r][TILE ? 0 : col] = amax;
        }
    }
    __syncthreads();
    if (TILE) {
        if (threadIdx.x < FMM_MAX_RANK) {
            const int r = threadIdx.x;
            blk_amax[r] = fmaxf(fmaxf(sub_amax[0][r][0], sub_amax[1][r][0]), fmaxf(sub_amax[2][r][0], sub_amax[3][r][0]));
        }
        fmmptx::cluster_sync();
        if (threadIdx.x < 8 * FMM_MAX_RANK) {       // thread: combination t / 8, block t % 8 of the cluster
            const int r = threadIdx.x >> 3;
            float a;
            asm volatile("{\n\t.reg .b32 m;\n\tmapa.shared::cluster.u32 m, %1, %2;\n\tld.shared::cluster.f32 %0, [m];\n\t}"
                         : "=f"(a) : "r"(fmmptx::smem_u32(&blk_amax[r])), "r"(threadIdx.x & 7) : "memory");
#pragma unroll
            for (int d = 4; d >= 1; d >>= 1) a = fmaxf(a, __shfl_xor_sync(FULL, a, d));
            if ((threadIdx.x & 7) == 0) tile_amax[r] = a;
        }
        __syncthreads();
        asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");       // this block has read its peers' maxima
    }
#pragma unroll
    for (int r = 0; r < FMM_MAX_RANK; ++r) {
        if (row_used<NZ>(r, p.R) && (only < 0 || r == only)) {
            const float amax = TILE ? tile_amax[r]
                                    : fmaxf(fmaxf(sub_amax[0][r][col], sub_amax[1][r][col]), fmaxf(sub_amax[2][r][col], sub_amax[3][r][col]));
            float sc; uint32_t e8;
            const float inv = block_scale<MODE>(amax, p.amax_floor, sc, e8);
            const int64_t t = (int64_t)b * p.R + r;
            // the upper half of the lanes writes the copy for the product kernels (the weight-tile kernel multiplies the two
            // scales first and needs none)
            if (warp == 0 && (!TILE || khalf == 0)) {
                float* sp = reinterpret_cast<float*>(reinterpret_cast<char*>(p.s_out) + t * p.s_term_stride + khalf * p.s_down) + (int64_t)kc * p.s_ld + j + r * p.s_step;
                if (FMM_GUARD(p.guard, sp, 4, 1201)) *sp = khalf ? sc * p.down : sc;
            }
            float v[16];
            combine(r, v);
            uint32_t wv[4];
#pragma unroll
            for (int g = 0; g < 4; ++g)
                wv[g] = scaled_pack4(make_float4(v[4 * g], v[4 * g + 1], v[4 * g + 2], v[4 * g + 3]), inv);
            uint8_t* qp = p.q_out + t * term_codes + (int64_t)j * p.rows + k0;
            if (FMM_GUARD(p.guard, qp, 16, 1204)) *reinterpret_cast<uint4*>(qp) = make_uint4(wv[0], wv[1], wv[2], wv[3]);
        }
    }
}

template <uint32_t NZ, bool TILE, bool PRE>
__global__ void __launch_bounds__(128, 4) encode_b128_kernel(const EncodeParams p)
{
    encode_b128_block<NZ, TILE, PRE>(p, blockIdx.z);
    end_of_b_side();
    if (TILE) asm volatile("barrier.cluster.wait.aligned;" ::: "memory");           // its own maxima are no longer read either
}

// Both sides of a call in one launch, for calls whose cost is their launches: the blocks of the B-side encoder (with ONE gridDim.z of them
// for each place, one per combination, otherwise one for all), and behind them (gridDim.y - pb.rows / BLK rows of blocks) warps for the A
// side's tasks.  ONE is a template argument: a combination chosen at run time keeps the compiler from interleaving the
// combinations of a block that makes all of them (encode, block 128, T*: 256 x 2048 x 2560 8.27 -> 7.48 us, 2048 x 512 x 3072 5.01 -> 4.57).  The
// panels of a plain pass have no combinations to interleave and take the registers that leave room for five blocks of 128 threads on an SM.
template <int BLK, int MODE, uint32_t NZA, uint32_t NZB, bool TILE, bool PRE, bool ONE>
__global__ void __launch_bounds__(BLK == 32 ? 32 : 128, BLK == 32 ? 16 : NZB == 0x00008421u ? 5 : 4) encode_both_kernel(const __grid_constant__ EncodeParams pa, const __grid_constant__ EncodeParams pb)
{
    const uint32_t b_rows = (uint32_t)pb.rows / BLK;
    const bool b_side = blockIdx.y < b_rows;
    if (b_side) {
        const int only = ONE ? (int)blockIdx.z : -1;
        if constexpr (BLK == 32) encode_b32_block<MODE, NZB>(pb, 0, only);
        else encode_b128_block<NZB, TILE, PRE>(pb, 0, only);
    } else {
        constexpr uint32_t WARPS = BLK / 32;
        encode_a_tasks<BLK, MODE, NZA>(pa, ((blockIdx.z * (gridDim.y - b_rows) + blockIdx.y - b_rows) * gridDim.x + blockIdx.x) * WARPS + fmmptx::warp_uniform(threadIdx.x >> 5),
                                       gridDim.z * (gridDim.y - b_rows) * gridDim.x * WARPS);
    }
    fmmptx::griddep_launch_dependents();           // as end_of_b_side (nothing to wait for: an ordinary launch)
    if (TILE && b_side) asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
}

// ---------------------------------------------------------------------------------------------
// Two recursion levels in one pass (levels >= 2): the combinations of the second-to-last level are formed in
// registers from the 16 sub-blocks and fed to the leaf-level arithmetic above, so the 7 fp32 intermediate
// matrices of that level are neither written nor read back.  The rounding sequence is the one of the
// level-by-level evaluation (Sec. 3: recursion = Kronecker power; each level a rounded multiply / FMA chain
// in fp32), so the bytes are identical.  p.rows x p.cols are the leaf dimensions, the input matrices are
// 4*rows x 4*cols, p.qoff_outer[] / p.qoff[] the block offsets of the two levels; terms are numbered
// (b * R + r1) * R + r2.
template <int BLK, int MODE, uint32_t NZ>
__global__ void __launch_bounds__(256) encode2_a_kernel(const EncodeParams p)
{
    fmmptx::griddep_wait();                        // as encode_a_kernel, ahead of the signal
    fmmptx::griddep_launch_dependents();
    constexpr int GROUP = BLK / 4;
    const int lane = threadIdx.x & 31;
    const uint32_t warp_gid = blockIdx.x * 8 + fmmptx::warp_uniform(threadIdx.x >> 5);
    const uint32_t nwarps = gridDim.x * 8;
    const uint32_t chunks = (uint32_t)(p.cols / 128);
    const uint32_t tasks = (uint32_t)p.batch * (uint32_t)p.rows * chunks;       // one 128-k chunk of one leaf row
    for (uint32_t task = warp_gid; task < tasks; task += nwarps) {
        const uint32_t row_id = task / chunks;
        const int c = (int)(task - row_id * chunks);
        const int b = (int)(row_id / (uint32_t)p.rows);
        const int i = (int)(row_id - (uint32_t)b * (uint32_t)p.rows);
        const float* base = p.in + (int64_t)b * p.in_batch_stride + (int64_t)i * p.ld + c * 128;
        float4 raw[4][4];                                   // [outer block][inner block]
#pragma unroll
        for (int q1 = 0; q1 < 4; ++q1)
#pragma unroll
            for (int q2 = 0; q2 < 4; ++q2)
                raw[q1][q2] = __ldcs(reinterpret_cast<const float4*>(base + p.qoff_outer[q1] + p.qoff[q2]) + lane);
#pragma unroll
        for (int r1 = 0; r1 < FMM_MAX_RANK; ++r1) {
            if (row_used<NZ>(r1, p.R)) {
                float4 x[4];
#pragma unroll
                for (int q2 = 0; q2 < 4; ++q2) x[q2] = combine_outer<NZ>(p, r1, raw, q2);
                float4 v[FMM_MAX_RANK];
                float inv, s; uint32_t e8;
                combine_chunk<GROUP, MODE, NZ>(p, x, lane, v, inv, s, e8);
                store_chunk_a<BLK, MODE, NZ>(p, v, inv, s, e8, b * p.R + r1, i, c, lane);
            }
        }
    }
}

// B side, block 32: a thread owns 4 consecutive k of one column, the 8 lanes (lane & 7) of a column hold one
// 32-element block, a warp covers 4 adjacent columns (16-byte row segments; the neighbouring warp of the block
// uses the other half of each 32-byte sector).  The eight lanes of a column write 32 contiguous code bytes of
// the K-major output.  Grid: (cols / 32, rows / 32, batch), 256 threads.
template <int MODE, uint32_t NZ>
__global__ void __launch_bounds__(256) encode2_b_kernel(const EncodeParams p)
{
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int j = blockIdx.x * 32 + warp * 4 + (lane >> 3);        // leaf column
    const int kb = blockIdx.y;                                      // 32-k block
    const int k0 = kb * 32 + (lane & 7) * 4;
    const int b = blockIdx.z;
    const int64_t term_codes = p.q_term;
    const int my_r = lane & 7;
    // The block's 32 k x 32 columns of each of the 16 sub-blocks go through shared memory: the global loads are
    // whole 128-byte row segments (a thread reading its own 4 k x 1 column directly touches eight lines per warp
    // instruction with 16 bytes each and is bound by L1 wavefronts), the transposed reads are conflict-free with
    // rows padded to 33 words.  Two passes of eight sub-blocks keep the buffer under the static 48 KB.
    __shared__ float tile[8][32][33];
    float4 raw[4][4];
    {
        const int lrow = threadIdx.x >> 3, lc = (threadIdx.x & 7) * 4;
        const float* blk = p.in + (int64_t)b * p.in_batch_stride + ((int64_t)kb * 32 + lrow) * p.ld + blockIdx.x * 32 + lc;
        const int rk = (lane & 7) * 4, rc = warp * 4 + (lane >> 3);
#pragma unroll
        for (int pass = 0; pass < 2; ++pass) {
            if (pass) __syncthreads();
            float4 v[8];
#pragma unroll
            for (int sblk = 0; sblk < 8; ++sblk)
                v[sblk] = __ldg(reinterpret_cast<const float4*>(blk + p.qoff_outer[2 * pass + (sblk >> 2)] + p.qoff[sblk & 3]));
#pragma unroll
            for (int sblk = 0; sblk < 8; ++sblk) {
                tile[sblk][lrow][lc] = v[sblk].x; tile[sblk][lrow][lc + 1] = v[sblk].y;
                tile[sblk][lrow][lc + 2] = v[sblk].z; tile[sblk][lrow][lc + 3] = v[sblk].w;
            }
            __syncthreads();
#pragma unroll
            for (int sblk = 0; sblk < 8; ++sblk)
                raw[2 * pass + (sblk >> 2)][sblk & 3] = make_float4(tile[sblk][rk][rc], tile[sblk][rk + 1][rc],
                                                                    tile[sblk][rk + 2][rc], tile[sblk][rk + 3][rc]);
        }
    }
#pragma unroll
    for (int r1 = 0; r1 < FMM_MAX_RANK; ++r1) {
        if (row_used<NZ>(r1, p.R)) {
            float4 x[4];
#pragma unroll
            for (int q2 = 0; q2 < 4; ++q2) x[q2] = combine_outer<NZ>(p, r1, raw, q2);
            float4 v[FMM_MAX_RANK];
            float inv, s; uint32_t e8;
            combine_chunk<8, MODE, NZ>(p, x, lane, v, inv, s, e8);
            const int64_t t0 = ((int64_t)b * p.R + r1) * p.R;
            // warp-uniform base; a lane's offset fits 32 bits: the operand has 16 times 4 bytes for every code of a term
            uint8_t* term = p.q_out + t0 * term_codes;
            const uint32_t at = (uint32_t)j * (uint32_t)p.rows + (uint32_t)k0;
#pragma unroll
            for (int r = 0; r < FMM_MAX_RANK; ++r) {
                if (row_used<NZ>(r, p.R)) {
                    const float inv_r = __shfl_sync(FULL, inv, (lane & 24) | r);
                    uint8_t* qp = term + at;
                    if (FMM_GUARD(p.guard, qp, 4, 1301))
                    *reinterpret_cast<uint32_t*>(qp) = scaled_pack4(v[r], inv_r);
                }
                term += term_codes;
            }
            if (my_r < p.R) {
                char* so = reinterpret_cast<char*>(p.s_out) + (t0 + my_r) * p.s_term_stride;
                if (MODE == FMM_SCALE_FP32_AMAX_DIV_448) {
                    float* sp = reinterpret_cast<float*>(so) + (int64_t)kb * p.s_ld + j;
                    if (FMM_GUARD(p.guard, sp, 4, 1302)) *sp = s;
                    float* sd = reinterpret_cast<float*>(reinterpret_cast<char*>(sp) + p.s_down);      // the copy for the product kernels
                    if (FMM_GUARD(p.guard, sd, 4, 1304)) *sd = s * p.down;
                } else {
                    const int64_t tile = (int64_t)(kb >> 2) * p.sf_blocks + (j >> 7);
                    char* sp = so + tile * 512 + (j & 31) * 16 + ((j & 127) >> 5) * 4 + (kb & 3);
                    if (FMM_GUARD(p.guard, sp, 1, 1303)) *reinterpret_cast<uint8_t*>(sp) = (uint8_t)e8;
                }
            }
        }
    }
    end_of_b_side();
}

// Streaming kernels of the outer recursion levels.  A block is 8 rows x 32 float4 of a matrix, a thread one float4 of every
// input block; the row and column come from one 32-bit division per thread (64-bit divisions took a third of the time of
// these kernels at the sizes where their data stays in L2).
struct OuterIndex { int row, col4; };
__device__ __forceinline__ OuterIndex outer_index(int cols)
{
    const uint32_t tiles = (uint32_t)cols / 128, by = blockIdx.x / tiles, bx = blockIdx.x - by * tiles;
    return {(int)(by * 8 + threadIdx.y), (int)(bx * 32 + threadIdx.x)};
}
__device__ __forceinline__ void axpy(float4& acc, float w, const float4& x)
{
    acc.x = __fmaf_rn(w, x.x, acc.x); acc.y = __fmaf_rn(w, x.y, acc.y);
    acc.z = __fmaf_rn(w, x.z, acc.z); acc.w = __fmaf_rn(w, x.w, acc.w);
}

// fp32 combinations of the outer recursion levels: out[b*R + r] = sum_j coef[r][j] X_j, first term a rounded multiply, later
// terms FMAs, zero coefficients skipped.  Both sides of a level in one launch (blockIdx.y).
__global__ void __launch_bounds__(256) comb_kernel(const CombParams pa, const CombParams pb)
{
    fmmptx::griddep_wait();                        // the level above, when this launch overlaps its tail
    const CombParams& p = blockIdx.y ? pb : pa;
    if (blockIdx.x * 8u >= (uint32_t)p.rows * ((uint32_t)p.cols / 128) || (int)blockIdx.z >= p.batch) return;
    const OuterIndex at = outer_index(p.cols);
    const int64_t qoff[4] = {0, (int64_t)p.cols, (int64_t)p.rows * p.ld, (int64_t)p.rows * p.ld + p.cols};
    const float* base = p.in + (int64_t)blockIdx.z * p.in_batch_stride + (int64_t)at.row * p.ld + at.col4 * 4;
    float4 x[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) x[j] = __ldcs(reinterpret_cast<const float4*>(base + qoff[j]));
    const int64_t term = (int64_t)p.rows * p.cols;
    float* o = p.out + (int64_t)blockIdx.z * p.R * term + (int64_t)at.row * p.cols + at.col4 * 4;
#pragma unroll
    for (int r = 0; r < FMM_MAX_RANK; ++r) {
        if (r >= p.R) break;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        bool set = false;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float cj = p.coef[r][j];
            if (cj != 0.0f) {
                if (!set) {
                    v.x = __fmul_rn(cj, x[j].x); v.y = __fmul_rn(cj, x[j].y);
                    v.z = __fmul_rn(cj, x[j].z); v.w = __fmul_rn(cj, x[j].w);
                    set = true;
                } else axpy(v, cj, x[j]);
            }
        }
        if (FMM_GUARD(p.guard, o, 16, 1401)) *reinterpret_cast<float4*>(o) = v;
        o += term;
    }
}

// Outward step of the decoder for levels >= 2: the R partially decoded products of a parent are
// combined into the four blocks of the parent's matrix, out_q = sum_r W[r][q] * in_r (fp32, r ascending).
__global__ void __launch_bounds__(256) decode_kernel(const DecodeParams p)
{
    fmmptx::griddep_wait();                        // the product kernel, whose tail this launch overlaps
    const OuterIndex at = outer_index(p.cols);
    const int64_t in_stride = (int64_t)p.rows * p.cols, out_ld = 2 * (int64_t)p.cols;
    const float* src = p.in + (int64_t)blockIdx.z * p.R * in_stride + (int64_t)at.row * p.cols + at.col4 * 4;
    // all R loads are issued before the first use (R x 16 bytes in flight per thread)
    float4 x[FMM_MAX_RANK];
#pragma unroll
    for (int r = 0; r < FMM_MAX_RANK; ++r)
        if (r < p.R) x[r] = __ldcs(reinterpret_cast<const float4*>(src + r * in_stride));
    float* dst = p.out + (int64_t)blockIdx.z * 4 * in_stride;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int r = 0; r < FMM_MAX_RANK; ++r) {
            const float w = p.W[r][q];             // zero for r >= R
            if (w != 0.0f) axpy(acc, w, x[r]);
        }
        float* o = dst + ((int64_t)(q >> 1) * p.rows + at.row) * out_ld + (q & 1) * p.cols + at.col4 * 4;
        if (FMM_GUARD(p.guard, o, 16, 1501)) *reinterpret_cast<float4*>(o) = acc;
    }
}

// Two outward steps at once (three levels): the R x R matrices of the second level go to the 16 blocks of the result with the
// first-level matrices in registers, in the order of two single steps.  The first-level matrices are neither written nor read
// back (n = 2048: 14 + 10 us as two launches).  Bound by memory latency: R loads in flight per thread and four blocks per SM (128 registers)
// keep more of it busy than the next R loads under the arithmetic and three (product kernel and decoder, n = 2048 39.1 -> 35.0 us, 4096 x 1024 x
// 4096 100.7 -> 97.7, 8192 x 1024 x 8192 377 -> 364); 8 bytes per load and up to eight blocks are slower.
__global__ void __launch_bounds__(128, 4) decode2_kernel(const DecodeParams p)
{
    fmmptx::griddep_wait();
    const uint32_t tiles = (uint32_t)p.cols / 128, by = blockIdx.x / tiles, bx = blockIdx.x - by * tiles;
    const int row = by * 4 + threadIdx.y, col = (bx * 32 + threadIdx.x) * 4;
    const int64_t in_stride = (int64_t)p.rows * p.cols, out_ld = 4 * (int64_t)p.cols;
    const float* src = p.in + (int64_t)row * p.cols + col;
    float4 acc[4][4];
#pragma unroll
    for (int i = 0; i < 16; ++i) acc[i >> 2][i & 3] = make_float4(0.f, 0.f, 0.f, 0.f);
    auto load = [&](int r1, float4 (&x)[FMM_MAX_RANK]) {
#pragma unroll
        for (int r = 0; r < FMM_MAX_RANK; ++r)
            if (r < p.R) x[r] = __ldcs(reinterpret_cast<const float4*>(src + (int64_t)(r1 * p.R + r) * in_stride));
    };
    auto add = [&](int r1, const float4 (&x)[FMM_MAX_RANK]) {
#pragma unroll
        for (int q2 = 0; q2 < 4; ++q2) {
            float4 y = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int r = 0; r < FMM_MAX_RANK; ++r) {
                const float w = p.W[r][q2];
                if (w != 0.0f) axpy(y, w, x[r]);
            }
#pragma unroll
            for (int q1 = 0; q1 < 4; ++q1) {
                const float w = p.W[r1][q1];
                if (w != 0.0f) axpy(acc[q1][q2], w, y);
            }
        }
    };
    float4 x[FMM_MAX_RANK];
#pragma unroll 1
    for (int r1 = 0; r1 < p.R; ++r1) {
        load(r1, x);
        add(r1, x);
    }
#pragma unroll
    for (int q1 = 0; q1 < 4; ++q1)
#pragma unroll
        for (int q2 = 0; q2 < 4; ++q2) {
            const int64_t r = (int64_t)(2 * (q1 >> 1) + (q2 >> 1)) * p.rows + row;
            float* o = p.out + r * out_ld + (2 * (q1 & 1) + (q2 & 1)) * (int64_t)p.cols + col;
            if (FMM_GUARD(p.guard, o, 16, 1502)) *reinterpret_cast<float4*>(o) = acc[q1][q2];
        }
}

}  // namespace

namespace {
// Launch that may begin under the tail of the kernel before it on the stream, one of the same call (which wrote what this one
// reads: it waits for it before its first load), so that its launch latency and set-up are hidden.
template <typename K, typename... A>
fmm_status_t launch_behind(K kernel, dim3 grid, dim3 block, cudaStream_t st, bool overlap, const A&... args)
{
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = grid; cfg.blockDim = block; cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at; cfg.numAttrs = overlap ? 1 : 0;
    cudaLaunchKernelEx(&cfg, kernel, args...);
    return cudaGetLastError() == cudaSuccess ? FMM_OK : FMM_ERR_CUDA;
}
}  // namespace

fmm_status_t fmm_launch_decode(const DecodeParams& p, int steps, cudaStream_t st)
{
    const unsigned tiles = (unsigned)(p.cols / 128);
    if (steps == 2) return launch_behind(decode2_kernel, dim3((unsigned)(p.rows / 4) * tiles), dim3(32, 4), st, true, p);
    return launch_behind(decode_kernel, dim3((unsigned)(p.rows / 8) * tiles, 1, (unsigned)p.batch), dim3(32, 8), st, true, p);
}

fmm_status_t fmm_launch_comb(const CombParams& a, const CombParams& b, bool overlap, cudaStream_t st)
{
    const unsigned ga = (unsigned)(a.rows / 8) * (unsigned)(a.cols / 128), gb = (unsigned)(b.rows / 8) * (unsigned)(b.cols / 128);
    return launch_behind(comb_kernel, dim3(ga > gb ? ga : gb, 2, (unsigned)(a.batch > b.batch ? a.batch : b.batch)), dim3(32, 8), st, overlap, a, b);
}

namespace {
uint32_t coef_mask(const EncodeParams& p)
{
    uint32_t m = 0;
    for (int r = 0; r < p.R; ++r)
        for (int j = 0; j < 4; ++j)
            if (p.coef[r][j] != 0.0f) m |= 1u << (4 * r + j);
    return m;
}

// zero patterns with pre-instantiated kernels: U and V of Strassen, the Winograd form and the
// Phi-optimal realization, and (one-level kernels) the identity used to quantize a matrix as four panels
#define FMM_REALIZATION_MASKS(X) X(0x0a5381c9u) X(0x0c385a19u) X(0x05dc8f21u) X(0x0ab3f841u) X(0x0f5fc5c9u) X(0x0cfc5f59u)
#define FMM_KNOWN_MASKS(X) FMM_REALIZATION_MASKS(X) X(0x00008421u)
// U and V of each
#define FMM_KNOWN_MASK_PAIRS(X) X(0x0a5381c9u, 0x0c385a19u) X(0x05dc8f21u, 0x0ab3f841u) X(0x0f5fc5c9u, 0x0cfc5f59u) X(0x00008421u, 0x00008421u)

// Launch of an encoder.  With `overlap` it carries the programmatic-serialization attribute.  B side: the kernel
// before it on the stream (the A-side encoder, which signals at its start) need not have drained when this one
// begins, so its blocks fill the SMs that the other's last wave leaves idle (6 % of the encode phase at n = 8192); what it
// reads, the caller's matrix or combinations of a kernel before the A-side one, is complete (encode_a_kernel).  A side: set up
// under the tail of the combinations of the same call.  The first kernel of a call is launched without: its wait would be
// for the caller's last kernel, which stands for the work before it only if it waited for that itself, and a caller's kernel that
// has the attribute need not (2 us of a call that follows another at every size).
template <typename K, typename... P>
void launch_encoder(K kernel, dim3 grid, unsigned threads, cudaStream_t st, unsigned cluster, bool overlap, const P&... p)
{
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = grid; cfg.blockDim = dim3(threads, 1, 1); cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cluster; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    // without a cluster only the second one, or none
    cfg.attrs = cluster > 1 ? at : at + 1; cfg.numAttrs = (cluster > 1 ? 1 : 0) + (overlap ? 1 : 0);
    cudaLaunchKernelEx(&cfg, kernel, p...);
}

template <int BLK, int MODE>
void launch_a(const EncodeParams& p, unsigned g, cudaStream_t st)
{
    const uint32_t m = (p.nq == 4) ? coef_mask(p) : 0u;
    switch (m) {
#define X(M) case M: launch_encoder(encode_a_kernel<BLK, MODE, M>, dim3(g), 256, st, 1, p.overlap_prev, p); return;
        FMM_KNOWN_MASKS(X)
#undef X
        default: launch_encoder(encode_a_kernel<BLK, MODE, 0u>, dim3(g), 256, st, 1, p.overlap_prev, p); return;
    }
}
template <int MODE>
void launch_b32(const EncodeParams& p, dim3 grid, cudaStream_t st)
{
    const uint32_t m = (p.nq == 4) ? coef_mask(p) : 0u;
    switch (m) {
#define X(M) case M: launch_encoder(encode_b32_kernel<MODE, M>, grid, 32, st, 1, p.overlap_prev, p); return;
        FMM_KNOWN_MASKS(X)
#undef X
        default: launch_encoder(encode_b32_kernel<MODE, 0u>, grid, 32, st, 1, p.overlap_prev, p); return;
    }
}
template <bool TILE, bool PRE>
void launch_b128(const EncodeParams& p, dim3 grid, cudaStream_t st)
{
    const uint32_t m = (p.nq == 4) ? coef_mask(p) : 0u;
    switch (m) {
#define X(M) case M: launch_encoder(encode_b128_kernel<M, TILE, PRE>, grid, 128, st, TILE ? 8 : 1, p.overlap_prev, p); return;
        FMM_KNOWN_MASKS(X)
#undef X
        default: launch_encoder(encode_b128_kernel<0u, TILE, PRE>, grid, 128, st, TILE ? 8 : 1, p.overlap_prev, p); return;
    }
}
template <int BLK, int MODE>
void launch_a2(const EncodeParams& p, unsigned g, cudaStream_t st)
{
    switch (coef_mask(p)) {
#define X(M) case M: launch_encoder(encode2_a_kernel<BLK, MODE, M>, dim3(g), 256, st, 1, p.overlap_prev, p); return;
        FMM_REALIZATION_MASKS(X)
#undef X
        default: launch_encoder(encode2_a_kernel<BLK, MODE, 0u>, dim3(g), 256, st, 1, p.overlap_prev, p); return;
    }
}
template <int MODE>
void launch_b2(const EncodeParams& p, dim3 grid, cudaStream_t st)
{
    switch (coef_mask(p)) {
#define X(M) case M: launch_encoder(encode2_b_kernel<MODE, M>, grid, 256, st, 1, p.overlap_prev, p); return;
        FMM_REALIZATION_MASKS(X)
#undef X
        default: launch_encoder(encode2_b_kernel<MODE, 0u>, grid, 256, st, 1, p.overlap_prev, p); return;
    }
}
template <int BLK, int MODE, bool TILE, bool PRE, bool ONE>
bool launch_both_as(const EncodeParams& a, const EncodeParams& b, unsigned a_warps, cudaStream_t st)
{
    constexpr unsigned THREADS = BLK == 32 ? 32 : 128;
    const unsigned gx = (unsigned)b.cols / 16, a_blocks = (a_warps + THREADS / 32 - 1) / (THREADS / 32);
    const unsigned gz = ONE ? (unsigned)b.R : 1u;
    const dim3 grid(gx, (unsigned)b.rows / BLK + (a_blocks + gx * gz - 1) / (gx * gz), gz);
    const uint32_t ma = coef_mask(a), mb = coef_mask(b);
#define X(U, V) if (ma == U && mb == V) { launch_encoder(encode_both_kernel<BLK, MODE, U, V, TILE, PRE, ONE>, grid, THREADS, st, TILE ? 8 : 1, false, a, b); return true; }
    FMM_KNOWN_MASK_PAIRS(X)
#undef X
    return false;
}
template <int BLK, int MODE, bool TILE, bool PRE>
bool launch_both(const EncodeParams& a, const EncodeParams& b, unsigned a_warps, bool one, cudaStream_t st)
{
    return one ? launch_both_as<BLK, MODE, TILE, PRE, true>(a, b, a_warps, st) : launch_both_as<BLK, MODE, TILE, PRE, false>(a, b, a_warps, st);
}

// Tasks of the A-side encoder, one per warp; sets their length.  Long tasks keep two steps of loads in flight, but a problem has
// to have tasks for about half the resident warps (n = 2048, block 32: one task per eight chunks 15 us for both sides, per two
// 10 us; n = 4096: per eight 36.8, per two 39).
int64_t a_side_tasks(EncodeParams& p, int blk, int mode)
{
    const int chunks = p.cols / 128, rpt = (mode == FMM_SCALE_FP32_AMAX_DIV_448 && blk == 32) ? 2 : 1;
    const int64_t row_tasks = (int64_t)p.batch * (p.rows / rpt);
    const int64_t want = (int64_t)fmm_sm_count() * 10;
    int64_t tpr = (chunks + 7) / 8;
    while (row_tasks * tpr < want && chunks > 2 * tpr) tpr *= 2;
    p.cpt = (int)((chunks + tpr - 1) / tpr);
    return row_tasks * ((chunks + p.cpt - 1) / p.cpt);
}
}  // namespace

fmm_status_t fmm_launch_encode_a(EncodeParams p, int blk, int mode, cudaStream_t st)
{
    // one task per warp; the block scheduler balances the SMs
    int64_t blocks = (a_side_tasks(p, blk, mode) + 7) / 8;
    if (blocks > 0x7fffffff) blocks = 0x7fffffff;
    const unsigned g = (unsigned)blocks;
    if (mode == FMM_SCALE_FP32_AMAX_DIV_448) {
        if (blk == 32) launch_a<32, FMM_SCALE_FP32_AMAX_DIV_448>(p, g, st);
        else launch_a<128, FMM_SCALE_FP32_AMAX_DIV_448>(p, g, st);
    } else {
        launch_a<32, FMM_SCALE_UE8M0_CEIL>(p, g, st);
    }
    return cudaGetLastError() == cudaSuccess ? FMM_OK : FMM_ERR_CUDA;
}

fmm_status_t fmm_launch_encode_b(EncodeParams p, int blk, int mode, cudaStream_t st)
{
    // A block loads everything first and then computes: the operand's next blocks come into L2 meanwhile, half of the resident ones
    // ahead (block 128, n = 8192: a quarter 141.6 us for both sides, half 133.9, three quarters 134.6, all 136.8, none 142.6; weight
    // tiles 177 -> 168, n = 4096 47.3 -> 44.1, block 128 37.4 -> 34.9, block 32 36.0 -> 34.5).  Only for an operand that is not in L2 already:
    // up to 51 MB it is 0 to 4 % slower (n = 3072 19.2, 20.0).  Panels of a plain pass, with less to compute, gain from twice that
    // on (n = 4096 28.5, 28.9; n = 8192 108.9, 108.1, weight tiles 137.1, 127.5).  The A side, whose warps keep loads in flight
    // while they compute, loses 3 % by it.
    const int64_t bytes = (int64_t)p.rows * p.cols * p.nq * 4;
    p.cpt = bytes >= (int64_t)(p.R > 4 ? 56 : 112) << 20 && p.batch == 1 ? fmm_sm_count() * (blk == 32 ? 8 : 2) : 0;

    dim3 grid((unsigned)(p.cols / 16), (unsigned)(p.rows / blk), (unsigned)p.batch);
    if (mode != FMM_SCALE_FP32_AMAX_DIV_448) launch_b32<FMM_SCALE_UE8M0_CEIL>(p, grid, st);
    else if (blk == 32) launch_b32<FMM_SCALE_FP32_AMAX_DIV_448>(p, grid, st);
    else if (p.b_tile && p.preround_bf16) launch_b128<true, true>(p, grid, st);
    else if (p.b_tile) launch_b128<true, false>(p, grid, st);
    else if (p.preround_bf16) launch_b128<false, true>(p, grid, st);
    else launch_b128<false, false>(p, grid, st);
    return cudaGetLastError() == cudaSuccess ? FMM_OK : FMM_ERR_CUDA;
}

// One launch for both sides where the call's cost is its launches (2.6 us of host time, up to 2 us of the device's): up to so
// many warps per SM.  Above that the A side is better off with the registers and blocks of its own kernel.  Calls with a launch a
// side and with one, in us, Phi-optimal, n = 256 / 512 / 1024 / 2048 / 3072: UE8M0 12.3, 10.8 / 12.3, 12.3 / 16.4, 14.4 / 31.2, 31.3 / 60.0,
// 63.5; weight tiles 10.8, 10.3 / 12.3, 10.7 / 16.4, 16.4 / 39.9, 38.6 / 78.0, 80.6; block 128 10.3, 8.2 / 10.6, 10.3 / 16.1, 15.3 /
// 41.0, 39.7 / 71.5, 74.1; block 32 10.3, 10.3 / 12.3, 12.3 / 18.5, 20.1 / 66.9, 67.2 / 111, 114.  The B side's blocks come first: they take
// longer (the other way round nothing is gained).
bool fmm_launch_encode_both(EncodeParams a, const EncodeParams& b, int blk, int mode, cudaStream_t st, fmm_status_t* status)
{
    if (a.nq != 4 || b.nq != 4 || a.batch != 1 || b.batch != 1) return false;
    const int64_t warps = a_side_tasks(a, blk, mode);
    const int64_t b_warps = (int64_t)(b.cols / 16) * (b.rows / 32);
    if (warps + b_warps > (int64_t)fmm_sm_count() * (blk == 128 ? 32 : mode != FMM_SCALE_FP32_AMAX_DIV_448 ? 16 : 4)) return false;
    const unsigned w = (unsigned)warps;
    // One combination per B-side block where that still leaves an SM few warps: a block of all R is a chain of 1250 instructions with a
    // warp or two per scheduler to hide it, but with a block for each the operand is read R / 2 times (by the four panels of a plain pass
    // once) and every warp's start and end are paid for.  What decides is all warps of that launch, the A side's included: the B side's alone misjudge
    // operands with many rows of A.  The bf16 pre-round lengthens the chain.  Of 973 problems (leaves of 64 to 1536, operands in L2 and not) the
    // other form would be faster by more than 2 % for 13.  us a call in a graph, Phi-optimal, all combinations and one per block (warps per SM): block
    // 32 n = 256 7.80, 7.46 (2); 512 x 256 x 512 9.33, 9.26 (3.9); n = 512 10.45, 11.06 (7).  UE8M0 n = 256 9.40, 8.26 (2); n = 512 9.99, 9.75 (7.8);
    // 512 x 1024 x 512 10.68, 11.70 (16); n = 1024 13.53, 16.21 (31).  Block 128 n = 256 7.54, 6.83 (2.4); 512 x 1536 x 256 9.36, 9.20 (14.3); n = 768 11.19,
    // 11.53 (18.8); n = 1024 13.76, 14.79 (31).  Weight tiles n = 256 8.46, 7.50; 512 x 1536 x 256 10.31, 10.13; 512 x 1024 x 512 10.73, 11.20 (15.6); n = 1024
    // 14.27, 16.53.  bf16 pre-round n = 256 8.31, 7.12; 512 x 1024 x 512 10.90, 10.49; n = 1024 14.46, 15.39.
    const bool panels = b.R == 4;
    const float most = blk == 128 ? (b.b_tile ? panels : b.preround_bf16 != 0) ? 18.5f : 15.5f
                     : mode != FMM_SCALE_FP32_AMAX_DIV_448 ? (panels ? 8.0f : 10.0f) : 4.0f;
    const bool one = (float)(warps + b_warps * b.R) < (float)fmm_sm_count() * most;
    bool known;
    if (mode != FMM_SCALE_FP32_AMAX_DIV_448) known = launch_both<32, FMM_SCALE_UE8M0_CEIL, false, false>(a, b, w, one, st);
    else if (blk == 32) known = launch_both<32, FMM_SCALE_FP32_AMAX_DIV_448, false, false>(a, b, w, one, st);
    else if (b.b_tile && b.preround_bf16) known = launch_both<128, FMM_SCALE_FP32_AMAX_DIV_448, true, true>(a, b, w, one, st);
    else if (b.b_tile) known = launch_both<128, FMM_SCALE_FP32_AMAX_DIV_448, true, false>(a, b, w, one, st);
    else if (b.preround_bf16) known = launch_both<128, FMM_SCALE_FP32_AMAX_DIV_448, false, true>(a, b, w, one, st);
    else known = launch_both<128, FMM_SCALE_FP32_AMAX_DIV_448, false, false>(a, b, w, one, st);
    if (known) *status = cudaGetLastError() == cudaSuccess ? FMM_OK : FMM_ERR_CUDA;
    return known;
}

bool fmm_encode2_supported(bool b_side, int blk, int b_tile, int preround_bf16)
{
    // A side: every block size; B side: block 32 (a 128-element block along the strided axis would leave one
    // column per warp), no weight-side options
    return !b_side || (blk == 32 && !b_tile && !preround_bf16);
}

fmm_status_t fmm_launch_encode2_a(const EncodeParams& p, int blk, int mode, cudaStream_t st)
{
    const int64_t tasks = (int64_t)p.batch * p.rows * (p.cols / 128);
    int64_t blocks = (tasks + 7) / 8;
    const int64_t cap = (int64_t)fmm_sm_count() * 64;
    if (blocks > cap) blocks = cap;
    const unsigned g = (unsigned)blocks;
    if (mode == FMM_SCALE_FP32_AMAX_DIV_448) {
        if (blk == 32) launch_a2<32, FMM_SCALE_FP32_AMAX_DIV_448>(p, g, st);
        else launch_a2<128, FMM_SCALE_FP32_AMAX_DIV_448>(p, g, st);
    } else {
        launch_a2<32, FMM_SCALE_UE8M0_CEIL>(p, g, st);
    }
    return cudaGetLastError() == cudaSuccess ? FMM_OK : FMM_ERR_CUDA;
}

fmm_status_t fmm_launch_encode2_b(const EncodeParams& p, int mode, cudaStream_t st)
{
    dim3 grid((unsigned)(p.cols / 32), (unsigned)(p.rows / 32), (unsigned)p.batch);
    if (mode == FMM_SCALE_FP32_AMAX_DIV_448) launch_b2<FMM_SCALE_FP32_AMAX_DIV_448>(p, grid, st);
    else launch_b2<FMM_SCALE_UE8M0_CEIL>(p, grid, st);
    return cudaGetLastError() == cudaSuccess ? FMM_OK : FMM_ERR_CUDA;
}
