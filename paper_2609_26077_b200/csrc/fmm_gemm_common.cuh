// What the product kernels share: tile constants, bounded barrier waits, tensor maps.
#pragma once
#include <string.h>
#include <atomic>
#include "fmm_internal.h"
#include "fmm_ptx.cuh"

namespace {
using namespace fmmptx;

// Internal third mode of the product kernel: FP32 scales whose B-side value is constant over each
// 128-column tile (the 128 x 128 weight tiles of App. E.5).  The promotion then needs one multiply per row
// and K block (s = sA * sB_tile) and one FMA per element, instead of a multiply and an FMA per element.
constexpr int MODE_FP32_SB_TILE = 2;

constexpr int BM = 128;                 // rows per CTA
constexpr int BK = 128;                 // K elements (= bytes) per pipeline stage: one swizzle row

constexpr unsigned long long WAIT_LIMIT_NS = 2000000000ull;   // 2 s: far beyond any legitimate wait

struct Ctl {
    volatile int* abort_flag;   // shared memory
    int* status;                // global status words
    unsigned long long limit_ns = WAIT_LIMIT_NS;
};

// Bounded mbarrier wait.  Returns false after WAIT_LIMIT_NS or when another role has given up.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, const Ctl& ctl, int where)
{
    uint32_t spins = 0;
    uint64_t t0 = 0;
    while (!mbar_try_wait(bar, parity)) {
        if ((++spins & 0x3FFu) == 0) {
            if (*ctl.abort_flag) return false;
            const uint64_t now = global_timer();
            if (t0 == 0) t0 = now;
            else if (now - t0 > ctl.limit_ns) {
                *ctl.abort_flag = 1;
                atomicCAS(ctl.status, 0, where);
                return false;
            }
        }
    }
    return true;
}
// Same, with a warp-uniform verdict (the epilogue warps execute .sync.aligned instructions afterwards).
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, const Ctl& ctl, int where)
{
    const bool ok = mbar_wait(bar, parity, ctl, where);
    return __all_sync(0xffffffffu, ok);
}

// --------------------------------------------------------------------------------- host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn get_encode_fn()
{
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* ptr = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qres) != cudaSuccess ||
            qres != cudaDriverEntryPointSuccess)
            return nullptr;
        fn = reinterpret_cast<EncodeTiledFn>(ptr);
    }
    return fn;
}

bool make_map_2d(CUtensorMap* tm, CUtensorMapDataType dt, int elt_bytes, const void* ptr, uint64_t inner, uint64_t outer,
                 uint32_t box_inner, uint32_t box_outer, CUtensorMapSwizzle swz, uint64_t pitch = 0)      // pitch in elements, 0: inner
{
    EncodeTiledFn fn = get_encode_fn();
    if (!fn) return false;
    cuuint64_t dims[2] = {inner, outer};
    cuuint64_t strides[1] = {(pitch ? pitch : inner) * (uint64_t)elt_bytes};
    cuuint32_t box[2] = {box_inner, box_outer};
    cuuint32_t estr[2] = {1, 1};
    return fn(tm, dt, 2, const_cast<void*>(ptr), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              swz, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace
