// Error measurement (paper App. E.2: relative Frobenius error against an fp64 product;
// Eq. (D.9) compares the RMS of that error across realizations).
//   fmm_ref_gemm_fp64 : Cref = A * B with fp64 multiply-accumulate of the fp32 inputs (DFMA tiles).
//   fmm_error_stats   : sum (C - Cref)^2, sum Cref^2, max |C - Cref| with fp64 accumulation,
//                       warp-shuffle + shared-memory tree per block, fixed block partition and a
//                       single-block second stage, hence bit-reproducible.
#include <mutex>
#include "fmm_internal.h"
#include "fmm_ptx.cuh"

// Scratch of fmm_error_stats_noalloc: one partial triple per reduction block.  It lives in the
// library image, so every GPU that loads the library carries these 24 KB until the process exits.
// In host code this name is only a stand-in for the symbol; the device address comes from
// cudaGetSymbolAddress (see noalloc_scratch below).
static __device__ __align__(256) double g_noalloc_partials[3 * 1024];
// where the statistics kernels of the FMM_DEBUG build report a store outside their output buffers
static __device__ int g_stats_guard_code;

namespace {

// 4 x 148 SMs, all resident at 512 threads; at most the 1024 slots of g_noalloc_partials.  A constant and not the device's count:
// the partition of the sums, and with it their bits, are the same on every device
constexpr int STAT_BLOCKS = 592;
constexpr int STAT_THREADS = 512;
constexpr int64_t STATS_MAX_DIM = (int64_t)1 << 30;    // per dimension, as for the product itself: M * N cannot overflow
static_assert(STAT_BLOCKS <= 1024, "one scratch slot per reduction block");

__device__ __forceinline__ void warp_reduce3(double& a, double& b, double& c)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        b += __shfl_xor_sync(0xffffffffu, b, o);
        c = fmax(c, __shfl_xor_sync(0xffffffffu, c, o));
    }
}

__device__ __forceinline__ void block_reduce3(double& a, double& b, double& c, double* sm)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    warp_reduce3(a, b, c);
    if (lane == 0) { sm[warp * 3] = a; sm[warp * 3 + 1] = b; sm[warp * 3 + 2] = c; }
    __syncthreads();
    if (warp == 0) {
        const int nw = blockDim.x >> 5;
        a = lane < nw ? sm[lane * 3] : 0.0;
        b = lane < nw ? sm[lane * 3 + 1] : 0.0;
        c = lane < nw ? sm[lane * 3 + 2] : 0.0;
        warp_reduce3(a, b, c);
    }
}

__global__ void __launch_bounds__(STAT_THREADS) error_partial_kernel(const float* __restrict__ C,
                                                                    const double* __restrict__ Cref,
                                                                    int64_t count, double* __restrict__ partial,
                                                                    const FmmGuard guard)
{
    __shared__ double sm[3 * (STAT_THREADS / 32)];
    double sd = 0.0, sr = 0.0, mx = 0.0;
    // each thread takes pairs: one 8-byte load of C, one 16-byte load of Cref (count is even); four pairs per
    // trip with all loads issued first, so that every thread keeps 96 bytes in flight
    const int64_t pairs = count >> 1;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const float2* C2 = reinterpret_cast<const float2*>(C);
    const double2* R2 = reinterpret_cast<const double2*>(Cref);
    auto add = [&](float2 c, double2 r) {
        const double d0 = (double)c.x - r.x, d1 = (double)c.y - r.y;
        sd = fma(d0, d0, sd); sd = fma(d1, d1, sd);
        sr = fma(r.x, r.x, sr); sr = fma(r.y, r.y, sr);
        mx = fmax(mx, fmax(fabs(d0), fabs(d1)));
    };
    // (the last trip is predicated, not a loop of single loads: at n = 4096 a thread makes 7 trips)
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < pairs; i += 4 * stride) {
        float2 c[4]; double2 r[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (i + u * stride < pairs) { c[u] = __ldcs(C2 + i + u * stride); r[u] = __ldcs(R2 + i + u * stride); }
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (i + u * stride < pairs) add(c[u], r[u]);
    }
    block_reduce3(sd, sr, mx, sm);
    if (threadIdx.x == 0 && FMM_GUARD(guard, partial + blockIdx.x * 3, 24, 1601)) {
        partial[blockIdx.x * 3] = sd; partial[blockIdx.x * 3 + 1] = sr; partial[blockIdx.x * 3 + 2] = mx;
    }
}

__global__ void __launch_bounds__(STAT_THREADS) error_final_kernel(const double* __restrict__ partial, int n,
                                                                  double* __restrict__ out3, const FmmGuard guard)
{
    __shared__ double sm[3 * (STAT_THREADS / 32)];
    double sd = 0.0, sr = 0.0, mx = 0.0;
    fmmptx::griddep_wait();                                  // launched under the first kernel's tail: its partials are complete now
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        sd += partial[i * 3]; sr += partial[i * 3 + 1]; mx = fmax(mx, partial[i * 3 + 2]);
    }
    block_reduce3(sd, sr, mx, sm);
    if (threadIdx.x == 0 && FMM_GUARD(guard, out3, 24, 1602)) { out3[0] = sd; out3[1] = sr; out3[2] = mx; }
}

// Both stages.  The second is launched with the programmatic-serialization attribute, so that its launch latency falls
// under the first (2 us of 38 at n = 4096).
fmm_status_t launch_stats(const float* C, const double* Cref, int64_t count, double* partial, double* out3, const FmmGuard& guard, cudaStream_t st)
{
    error_partial_kernel<<<STAT_BLOCKS, STAT_THREADS, 0, st>>>(C, Cref, count, partial, guard);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(1); cfg.blockDim = dim3(STAT_THREADS); cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at; cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, error_final_kernel, static_cast<const double*>(partial), STAT_BLOCKS, out3, guard);
    return cudaGetLastError() == cudaSuccess ? FMM_OK : FMM_ERR_CUDA;
}

// fp64 product of fp32 operands on the fp64 tensor path: T x T outputs per block of four warps (each T/2 x T/2, as
// m16n8k4 fragments), K in steps of 16 through a ring of shared-memory stages filled by cp.async.  Operands stay fp32 in
// shared memory and are widened (exactly) when a fragment is read: half the shared-memory bytes of a double copy, and the
// conversions run beside the multiply-adds.  Rows are padded to 20 and T + 8 words so that a fragment read touches all 32
// banks.  Bound: the fp64 pipe, 37 TFLOP/s measured with DFMA and with mma alike; fragments feed it with a fourth of the
// operand reads of a 4 x 4 register tile (which took 1.12 ms at n = 2048).  T = 64 keeps the last wave full at the usual
// sizes (7 tiles per SM at n = 2048); T = 32 spreads problems of fewer 64 x 64 tiles than SMs.  ALIGNED: both operands
// 16-byte aligned (16-byte copies; 4-byte ones otherwise).
constexpr int REF_BK = 16, REF_STAGES = 4;

__device__ __forceinline__ void ref_mma(double (&c)[4], double a0, double a1, double b)
{
    asm volatile("mma.sync.aligned.m16n8k4.row.col.f64.f64.f64.f64 {%0, %1, %2, %3}, {%4, %5}, {%6}, {%0, %1, %2, %3};"
                 : "+d"(c[0]), "+d"(c[1]), "+d"(c[2]), "+d"(c[3]) : "d"(a0), "d"(a1), "d"(b));
}
template <bool ALIGNED>
__device__ __forceinline__ void ref_copy16(float* dst, const float* src)
{
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    if (ALIGNED) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
    else
#pragma unroll
        for (int i = 0; i < 4; ++i) asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d + 4 * i), "l"(src + i) : "memory");
}

template <int T, bool ALIGNED>
__global__ void __launch_bounds__(128, T == 64 ? 4 : 8)
ref_gemm_fp64_kernel(const float* __restrict__ A, const float* __restrict__ B, double* __restrict__ C, int64_t M, int64_t N, int64_t K,
                     const FmmGuard guard)
{
    constexpr int LDA = REF_BK + 4, LDB = T + 8;
    constexpr int MF = T / 32, NF = T / 16;               // m16 and n8 fragments of a warp's T/2 x T/2 outputs
    __shared__ __align__(16) float As[REF_STAGES][T][LDA];          // [m][k]
    __shared__ __align__(16) float Bs[REF_STAGES][REF_BK][LDB];     // [k][n]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int wm = (warp >> 1) * (T / 2), wn = (warp & 1) * (T / 2);
    const int64_t m0 = (int64_t)blockIdx.y * T, n0 = (int64_t)blockIdx.x * T;
    auto load = [&](int stage, int64_t k0) {
#pragma unroll
        for (int i = threadIdx.x; i < T * (REF_BK / 4); i += 128) {
            const int r = i / (REF_BK / 4), c = i % (REF_BK / 4) * 4;
            ref_copy16<ALIGNED>(&As[stage][r][c], A + (m0 + r) * K + k0 + c);
        }
#pragma unroll
        for (int i = threadIdx.x; i < REF_BK * (T / 4); i += 128) {
            const int r = i / (T / 4), c = i % (T / 4) * 4;
            ref_copy16<ALIGNED>(&Bs[stage][r][c], B + (k0 + r) * N + n0 + c);
        }
    };
    double acc[MF][NF][4];
#pragma unroll
    for (int i = 0; i < MF; ++i)
#pragma unroll
        for (int j = 0; j < NF; ++j)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[i][j][e] = 0.0;
    const int steps = (int)(K / REF_BK);
#pragma unroll
    for (int s = 0; s < REF_STAGES - 1; ++s) {
        if (s < steps) load(s, (int64_t)s * REF_BK);
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    for (int s = 0; s < steps; ++s) {
        asm volatile("cp.async.wait_group %0;" ::"n"(REF_STAGES - 2) : "memory");
        __syncthreads();                                   // stage s has landed, stage s - 1 has been read by every warp
        if (s + REF_STAGES - 1 < steps) load((s + REF_STAGES - 1) % REF_STAGES, (int64_t)(s + REF_STAGES - 1) * REF_BK);
        asm volatile("cp.async.commit_group;" ::: "memory");
        const int st = s % REF_STAGES;
#pragma unroll
        for (int kk = 0; kk < REF_BK; kk += 4) {
            double a[MF][2], b[NF];
#pragma unroll
            for (int i = 0; i < MF; ++i)
#pragma unroll
                for (int h = 0; h < 2; ++h) a[i][h] = (double)As[st][wm + 16 * i + 8 * h + (lane >> 2)][kk + (lane & 3)];
#pragma unroll
            for (int j = 0; j < NF; ++j) b[j] = (double)Bs[st][kk + (lane & 3)][wn + 8 * j + (lane >> 2)];
#pragma unroll
            for (int i = 0; i < MF; ++i)
#pragma unroll
                for (int j = 0; j < NF; ++j) ref_mma(acc[i][j], a[i][0], a[i][1], b[j]);
        }
    }
#pragma unroll
    for (int i = 0; i < MF; ++i)
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int j = 0; j < NF; ++j) {
                double* c = C + (m0 + wm + 16 * i + 8 * h + (lane >> 2)) * N + n0 + wn + 8 * j + 2 * (lane & 3);
                if (FMM_GUARD(guard, c, 16, 1603)) *reinterpret_cast<double2*>(c) = make_double2(acc[i][j][2 * h], acc[i][j][2 * h + 1]);
            }
}

template <int T>
void launch_ref(const float* A, const float* B, double* C, int64_t M, int64_t N, int64_t K, const FmmGuard& guard, cudaStream_t st)
{
    const dim3 grid((unsigned)(N / T), (unsigned)(M / T));
    if ((((uintptr_t)A | (uintptr_t)B) & 15) == 0) ref_gemm_fp64_kernel<T, true><<<grid, 128, 0, st>>>(A, B, C, M, N, K, guard);
    else ref_gemm_fp64_kernel<T, false><<<grid, 128, 0, st>>>(A, B, C, M, N, K, guard);
}

// Device address of g_stats_guard_code on the current device (FMM_DEBUG build; the release build passes no word and
// never resolves the symbol, so its calls stay free of runtime lookups).
int* stats_guard_word()
{
#ifdef FMM_DEBUG
    int* ptr = nullptr;
    if (cudaGetSymbolAddress((void**)&ptr, g_stats_guard_code) != cudaSuccess) { cudaGetLastError(); return nullptr; }
    return ptr;
#else
    return nullptr;
#endif
}

}  // namespace

// Self-test of the store guard: one thread stores to status word 40 under a guard that allows words 32..39 only.
// Both addresses lie inside the plan's 64-word status array, so nothing is ever written out of bounds; the checked
// build must skip the store and record code 1901, the normal build has no guard and simply writes the spare word.
__global__ void guard_selftest_kernel(int* status, const FmmGuard guard)
{
    int* target = status + 40;
    if (FMM_GUARD(guard, target, sizeof(int), 1901)) *target = 1;
}

fmm_status_t fmm_launch_guard_selftest(int* status, cudaStream_t st)
{
    const FmmGuard guard = fmm_make_guard(status + 32, 8 * sizeof(int), nullptr, 0, status + FMM_GUARD_WORD);
    guard_selftest_kernel<<<1, 1, 0, st>>>(status, guard);
    return cudaGetLastError() == cudaSuccess ? FMM_OK : FMM_ERR_CUDA;
}

fmm_status_t fmm_stats_guard_read(int* code)
{
    *code = 0;
#ifdef FMM_DEBUG
    if (cudaDeviceSynchronize() != cudaSuccess) { cudaGetLastError(); return FMM_ERR_CUDA; }
    if (cudaMemcpyFromSymbol(code, g_stats_guard_code, sizeof(int)) != cudaSuccess) { cudaGetLastError(); return FMM_ERR_CUDA; }
#endif
    return FMM_OK;
}

extern "C" {

size_t fmm_error_stats_scratch_bytes(void) { return sizeof(double) * 3 * STAT_BLOCKS; }

fmm_status_t fmm_error_stats(const float* C, const double* Cref, int64_t M, int64_t N, double* out3,
                             void* scratch, size_t scratch_bytes, void* stream)
{
    if (!C || !Cref || !out3 || !scratch) return FMM_ERR_INVALID_ARG;
    // bound each factor before forming the product (signed overflow otherwise)
    if (M <= 0 || N <= 0 || M > STATS_MAX_DIM || N > STATS_MAX_DIM || ((M * N) & 1)) return FMM_ERR_SHAPE;
    if (scratch_bytes < fmm_error_stats_scratch_bytes() || ((uintptr_t)scratch & 15)) return FMM_ERR_WORKSPACE;
    if (((uintptr_t)C & 7) || ((uintptr_t)Cref & 15)) return FMM_ERR_INVALID_ARG;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    double* partial = static_cast<double*>(scratch);
    const FmmGuard guard = fmm_make_guard(partial, sizeof(double) * 3 * STAT_BLOCKS, out3, sizeof(double) * 3, stats_guard_word());
    return launch_stats(C, Cref, M * N, partial, out3, guard, st);
}

fmm_status_t fmm_ref_gemm_fp64(const float* A, const float* B, double* Cref, int64_t M, int64_t N, int64_t K,
                               void* stream)
{
    if (!A || !B || !Cref) return FMM_ERR_INVALID_ARG;
    if (M <= 0 || N <= 0 || K <= 0 || (M % 64) || (N % 64) || (K % 16)) return FMM_ERR_SHAPE;
    if ((uintptr_t)Cref & 15) return FMM_ERR_INVALID_ARG;
    const FmmGuard guard = fmm_make_guard(Cref, sizeof(double) * (size_t)M * (size_t)N, nullptr, 0, stats_guard_word());
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    // tiles of 64 only where they fill the device (the same bits either way)
    if ((M / 64) * (N / 64) < fmm_sm_count()) launch_ref<32>(A, B, Cref, M, N, K, guard, st);
    else launch_ref<64>(A, B, Cref, M, N, K, guard, st);
    return cudaGetLastError() == cudaSuccess ? FMM_OK : FMM_ERR_CUDA;
}

// ---- variant of fmm_error_stats for callers that cannot allocate device memory ----------------
namespace {
constexpr int NOALLOC_MAX_DEVICES = 64;
constexpr int64_t NOALLOC_MAX_ELEMS = (int64_t)1 << 28;    // a constant of the interface, not of the array: the kernels handle any count
std::mutex g_noalloc_mutex;
double* g_noalloc_ptr[NOALLOC_MAX_DEVICES] = {nullptr};

// Device address of the static scratch on the current device, resolved once per device.
fmm_status_t noalloc_scratch(double** out)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) { cudaGetLastError(); return FMM_ERR_CUDA; }
    if (dev < 0 || dev >= NOALLOC_MAX_DEVICES) return FMM_ERR_INVALID_ARG;
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (!g_noalloc_ptr[dev]) {
        double* ptr = nullptr;
        if (cudaGetSymbolAddress((void**)&ptr, g_noalloc_partials) != cudaSuccess || !ptr) {
            cudaGetLastError();
            return FMM_ERR_CUDA;
        }
        g_noalloc_ptr[dev] = ptr;
    }
    *out = g_noalloc_ptr[dev];
    return FMM_OK;
}
}  // namespace

fmm_status_t fmm_error_stats_noalloc(const float* C, const double* Cref, int64_t M, int64_t N, double* out3,
                                     void* stream)
{
    if (!C || !Cref || !out3) return FMM_ERR_INVALID_ARG;
    if (M <= 0 || N <= 0 || M > NOALLOC_MAX_ELEMS || N > NOALLOC_MAX_ELEMS) return FMM_ERR_SHAPE;
    if (M * N > NOALLOC_MAX_ELEMS || ((M * N) & 1)) return FMM_ERR_SHAPE;
    if (((uintptr_t)C & 7) || ((uintptr_t)Cref & 15)) return FMM_ERR_INVALID_ARG;
    double* partial = nullptr;
    fmm_status_t s = noalloc_scratch(&partial);
    if (s != FMM_OK) return s;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    // every one of the STAT_BLOCKS slots is rewritten by the first kernel, so nothing left behind by
    // an earlier call is ever read and no clearing is needed
    const FmmGuard guard = fmm_make_guard(partial, sizeof(double) * 3 * STAT_BLOCKS, out3, sizeof(double) * 3, stats_guard_word());
    return launch_stats(C, Cref, M * N, partial, out3, guard, st);
}

int64_t fmm_error_stats_noalloc_max_elements(void) { return NOALLOC_MAX_ELEMS; }

}  // extern "C"
