// Host side of the C ABI: plan validation, workspace layout, the recursion driver that turns
// (levels, realization) into kernel launches.  No device allocation happens after plan creation.
#include <math.h>
#include <stdlib.h>
#include <string.h>
#include <mutex>
#include <new>
#include <vector>
#include "fmm_internal.h"

constexpr int HOST_STRIPS = 8;

// Side streams and events of one fmm_matmul_host call in flight.
struct HostLane {
    cudaStream_t comp = nullptr, down = nullptr;
    cudaEvent_t up[HOST_STRIPS + 1] = {}, mul[HOST_STRIPS] = {}, done[2] = {};
    bool taken = false;           // a host thread is enqueuing on it
    bool create()
    {
        bool ok = cudaStreamCreateWithFlags(&comp, cudaStreamNonBlocking) == cudaSuccess && cudaStreamCreateWithFlags(&down, cudaStreamNonBlocking) == cudaSuccess;
        auto make = [&](cudaEvent_t& e) { ok = ok && cudaEventCreateWithFlags(&e, cudaEventDisableTiming) == cudaSuccess; };
        for (auto& e : up) make(e);
        for (auto& e : mul) make(e);
        for (auto& e : done) make(e);
        if (!ok) cudaGetLastError();
        return ok;
    }
    ~HostLane()
    {
        for (auto& e : up) if (e) cudaEventDestroy(e);
        for (auto& e : mul) if (e) cudaEventDestroy(e);
        for (auto& e : done) if (e) cudaEventDestroy(e);
        if (comp) cudaStreamDestroy(comp);
        if (down) cudaStreamDestroy(down);
    }
    bool idle() const
    {
        for (auto& e : done) if (cudaEventQuery(e) != cudaSuccess) { cudaGetLastError(); return false; }
        return true;
    }
};

// A plan's lanes, made when first needed, at most MAX of them, destroyed with the plan.  A lane serves one call at a time: one
// whose last call has drained if there is one, else a new one, else the longest unused (its streams keep the order then).
// nullptr when every lane is being enqueued on by another thread: the caller then does without.
struct FmmHostLanes {
    static constexpr int MAX = 4;
    std::mutex mutex;
    std::vector<HostLane*> lanes;          // least recently used first
    HostLane* acquire()
    {
        std::lock_guard<std::mutex> lock(mutex);
        HostLane* pick = nullptr;
        for (HostLane* l : lanes) if (!l->taken && l->idle()) { pick = l; break; }
        if (!pick && (int)lanes.size() < MAX) {
            pick = new (std::nothrow) HostLane;
            if (!pick || !pick->create()) { delete pick; return nullptr; }
            lanes.push_back(pick);
        }
        if (!pick) for (HostLane* l : lanes) if (!l->taken) { pick = l; break; }
        if (!pick) return nullptr;
        pick->taken = true;
        for (size_t i = 0; i + 1 < lanes.size(); ++i) if (lanes[i] == pick) std::swap(lanes[i], lanes[i + 1]);
        return pick;
    }
    void release(HostLane* l)
    {
        std::lock_guard<std::mutex> lock(mutex);
        l->taken = false;
    }
    ~FmmHostLanes() { for (HostLane* l : lanes) delete l; }
};

namespace {

size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

bool finite_all(const float* p, int n)
{
    for (int i = 0; i < n; ++i)
        if (!isfinite(p[i])) return false;
    return true;
}

// Largest residual of the Brent equations of <2,2,2> (Sec. 2.1: the decomposition must equal the
// matrix-multiplication tensor): sum_r U[r][ij] V[r][kl] W[r][mn] = [j==k][i==m][l==n].
double brent_residual(int rank, const float* U, const float* V, const float* W)
{
    double worst = 0.0;
    for (int a = 0; a < 4; ++a)
        for (int b = 0; b < 4; ++b)
            for (int c = 0; c < 4; ++c) {
                double s = 0.0;
                for (int r = 0; r < rank; ++r)
                    s += (double)U[r * 4 + a] * (double)V[r * 4 + b] * (double)W[r * 4 + c];
                const int i = a >> 1, j = a & 1, k = b >> 1, l = b & 1, m = c >> 1, n = c & 1;
                const double target = (j == k && i == m && l == n) ? 1.0 : 0.0;
                worst = fmax(worst, fabs(s - target));
            }
    return worst;
}

fmm_status_t check_shape(const fmm_plan* plan, int64_t M, int64_t N, int64_t K)
{
    if (M <= 0 || N <= 0 || K <= 0) return FMM_ERR_SHAPE;
    const int64_t d = (int64_t)1 << plan->levels;
    if (M % d || N % d || K % d) return FMM_ERR_SHAPE;
    if ((M / d) % 128 || (N / d) % 128 || (K / d) % 128) return FMM_ERR_SHAPE;
    if (M > (1 << 30) || N > (1 << 30) || K > (1 << 30)) return FMM_ERR_SHAPE;
    return FMM_OK;
}

void make_layout(const fmm_plan* plan, int64_t M, int64_t N, int64_t K, FmmLayout* L)
{
    const int64_t d = (int64_t)1 << plan->levels;
    L->m = M / d; L->n = N / d; L->k = K / d;
    L->terms = plan->terms;
    const int64_t nkb = L->k / plan->qp.block_k;
    size_t off = 0;
    L->qa = off; off = align_up(off + (size_t)(L->terms * L->m * L->k), 1024);
    L->qb = off; off = align_up(off + (size_t)(L->terms * L->n * L->k), 1024);
    const size_t sbytes = plan->qp.scale_mode == FMM_SCALE_FP32_AMAX_DIV_448 ? 4 : 1;
    L->sa_term = (size_t)(L->m * nkb) * sbytes;
    L->sb_term = (size_t)(L->n * nkb) * sbytes;
    L->sa = off; off = align_up(off + L->sa_term * L->terms, 1024);
    L->sb = off; off = align_up(off + L->sb_term * L->terms, 1024);
    L->sb_down = L->sb;
    if (fmm_scale_per_column(plan->qp)) { L->sb_down = off; off = align_up(off + L->sb_term * L->terms, 1024); }
    for (int lv = 0; lv < FMM_MAX_LEVELS; ++lv) { L->inter_a[lv] = 0; L->inter_b[lv] = 0; L->dec[lv] = 0; }
    // fp32 combinations of the outer levels 1 .. levels-1
    for (int lv = 1; lv < plan->levels; ++lv) {
        const int64_t cnt = fmm_ipow(plan->rank, lv);
        const int64_t dd = (int64_t)1 << lv;
        // the innermost of these levels is formed in registers by the two-level encoder where that exists
        const bool last = (lv == plan->levels - 1);
        const bool need_a = !(last && fmm_encode2_supported(false, plan->qp.block_k, 0, 0));
        const bool need_b = !(last && fmm_encode2_supported(true, plan->qp.block_k, plan->qp.b_tile_n, plan->qp.b_preround_bf16));
        if (need_a) { L->inter_a[lv] = off; off = align_up(off + (size_t)(cnt * (M / dd) * (K / dd)) * 4, 1024); }
        if (need_b) { L->inter_b[lv] = off; off = align_up(off + (size_t)(cnt * (K / dd) * (N / dd)) * 4, 1024); }
        // (three levels: the first-level matrices stay in the registers of the two-step decoder)
        if (last) { L->dec[lv] = off; off = align_up(off + (size_t)(cnt * (M / dd) * (N / dd)) * 4, 1024); }
    }
    L->total = off;
}

// the kernels read the operands with 16-byte vector loads and write C through a tensor map
bool aligned16(const void* p) { return ((uintptr_t)p & 15) == 0; }

// a plan's device tables live on the device that was current at fmm_plan_create
fmm_status_t check_device(const fmm_plan* plan)
{
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) { cudaGetLastError(); return FMM_ERR_CUDA; }
    return dev == plan->device ? FMM_OK : FMM_ERR_WRONG_DEVICE;
}

fmm_status_t check_ws(const fmm_plan* plan, int64_t M, int64_t N, int64_t K, void* ws, size_t ws_bytes,
                      FmmLayout* L)
{
    fmm_status_t s = check_device(plan);
    if (s != FMM_OK) return s;
    s = check_shape(plan, M, N, K);
    if (s != FMM_OK) return s;
    make_layout(plan, M, N, K, L);
    if (!ws || ((uintptr_t)ws & 1023) || ws_bytes < L->total) return FMM_ERR_WORKSPACE;
    return FMM_OK;
}

void fill_coef(float dst[FMM_MAX_RANK][4], const float src[FMM_MAX_RANK][4], int R)
{
    memset(dst, 0, sizeof(float) * FMM_MAX_RANK * 4);
    for (int r = 0; r < R; ++r)
        for (int j = 0; j < 4; ++j) dst[r][j] = src[r][j];
}

// A strip of the leaf rows of A and C (m0 .. m1) or of the leaf columns of B and C (n0 .. n1), in every block.
struct Strip { int64_t m0, m1, n0, n1; };

// Levels whose combinations are formed as fp32 matrices in the workspace (the innermost one or two are not).
int outer_levels(const fmm_plan* plan, bool b_side)
{
    if (plan->levels < 2) return 0;
    const bool fused2 = fmm_encode2_supported(b_side, plan->qp.block_k, b_side ? plan->qp.b_tile_n : 0, b_side ? plan->qp.b_preround_bf16 : 0);
    return fused2 ? plan->levels - 2 : plan->levels - 1;
}

// Those combinations, level by level, both sides of a level in one launch.
fmm_status_t encode_outer(const fmm_plan* plan, const FmmLayout& L, char* ws, const float* A, const float* B, int64_t M, int64_t N, int64_t K,
                          cudaStream_t st, int* launches)
{
    const int deepest[2] = {outer_levels(plan, false), outer_levels(plan, true)};
    for (int level = 1; level <= deepest[0] || level <= deepest[1]; ++level) {
        CombParams c[2];
        memset(c, 0, sizeof(c));
        for (int side = 0; side < 2; ++side) {
            if (level > deepest[side]) continue;
            const size_t* inter = side ? L.inter_b : L.inter_a;
            const int64_t rows = (side ? K : M) >> (level - 1), cols = (side ? N : K) >> (level - 1);
            CombParams& s = c[side];
            s.in = level > 1 ? reinterpret_cast<const float*>(ws + inter[level - 1]) : (side ? B : A);
            s.in_batch_stride = level > 1 ? rows * cols : 0; s.ld = cols; s.batch = (int)fmm_ipow(plan->rank, level - 1);
            s.rows = (int)(rows / 2); s.cols = (int)(cols / 2); s.R = plan->rank;
            fill_coef(s.coef, side ? plan->V : plan->U, plan->rank);
            s.out = reinterpret_cast<float*>(ws + inter[level]);
            s.guard = fmm_make_guard(s.out, (size_t)s.batch * s.R * (size_t)(s.rows * (int64_t)s.cols) * 4, nullptr, 0, plan->d_status + FMM_GUARD_WORD);
        }
        const fmm_status_t s = fmm_launch_comb(c[0], c[1], level > 1, st);
        if (s != FMM_OK) return s;
        ++*launches;
    }
    return FMM_OK;
}

// Parameters of one side of steps 1-2, behind encode_outer: the innermost one or two levels and the quantizer.  [lo, hi) is the
// strip of leaf rows (A) or columns (B) to encode: everything, or with at most one level a part of it (multiples of 128).
EncodeParams encode_params(const fmm_plan* plan, const FmmLayout& L, char* ws, const float* X,
                           int64_t rows, int64_t cols, bool b_side, int64_t lo, int64_t hi, bool overlap)
{
    const int R = plan->rank, lv = plan->levels;
    const int blk = plan->qp.block_k, mode = (int)plan->qp.scale_mode;
    const float (*coef)[4] = b_side ? plan->V : plan->U;
    EncodeParams e;
    memset(&e, 0, sizeof(e));
    e.q_out = reinterpret_cast<uint8_t*>(ws + (b_side ? L.qb : L.qa));
    e.s_out = ws + (b_side ? L.sb : L.sa);
    e.s_term_stride = (int64_t)(b_side ? L.sb_term : L.sa_term);
    e.amax_floor = plan->qp.amax_floor;
    e.s_down = (int64_t)(L.sb_down - L.sb); e.down = fmm_scale_down(plan->qp);
    e.b_tile = (short)(b_side ? plan->qp.b_tile_n : 0);
    e.preround_bf16 = (b_side && plan->qp.b_preround_bf16) ? 1 : 0;
    e.guard = fmm_make_guard(e.q_out, (size_t)L.terms * (size_t)((b_side ? L.n : L.m) * L.k),
                             e.s_out, (size_t)L.terms * (b_side ? L.sb_term : L.sa_term) + (b_side ? L.sb_down - L.sb : 0), plan->d_status + FMM_GUARD_WORD);
    // first element of the strip in every array
    const int64_t strip_in = b_side ? lo : lo * cols;
    e.q_out += lo * L.k;
    e.s_out = static_cast<char*>(e.s_out) + (mode == FMM_SCALE_UE8M0_CEIL ? lo / 128 * 512 : lo * 4 * (b_side ? 1 : 128 / blk));
    if (lv == 0) {
        // Plain quantization of the matrix itself.  The matrix is cut into four panels (row panels of A,
        // column panels of B) that are handled like four "combinations" with identity coefficients, so
        // each thread keeps four independent loads in flight; the outputs land where the unsplit
        // matrix would put them.
        const int64_t ext = hi - lo;               // rows of A / columns of B in this launch
        const bool panels = b_side ? (ext % (e.b_tile ? 512 : 256) == 0) : (ext % 4 == 0);
        e.in = X + strip_in; e.in_batch_stride = 0; e.ld = cols; e.batch = 1;
        e.overlap_prev = overlap ? 1 : 0;
        e.s_ld = (int)(b_side ? cols : rows); e.sf_blocks = (int)((b_side ? cols : rows) / 128);
        if (panels) {
            e.nq = 4; e.R = 4;
            for (int r = 0; r < 4; ++r) e.coef[r][r] = 1.0f;
            if (b_side) {
                e.rows = (int)rows; e.cols = (int)(ext / 4);
                for (int j = 0; j < 4; ++j) e.qoff[j] = (int64_t)j * (ext / 4);
            } else {
                e.rows = (int)(ext / 4); e.cols = (int)cols;
                for (int j = 0; j < 4; ++j) e.qoff[j] = (int64_t)j * (ext / 4) * cols;
            }
            e.s_step = (int)(ext / 4);
            // the four panels share one scale array (panel r is shifted by r * s_step rows / columns inside it)
            e.s_term_stride = 0;
        } else {
            e.rows = (int)(b_side ? rows : ext); e.cols = (int)(b_side ? ext : cols); e.nq = 1; e.R = 1;
            e.coef[0][0] = 1.0f;
            e.s_step = 0;
        }
        e.q_term = (int64_t)e.rows * e.cols;
    } else {
        // the last two levels run as one kernel where that is supported: the combinations of level lv-1 stay
        // in registers
        const bool fused2 = lv >= 2 && fmm_encode2_supported(b_side, blk, e.b_tile, e.preround_bf16);
        const int level = outer_levels(plan, b_side);
        const float* cur = level ? reinterpret_cast<const float*>(ws + (b_side ? L.inter_b[level] : L.inter_a[level])) : X;
        const int64_t cur_rows = rows >> level, cur_cols = cols >> level, cur_ld = cur_cols, cur_stride = level ? cur_rows * cur_cols : 0;
        const int batch = (int)fmm_ipow(R, level);
        e.in = cur + strip_in; e.in_batch_stride = cur_stride; e.ld = cur_ld; e.batch = batch;
        e.overlap_prev = overlap ? 1 : 0;
        const int div = fused2 ? 4 : 2;
        e.rows = (int)(cur_rows / div); e.cols = (int)(cur_cols / div); e.nq = 4; e.R = R;
        e.qoff[0] = 0; e.qoff[1] = e.cols; e.qoff[2] = (int64_t)e.rows * e.ld; e.qoff[3] = (int64_t)e.rows * e.ld + e.cols;
        for (int j = 0; j < 4; ++j) e.qoff_outer[j] = 2 * e.qoff[j];
        fill_coef(e.coef, coef, R);
        e.s_step = 0; e.s_ld = b_side ? e.cols : e.rows; e.sf_blocks = (b_side ? e.cols : e.rows) / 128;
        e.q_term = (int64_t)e.rows * e.cols;
        if (b_side) e.cols = (int)(hi - lo); else e.rows = (int)(hi - lo);
    }
    return e;
}

fmm_status_t encode_side(const fmm_plan* plan, const FmmLayout& L, char* ws, const float* X,
                         int64_t rows, int64_t cols, bool b_side, int64_t lo, int64_t hi, bool overlap, cudaStream_t st, int* launches)
{
    const int blk = plan->qp.block_k, mode = (int)plan->qp.scale_mode;
    const EncodeParams e = encode_params(plan, L, ws, X, rows, cols, b_side, lo, hi, overlap);
    fmm_status_t s;
    if (plan->levels >= 2 && fmm_encode2_supported(b_side, blk, e.b_tile, e.preround_bf16))
        s = b_side ? fmm_launch_encode2_b(e, mode, st) : fmm_launch_encode2_a(e, blk, mode, st);
    else
        s = b_side ? fmm_launch_encode_b(e, blk, mode, st) : fmm_launch_encode_a(e, blk, mode, st);
    if (s == FMM_OK) ++*launches;
    return s;
}

// Steps 1-2 of a whole call.
fmm_status_t encode_all(const fmm_plan* plan, const FmmLayout& L, char* ws, const float* A, const float* B, int64_t M, int64_t N, int64_t K,
                        cudaStream_t st, int* launches)
{
    if (plan->levels <= 1) {
        fmm_status_t s;
        if (fmm_launch_encode_both(encode_params(plan, L, ws, A, M, K, false, 0, L.m, false), encode_params(plan, L, ws, B, K, N, true, 0, L.n, false),
                                   plan->qp.block_k, (int)plan->qp.scale_mode, st, &s)) {
            if (s == FMM_OK) ++*launches;
            return s;
        }
    }
    fmm_status_t s = encode_outer(plan, L, ws, A, B, M, N, K, st, launches);
    if (s == FMM_OK) s = encode_side(plan, L, ws, A, M, K, false, 0, L.m, *launches > 0, st, launches);     // behind combinations
    if (s == FMM_OK) s = encode_side(plan, L, ws, B, K, N, true, 0, L.n, true, st, launches);
    return s;
}

// The part of the product kernel's parameters that its tile shape depends on.
GemmParams product_params(const fmm_plan* plan, const FmmLayout& L, const Strip& strip)
{
    GemmParams g;
    memset(&g, 0, sizeof(g));
    g.msub = (int)(strip.m1 - strip.m0); g.nsub = (int)(strip.n1 - strip.n0);
    g.m = (int)L.m; g.n = (int)L.n; g.k = (int)L.k; g.terms = (int)L.terms;
    g.terms_per_group = plan->levels >= 2 ? plan->rank : (int)L.terms;
    g.device = plan->device; g.sms = plan->sms;
    g.R = plan->levels >= 1 ? plan->rank : 1; g.nq = plan->levels >= 1 ? 4 : 1; g.W = plan->W;
    g.sb_tile = plan->qp.b_tile_n == 128 ? 1 : 0; g.updates = plan->updates;
    g.forced = plan->forced;
    return g;
}

fmm_status_t multiply(const fmm_plan* plan, const FmmLayout& L, char* ws, float* C, int64_t M, int64_t N, const Strip& strip,
                      cudaStream_t st, int* launches, bool after_encode)
{
    GemmParams g = product_params(plan, L, strip);
    g.overlap_prev = after_encode ? 1 : 0;
    g.qa = reinterpret_cast<const uint8_t*>(ws + L.qa) + strip.m0 * L.k;
    g.qb = reinterpret_cast<const uint8_t*>(ws + L.qb) + strip.n0 * L.k;
    const bool e8 = plan->qp.scale_mode == FMM_SCALE_UE8M0_CEIL;
    g.sa = ws + L.sa + (e8 ? strip.m0 / 128 * 512 : strip.m0 * 4 * (128 / plan->qp.block_k));
    g.sb = ws + L.sb_down + (e8 ? strip.n0 / 128 * 512 : strip.n0 * 4);
    g.sa_term = (int64_t)L.sa_term; g.sb_term = (int64_t)L.sb_term;
    g.up = fmm_scale_up(plan->qp); g.small_weights = plan->small_weights;
    // The product kernel applies the innermost decoder only: leaf products of parent p land in the four
    // blocks of parent p's (2m x 2n) matrix.  For one level that matrix is C itself; for more levels the
    // parents' matrices are stacked in the workspace and decoded outwards level by level (the same
    // two-stage order as the recursion in Sec. 3), which moves far fewer bytes than scattering every
    // leaf product into all of its R^(levels-1)-fold weighted destinations.
    const int lv = plan->levels;
    const int64_t parents = lv >= 2 ? fmm_ipow(plan->rank, lv - 1) : 1;
    const int64_t pm = lv >= 1 ? 2 * L.m : L.m, pn = lv >= 1 ? 2 * L.n : L.n;      // a parent's matrix
    float* dest = lv >= 2 ? reinterpret_cast<float*>(ws + L.dec[lv - 1]) : C;
    g.C = dest + strip.m0 * pn + strip.n0; g.ldc = pn; g.Mfull = parents * pm; g.Nfull = pn;
    g.walk = plan->d_walk; g.out = plan->d_out; g.status = plan->d_status;
    g.pair_start = plan->d_pair_start; g.pair = plan->d_pair; g.steps = plan->steps;
    for (int r = 0; r < FMM_MAX_RANK; ++r) g.order[r] = plan->order[r];
    g.guard = fmm_make_guard(dest, (size_t)g.Mfull * (size_t)g.Nfull * 4, nullptr, 0, plan->d_status + FMM_GUARD_WORD);
    fmm_status_t s = fmm_launch_gemm(g, plan->qp.block_k, (int)plan->qp.scale_mode, st, launches);
    if (s != FMM_OK) return s;
    for (int l = lv - 1, steps; l >= 1; l -= steps) {
        steps = l == 2 ? 2 : 1;
        DecodeParams d;
        memset(&d, 0, sizeof(d));
        d.in = reinterpret_cast<const float*>(ws + L.dec[l]);
        d.out = l == steps ? C : reinterpret_cast<float*>(ws + L.dec[l - steps]);
        d.batch = (int)fmm_ipow(plan->rank, l - steps);
        d.rows = (int)(M >> l); d.cols = (int)(N >> l); d.R = plan->rank;
        for (int r = 0; r < plan->rank; ++r)
            for (int q = 0; q < 4; ++q) d.W[r][q] = plan->W[r][q];
        d.guard = fmm_make_guard(d.out, (size_t)d.batch * ((size_t)d.rows << steps) * ((size_t)d.cols << steps) * 4, nullptr, 0,
                                 plan->d_status + FMM_GUARD_WORD);
        s = fmm_launch_decode(d, steps, st);
        if (s != FMM_OK) return s;
        ++*launches;
    }
    return FMM_OK;
}

}  // namespace

extern "C" {

const char* fmm_status_string(fmm_status_t s)
{
    switch (s) {
        case FMM_OK: return "ok";
        case FMM_ERR_INVALID_ARG: return "invalid argument";
        case FMM_ERR_SHAPE: return "shape not supported (M, N, K must be 2^levels * multiples of 128)";
        case FMM_ERR_NOT_EXACT: return "realization violates the Brent equations";
        case FMM_ERR_WORKSPACE: return "workspace missing, misaligned or too small";
        case FMM_ERR_ALLOC: return "allocation failed";
        case FMM_ERR_CUDA: return "CUDA call failed";
        case FMM_ERR_ARCH: return "device is not compute capability 10.x (B200)";
        case FMM_ERR_DEVICE_TIMEOUT: return "a bounded device-side wait timed out";
        case FMM_ERR_WRONG_DEVICE: return "the current device is not the one the plan was created on";
    }
    return "unknown status";
}

fmm_status_t fmm_phi_gamma(int rank, const float* U, const float* V, const float* W, double* phi, double* gamma)
{
    if (rank < 1 || rank > FMM_MAX_RANK || !U || !V || !W || !phi || !gamma) return FMM_ERR_INVALID_ARG;
    double p = 0.0, g = 0.0;
    for (int r = 0; r < rank; ++r) {
        double nu = 0, nv = 0, nw = 0;
        for (int j = 0; j < 4; ++j) {
            nu += (double)U[r * 4 + j] * U[r * 4 + j];
            nv += (double)V[r * 4 + j] * V[r * 4 + j];
            nw += (double)W[r * 4 + j] * W[r * 4 + j];
        }
        p += nu * nv * nw;
        g += sqrt(nu * nv * nw);
    }
    *phi = p; *gamma = g;
    return FMM_OK;
}

fmm_status_t fmm_brent_residual(int rank, const float* U, const float* V, const float* W, double* out)
{
    if (rank < 1 || rank > FMM_MAX_RANK || !U || !V || !W || !out) return FMM_ERR_INVALID_ARG;
    *out = brent_residual(rank, U, V, W);
    return FMM_OK;
}

fmm_status_t fmm_plan_create(fmm_plan_t** out, int rank, const float* U, const float* V, const float* W,
                             int levels, const fmm_quant_params_t* qp)
{
    if (!out) return FMM_ERR_INVALID_ARG;
    *out = nullptr;
    if (!qp || levels < 0 || levels > FMM_MAX_LEVELS) return FMM_ERR_INVALID_ARG;
    if (qp->block_k != 32 && qp->block_k != 128) return FMM_ERR_INVALID_ARG;
    if (qp->scale_mode != FMM_SCALE_FP32_AMAX_DIV_448 && qp->scale_mode != FMM_SCALE_UE8M0_CEIL) return FMM_ERR_INVALID_ARG;
    if (qp->scale_mode == FMM_SCALE_UE8M0_CEIL && qp->block_k != 32) return FMM_ERR_INVALID_ARG;
    if (qp->fp8_max != 448.0f || !(qp->amax_floor > 0.0f) || !isfinite(qp->amax_floor)) return FMM_ERR_INVALID_ARG;
    if (qp->b_tile_n != 0 && qp->b_tile_n != 128) return FMM_ERR_INVALID_ARG;
    if ((qp->b_tile_n == 128 || qp->b_preround_bf16) &&
        (qp->block_k != 128 || qp->scale_mode != FMM_SCALE_FP32_AMAX_DIV_448)) return FMM_ERR_INVALID_ARG;
    if (levels > 0) {
        if (rank < 1 || rank > FMM_MAX_RANK || !U || !V || !W) return FMM_ERR_INVALID_ARG;
        if (!finite_all(U, rank * 4) || !finite_all(V, rank * 4) || !finite_all(W, rank * 4)) return FMM_ERR_INVALID_ARG;
        if (brent_residual(rank, U, V, W) > 1e-5) return FMM_ERR_NOT_EXACT;
    } else {
        rank = 1;
    }
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) { cudaGetLastError(); return FMM_ERR_CUDA; }
    int major = 0;
    if (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess) { cudaGetLastError(); return FMM_ERR_CUDA; }
    if (major != 10) return FMM_ERR_ARCH;

    int sms = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0) { cudaGetLastError(); return FMM_ERR_CUDA; }

    fmm_plan* p = new (std::nothrow) fmm_plan;
    if (!p) return FMM_ERR_ALLOC;
    memset(static_cast<void*>(p), 0, sizeof(*p));
    p->last_launches.store(0, std::memory_order_relaxed);
    p->rank = rank; p->levels = levels; p->qp = *qp; p->device = dev; p->sms = sms;
    if (levels > 0)
        for (int r = 0; r < rank; ++r)
            for (int j = 0; j < 4; ++j) { p->U[r][j] = U[r * 4 + j]; p->V[r][j] = V[r * 4 + j]; p->W[r][j] = W[r * 4 + j]; }
    p->terms = (int)fmm_ipow(rank, levels);

    // Walks and decoder table of the fp32-scale product kernel (Sec. 2.1 decode, innermost level; outer levels are decoded
    // afterwards), with carried sums and after them without.  row_off / col_off are in units of leaf blocks inside the stack
    // of parent matrices.
    std::vector<FmmWalkEntry> walk(2 * (size_t)p->terms);
    std::vector<FmmOutEntry> entries;
    const int parents = levels >= 1 ? p->terms / rank : 1;
    for (int carried = 1; carried >= 0; --carried) {
        int order[FMM_MAX_RANK];
        float carry[FMM_MAX_RANK] = {0.0f};
        for (int r = 0; r < FMM_MAX_RANK; ++r) order[r] = r;
        if (carried && levels >= 1 && qp->scale_mode == FMM_SCALE_FP32_AMAX_DIV_448) fmm_choose_walk(rank, p->U, p->V, p->W, order, carry);
        std::vector<int> touched((size_t)parents * 4, -1);         // the last update of a block
        for (int t = 0; t < p->terms; ++t) {
            FmmWalkEntry& step = walk[t + (carried ? 0 : p->terms)];
            step.out0 = (int)entries.size();
            const int parent = levels ? t / rank : 0, s = levels ? t % rank : 0, r = order[s];
            step.term = levels ? parent * rank + r : 0; step.carry = carry[s];
            for (int q = 0; q < (levels ? 4 : 1); ++q) {
                const float w = !levels ? 1.0f : s + 1 < rank ? fmm_emitted_weight(p->W[r][q], carry[s + 1], p->W[order[s + 1]][q]) : p->W[r][q];
                if (w == 0.0f) continue;
                if (carried && levels && fabsf(w) < 1.0f) p->small_weights |= 1u << s;
                FmmOutEntry e;
                e.row_off = parent * 2 + (q >> 1); e.col_off = q & 1;
                e.w = w;
                int& last = touched[(size_t)parent * 4 + q];
                e.gap = last < 0 ? 0 : (int)entries.size() - last;
                last = (int)entries.size();
                entries.push_back(e);
            }
            step.out1 = (int)entries.size();
        }
    }

    // Pair-fused decoder: pair up the R products of a parent so that the pairs' unions of destination blocks are as
    // small as possible in total (exhaustive over the matchings: R <= 8), walk the pairs one after the other.
    for (int r = 0; r < FMM_MAX_RANK; ++r) p->order[r] = r;
    p->steps = levels >= 1 ? (rank + 1) / 2 : 1;
    std::vector<int> pstart;
    std::vector<FmmPairEntry> pentries;
    if (levels >= 1) {
        auto mask = [&](int r) { int m = 0; for (int q = 0; q < 4; ++q) if (p->W[r][q] != 0.0f) m |= 1 << q; return m; };
        auto bits = [](int m) { return (m & 1) + ((m >> 1) & 1) + ((m >> 2) & 1) + ((m >> 3) & 1); };
        int best_cost = 1 << 30, best[FMM_MAX_RANK], cur[FMM_MAX_RANK];
        bool used[FMM_MAX_RANK] = {false};
        // recursive matching: always pair the lowest unused product with some other one (or leave it single once)
        struct Rec {
            static void go(int n, int R, int cost, bool single_used, bool* used, int* cur, int& best_cost, int* best,
                           const int* masks, int (*bitsf)(int))
            {
                if (cost >= best_cost) return;
                int a = -1;
                for (int r = 0; r < R; ++r) if (!used[r]) { a = r; break; }
                if (a < 0) { best_cost = cost; for (int i = 0; i < R; ++i) best[i] = cur[i]; return; }
                used[a] = true;
                for (int b = a + 1; b < R; ++b) {
                    if (used[b]) continue;
                    used[b] = true; cur[n] = a; cur[n + 1] = b;
                    go(n + 2, R, cost + bitsf(masks[a] | masks[b]), single_used, used, cur, best_cost, best, masks, bitsf);
                    used[b] = false;
                }
                if ((R & 1) && !single_used) {
                    // the single product goes last in the walk: remember it at the end of cur
                    cur[R - 1] = a;
                    // shift: pairs fill cur[0 .. R-2]
                    go(n, R, cost + bitsf(masks[a]), true, used, cur, best_cost, best, masks, bitsf);
                }
                used[a] = false;
            }
        };
        int masks[FMM_MAX_RANK];
        for (int r = 0; r < rank; ++r) masks[r] = mask(r);
        Rec::go(0, rank, 0, false, used, cur, best_cost, best, masks, +bits);
        for (int r = 0; r < rank; ++r) p->order[r] = best[r];
        std::vector<char> ptouched((size_t)parents * 4, 0);
        for (int parent = 0; parent < parents; ++parent)
            for (int s = 0; s < p->steps; ++s) {
                pstart.push_back((int)pentries.size());
                const bool pairstep = 2 * s + 1 < rank;
                const int ra = pairstep ? p->order[2 * s] : -1, rb = pairstep ? p->order[2 * s + 1] : p->order[2 * s];
                for (int q = 0; q < 4; ++q) {
                    const float wa = ra >= 0 ? p->W[ra][q] : 0.0f, wb = p->W[rb][q];
                    if (wa == 0.0f && wb == 0.0f) continue;
                    FmmPairEntry e;
                    e.row_off = parent * 2 + (q >> 1); e.col_off = q & 1; e.wA = wa; e.wB = wb;
                    e.first = ptouched[(size_t)parent * 4 + q] ? 0 : 1;
                    ptouched[(size_t)parent * 4 + q] = 1;
                    pentries.push_back(e);
                }
            }
    } else {
        pstart.push_back(0);
        FmmPairEntry e; e.row_off = 0; e.col_off = 0; e.wA = 0.0f; e.wB = 1.0f; e.first = 1;
        pentries.push_back(e);
    }
    pstart.push_back((int)pentries.size());

    p->updates = qp->scale_mode == FMM_SCALE_UE8M0_CEIL ? (int)(pentries.size() / parents) : walk[levels ? rank - 1 : 0].out1;

    p->lanes = new (std::nothrow) FmmHostLanes;
    if (!p->lanes) { delete p; return FMM_ERR_ALLOC; }
    cudaError_t ce = cudaMalloc(&p->d_status, 64 * sizeof(int));
    if (ce == cudaSuccess) ce = cudaMalloc(&p->d_walk, sizeof(FmmWalkEntry) * walk.size());
    if (ce == cudaSuccess) ce = cudaMalloc(&p->d_out, sizeof(FmmOutEntry) * (entries.size() + 1));
    if (ce == cudaSuccess) ce = cudaMemset(p->d_status, 0, 64 * sizeof(int));
    if (ce == cudaSuccess) ce = cudaMemcpy(p->d_walk, walk.data(), sizeof(FmmWalkEntry) * walk.size(), cudaMemcpyHostToDevice);
    if (ce == cudaSuccess && !entries.empty())
        ce = cudaMemcpy(p->d_out, entries.data(), sizeof(FmmOutEntry) * entries.size(), cudaMemcpyHostToDevice);
    if (ce == cudaSuccess) ce = cudaMalloc(&p->d_pair_start, sizeof(int) * pstart.size());
    if (ce == cudaSuccess) ce = cudaMalloc(&p->d_pair, sizeof(FmmPairEntry) * (pentries.size() + 1));
    if (ce == cudaSuccess) ce = cudaMemcpy(p->d_pair_start, pstart.data(), sizeof(int) * pstart.size(), cudaMemcpyHostToDevice);
    if (ce == cudaSuccess) ce = cudaMemcpy(p->d_pair, pentries.data(), sizeof(FmmPairEntry) * pentries.size(), cudaMemcpyHostToDevice);
    if (ce != cudaSuccess) {
        cudaGetLastError();
        fmm_plan_destroy(p);
        return ce == cudaErrorMemoryAllocation ? FMM_ERR_ALLOC : FMM_ERR_CUDA;
    }
    *out = p;
    return FMM_OK;
}

fmm_status_t fmm_plan_destroy(fmm_plan_t* p)
{
    if (!p) return FMM_ERR_INVALID_ARG;
    delete p->lanes;
    if (p->d_status) cudaFree(p->d_status);
    if (p->d_walk) cudaFree(p->d_walk);
    if (p->d_out) cudaFree(p->d_out);
    if (p->d_pair_start) cudaFree(p->d_pair_start);
    if (p->d_pair) cudaFree(p->d_pair);
    delete p;
    return FMM_OK;
}

fmm_status_t fmm_workspace_bytes(const fmm_plan_t* plan, int64_t M, int64_t N, int64_t K, size_t* bytes)
{
    if (!plan || !bytes) return FMM_ERR_INVALID_ARG;
    fmm_status_t s = check_shape(plan, M, N, K);
    if (s != FMM_OK) return s;
    FmmLayout L;
    make_layout(plan, M, N, K, &L);
    *bytes = L.total;
    return FMM_OK;
}

fmm_status_t fmm_quantized_view(const fmm_plan_t* plan, int64_t M, int64_t N, int64_t K, int term, char side,
                                size_t* q_offset, int64_t* q_rows, int64_t* q_cols,
                                size_t* scale_offset, int64_t* scale_rows, int64_t* scale_cols)
{
    if (!plan || !q_offset || !q_rows || !q_cols || !scale_offset || !scale_rows || !scale_cols) return FMM_ERR_INVALID_ARG;
    if (side != 'A' && side != 'B') return FMM_ERR_INVALID_ARG;
    fmm_status_t s = check_shape(plan, M, N, K);
    if (s != FMM_OK) return s;
    if (term < 0 || term >= plan->terms) return FMM_ERR_INVALID_ARG;
    FmmLayout L;
    make_layout(plan, M, N, K, &L);
    const int64_t nkb = L.k / plan->qp.block_k;
    const bool fp32 = plan->qp.scale_mode == FMM_SCALE_FP32_AMAX_DIV_448;
    if (side == 'A') {
        *q_offset = L.qa + (size_t)term * L.m * L.k; *q_rows = L.m; *q_cols = L.k;
        *scale_offset = L.sa + (size_t)term * L.sa_term;
        if (fp32) { *scale_rows = L.k / 128; *scale_cols = L.m * (128 / plan->qp.block_k); } else { *scale_rows = L.m; *scale_cols = nkb; }
    } else {
        *q_offset = L.qb + (size_t)term * L.n * L.k; *q_rows = L.n; *q_cols = L.k;
        *scale_offset = L.sb + (size_t)term * L.sb_term;
        if (fp32) { *scale_rows = nkb; *scale_cols = L.n; } else { *scale_rows = L.n; *scale_cols = nkb; }
    }
    return FMM_OK;
}

fmm_status_t fmm_encode_only(const fmm_plan_t* plan, const float* A, const float* B, int64_t M, int64_t N, int64_t K,
                             void* ws, size_t ws_bytes, void* stream)
{
    if (!plan || !A || !B || !aligned16(A) || !aligned16(B)) return FMM_ERR_INVALID_ARG;
    FmmLayout L;
    fmm_status_t s = check_ws(plan, M, N, K, ws, ws_bytes, &L);
    if (s != FMM_OK) return s;
    int launches = 0;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    s = encode_all(plan, L, static_cast<char*>(ws), A, B, M, N, K, st, &launches);
    plan->last_launches.store(launches, std::memory_order_relaxed);
    return s;
}

fmm_status_t fmm_multiply_only(const fmm_plan_t* plan, float* C, int64_t M, int64_t N, int64_t K,
                               void* ws, size_t ws_bytes, void* stream)
{
    if (!plan || !C || !aligned16(C)) return FMM_ERR_INVALID_ARG;
    FmmLayout L;
    fmm_status_t s = check_ws(plan, M, N, K, ws, ws_bytes, &L);
    if (s != FMM_OK) return s;
    int launches = 0;
    s = multiply(plan, L, static_cast<char*>(ws), C, M, N, {0, L.m, 0, L.n}, reinterpret_cast<cudaStream_t>(stream), &launches, false);
    plan->last_launches.store(launches, std::memory_order_relaxed);
    return s;
}

fmm_status_t fmm_matmul(const fmm_plan_t* plan, const float* A, const float* B, float* C,
                        int64_t M, int64_t N, int64_t K, void* ws, size_t ws_bytes, void* stream)
{
    if (!plan || !A || !B || !C || !aligned16(A) || !aligned16(B) || !aligned16(C)) return FMM_ERR_INVALID_ARG;
    FmmLayout L;
    fmm_status_t s = check_ws(plan, M, N, K, ws, ws_bytes, &L);
    if (s != FMM_OK) return s;
    int launches = 0;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    s = encode_all(plan, L, static_cast<char*>(ws), A, B, M, N, K, st, &launches);
    if (s == FMM_OK) s = multiply(plan, L, static_cast<char*>(ws), C, M, N, {0, L.m, 0, L.n}, st, &launches, true);
    plan->last_launches.store(launches, std::memory_order_relaxed);
    return s;
}

fmm_status_t fmm_product_shape(const fmm_plan_t* plan, int64_t M, int64_t N, int64_t K, fmm_product_shape_t* shape)
{
    if (!plan || !shape) return FMM_ERR_INVALID_ARG;
    fmm_status_t s = check_device(plan);
    if (s == FMM_OK) s = check_shape(plan, M, N, K);
    if (s != FMM_OK) return s;
    FmmLayout L;
    make_layout(plan, M, N, K, &L);
    const GemmParams g = product_params(plan, L, {0, L.m, 0, L.n});
    *shape = fmm_choose_product(g, plan->qp.block_k, (int)plan->qp.scale_mode);
    return shape->k_shares <= L.k / 128 ? FMM_OK : FMM_ERR_SHAPE;
}

fmm_status_t fmm_force_product_shape(fmm_plan_t* plan, const fmm_product_shape_t* shape)
{
    if (!plan) return FMM_ERR_INVALID_ARG;
    if (!shape) { memset(&plan->forced, 0, sizeof(plan->forced)); return FMM_OK; }
    if (!fmm_product_shape_exists(*shape, plan->qp.block_k, (int)plan->qp.scale_mode, plan->qp.b_tile_n == 128, plan->levels >= 1 ? plan->rank : 1))
        return FMM_ERR_INVALID_ARG;
    plan->forced = *shape;
    return FMM_OK;
}

// Host-operand variant: [product workspace | A | B | C] in the caller's device buffer, 1024-byte aligned parts.
static size_t host_align(size_t x) { return (x + 1023) & ~(size_t)1023; }

fmm_status_t fmm_host_workspace_bytes(const fmm_plan_t* plan, int64_t M, int64_t N, int64_t K, size_t* bytes)
{
    if (!bytes) return FMM_ERR_INVALID_ARG;
    size_t ws = 0;
    fmm_status_t s = fmm_workspace_bytes(plan, M, N, K, &ws);
    if (s != FMM_OK) return s;
    *bytes = host_align(ws) + host_align((size_t)M * K * 4) + host_align((size_t)K * N * 4) + host_align((size_t)M * N * 4);
    return FMM_OK;
}

// The strip [lo, hi) of the rows (columns) of each of the `blocks` leaf blocks of a rows x cols matrix, as one copy.
static bool copy_strip(float* dst, const float* src, int64_t rows, int64_t cols, int blocks, bool by_rows, int64_t lo, int64_t hi,
                       cudaMemcpyKind kind, cudaStream_t st)
{
    if (by_rows) {
        // a "row" of this copy is the strip's rows of one block, which are contiguous
        const size_t pitch = (size_t)(rows / blocks) * (size_t)cols * 4, width = (size_t)((hi - lo) * cols) * 4;
        const int64_t at = lo * cols;
        if (blocks == 1 || pitch > 0x7fffffff) {
            for (int b = 0; b < blocks; ++b)
                if (cudaMemcpyAsync(dst + b * (int64_t)(pitch / 4) + at, src + b * (int64_t)(pitch / 4) + at, width, kind, st) != cudaSuccess) { cudaGetLastError(); return false; }
        } else if (cudaMemcpy2DAsync(dst + at, pitch, src + at, pitch, width, (size_t)blocks, kind, st) != cudaSuccess) { cudaGetLastError(); return false; }
        return true;
    }
    for (int b = 0; b < blocks; ++b) {
        const int64_t at = b * (cols / blocks) + lo;
        if (cudaMemcpy2DAsync(dst + at, (size_t)cols * 4, src + at, (size_t)cols * 4, (size_t)(hi - lo) * 4, (size_t)rows, kind, st) != cudaSuccess) { cudaGetLastError(); return false; }
    }
    return true;
}

// Borders of the strips in sixteenths of the leaf extent.  A copy costs about 12 us besides its bytes while the link is used
// both ways, so strips are few where the upload bounds the call and more where the download, which cannot begin before the
// first strip has been multiplied, does too (n = 4096: eight 2.88 ms, five 3.13).  Of the
// few, the first is short to start the download, the last short because its products and download follow the upload; more
// equal or smaller strips cost more copies than they gain (n = 4096: nine with a shorter end 2.90, eleven 2.98, sixteen 3.34).
static const int* strip_borders(int64_t upload, int64_t download, int* count)
{
    static const int eight[] = {0, 2, 4, 6, 8, 10, 12, 14, 16}, five[] = {0, 2, 6, 10, 14, 16}, four[] = {0, 8, 12, 14, 16}, two[] = {0, 8, 16};
    if (upload >= (32 << 20) && 5 * download > 3 * upload) { *count = 8; return eight; }
    if (upload >= (32 << 20)) { *count = 5; return five; }
    if (upload >= (12 << 20)) { *count = 4; return four; }
    *count = upload >= (8 << 20) ? 2 : 1;
    return two;
}

// Host operands, at most one level: the transfers bound the call (n = 4096: 134 MB up at 55 GB/s = 2.4 ms, 67 MB down, against
// 0.33 ms of kernels), and the link is full duplex.  So the smaller operand goes up first, the larger one in strips of leaf
// rows (A) or columns (B); a strip is encoded and multiplied on one side stream while the next one is on its way, and its part
// of C goes down on another while later strips still come up.  What remains beside the upload is the last strip's kernels
// and download.  A strip is computed by the kernel that the whole product would take, so the results are the same bits.
static fmm_status_t matmul_host_strips(const fmm_plan* plan, const FmmLayout& L, char* ws, const float* A, const float* B, float* C,
                                       float* dA, float* dB, float* dC, int64_t M, int64_t N, int64_t K, int strips, const int* borders, bool by_rows,
                                       HostLane& lane, cudaStream_t st)
{
    const int blocks = 1 << plan->levels;
    const cudaMemcpyKind up = cudaMemcpyHostToDevice, down = cudaMemcpyDeviceToHost;
    int launches = 0;
    auto sig = [](cudaEvent_t e, cudaStream_t from, cudaStream_t to) {
        if (cudaEventRecord(e, from) == cudaSuccess && cudaStreamWaitEvent(to, e, 0) == cudaSuccess) return true;
        cudaGetLastError();
        return false;
    };
    // whatever happens below, the caller's stream waits for what has been enqueued on the side streams
    auto join = [&](fmm_status_t s) {
        const bool ok = sig(lane.done[0], lane.comp, st) && sig(lane.done[1], lane.down, st);
        return s == FMM_OK && !ok ? FMM_ERR_CUDA : s;
    };
    const int64_t units = (by_rows ? L.m : L.n) / 128;
    if (cudaMemcpyAsync(by_rows ? dB : dA, by_rows ? B : A, (size_t)(by_rows ? K * N : M * K) * 4, up, st) != cudaSuccess) { cudaGetLastError(); return FMM_ERR_CUDA; }
    if (!sig(lane.up[strips], st, lane.comp)) return join(FMM_ERR_CUDA);
    fmm_status_t s = by_rows ? encode_side(plan, L, ws, dB, K, N, true, 0, L.n, false, lane.comp, &launches)
                             : encode_side(plan, L, ws, dA, M, K, false, 0, L.m, false, lane.comp, &launches);
    // Where the uploads are the longer part, a strip of C goes down behind its product and the next strip's upload, that is with the
    // upload after that one: a copy that starts while the other direction is busy takes some 45 us to get going, two that start
    // together do not.  Where the downloads are, each one goes as soon as it can (8192 x 2048 x 4096 3.40 ms,
    // behind the next upload 3.46; 16384 x 512 x 2048 2.68, 2.70; 4096 x 1024 x 4096 1.75, 1.76 to 1.80).
    const bool with_upload = (M + N) * K > M * N;
    int last = -1;                             // the strip whose product was enqueued last
    int64_t c_lo = 0, c_hi = 0;
    auto send_down = [&]() {
        return last < 0 || (sig(lane.mul[last], lane.comp, lane.down) && copy_strip(C, dC, M, N, blocks, by_rows, c_lo, c_hi, down, lane.down));
    };
    for (int i = 0; i < strips && s == FMM_OK; ++i) {
        const int64_t lo = units * borders[i] / 16 * 128, hi = units * borders[i + 1] / 16 * 128;
        if (lo == hi) continue;
        Strip part = {0, L.m, 0, L.n};
        if (by_rows) { part.m0 = lo; part.m1 = hi; } else { part.n0 = lo; part.n1 = hi; }
        if (!copy_strip(by_rows ? dA : dB, by_rows ? A : B, by_rows ? M : K, by_rows ? K : N, blocks, by_rows, lo, hi, up, st) ||
            !sig(lane.up[i], st, lane.comp) || (with_upload && !send_down())) return join(FMM_ERR_CUDA);
        s = by_rows ? encode_side(plan, L, ws, dA, M, K, false, lo, hi, false, lane.comp, &launches)
                    : encode_side(plan, L, ws, dB, K, N, true, lo, hi, false, lane.comp, &launches);
        if (s == FMM_OK) s = multiply(plan, L, ws, dC, M, N, part, lane.comp, &launches, false);
        last = i; c_lo = lo; c_hi = hi;
        if (s == FMM_OK && !with_upload && !send_down()) s = FMM_ERR_CUDA;
    }
    if (s == FMM_OK && with_upload && !send_down()) s = FMM_ERR_CUDA;
    plan->last_launches.store(launches, std::memory_order_relaxed);
    return join(s);
}

fmm_status_t fmm_matmul_host(const fmm_plan_t* plan, const float* A, const float* B, float* C,
                             int64_t M, int64_t N, int64_t K, void* ws, size_t ws_bytes, void* stream)
{
    if (!plan || !A || !B || !C) return FMM_ERR_INVALID_ARG;
    size_t need = 0, inner = 0;
    fmm_status_t s = fmm_host_workspace_bytes(plan, M, N, K, &need);
    if (s != FMM_OK) return s;
    if (!ws || ((uintptr_t)ws & 1023) || ws_bytes < need) return FMM_ERR_WORKSPACE;
    fmm_workspace_bytes(plan, M, N, K, &inner);
    char* base = static_cast<char*>(ws);
    float* dA = reinterpret_cast<float*>(base + host_align(inner));
    float* dB = reinterpret_cast<float*>(reinterpret_cast<char*>(dA) + host_align((size_t)M * K * 4));
    float* dC = reinterpret_cast<float*>(reinterpret_cast<char*>(dB) + host_align((size_t)K * N * 4));
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    if (plan->levels <= 1) {
        FmmLayout L;
        s = check_ws(plan, M, N, K, ws, inner, &L);
        if (s != FMM_OK) return s;
        const bool by_rows = M >= N;                         // the larger operand of the two
        int strips = 1;
        const int* borders = strip_borders((by_rows ? M : N) * K * 4, M * N * 4, &strips);
        if ((by_rows ? L.m : L.n) < 256) strips = 1;
        cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
        // pageable copies block the host in order, so they would gain nothing from the strips
        auto pinned = [](const void* p) {
            cudaPointerAttributes a;
            return cudaPointerGetAttributes(&a, p) == cudaSuccess && a.type == cudaMemoryTypeHost;
        };
        if (strips > 1 && pinned(A) && pinned(B) && pinned(C) && cudaStreamIsCapturing(st, &capture) == cudaSuccess &&
            capture == cudaStreamCaptureStatusNone) {
            if (HostLane* lane = plan->lanes->acquire()) {
                s = matmul_host_strips(plan, L, base, A, B, C, dA, dB, dC, M, N, K, strips, borders, by_rows, *lane, st);
                plan->lanes->release(lane);
                return s;
            }
        }
        cudaGetLastError();
    }
    if (cudaMemcpyAsync(dA, A, (size_t)M * K * 4, cudaMemcpyHostToDevice, st) != cudaSuccess ||
        cudaMemcpyAsync(dB, B, (size_t)K * N * 4, cudaMemcpyHostToDevice, st) != cudaSuccess) {
        cudaGetLastError();
        return FMM_ERR_CUDA;
    }
    s = fmm_matmul(plan, dA, dB, dC, M, N, K, ws, inner, stream);
    if (s != FMM_OK) return s;
    if (cudaMemcpyAsync(C, dC, (size_t)M * N * 4, cudaMemcpyDeviceToHost, st) != cudaSuccess) {
        cudaGetLastError();
        return FMM_ERR_CUDA;
    }
    return FMM_OK;
}

fmm_status_t fmm_device_status(const fmm_plan_t* plan, int* code)
{
    if (!plan || !code) return FMM_ERR_INVALID_ARG;
    fmm_status_t sd = check_device(plan);
    if (sd != FMM_OK) return sd;
    int h[4] = {0, 0, 0, 0};
    // every stream, including non-blocking ones that the copy below would not wait for
    if (cudaDeviceSynchronize() != cudaSuccess) { cudaGetLastError(); return FMM_ERR_CUDA; }
    if (cudaMemcpy(h, plan->d_status, sizeof(h), cudaMemcpyDeviceToHost) != cudaSuccess) { cudaGetLastError(); return FMM_ERR_CUDA; }
    *code = h[0];
    return h[0] ? FMM_ERR_DEVICE_TIMEOUT : FMM_OK;
}

int fmm_debug_build(void)
{
#ifdef FMM_DEBUG
    return 1;
#else
    return 0;
#endif
}

fmm_status_t fmm_debug_violation(const fmm_plan_t* plan, int* code)
{
    if (!code) return FMM_ERR_INVALID_ARG;
    if (!plan) return fmm_stats_guard_read(code);
    fmm_status_t sd = check_device(plan);
    if (sd != FMM_OK) return sd;
    if (cudaDeviceSynchronize() != cudaSuccess) { cudaGetLastError(); return FMM_ERR_CUDA; }
    if (cudaMemcpy(code, plan->d_status + FMM_GUARD_WORD, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) { cudaGetLastError(); return FMM_ERR_CUDA; }
    return FMM_OK;
}

fmm_status_t fmm_device_status_clear(const fmm_plan_t* plan)
{
    if (!plan) return FMM_ERR_INVALID_ARG;
    fmm_status_t sd = check_device(plan);
    if (sd != FMM_OK) return sd;
    if (cudaDeviceSynchronize() != cudaSuccess) { cudaGetLastError(); return FMM_ERR_CUDA; }
    if (cudaMemset(plan->d_status, 0, 64 * sizeof(int)) != cudaSuccess) { cudaGetLastError(); return FMM_ERR_CUDA; }
    return FMM_OK;
}

fmm_status_t fmm_selftest_bounded_wait(const fmm_plan_t* plan, int64_t limit_ns, void* stream)
{
    if (!plan || limit_ns <= 0 || limit_ns > 2000000000ll) return FMM_ERR_INVALID_ARG;
    fmm_status_t sd = check_device(plan);
    if (sd != FMM_OK) return sd;
    return fmm_launch_bounded_wait_selftest(plan->d_status, (unsigned long long)limit_ns, reinterpret_cast<cudaStream_t>(stream));
}

fmm_status_t fmm_selftest_store_guard(const fmm_plan_t* plan, void* stream)
{
    if (!plan) return FMM_ERR_INVALID_ARG;
    fmm_status_t sd = check_device(plan);
    if (sd != FMM_OK) return sd;
    return fmm_launch_guard_selftest(plan->d_status, reinterpret_cast<cudaStream_t>(stream));
}

fmm_status_t fmm_last_launch_count(const fmm_plan_t* plan, int* launches)
{
    if (!plan || !launches) return FMM_ERR_INVALID_ARG;
    *launches = plan->last_launches.load(std::memory_order_relaxed);
    return FMM_OK;
}

}  // extern "C"
