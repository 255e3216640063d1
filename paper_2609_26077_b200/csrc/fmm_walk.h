// Order in which the fp32-scale product kernel walks the products of a parent (plain host C++, no CUDA).
#pragma once
#include <math.h>
#include <string.h>

#define FMM_MAX_RANK 8

// Weight with which the running sum of a step goes to a block: w - c * w_next, c being the next step's carry; exactly zero
// where that cancels but for the rounding of the coefficients (two units in the last place).
static inline float fmm_emitted_weight(float w, float carry, float w_next)
{
    const double x = (double)w - (double)carry * (double)w_next;
    return fabs(x) <= 2.5e-7 * fabs((double)w) ? 0.0f : (float)x;
}

// The order in which the fp32-scale product kernel walks the R products of a parent, and what it carries from one to the
// next.  A product's sum need not stand alone: with S_t = M_t + c_t * S_{t-1} (the previous sum is still on chip)
// C_q = sum_t W_t[q] M_t = sum_t (W_t[q] - c_{t+1} W_{t+1}[q]) S_t, so a ratio c that two neighbouring rows of W share in
// several blocks saves an update of C in all but one of them: 18 -> 12 block updates for the Phi-optimal realization, 14 -> 7
// for the Winograd form, 12 -> 10 for Strassen, 28 -> 17 where W has no zeros.
//
// Two conditions keep the sums as good as the products:
//   |c| <= 1      A kernel that starts its accumulators from c * S_{t-1} rounds every later addition at the size of the
//                 running sum.  Steps of up to 2 in magnitude, whose product along a walk can reach 2^6, made the error of C
//                 2.0 to 2.8 times the one of separate sums for realizations without zeros.  With this bound it is 1.05
//                 (Strassen), 1.19 (Winograd), 1.20 (Phi-optimal), 1.05 to 1.13 (without zeros) at block 32, and 1.03, 1.13,
//                 1.15, 1.05 to 1.09 at block 128 (K = 4096, measured against the exact product of the quantized operands; 3.1e-7,
//                 4.6e-7 and 3.0e-7 for the named ones at block 32), with the same numbers of updates.
//   nested rows   A step may be carried only into a product that feeds no other blocks, so that a block never sees a product
//                 that its own sum does not contain (and would have to cancel: products of blocks of very different size, or
//                 an infinity).
// Of the walks that save most, the search (10 to 50 us) takes the first one, from the last product backwards and in the order of
// the rows, unless another one's sums round clearly less: a third less of what carrying adds to the error's variance.  (For the
// named realizations the gain would be smaller than that and does not show in the error of C, while the walks found first are
// 0.5 % faster at block 128, n = 4096; for realizations without zeros it halves the excess.)  Model: independent products, M_t
// of variance s_t = |U_t|^2 |V_t|^2 as operands of independent elements give it.  The running sum then holds
// v_t = s_t + c_t^2 v_{t-1}, adding M_t to it in small steps rounds at s_t / 2 + c_t^2 v_{t-1} in the mean instead of s_t / 2,
// and an error of S_t reaches C_q with the factor W_t[q], as M_t itself does.
struct FmmWalkSearch {
    int R;
    int save[FMM_MAX_RANK][FMM_MAX_RANK];              // updates saved by carrying from the first row into the second
    float ratio[FMM_MAX_RANK][FMM_MAX_RANK];
    double norm2[FMM_MAX_RANK], size[FMM_MAX_RANK];    // |W_r|^2, |U_r|^2 |V_r|^2
    signed char left[1 << FMM_MAX_RANK][FMM_MAX_RANK]; // [rows placed][first of them]: most updates that the rows before can save
    int cur[FMM_MAX_RANK], best[FMM_MAX_RANK];
    double best_extra;

    void bound()
    {
        for (int set = (1 << R) - 1; set > 0; --set)
            for (int b = 0; b < R; ++b) {
                int most = 0;
                for (int a = 0; a < R; ++a)
                    if (!(set >> a & 1) && save[a][b] + left[set | 1 << a][a] > most) most = save[a][b] + left[set | 1 << a][a];
                left[set][b] = (signed char)most;
            }
    }
    // cur[n ..] is placed; goes on to every walk that saves `most` more.  Walks fall into runs of rows that carry into one
    // another, whose order does not matter: `tail`, the last row of the run that cur[n] begins or belongs to, rises from run to run
    void go(int n, int set, int most, int tail)
    {
        if (n == 0) {
            double v = 0.0, extra = 0.0;
            for (int i = 0; i < R; ++i) {
                const double c = i ? ratio[cur[i - 1]][cur[i]] : 0.0, c2v = c * c * v;
                v = size[cur[i]] + c2v;
                extra += norm2[cur[i]] * c2v;
            }
            if (extra >= 0.67 * best_extra) return;
            best_extra = extra;
            memcpy(best, cur, sizeof(best));
            return;
        }
        for (int r = 0; r < R; ++r) {
            const int saved = n < R ? save[r][cur[n]] : 0;
            if (set >> r & 1 || saved + left[set | 1 << r][r] < most || (saved == 0 && r < tail)) continue;
            cur[n - 1] = r;
            go(n - 1, set | 1 << r, most - saved, saved ? tail : r);
        }
    }
};

static inline void fmm_choose_walk(int R, const float (*U)[4], const float (*V)[4], const float (*W)[4], int* order, float* carry)
{
    auto square = [](const float (&x)[4]) { return (double)x[0] * x[0] + (double)x[1] * x[1] + (double)x[2] * x[2] + (double)x[3] * x[3]; };
    FmmWalkSearch s;
    s.R = R; s.best_extra = HUGE_VAL;
    for (int a = 0; a < R; ++a) {
        s.norm2[a] = square(W[a]); s.size[a] = square(U[a]) * square(V[a]);
        for (int b = 0; b < R; ++b) {
            s.save[a][b] = 0; s.ratio[a][b] = 0.0f;
            bool nested = a != b;
            for (int q = 0; q < 4; ++q) nested = nested && (W[b][q] == 0.0f || W[a][q] != 0.0f);
            for (int q = 0; q < 4 && nested; ++q) {
                if (W[a][q] == 0.0f || W[b][q] == 0.0f) continue;
                const float c = W[a][q] / W[b][q];
                if (!(fabsf(c) <= 1.000001f)) continue;            // 1, but for the rounding of the coefficients
                int n = 0;
                for (int k = 0; k < 4; ++k) n += (W[a][k] != 0.0f) - (fmm_emitted_weight(W[a][k], c, W[b][k]) != 0.0f);
                if (n > s.save[a][b] || (n == s.save[a][b] && n > 0 && fabsf(c) < fabsf(s.ratio[a][b]))) { s.save[a][b] = n; s.ratio[a][b] = c; }
            }
        }
    }
    s.bound();
    int most = 0;
    for (int r = 0; r < R; ++r) if (s.left[1 << r][r] > most) most = s.left[1 << r][r];
    s.go(R, 0, most, -1);
    for (int i = 0; i < R; ++i) {
        order[i] = s.best[i];
        carry[i] = i ? s.ratio[order[i - 1]][order[i]] : 0.0f;
    }
}
