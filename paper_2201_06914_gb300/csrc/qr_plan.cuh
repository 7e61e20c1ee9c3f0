// Which cluster size the thin QR of the range finder takes (cgs2_qr_kernel, range_finder.cu).
// Host code without device types, so that the rule is tested on the CPU (tests/test_qr_plan.py).
#pragma once

#include <cstddef>

namespace wp {

constexpr int QR_THREADS = 512;
constexpr int QR_MAXR = 512;
constexpr int QR_MAXC = 8;                    // portable cluster size
constexpr size_t QR_SMEM = 227 * 1024;

// Dynamic shared memory before the CTA's rows: partial dot products of two steps, coefficients,
// reciprocal squared norms, per-thread partial sums.
constexpr size_t QR_HEAD = (size_t)(2 * (QR_MAXR + 1) + 2 * QR_MAXR + QR_THREADS) * sizeof(double);

// Dynamic shared memory of a CTA whose rows lie there (clusters of c), or 0 if they do not fit.
inline size_t qr_rows_smem(int nt, int r, int c)
{
    const size_t rows = ((size_t)nt + c - 1) / c;
    const size_t need = QR_HEAD + (rows | 1) * r * sizeof(double);
    return need <= QR_SMEM ? need : 0;
}

// CTAs per shot.  The FP64 multiply-adds of a shot are shared by c CTAs; nshots clusters run in
// rounds of fit(c, smem), the clusters resident at once.  With the rows in shared memory an SM counts
// for one CTA, whatever its memory holds: two share the SM's FP64 units, so a second CTA costs what
// a second round does.  With the rows in global memory a CTA waits for its loads most of the time:
// twice the time a product, and every resident CTA counts.  The two barriers a column are not in
// the rule: clusters of two and more were never slower than one CTA for the shots that fit in a round.
// Measured for nt 300 .. 4000, r 2 .. 256, 1 .. 64 shots: within 0.4 % of the best size on average,
// 8 % at most; 7 % and 57 % with the former rule, which charged 2500 cycles a barrier, took the
// global-memory form for free and counted co-resident CTAs as parallel (2000 x 96, 16 shots: 3.61 ms
// in clusters of 8, 4.87 in the clusters of 7 it took; 1000 x 4, one shot 90 us in clusters of 8,
// 137 with the one CTA it took).
template <class Fit>
inline int qr_cluster(int nt, int r, int nshots, Fit fit)
{
    int best = 1;
    double cost = 1e300;
    for (int c = 1; c <= QR_MAXC; c++) {
        const bool smem = qr_rows_smem(nt, r, c) > 0;
        const int n = fit(c, smem);
        if (n < 1) continue;
        const double t = (double)((nshots + n - 1) / n) * (smem ? 1.0 : 2.0) / c;
        if (t < cost) {
            cost = t;
            best = c;
        }
    }
    return best;
}

}  // namespace wp
