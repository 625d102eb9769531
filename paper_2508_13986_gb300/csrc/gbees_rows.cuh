// The rows of an initial Gaussian's box in single precision: whether a cell is in the
// set p > pstar, or too near the limit to tell. Pure functions that the device code uses
// and that a host compiler can build too (the host tests compare them with FP64 over
// scales, origins and shapes of the prior).
//
// Everything is in units of the cells: distances from the mean divided by the widths,
// the inverse covariance times the widths of its row and column. Distances are below
// 2^33 then, so that entries below single precision's normal range (2^-126), flushed or
// rounded coarsely, move the quadratic form by less than 36 2^-126 2^66 < 1e-16 whatever
// the prior's scale; one that overflows gives an infinite bound or no number: FP64 decides.
#pragma once

#include <math.h>

#if defined(__CUDACC__)
#define GBEES_ROWS_HD __host__ __device__ __forceinline__
#else
#define GBEES_ROWS_HD inline
#endif

namespace gbees {

// The smallest pstar that the rows may decide on: below 2^-1022 a density loses bits,
// and -2 ln pstar no longer tells which densities exceed pstar. With an infinite limit
// nothing is decided (FP64 decides on every cell).
constexpr double ROWS_MIN_PSTAR = 1e-290;

// Rounding of the cells' centres along an axis, in cells. A distance from the mean
// fl(fl(x0 + fl(i h)) - mean), |mean| about |x0 + i h|, is off by at most 4 2^-53 W, W =
// |x0| + max |i| h, and so is another of the same row: their difference (and that of
// two evaluations, one with a fused multiply-add) by at most 2^-50 W.
GBEES_ROWS_HD double centre_slack(double x0, double h, double max_abs_i) {
    return 8.8817841970012523e-16 * (fabs(x0) / h + max_abs_i);  // 2^-50
}

// An upper bound of the quadratic form at a cell whose distances from the mean are dx
// (in cells) up to slack.
inline double form_above(int n, const double* icov, const double* h, const double* dx, const double* slack) {
    double q = 0.0, e = 0.0;
    for (int a = 0; a < n; ++a)
        for (int c = 0; c < n; ++c) {
            const double w = icov[a * n + c] * h[a] * h[c];
            q += dx[a] * w * dx[c];
            e += fabs(w) * (fabs(dx[a]) * slack[c] + slack[a] * fabs(dx[c]) + slack[a] * slack[c]);
        }
    return q + e;
}

struct InitRow {
    float A, B, C;   // q = A + B dx + C dx^2
    float Aa, Ba;    // the same sums of absolute values
    float dx0, err;  // dx of the row's first cell, error bound of a cell's dx
};

// dx: distances of the row's first cell from the mean; w: the inverse covariance (both
// in cells); len: cells of the row; slack: of the last dimension.
template <int N>
GBEES_ROWS_HD InitRow row_form(const float* dx, const float* w, float len, float slack) {
    InitRow r;
    r.A = r.Aa = r.B = r.Ba = 0.0f;
#pragma unroll
    for (int a = 0; a < N - 1; ++a) {
#pragma unroll
        for (int c = 0; c < N - 1; ++c) {
            const float t = dx[a] * w[a * N + c] * dx[c];
            r.A += t;
            r.Aa += fabsf(t);
        }
        const float t = dx[a] * (w[a * N + N - 1] + w[(N - 1) * N + a]);
        r.B += t;
        r.Ba += fabsf(t);
    }
    r.C = w[N * N - 1];
    r.dx0 = dx[N - 1];
    // dx of a cell of the row as dx0 + i: the roundings of dx0 and of the sum, and the
    // centres'
    r.err = 5e-7f * (fabsf(r.dx0) + len) + 1.01f * slack;
    return r;
}

// q of cell i of the row and a bound of its error: fewer than 64 roundings of
// relative size 2^-24 on sums of absolute value S (1e-5 is 2.5 times that), and
// the error of dx.
GBEES_ROWS_HD float row_q(const InitRow& r, int i, float& e) {
    const float dx = r.dx0 + (float)i, ad = fabsf(dx);
    e = 1e-5f * (r.Aa + (r.Ba + r.C * ad) * ad) + (r.Ba + 2.0f * r.C * (ad + r.err)) * r.err + 1e-6f;
    return r.A + (r.B + r.C * dx) * dx;
}

// q of cell i less the limit qlim (rounded to float), and a bound of its error: above
// the limit when d > e, below it when d < -e, else too near it (or not a number).
GBEES_ROWS_HD float row_gap(const InitRow& r, int i, float qlim, float& e) {
    const float q = row_q(r, i, e);
    e += 1e-6f * fabsf(qlim);
    return q - qlim;
}

}  // namespace gbees
