// Small dense algebra of the compact limited-memory BFGS representation
// (Byrd, Nocedal & Schnabel, Math. Prog. 63, 1994):
//     H = gamma I + [S  gamma Y] M [S^T; gamma Y^T],
//     M = [[R^-T (D + gamma Y^T Y) R^-1, -R^-T], [-R^-1, 0]],
// with S, Y the n x k matrices of the stored pairs (oldest first),
// R_ij = s_i^T y_j (i <= j, upper triangle of S^T Y), D = diag(s_i^T y_i).
// Given u = S^T g and v = Y^T g, H g = gamma g + S p - gamma Y t with
//     t = R^-1 u,   p = R^-T ((D + gamma Y^T Y) t - gamma v).
// Plain C++ usable from host and device code (k <= kLbfgsMax).
#pragma once

#if defined(__CUDACC__)
#define NN_HD __host__ __device__
#else
#define NN_HD
#endif

namespace nnqp {

constexpr int kLbfgsMax = 16;

// SY[i][j] = s_i^T y_j, YY[i][j] = y_i^T y_j (k x k, row stride kLbfgsMax).
// Outputs coefficients cs[k] (of S) and cy[k] (of Y) such that
// H g = gamma g + sum_j cs[j] s_j + sum_j cy[j] y_j.  Returns false if R is
// singular (then the caller falls back to a gradient step).
NN_HD inline bool lbfgs_coefficients(int k, const double *SY, const double *YY, const double *u,
                                     const double *v, double gamma, double *cs, double *cy) {
    double t[kLbfgsMax], w[kLbfgsMax], rinv[kLbfgsMax];
    // reciprocals of R's diagonal first: k independent divisions instead of
    // one division on every step of both substitution chains
    for (int i = 0; i < k; ++i) {
        const double rii = SY[i * kLbfgsMax + i];
        if (!(rii > 0.0)) return false;
        rinv[i] = 1.0 / rii;
    }
    // back substitution R t = u, R upper triangular with R_ij = SY[i][j]
    for (int i = k - 1; i >= 0; --i) {
        double s = u[i];
        for (int j = i + 1; j < k; ++j) s -= SY[i * kLbfgsMax + j] * t[j];
        t[i] = s * rinv[i];
    }
    // w = (D + gamma Y^T Y) t - gamma v
    for (int i = 0; i < k; ++i) {
        double s = SY[i * kLbfgsMax + i] * t[i] - gamma * v[i];
        for (int j = 0; j < k; ++j) s += gamma * YY[i * kLbfgsMax + j] * t[j];
        w[i] = s;
    }
    // forward substitution R^T p = w
    for (int i = 0; i < k; ++i) {
        double s = w[i];
        for (int j = 0; j < i; ++j) s -= SY[j * kLbfgsMax + i] * cs[j];
        cs[i] = s * rinv[i];
    }
    for (int i = 0; i < k; ++i) cy[i] = -gamma * t[i];
    return true;
}

#if defined(__CUDACC__)
// The same by one warp, lane i for row i (every lane calls it; u, v: the lane's
// entries).  One thread took some 9,000 cycles for k = 5, an FP64 operation being
// 64; here the divisions and the rows of w go side by side and a substitution
// step is one multiplication, one broadcast and one multiply-add.
__device__ inline bool lbfgs_coefficients_warp(int k, const double *SY, const double *YY, double u, double v,
                                               double gamma, double *cs, double *cy) {
    const unsigned all = 0xffffffffu;
    const int i = threadIdx.x & 31;
    const bool in = i < k;
    const double rii = in ? SY[i * kLbfgsMax + i] : 1.0;
    if (!__all_sync(all, rii > 0.0)) return false;
    const double rinv = 1.0 / rii;
    double s = in ? u : 0.0, t = 0.0;
    for (int j = k - 1; j >= 0; --j) {       // R t = u
        const double tj = __shfl_sync(all, s * rinv, j);
        if (i == j) t = tj;
        if (i < j) s -= SY[i * kLbfgsMax + j] * tj;
    }
    double w = in ? rii * t - gamma * v : 0.0;   // w = (D + gamma Y^T Y) t - gamma v
    for (int j = 0; j < k; ++j) {
        const double tj = __shfl_sync(all, t, j);
        if (in) w += gamma * YY[i * kLbfgsMax + j] * tj;
    }
    for (int j = 0; j < k; ++j) {            // R^T p = w
        const double pj = __shfl_sync(all, w * rinv, j);
        if (i == j) cs[j] = pj;
        if (in && i > j) w -= SY[j * kLbfgsMax + i] * pj;
    }
    if (in) cy[i] = -gamma * t;
    return true;
}
#endif

}  // namespace nnqp
