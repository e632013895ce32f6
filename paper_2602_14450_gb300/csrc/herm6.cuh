// Inverses of the Hermitian 6 x 6 blocks of the clover term (clover.cu), stored as 36 reals: the diagonal, then the
// upper triangle row by row, (re, im).
#pragma once

#include <math.h>

#ifdef __CUDACC__
#define WD_NOINLINE __noinline__
#else
#define WD_NOINLINE
#define __host__
#define __device__
#define __forceinline__ inline
#endif

namespace wd {
namespace herm6 {

// Inverse of a Hermitian 6 x 6 block by Gauss-Jordan with partial pivoting; false when a pivot vanishes. For
// the blocks that are not positive definite, or nearly singular (a large c_sw).
__host__ __device__ WD_NOINLINE bool invert_pivoted(const double* S, double* out) {
    double a[6][12], inv[6][12];
    for (int i = 0; i < 6; ++i)
        for (int j = 0; j < 6; ++j) {
            const int lo = i < j ? i : j, hi = i < j ? j : i;
            const int q = 6 + 2 * (lo * 5 - lo * (lo - 1) / 2 + hi - lo - 1);
            a[i][2 * j] = i == j ? S[i] : S[q];
            a[i][2 * j + 1] = i == j ? 0.0 : i < j ? S[q + 1] : -S[q + 1];
            inv[i][2 * j] = i == j ? 1.0 : 0.0;
            inv[i][2 * j + 1] = 0.0;
        }
    for (int col = 0; col < 6; ++col) {
        int piv = col;
        double best = -1.0;
        for (int i = col; i < 6; ++i) {
            const double m = a[i][2 * col] * a[i][2 * col] + a[i][2 * col + 1] * a[i][2 * col + 1];
            if (m > best) { best = m; piv = i; }
        }
        if (!(best > 0.0)) return false;
        for (int j = 0; j < 12 && piv != col; ++j) {
            double t = a[col][j]; a[col][j] = a[piv][j]; a[piv][j] = t;
            t = inv[col][j]; inv[col][j] = inv[piv][j]; inv[piv][j] = t;
        }
        const double dr = a[col][2 * col] / best, di = -a[col][2 * col + 1] / best;   // 1 / pivot
        for (int j = 0; j < 6; ++j) {
            double r = a[col][2 * j], i = a[col][2 * j + 1];
            a[col][2 * j] = r * dr - i * di;
            a[col][2 * j + 1] = r * di + i * dr;
            r = inv[col][2 * j];
            i = inv[col][2 * j + 1];
            inv[col][2 * j] = r * dr - i * di;
            inv[col][2 * j + 1] = r * di + i * dr;
        }
        for (int i = 0; i < 6; ++i) {
            if (i == col) continue;
            const double fr = a[i][2 * col], fi = a[i][2 * col + 1];
            for (int j = 0; j < 6; ++j) {
                a[i][2 * j] -= fr * a[col][2 * j] - fi * a[col][2 * j + 1];
                a[i][2 * j + 1] -= fr * a[col][2 * j + 1] + fi * a[col][2 * j];
                inv[i][2 * j] -= fr * inv[col][2 * j] - fi * inv[col][2 * j + 1];
                inv[i][2 * j + 1] -= fr * inv[col][2 * j + 1] + fi * inv[col][2 * j];
            }
        }
    }
    for (int i = 0, q = 6; i < 6; ++i) {
        out[i] = inv[i][2 * i];
        for (int j = i + 1; j < 6; ++j, q += 2) {
            out[q] = inv[i][2 * j];
            out[q + 1] = inv[i][2 * j + 1];
        }
    }
    return true;
}

// Element (i, j), i != j, of a Hermitian matrix stored as 6 reals and the upper triangle (row by row).
__host__ __device__ constexpr int tri(int i, int j) { return 6 + 2 * (i * 5 - i * (i - 1) / 2 + j - i - 1); }
__host__ __device__ __forceinline__ void element(const double (&s)[36], int i, int j, double& re, double& im) {
    re = s[i < j ? tri(i, j) : tri(j, i)];
    im = i < j ? s[tri(i, j) + 1] : -s[tri(j, i) + 1];
}

// s := s^-1 for a Hermitian 6 x 6 block by the sweep operator (each sweep keeps the matrix Hermitian, so only the
// triangle is held; after all six it is -s^-1). Pivots are not exchanged; false unless all are positive and at least
// 1e-3 of the block's scale 1/2 (the trace of the block is 3). Positive pivots make the block positive definite, whose
// elimination grows no element: over random blocks of up to 1e3 in condition the errors are those of the elimination
// with exchanged pivots, 3e-16 times the condition number (pivots of either sign, 5e-13 times).
__host__ __device__ __forceinline__ bool sweep_inverse(double (&s)[36]) {
    bool good = true;
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        good = good && s[k] > 5e-4;
        const double rd = 1.0 / s[k];
        double cr[6], ci[6];   // column k
#pragma unroll
        for (int i = 0; i < 6; ++i)
            if (i != k) element(s, i, k, cr[i], ci[i]);
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            if (i == k) continue;
            const double br = cr[i] * rd, bi = ci[i] * rd;   // s_ik / s_kk
            s[i] = fma(-br, cr[i], fma(-bi, ci[i], s[i]));
#pragma unroll
            for (int j = i + 1; j < 6; ++j) {
                if (j == k) continue;                        // s_ij -= s_ik conj(s_jk) / s_kk
                s[tri(i, j)] = fma(-br, cr[j], fma(-bi, ci[j], s[tri(i, j)]));
                s[tri(i, j) + 1] = fma(-bi, cr[j], fma(br, ci[j], s[tri(i, j) + 1]));
            }
            if (i < k) {
                s[tri(i, k)] = br;
                s[tri(i, k) + 1] = bi;
            } else {
                s[tri(k, i)] = br;
                s[tri(k, i) + 1] = -bi;
            }
        }
        s[k] = -rd;
    }
#pragma unroll
    for (int i = 0; i < 36; ++i) s[i] = -s[i];
    return good;
}

}  // namespace herm6
}  // namespace wd
