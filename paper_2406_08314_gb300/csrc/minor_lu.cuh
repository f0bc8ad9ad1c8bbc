// The LU of one excitation string's minor, and its inverse.
#pragma once

#include "common.cuh"

// sign * det A of the K x K block A[i][j] = g(i, j) by an LU with partial pivoting (by the
// larger of |Re|, |Im|) in FP64; B (may be NULL): A^-1 from its factors, K K entries (B[i][j]
// at i K + j) and the pad entry of b_stride(K). Zero pivots: determinant 0, finite B.
//
// FP64 issue rate is the bound here (a few FP64 operations per clock per SM), so the LU
// spends FP64 operations on the elimination and the determinant only: the pivot search
// compares integer magnitude keys, the row swaps count parity in an integer, and the pivot
// reciprocals are Newton-Raphson iterations from an FP32 seed.
template <int K, class G>
__device__ __forceinline__ double2 minor_lu(double sign, G g, double2* __restrict__ B)
{
    double2 a[K][K];
#pragma unroll
    for (int i = 0; i < K; ++i)
#pragma unroll
        for (int j = 0; j < K; ++j) a[i][j] = g(i, j);
    int perm[K];
#pragma unroll
    for (int i = 0; i < K; ++i) perm[i] = i;
    double2 det = cz(sign, 0);
    double2 dinv[K];
    bool sing = false;
    int odd = 0;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        int p = k, best = mag_key(a[k][k]);
        double2 pv = a[k][k];
#pragma unroll
        for (int i = k + 1; i < K; ++i) {
            const int v = mag_key(a[i][k]);
            if (v > best) { best = v; p = i; pv = a[i][k]; }
        }
        if (pv.x == 0.0 && pv.y == 0.0) sing = true;
#pragma unroll
        for (int i = k + 1; i < K; ++i) {
            if (i == p) {
#pragma unroll
                for (int j = 0; j < K; ++j) { double2 tt = a[k][j]; a[k][j] = a[i][j]; a[i][j] = tt; }
                int tp = perm[k]; perm[k] = perm[i]; perm[i] = tp;
                odd ^= 1;
            }
        }
        det = cmul(det, a[k][k]);
        dinv[k] = sing ? cz(0, 0) : crecip(a[k][k]);
        if (k + 1 < K) {
#pragma unroll
            for (int i = k + 1; i < K; ++i) {
                const double2 f = cmul(a[i][k], dinv[k]);
                a[i][k] = f;
#pragma unroll
                for (int j = k + 1; j < K; ++j) a[i][j] = cfms(f, a[k][j], a[i][j]);
            }
        }
    }
    if (odd) det = cz(-det.x, -det.y);
    if (sing) det = cz(0, 0);
    if (!B) return det;
    // B = A^-1 from P A = L U: column c solves L U x = P e_c
    if (K & 1) B[K * K] = cz(0, 0);   // the pad entry
#pragma unroll
    for (int c = 0; c < K; ++c) {
        double2 x[K];
#pragma unroll
        for (int i = 0; i < K; ++i) x[i] = cz(perm[i] == c ? 1 : 0, 0);
#pragma unroll
        for (int i = 0; i < K; ++i)
#pragma unroll
            for (int k = 0; k < i; ++k) x[i] = cfms(a[i][k], x[k], x[i]);
#pragma unroll
        for (int i = K - 1; i >= 0; --i) {
#pragma unroll
            for (int k = i + 1; k < K; ++k) x[i] = cfms(a[i][k], x[k], x[i]);
            x[i] = cmul(x[i], dinv[i]);
        }
#pragma unroll
        for (int i = 0; i < K; ++i) B[i * K + c] = x[i];
    }
    return det;
}
