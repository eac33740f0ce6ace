// roks_chol.cuh -- Cholesky inverse of a small Hermitian matrix by one block,
// in shared memory, FP64 (internal).
#pragma once

#include "roks_impl.cuh"

namespace roks {

// L (n x n, column major, lower triangle of O on entry) becomes its Cholesky
// factor and X (zero on entry) the factor's inverse, both lower triangles;
// dinv: n values of scratch.  Returns 0, or 1 + the first column whose pivot
// is not positive (the column then goes on with a pivot of 1), to every thread.
//
// Bound by the chain of pivots for a few bands and by the SM's FP64 pipe (two
// multiply-adds a cycle) from some 30 on.  So factor and inverse advance
// together, right-looking: with column j final, one barrier step scales it
// and row j of X, the next updates all that lies below, elements spread over
// all lanes (predicated lanes would cost as much), and the thread that
// finishes element (j + 1, j + 1) takes its root and reciprocal at once.
template <int NT>
__device__ int chol_inverse_block(int n, double2* L, double2* X, double* dinv) {
    __shared__ int bad;
    const int tid = threadIdx.x;
    auto pivot = [&](int j, double d) {
        if (!(d > 0.0)) {
            if (!bad) bad = j + 1;
            d = 1.0;
        }
        const double piv = sqrt(d);
        L[j * n + j] = make_double2(piv, 0.0);
        dinv[j] = 1.0 / piv;
    };
    if (tid == 0) {
        bad = 0;
        pivot(0, L[0].x);
    }
    __syncthreads();
    for (int j = 0; j < n; ++j) {
        const int m = n - j - 1;
        // column j below the diagonal, row j of X
        for (int t = tid; t < n; t += NT) {
            const double inv = dinv[j];
            if (t > j) {
                const double2 v = L[j * n + t];
                L[j * n + t] = make_double2(v.x * inv, v.y * inv);
            } else {
                const double2 v = t == j ? make_double2(1.0, 0.0) : X[t * n + j];
                X[t * n + j] = make_double2(v.x * inv, v.y * inv);
            }
        }
        __syncthreads();
        // A_ik -= L_ij conj(L_kj), j < k <= i; then X_ic -= L_ij X_jc, c <= j
        const int tri = m * (m + 1) / 2, all = tri + m * (j + 1);
        for (int t = tid; t < all; t += NT) {
            double2 a, b, *c;
            int i, k = 0;
            if (t < tri) {
                i = (int)((sqrtf(8.f * t + 1.f) - 1.f) * 0.5f);
                i += (i + 1) * (i + 2) / 2 <= t;
                i -= i * (i + 1) / 2 > t;
                k = t - i * (i + 1) / 2;
                a = L[j * n + j + 1 + i];
                b = L[j * n + j + 1 + k];
                b.y = -b.y;
                c = L + (j + 1 + k) * n + j + 1 + i;
            } else {
                const int u = t - tri, col = u / m;
                i = u - col * m;
                a = L[j * n + j + 1 + i];
                b = X[col * n + j];
                c = X + col * n + j + 1 + i;
            }
            double2 v = *c;
            v.x -= a.x * b.x - a.y * b.y;
            v.y -= a.x * b.y + a.y * b.x;
            if (t == 0) pivot(j + 1, v.x);   // (i = k = 0: element (j + 1, j + 1))
            else *c = v;
        }
        __syncthreads();
    }
    return bad;
}

}  // namespace roks
