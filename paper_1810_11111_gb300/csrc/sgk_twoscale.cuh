// Two-scale (pyramid) steps between a cell and its halves, shared by the
// transforms along one direction (fiber.cu) and the fused pass
// (sgk_pencil.cuh).
//
// The two halves of a cell mirror each other, so the filters of the right
// child are those of the left one up to the sign (-1)^{r+s} (wavelets:
// (-1)^{p+k+1+s}): with A the sum of the terms of equal sign and B that of
// the others, the children are A + B and A - B, and transposed the parent
// comes from the sum and the difference of the children.  H is triangular (a
// degree-r polynomial has degree r on the halves); against constants the even
// degrees above 0 vanish (their mean over a half is that over the cell) and so
// do the even wavelets (their mean is 0).  At k = 2 that leaves 13
// multiply-adds and 6 additions per parent and fiber instead of 36
// multiply-adds, 168 FP32 operations instead of 432 in double-float.
#pragma once
#include "sgk_lanes.h"

namespace sgk_ts {

using namespace lanes;

// Left-half two-scale filters: H[r][s] = <phi_r, phi^0_s>, G[p][s] =
// <psi_p, phi^0_s> (parent Legendre and wavelet against the child's basis).
template <typename T, int K>
struct Filt {
    Cst<T> H[K][K];
    Cst<T> G[K][K];
};
// terms that are not zero by structure, and whether the right half has the
// same sign
__host__ __device__ constexpr bool h_term(int r, int s) { return r >= s && !(s == 0 && r > 0 && r % 2 == 0); }
__host__ __device__ constexpr bool g_term(int k1, int p, int s) { return !(s == 0 && (p + k1) % 2 == 0); }
__host__ __device__ constexpr bool h_even(int r, int s) { return (r + s) % 2 == 0; }
__host__ __device__ constexpr bool g_even(int k1, int p, int s) { return (p + k1 + s) % 2 == 0; }

// two_scale: [H_0, H_1, G_0, G_1], each K x K (Tables1D::two_scale)
template <typename T, int K>
Filt<T, K> make_filt(const double* two_scale) {
    Filt<T, K> F{};
    for (int r = 0; r < K; ++r)
        for (int s = 0; s < K; ++s) {
            cst_set(F.H[r][s], two_scale[r * K + s]);
            cst_set(F.G[r][s], two_scale[2 * K * K + r * K + s]);
        }
    return F;
}

// One two-scale step down: A and B of a parent with scaling coefficients p
// and details d; its children are A + B (left) and A - B (right).
template <typename T, int K>
__device__ __forceinline__ void split_node(const T (&p)[K], const T (&d)[K], const Filt<T, K>& F, T (&A)[K],
                                           T (&B)[K]) {
#pragma unroll
    for (int s = 0; s < K; ++s) {
        bool a0 = true, b0 = true;
        A[s] = zero<T>();
        B[s] = zero<T>();
#pragma unroll
        for (int r = 0; r < K; ++r)
            if (h_term(r, s)) {
                if (h_even(r, s)) {
                    A[s] = a0 ? mulc(F.H[r][s], p[r]) : maddc(F.H[r][s], p[r], A[s]);
                    a0 = false;
                } else {
                    B[s] = b0 ? mulc(F.H[r][s], p[r]) : maddc(F.H[r][s], p[r], B[s]);
                    b0 = false;
                }
            }
#pragma unroll
        for (int q = 0; q < K; ++q)
            if (g_term(K, q, s)) {
                if (g_even(K, q, s)) {
                    A[s] = a0 ? mulc(F.G[q][s], d[q]) : maddc(F.G[q][s], d[q], A[s]);
                    a0 = false;
                } else {
                    B[s] = b0 ? mulc(F.G[q][s], d[q]) : maddc(F.G[q][s], d[q], B[s]);
                    b0 = false;
                }
            }
    }
}

// The transposed step: scaling coefficients p and details d of the parent
// from the sum x0 + x1 and the difference x0 - x1 of its children.
template <typename T, int K>
__device__ __forceinline__ void merge_node(const T (&sum)[K], const T (&dif)[K], const Filt<T, K>& F, T (&p)[K],
                                           T (&d)[K]) {
#pragma unroll
    for (int r = 0; r < K; ++r) {
        bool p0 = true, d0 = true;
        p[r] = zero<T>();
        d[r] = zero<T>();
#pragma unroll
        for (int s = 0; s < K; ++s) {
            if (h_term(r, s)) {
                const T x = h_even(r, s) ? sum[s] : dif[s];
                p[r] = p0 ? mulc(F.H[r][s], x) : maddc(F.H[r][s], x, p[r]);
                p0 = false;
            }
            if (g_term(K, r, s)) {
                const T x = g_even(K, r, s) ? sum[s] : dif[s];
                d[r] = d0 ? mulc(F.G[r][s], x) : maddc(F.G[r][s], x, d[r]);
                d0 = false;
            }
        }
    }
}

}  // namespace sgk_ts
