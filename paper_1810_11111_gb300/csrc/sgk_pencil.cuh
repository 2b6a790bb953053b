// Fused last-direction pass of the reaction term (Section 4: reconstruction
// at the finest-mesh Gauss points and quadrature): device code and launch
// templates; pencil_<type>_d<d>.cu instantiate them, pencil.cu dispatches.
//
// After directions 0..d-2 have been changed to the finest-cell Legendre basis
// (fiber engine), direction d-1 still holds 1D hierarchical coefficients.
// A pencil is a fixed finest cell in directions 0..d-2, i.e. the (k+1)^{d-1}
// fibers of that cell's Legendre degrees, each of length H = (k+1) 2^N along
// direction d-1.  A CTA takes a few pencils at a time; in shared memory it
//   1. reconstructs each fiber in the finest-cell Legendre basis with the
//      two-scale relations (subtrees of up to 3 levels expanded in registers,
//      one barrier per stage and set);
//   2. runs the cell quadrature: Legendre -> q^d Gauss points -> f(u) or
//      f'(u) w -> Legendre moments, as nested sum-factorised loops whose
//      indices are compile-time constants; f and f' are polynomials evaluated
//      by Horner's rule;
//   3. decomposes the moments back to hierarchical coefficients with the
//      transposed two-scale relations (subtrees of up to 3 levels reduced in
//      registers, one barrier per 3 levels) and stores them.
// Specialised for (d, k+1, q, species); other shapes use the unfused path.
//
// The operation count is what bounds the pass (FP64: one warp instruction per
// 64 clocks and scheduler; double-float: 12 FP32 operations per
// multiply-add), so both parts use every symmetry of their tables:
//   * the Gauss points are symmetric and P_r(-x) = (-1)^r P_r(x): the values
//     at a pair of points are E + O and E - O of the even and odd partial
//     sums, the moments come from the sum and the difference of the pair;
//   * the basis is scaled to P_0 = 1 (h^{-d/2} goes into the coefficients of
//     f) and the weights into the table of the moments: no multiplications
//     by either at the points;
//   * the two-scale steps share their terms between the children
//     (sgk_twoscale.cuh).
// Multiply-adds per finest cell at d = 3, k = 2, q = 5: quadrature 1470 ->
// 931, transforms 648 -> 360 additions and multiply-adds.
//
// Lanes: with a packed element type (sgk_lanes.h) a thread works on two
// cells, c and c + 2^{N-1}: the two halves of the pencil, so the subtrees and
// cells of the lanes pair up at every level above the first split.  A shared
// memory slot holds both lanes; the coefficients of levels 0 and 1, which
// belong to the whole pencil, are stored in both.
#pragma once
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "sgk_pencil.h"
#include "sgk_twoscale.cuh"

namespace sgk_pen {

using namespace lanes;
using namespace sgk_ts;

template <int B, int E>
struct Pow {
    static constexpr int v = B * Pow<B, E - 1>::v;
};
template <int B>
struct Pow<B, 0> {
    static constexpr int v = 1;
};

constexpr int PDEG = 5;  // exponents 0..4 per species
// levels of a subtree expanded or reduced in registers: 8 cells, in
// double-float 4 (8 cells of 4 registers a value spill at the register cap)
template <typename T>
constexpr int PD = std::is_same<T, df2>::value ? 2 : 3;
constexpr int QMAX = 8;  // Gauss points per direction

// Gauss tables of the scaled basis sqrt(2r+1) P_r: point 0 is the middle one
// for odd q, then pairs (+xi_g, -xi_g).  B, WB: positive point of pair g (the
// middle point last, index q / 2), WB with the weight h w_g / 2 folded in;
// TB, TWB: all q points in that order, signed.
template <typename T, int K, int Q>
struct QuadTab {
    Cst<T> B[(Q + 1) / 2][K], WB[(Q + 1) / 2][K];
    Cst<T> TB[Q][K], TWB[Q][K];
};

// Polynomials of the reaction, dense with bit masks of the non-zero
// coefficients: F passes hold f_s, Jacobian passes the derivatives d f_s / d
// u_r (index s S + r).  One species: c[e] u^e; two: c[a 5 + b] u^a v^b, mask[a]
// the bits of b and rows the bits of a.
template <typename T, int S, int NP>
struct Poly {
    Cst<T> c[NP][Pow<PDEG, S>::v];
    unsigned char rows[NP], mask[NP][PDEG], monic;
};

// The largest total degree of f whose pass has q points at k + 1 = K: q =
// ceil((p k + k + 1) / 2).
__host__ __device__ constexpr int max_degree(int K, int Q) { return (2 * Q - K) / (K - 1); }

// One species in FP64: the polynomial is divided by its leading coefficient,
// which goes into the outermost table of the moments (one multiplication less
// at every point: -c u^3 takes two), where that stays in range: with a leading
// coefficient of at least 1 no bare power overflows where the term does not,
// below 2^128 it underflows only where the term does by 2^-894, and the other
// coefficients keep their digits in the quotients (Poly::monic).  Not in the
// narrower types, whose range would not hold the bare powers of a decayed
// state.
template <typename T, int S>
constexpr bool MONIC = std::is_same<T, double>::value && S == 1;

// Horner's rule over total degree <= PM.  FP64 and double-float skip the zero
// coefficients (the reactions are sparse polynomials, e.g. -c u^3; the tests
// are uniform over the grid and cheaper than the multiply-adds); in FP32 a
// multiply-add is cheaper than a test.
template <typename T, int PM, int NP>
__device__ __forceinline__ T poly_value(const Poly<T, 1, NP>& P, int i, const T (&u)[1]) {
    constexpr bool SKIP = !std::is_same<T, float>::value;
    T f = zero<T>();
    int state = 0;  // 0 above the leading term, 1 at it (monic: f stands for 1), 2 below
#pragma unroll
    for (int e = PM < PDEG ? PM : PDEG - 1; e >= 0; --e) {
        if (state == 2) {
            f = mul(f, u[0]);
        } else if (state == 1) {
            f = u[0];
            state = 2;
        }
        if (!SKIP || ((P.rows[i] >> e) & 1)) {
            if (state == 0) {
                f = cvalue(P.c[i][e]);
                state = MONIC<T, 1> && P.monic ? 1 : 2;
            } else {
                f = add(f, cvalue(P.c[i][e]));
            }
        }
    }
    return f;
}
template <typename T, int PM, int NP>
__device__ __forceinline__ T poly_value(const Poly<T, 2, NP>& P, int i, const T (&u)[2]) {
    constexpr bool SKIP = !std::is_same<T, float>::value;
    T f = zero<T>();
    bool started = false;
#pragma unroll
    for (int a = PM < PDEG ? PM : PDEG - 1; a >= 0; --a) {
        if (started) f = mul(f, u[0]);
        if (!SKIP || ((P.rows[i] >> a) & 1)) {
            T g = zero<T>();
            bool gst = false;
#pragma unroll
            for (int b = PM - a < PDEG ? PM - a : PDEG - 1; b >= 0; --b) {
                if (gst) g = mul(g, u[1]);
                if (!SKIP || ((P.mask[i][a] >> b) & 1)) {
                    const T c = cvalue(P.c[i][a * PDEG + b]);
                    g = gst ? add(g, c) : c;
                    gst = true;
                }
            }
            f = started ? add(f, g) : g;
            started = true;
        }
    }
    return f;
}

template <typename T, int PM, int S, bool JAC>
struct PointEval {
    static constexpr int NP = JAC ? S * S : S;
    __device__ __forceinline__ static void run(const Poly<T, S, NP>& P, const T (&u)[S], const T (&w)[S], T (&o)[S]) {
#pragma unroll
        for (int s = 0; s < S; ++s) {
            if constexpr (!JAC) {
                o[s] = poly_value<T, PM, NP>(P, s, u);
            } else {
                T acc = mul(poly_value<T, PM - 1, NP>(P, s * S, u), w[0]);
#pragma unroll
                for (int r = 1; r < S; ++r) acc = add(acc, mul(poly_value<T, PM - 1, NP>(P, s * S + r, u), w[r]));
                o[s] = acc;
            }
        }
    }
};

// Sum-factorised quadrature over directions DIM..D-1 (see header): the
// moments M of f over the values with Legendre coefficients C in those
// directions.  The innermost level is unrolled, its table entries being
// compile-time operands, with both points of a pair evaluated side by side
// (two independent chains).  The outer levels loop over the points with one
// copy of the inner level (the positive point of a pair leaves the negative
// point's values and its own moments behind): unrolled, the code outgrows the
// instruction cache.
template <typename T, int D, int K, int Q, int S, bool JAC, int DIM>
struct Quad {
    static constexpr int N = Pow<K, D - DIM>::v;
    static constexpr int NS = N / K;
    static constexpr int ODD = Q & 1;
    static constexpr int NP = JAC ? S * S : S;
    __device__ __forceinline__ static void halves(const QuadTab<T, K, Q>& tb, int g, const T (&C)[S][N], bool mid,
                                                  T (&a)[S][NS], T (&b)[S][NS]) {
#pragma unroll
        for (int s = 0; s < S; ++s)
#pragma unroll
            for (int i = 0; i < NS; ++i) {
                T e = C[s][i];
#pragma unroll
                for (int r = 2; r < K; r += 2) e = maddc(tb.B[g][r], C[s][r * NS + i], e);
                if (mid) {
                    a[s][i] = e;
                } else if constexpr (K <= 3 && !std::is_same<T, df2>::value) {
                    a[s][i] = maddc(tb.B[g][1], C[s][NS + i], e);
                    b[s][i] = nmaddc(tb.B[g][1], C[s][NS + i], e);
                } else {
                    T o = mulc(tb.B[g][1], C[s][NS + i]);
#pragma unroll
                    for (int r = 3; r < K; r += 2) o = maddc(tb.B[g][r], C[s][r * NS + i], o);
                    a[s][i] = add(e, o);
                    b[s][i] = sub(e, o);
                }
            }
    }
    // innermost level (NS = 1)
    __device__ __forceinline__ static void run_points(const QuadTab<T, K, Q>& tb, const Poly<T, S, NP>& P,
                                                      const T (&Cu)[S][N], const T (&Cw)[S][N], T (&M)[S][N]) {
        using PE = PointEval<T, max_degree(K, Q), S, JAC>;
        auto points = [](const T (&x)[S][1], T (&y)[S]) {
#pragma unroll
            for (int s = 0; s < S; ++s) y[s] = x[s][0];
        };
        if constexpr (ODD) {
            constexpr int g = Q / 2;
            T u[S][1], ub[S][1], w[S][1], wb[S][1], uv[S], wv[S], m[S];
            halves(tb, g, Cu, true, u, ub);
            points(u, uv);
            if constexpr (JAC) {
                halves(tb, g, Cw, true, w, wb);
                points(w, wv);
            }
            PE::run(P, uv, wv, m);
#pragma unroll
            for (int s = 0; s < S; ++s)
#pragma unroll
                for (int r = 0; r < K; r += 2) M[s][r] = mulc(tb.WB[g][r], m[s]);
        }
#pragma unroll
        for (int g = 0; g < Q / 2; ++g) {
            T ua[S][1], ub[S][1], wa[S][1], wb[S][1], uv[S], wv[S], ma[S], mb[S];
            halves(tb, g, Cu, false, ua, ub);
            if constexpr (JAC) halves(tb, g, Cw, false, wa, wb);
            points(ua, uv);
            if constexpr (JAC) points(wa, wv);
            PE::run(P, uv, wv, ma);
            points(ub, uv);
            if constexpr (JAC) points(wb, wv);
            PE::run(P, uv, wv, mb);
#pragma unroll
            for (int s = 0; s < S; ++s) {
                const T sp = add(ma[s], mb[s]), sd = sub(ma[s], mb[s]);
#pragma unroll
                for (int r = 0; r < K; ++r) {
                    const T x = (r & 1) ? sd : sp;
                    const bool first = g == 0 && (!ODD || (r & 1));
                    M[s][r] = first ? mulc(tb.WB[g][r], x) : maddc(tb.WB[g][r], x, M[s][r]);
                }
            }
        }
    }
    __device__ __forceinline__ static void run(const QuadTab<T, K, Q>& tb, const Poly<T, S, NP>& P,
                                               const T (&Cu)[S][N], const T (&Cw)[S][N], T (&M)[S][N]) {
        if constexpr (DIM == D - 1) {
            run_points(tb, P, Cu, Cw, M);
        } else {
            run_loop(tb, P, Cu, Cw, M);
        }
    }
    __device__ __forceinline__ static void run_loop(const QuadTab<T, K, Q>& tb, const Poly<T, S, NP>& P,
                                                    const T (&Cu)[S][N], const T (&Cw)[S][N], T (&M)[S][N]) {
        T ub[S][NS], wb[S][NS], ma[S][NS];
#pragma unroll 1
        for (int it = 0; it < Q; ++it) {
            const bool mid = ODD && it == 0;
            const int g = mid ? Q / 2 : (it - ODD) >> 1;
            const bool second = !mid && ((it - ODD) & 1);
            T u[S][NS], w[S][NS], m[S][NS];
            if (!second) {
                halves(tb, g, Cu, mid, u, ub);
                if constexpr (JAC) halves(tb, g, Cw, mid, w, wb);
            } else {
#pragma unroll
                for (int s = 0; s < S; ++s)
#pragma unroll
                    for (int i = 0; i < NS; ++i) {
                        u[s][i] = ub[s][i];
                        if (JAC) w[s][i] = wb[s][i];
                    }
            }
            Quad<T, D, K, Q, S, JAC, DIM + 1>::run(tb, P, u, w, m);
            const bool first_even = it == 0 || (!ODD && it == 1);
            const bool first_odd = it == (ODD ? 2 : 1);
#pragma unroll
            for (int s = 0; s < S; ++s)
#pragma unroll
                for (int i = 0; i < NS; ++i) {
                    if (mid) {
#pragma unroll
                        for (int r = 0; r < K; r += 2) M[s][r * NS + i] = mulc(tb.WB[g][r], m[s][i]);
                    } else if (!second) {
                        ma[s][i] = m[s][i];
                    } else {
                        const T sp = add(ma[s][i], m[s][i]), sd = sub(ma[s][i], m[s][i]);
#pragma unroll
                        for (int r = 0; r < K; ++r) {
                            const T x = (r & 1) ? sd : sp;
                            T& acc = M[s][r * NS + i];
                            if ((r & 1) ? first_odd : first_even) acc = mulc(tb.WB[g][r], x);
                            else acc = maddc(tb.WB[g][r], x, acc);
                        }
                    }
                }
        }
    }
};

// Outermost quadrature level: the cell's coefficients are read from shared
// memory at every Gauss point (coefficient e = f (k+1) + r of the cell at
// pu[r PS + f]: fiber f, position r along the pencil) and the moments of
// species s accumulated in shared memory (moment e at ms[s][e mstride]; in
// registers for a species whose ms is null), so that only the inner levels'
// partial sums are live across the point loop.
template <typename T, int D, int K, int Q, int S, bool JAC, int PS, int NSH>
struct QuadTop {
    static constexpr int NC = Pow<K, D>::v;
    static constexpr int NS = NC / K;
    static constexpr int NP = JAC ? S * S : S;
    static constexpr int NR = S > NSH ? S - NSH : 1;  // species with moments in registers
    __device__ __forceinline__ static T at(const T* p, int e) { return vread(p + (e % K) * PS + e / K); }
    __device__ __forceinline__ static void values(const QuadTab<T, K, Q>& tb, int it, const T* const (&p)[S],
                                                  T (&u)[S][NS]) {
#pragma unroll
        for (int s = 0; s < S; ++s)
#pragma unroll
            for (int i = 0; i < NS; ++i) {
                T a = at(p[s], i);
#pragma unroll
                for (int r = 1; r < K; ++r) a = maddc(tb.TB[it][r], at(p[s], r * NS + i), a);
                u[s][i] = a;
            }
    }
    __device__ __forceinline__ static void run(const QuadTab<T, K, Q>& tb, const Poly<T, S, NP>& P,
                                               const T* const (&pu)[S], const T* const (&pw)[S], T* const (&ms)[S],
                                               int mstride, T (&M)[NR][NC]) {
#pragma unroll 1
        for (int it = 0; it < Q; ++it) {
            T u[S][NS], w[S][NS], m[S][NS];
            values(tb, it, pu, u);
            if constexpr (JAC) values(tb, it, pw, w);
            Quad<T, D, K, Q, S, JAC, 1>::run(tb, P, u, w, m);
#pragma unroll
            for (int s = 0; s < S; ++s)
#pragma unroll
                for (int r = 0; r < K; ++r)
#pragma unroll
                    for (int i = 0; i < NS; ++i) {
                        const int e = r * NS + i;
                        if (s < NSH) {
                            T* p = ms[s] + e * mstride;
                            vwrite(p, it == 0 ? mulc(tb.TWB[it][r], m[s][i]) : maddc(tb.TWB[it][r], m[s][i], vread(p)));
                        } else {
                            T& acc = M[s < NSH ? 0 : s - NSH][e];
                            acc = it == 0 ? mulc(tb.TWB[it][r], m[s][i]) : maddc(tb.TWB[it][r], m[s][i], acc);
                        }
                    }
        }
    }
};

// Slot position of detail r of parent par (counted within the half for two
// lanes) for children of level n.
template <int LANES, int K>
__device__ __forceinline__ int detail_pos(int n, int par, int r) {
    if (LANES == 1) return (K << (n - 1)) + par * K + r;
    return n == 1 ? K + r : K * ((1 << (n - 2)) + 1) + par * K + r;
}

// In shared memory a buffer holds the P fibers of one set interleaved,
// position pos of fiber f at slot pos PS + f (PS = P rounded up to odd:
// threads on consecutive fibers, or on consecutive cells of one fiber, hit
// distinct banks).
//
// Forward stage (hierarchical coefficients in X -> Legendre coefficients of
// the cells of level a + de in Y) for the subtree under node j of level a of
// fiber f (j within the half for two lanes): node m of level l is stored at
// position m (k+1) 2^{N - l} of Y, so a stage works in place and the finest
// cells come out contiguous.  The first stage starts from the level-0
// coefficients, for two lanes from the halves that the first split makes of
// them (left in lane 0, right in lane 1).
template <typename T, int K, int PS>
__device__ __forceinline__ void fwd_subtree(const T* X, T* Y, int f, int j, int N, int a, int de, bool first,
                                            const Filt<T, K>& F) {
    constexpr int LANES = LaneTraits<T>::LANES, LV = PD<T>;
    T cell[1 << LV][K];
    if (!first) {
#pragma unroll
        for (int r = 0; r < K; ++r) cell[0][r] = Y[(j * (K << (N - a)) + r) * PS + f];
    } else {
#pragma unroll
        for (int r = 0; r < K; ++r) cell[0][r] = X[r * PS + f];
        if constexpr (LANES == 2) {
            T d[K], A[K], B[K];
#pragma unroll
            for (int r = 0; r < K; ++r) d[r] = X[(K + r) * PS + f];
            split_node<T, K>(cell[0], d, F, A, B);
#pragma unroll
            for (int r = 0; r < K; ++r) cell[0][r] = add_signed(A[r], B[r], false, true);
        }
    }
#pragma unroll
    for (int l = 0; l < LV; ++l) {
        if (l < de) {
            const int n = a + l + 1;
#pragma unroll
            for (int i = (1 << l) - 1; i >= 0; --i) {
                const int par = (j << l) + i;
                T d[K], A[K], B[K];
#pragma unroll
                for (int r = 0; r < K; ++r) d[r] = X[detail_pos<LANES, K>(n, par, r) * PS + f];
                split_node<T, K>(cell[i], d, F, A, B);
#pragma unroll
                for (int s = 0; s < K; ++s) {
                    cell[2 * i][s] = add(A[s], B[s]);
                    cell[2 * i + 1][s] = sub(A[s], B[s]);
                }
            }
        }
    }
    const int stride = K << (N - a - de);
#pragma unroll
    for (int i = 0; i < (1 << LV); ++i)
        if (i < (1 << de))
#pragma unroll
            for (int s = 0; s < K; ++s) Y[(((j << de) + i) * stride + s) * PS + f] = cell[i][s];
}

// Transposed step for subtree j of fiber f: its 2^De nodes of level Lhi,
// node m stored at position m stride of Mb (stride = (k+1) 2^{N - Lhi};
// the finest cells are contiguous), reduced over De levels; the details of
// levels Lhi - De + 1 .. Lhi go to Y (hierarchical layout) and the root
// (level Lhi - De) in place over the first node, or to Y when it is level 0
// (one lane; two lanes stop at level 1, whose nodes are the halves).
template <typename T, int K, int PS>
__device__ __forceinline__ void bwd_subtree(T* Mb, T* Y, int f, int j, int Lhi, int De, int stride,
                                            const Filt<T, K>& F) {
    constexpr int LANES = LaneTraits<T>::LANES, LV = PD<T>;
    T cell[1 << LV][K];
#pragma unroll
    for (int i = 0; i < (1 << LV); ++i)
        if (i < (1 << De))
#pragma unroll
            for (int s = 0; s < K; ++s) cell[i][s] = Mb[(((j << De) + i) * stride + s) * PS + f];
#pragma unroll
    for (int l = LV - 1; l >= 0; --l) {
        if (l < De) {
            const int n = Lhi - De + l + 1;  // level of the children
#pragma unroll
            for (int i = 0; i < (1 << l); ++i) {
                T sum[K], dif[K], d[K];
#pragma unroll
                for (int s = 0; s < K; ++s) {
                    sum[s] = add(cell[2 * i][s], cell[2 * i + 1][s]);
                    dif[s] = sub(cell[2 * i][s], cell[2 * i + 1][s]);
                }
                const int par = (j << l) + i;
                merge_node<T, K>(sum, dif, F, cell[i], d);
#pragma unroll
                for (int r = 0; r < K; ++r) Y[detail_pos<LANES, K>(n, par, r) * PS + f] = d[r];
            }
        }
    }
    const bool top = LANES == 1 && Lhi == De;
#pragma unroll
    for (int r = 0; r < K; ++r) {
        if (top) Y[r * PS + f] = cell[0][r];
        else Mb[((j << De) * stride + r) * PS + f] = cell[0][r];
    }
}

// the last split of two lanes: the halves of fiber f
template <typename T, int K, int PS>
__device__ __forceinline__ void bwd_root(const T* Mb, T* Y, int f, const Filt<T, K>& F) {
    T sum[K], dif[K], p[K], d[K];
#pragma unroll
    for (int s = 0; s < K; ++s) {
        const T x = Mb[s * PS + f], y = swap_lanes(x);
        sum[s] = add(x, y);
        dif[s] = sub(x, y);  // left minus right in lane 0, the one stored
    }
    merge_node<T, K>(sum, dif, F, p, d);
#pragma unroll
    for (int r = 0; r < K; ++r) {
        Y[r * PS + f] = p[r];
        Y[(K + r) * PS + f] = d[r];
    }
}

// Shared memory of one pencil, in slots: NSETS hierarchical buffers, one
// nodal buffer, and for two species from d = 3 on one more for the second
// species' moments (at d = 2 they fit in registers).
template <typename T, int D, int K, int S, bool JAC>
struct PencilShape {
    static constexpr int LANES = LaneTraits<T>::LANES;
    static constexpr int P = Pow<K, D - 1>::v;  // fibers per species and set
    static constexpr int PS = P | 1;            // odd fiber stride in shared memory
    static constexpr int NC = Pow<K, D>::v;     // coefficients per cell
    static constexpr int NSETS = JAC ? 2 * S : S;
    static constexpr int NSH = (S == 2 && D >= 3) ? 2 : 1;  // species with moments in shared memory
    // positions per fiber of a hierarchical and of a nodal buffer
    __host__ __device__ static int hier(int H) { return LANES == 1 ? H : H / 2 + K; }
    __host__ __device__ static int nodal(int H) { return H / LANES; }
    __host__ __device__ static size_t bytes(int H) {
        return sizeof(T) * (size_t)PS * ((size_t)NSETS * hier(H) + (size_t)NSH * nodal(H)) + sizeof(long long) * (P + 1);
    }
};

// Register limits.  FP64 fills its pipe with four warps per SM and
// double-float runs the eight that shared memory admits, so both take what
// they want; FP32 wants warps (128 registers, ten to sixteen of them).
template <typename T>
constexpr int MAX_REGS = std::is_same<T, float>::value ? 128 : 255;

template <typename T, int D, int K, int Q, int S, bool JAC>
__global__ void __maxnreg__(MAX_REGS<T>)
    pencil_kernel(const PencilArgs args, const int ppc, const __grid_constant__ QuadTab<T, K, Q> tb,
                  const __grid_constant__ Filt<T, K> F,
                  const __grid_constant__ Poly<T, S, (JAC ? S * S : S)> poly) {
    using Sh = PencilShape<T, D, K, S, JAC>;
    using Elem = typename LaneTraits<T>::Elem;
    constexpr int LANES = Sh::LANES, P = Sh::P, PS = Sh::PS, NC = Sh::NC, NSETS = Sh::NSETS, NSH = Sh::NSH;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* const sm = reinterpret_cast<T*>(smem_raw);
    const int H = args.H, N = args.N;
    const int bsh = Sh::hier(H) * PS, bsn = Sh::nodal(H) * PS;
    const size_t per_pencil = (size_t)NSETS * bsh + (size_t)NSH * bsn;
    // ppc P fiber offsets behind the slots
    long long* const s_of = reinterpret_cast<long long*>(smem_raw + (ppc * per_pencil * sizeof(T) + 7) / 8 * 8);
    // buffer i of pencil pp: the NSETS hierarchical ones, then the nodal ones
    auto buf = [&](int pp, int i) {
        return sm + pp * per_pencil + (i <= NSETS ? (size_t)i * bsh : (size_t)NSETS * bsh + (size_t)(i - NSETS) * bsn);
    };
    const int half = LANES == 2 ? 1 : 0;     // the unit counts below are per half for two lanes
    // levels of the first forward stage: the rest takes PD levels a stage
    const int levels = N - half, de0 = levels % PD<T> ? levels % PD<T> : (levels ? PD<T> : 0);
    for (long long pen0 = blockIdx.x * (long long)ppc; pen0 < args.npencils; pen0 += (long long)gridDim.x * ppc) {
        const int np = (int)(args.npencils - pen0 < ppc ? args.npencils - pen0 : ppc);
        // source offset of every fiber: o_f = obase + sum_m r_m H^{d-2-m}
        for (int i = threadIdx.x; i < np * P; i += blockDim.x) {
            long long o = 0, rem = pen0 + i / P, mul = 1;
            for (int m = D - 2; m >= 0; --m) {
                const long long c = rem % args.ncell1;
                rem /= args.ncell1;
                o += c * K * mul;
                mul *= H;
            }
            int rr = i % P;
            mul = 1;
            for (int m = D - 2; m >= 0; --m) {
                o += (rr % K) * mul;
                rr /= K;
                mul *= H;
            }
            s_of[i] = o;
        }
        __syncthreads();
        // position a of a fiber with offset o lives in the level-l chunk at
        // cbase[l] + o n_l + (a - off); body(pp, slot position, lane, level,
        // address base, n_l); levels 0 and 1 belong to both lanes
        auto each_position = [&](auto&& body) {
            for (int i = threadIdx.x; i < np * H; i += blockDim.x) {
                const int cr = i / K, r = i - cr * K;
                const int q = cr & ((1 << N) - 1), pp = cr >> N;
                const int l = q == 0 ? 0 : 32 - __clz(q);
                const int node = l ? q - (1 << (l - 1)) : 0;
                const int nl = l ? (K << (l - 1)) : K;
                int pos = q * K + r, lane = 0;
                if (LANES == 2 && l >= 2) {
                    const int hn = 1 << (l - 2);
                    lane = node >= hn;
                    pos = K * (hn + 1) + (node - lane * hn) * K + r;
                }
                body(pp, pos, lane, l, args.cbase[l] + node * K + r, nl);
            }
        };
        // 1. load every set's hierarchical fibers into buffers 0..NSETS-1
        each_position([&](int pp, int pos, int lane, int l, long long base, int nl) {
#pragma unroll
            for (int set = 0; set < NSETS; ++set) {
                const Elem* src = reinterpret_cast<const Elem*>(set < S ? args.u[set] : args.w[set - S]) + base;
                T* dst = buf(pp, set) + pos * PS;
#pragma unroll
                for (int f = 0; f < P; ++f) {
                    const Elem* e = src + s_of[pp * P + f] * nl;
                    slot_load(dst + f, lane, e);
                    if (LANES == 2 && l < 2) slot_load(dst + f, 1, e);
                }
            }
        });
        async_wait_all();
        __syncthreads();
        // 2. forward pyramids, one set after the other: set 0 into the nodal
        //    buffer NSETS, set k >= 1 into buffer k-1 (freed by set k-1)
#pragma unroll 1
        for (int set = 0; set < NSETS; ++set) {
#pragma unroll 1
            for (int a = half, de = de0;; a += de, de = PD<T>) {
                const int ush = a - half;  // log2 of the subtrees of a fiber
                for (int u = threadIdx.x; u < np * (P << ush); u += blockDim.x) {
                    const int f = u % P, jj = u / P, j = jj & ((1 << ush) - 1), pp = jj >> ush;
                    fwd_subtree<T, K, PS>(buf(pp, set), buf(pp, set == 0 ? NSETS : set - 1), f, j, N, a, de,
                                          a == half, F);
                }
                __syncthreads();
                if (a + de >= N) break;
            }
        }
        // nodal buffer of set k: NSETS for k = 0, k - 1 otherwise; buffer
        // NSETS - 1 is free
        // 3. cell quadrature, one thread per finest cell along the pencil (two
        //    cells for two lanes).  The moments of the first species (both
        //    from d = 3 on) accumulate in buffer NSETS - 1 (and NSETS + 1),
        //    moment e of cell c at e ncell + c, then overwrite the nodal u
        //    values (each thread reads and writes only its own cells)
        const int lc = N - half, ncell = 1 << lc;
        for (int u = threadIdx.x; u < np << lc; u += blockDim.x) {
            const int c = u & (ncell - 1), pp = u >> lc;
            const T* pu[S];
            const T* pw[S];
            T* ms[S];
            T M[QuadTop<T, D, K, Q, S, JAC, PS, NSH>::NR][NC];
#pragma unroll
            for (int s = 0; s < S; ++s) {
                pu[s] = buf(pp, s == 0 ? NSETS : s - 1) + c * K * PS;
                pw[s] = JAC ? buf(pp, S + s - 1) + c * K * PS : pu[s];
                ms[s] = s < NSH ? buf(pp, s == 0 ? NSETS - 1 : NSETS + s) + c : nullptr;
            }
            QuadTop<T, D, K, Q, S, JAC, PS, NSH>::run(tb, poly, pu, pw, ms, ncell, M);
#pragma unroll
            for (int s = 0; s < S; ++s) {
                T* mo = const_cast<T*>(pu[s]);
#pragma unroll
                for (int i = 0; i < NC; ++i)
                    mo[(i % K) * PS + i / K] = s < NSH ? vread(ms[s] + i * ncell) : M[s < NSH ? 0 : s - NSH][i];
            }
        }
        __syncthreads();
        // 4. per species: backward pyramid (stages of up to PD levels, roots
        //    kept in place between them) into the free buffer, then store
#pragma unroll 1
        for (int s = 0; s < S; ++s) {
            const int mbuf = s == 0 ? NSETS : s - 1;
            for (int Lhi = N; Lhi > half;) {
                const int de = Lhi - half < PD<T> ? Lhi - half : PD<T>;
                const int sh = Lhi - de - half, stride = K << (N - Lhi);
                for (int u = threadIdx.x; u < np * (P << sh); u += blockDim.x) {
                    const int f = u % P, jj = u / P, j = jj & ((1 << sh) - 1), pp = jj >> sh;
                    bwd_subtree<T, K, PS>(buf(pp, mbuf), buf(pp, NSETS - 1), f, j, Lhi, de, stride, F);
                }
                __syncthreads();
                Lhi -= de;
            }
            if constexpr (LANES == 2) {
                for (int u = threadIdx.x; u < np * P; u += blockDim.x)
                    bwd_root<T, K, PS>(buf(u / P, mbuf), buf(u / P, NSETS - 1), u % P, F);
                __syncthreads();
            }
            Elem* dst = reinterpret_cast<Elem*>(args.out[s]);
            each_position([&](int pp, int pos, int lane, int, long long base, int nl) {
                const T* y = buf(pp, NSETS - 1) + pos * PS;
#pragma unroll
                for (int f = 0; f < P; ++f) dst[base + s_of[pp * P + f] * nl] = slot_value(y + f, lane);
            });
            __syncthreads();
        }
    }
}

// ------------------------------------------------------------- host side

// Reaction coefficients by exponents, scaled for the basis without h^{-1/2}
// (u = s u~ with s = h^{-d/2} at the points, the moments times s): c s^{deg+1}.
// lead: the leading coefficient that a monic polynomial leaves out (else 1).
template <typename T, int S, bool JAC>
Poly<T, S, (JAC ? S * S : S)> make_poly(const ReactionDev& rx, double s, double* lead) {
    constexpr int NP = JAC ? S * S : S, NCOEF = Pow<PDEG, S>::v;
    double c[NP][NCOEF] = {};
    for (int m = 0; m < rx.nmono; ++m) {
        int deg = 0;
        for (int r = 0; r < S; ++r) deg += rx.exps[m][r];
        double v = rx.coef[m];
        for (int i = 0; i <= deg; ++i) v *= s;
        if (!JAC) {
            int idx = 0;
            for (int r = 0; r < S; ++r) idx = idx * PDEG + rx.exps[m][r];
            c[rx.species[m]][idx] += v;
        } else {
            for (int q = 0; q < S; ++q) {  // derivative by u_q
                if (rx.exps[m][q] == 0) continue;
                int idx = 0;
                for (int r = 0; r < S; ++r) idx = idx * PDEG + rx.exps[m][r] - (r == q ? 1 : 0);
                c[rx.species[m] * S + q][idx] += v * rx.exps[m][q];
            }
        }
    }
    *lead = 1.0;
    Poly<T, S, NP> p{};
    if (MONIC<T, S>)
        for (int j = NCOEF - 1; j >= 0; --j)
            if (c[0][j] != 0.0) {
                const double a = std::fabs(c[0][j]);
                bool fits = a >= 1.0 && a <= 0x1p128;
                for (int l = 0; l < j; ++l) fits = fits && (c[0][l] == 0.0 || std::fabs(c[0][l]) / a >= 0x1p-900);
                if (fits) {
                    p.monic = 1;
                    *lead = c[0][j];
                    for (int l = 0; l < j; ++l) c[0][l] /= *lead;
                    c[0][j] = 1.0;
                }
                break;
            }
    for (int i = 0; i < NP; ++i)
        for (int j = 0; j < NCOEF; ++j) {
            cst_set(p.c[i][j], c[i][j]);
            if (c[i][j] == 0.0) continue;
            if (S == 1) p.rows[i] |= 1u << j;
            else {
                p.rows[i] |= 1u << (j / PDEG);
                p.mask[i][j / PDEG] |= 1u << (j % PDEG);
            }
        }
    return p;
}

// B: q x (k+1), sqrt(2r+1) P_r(xi_g) at ascending points; w: h w_g / 2; lead:
// see make_poly
template <typename T, int K, int Q>
QuadTab<T, K, Q> make_tab(const double* B, const double* w, double lead) {
    QuadTab<T, K, Q> t{};
    auto fill = [&](int g, int src) {
        for (int r = 0; r < K; ++r) {
            cst_set(t.B[g][r], B[src * K + r]);
            cst_set(t.WB[g][r], w[src] * B[src * K + r]);
        }
    };
    for (int g = 0; g < Q / 2; ++g) fill(g, Q - 1 - g);
    if (Q & 1) fill(Q / 2, Q / 2);
    for (int it = 0; it < Q; ++it) {
        const bool mid = (Q & 1) && it == 0;
        const int k2 = it - (Q & 1), g = mid ? Q / 2 : k2 / 2;
        const int src = mid ? Q / 2 : Q - 1 - g;
        const double sign = !mid && (k2 & 1) ? -1.0 : 1.0;
        for (int r = 0; r < K; ++r) {
            const double sr = (r & 1) ? sign : 1.0;
            cst_set(t.TB[it][r], sr * B[src * K + r]);
            cst_set(t.TWB[it][r], sr * w[src] * B[src * K + r] * lead);
        }
    }
    return t;
}

template <typename T, int D, int K, int Q, int S, bool JAC>
void launch_one(sgk_ctx* ctx, const PencilArgs& a, const double* B, const double* w, const double* two_scale,
                const ReactionDev& rx, double scale) {
    using Sh = PencilShape<T, D, K, S, JAC>;
    const Filt<T, K> F = make_filt<T, K>(two_scale);
    double lead = 1.0;
    const auto poly = make_poly<T, S, JAC>(rx, scale, &lead);
    const auto tab = make_tab<T, K, Q>(B, w, lead);
    const size_t smem1 = Sh::bytes(a.H);
    SGK_REQUIRE(smem1 <= ctx->smem_optin, SGK_EUNSUPPORTED, "pencil exceeds shared memory");
    // Pencils per CTA: as many cells (pairs of cells) as threads, two a
    // thread in FP32 where a pencil is light, as long as shared memory still
    // holds four CTAs (FP64: two, of 128 threads) and every SM gets four.
    // Level 6, degree 2: FP64 F 1.15 ms with two pencils and 128 threads, 1.19
    // with one and 64; FP32 Jacobian 73.6 and 76 us; level 7, degree 1, where
    // a cell has 27 points: 149 us with two cells a thread, 186 with one.
    constexpr bool F64 = std::is_same<T, double>::value, F32 = std::is_same<T, float>::value;
    const int want = F32 ? 256 : F64 ? 128 : 64;
    const size_t cap = (F64 ? 112 : 57) * 1024;
    const int cells = std::max(1, (1 << a.N) / Sh::LANES);
    int ppc = 1;
    while (ppc < 16 && ppc * cells < want && smem1 * (2 * ppc) <= cap &&
           a.npencils >= (long long)ctx->num_sms * 4 * ppc)
        ppc *= 2;
    const size_t smem = smem1 * ppc;
    const int threads = std::min(128, std::max(64, (cells * ppc + 31) / 32 * 32));
    const int grid = (int)std::min<long long>((a.npencils + ppc - 1) / ppc, (long long)ctx->num_sms * 16);
    auto kern = pencil_kernel<T, D, K, Q, S, JAC>;
    allow_max_dynamic_smem(ctx->smem_optin, kern);
    kern<<<grid, threads, smem, ctx->stream>>>(a, ppc, tab, F, poly);
}

}  // namespace sgk_pen

// (d, k+1, q, species): the shapes of the fused pass.  DF: their F passes of
// mixed mode run in double-float; the other shapes keep FP64 there.
#define SGK_PENCIL_DF_D2(X) X(2, 3, 5, 2) X(2, 2, 3, 1) X(2, 2, 3, 2) X(2, 3, 5, 1)
#define SGK_PENCIL_DF_D34(X) X(3, 3, 5, 1) X(3, 2, 3, 1) X(4, 2, 3, 1)
#define SGK_PENCIL_D2(X) SGK_PENCIL_DF_D2(X) X(2, 4, 7, 1) X(2, 4, 7, 2) X(2, 2, 2, 1) X(2, 3, 4, 1) X(2, 4, 5, 1)
#define SGK_PENCIL_D34(X)                                                                                   \
    SGK_PENCIL_DF_D34(X) X(3, 2, 3, 2) X(3, 3, 5, 2) X(3, 4, 7, 1) X(3, 4, 7, 2) X(3, 2, 2, 1) X(3, 3, 4, 1) \
    X(4, 3, 5, 1) X(4, 2, 3, 2)

// Launches the shape's kernel, or returns false when the list has none.
#define SGK_PENCIL_DISPATCH(NAME, T, JAC, LIST)                                                                   \
    bool NAME(sgk_ctx* ctx, int d, int kp1, int q, int S, const PencilArgs& a, const double* B, const double* w, \
              const double* two_scale, const ReactionDev& rx, double scale) {                                    \
        LIST(SGK_PENCIL_CASE_##JAC##_##T)                                                                         \
        return false;                                                                                             \
    }
#define SGK_PENCIL_CASE(T, JAC, DD, KK, QQ, SS)                                                         \
    if (d == DD && kp1 == KK && q == QQ && S == SS) {                                                   \
        sgk_pen::launch_one<T, DD, KK, QQ, SS, JAC>(ctx, a, B, w, two_scale, rx, scale);                \
        return true;                                                                                    \
    }
#define SGK_PENCIL_CASE_false_double(DD, KK, QQ, SS) SGK_PENCIL_CASE(double, false, DD, KK, QQ, SS)
#define SGK_PENCIL_CASE_true_double(DD, KK, QQ, SS) SGK_PENCIL_CASE(double, true, DD, KK, QQ, SS)
#define SGK_PENCIL_CASE_false_float(DD, KK, QQ, SS) SGK_PENCIL_CASE(float, false, DD, KK, QQ, SS)
#define SGK_PENCIL_CASE_true_float(DD, KK, QQ, SS) SGK_PENCIL_CASE(float, true, DD, KK, QQ, SS)
#define SGK_PENCIL_CASE_false_df2(DD, KK, QQ, SS) SGK_PENCIL_CASE(df2, false, DD, KK, QQ, SS)
