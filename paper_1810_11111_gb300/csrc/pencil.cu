// Fused last-direction reaction pass: which shapes it serves, and dispatch to
// the kernels (sgk_pencil.cuh) by element type, dimension and pass.
#include <cmath>
#include <type_traits>

#include "sgk_pencil.cuh"

#define SGK_PENCIL_DECLARE(NAME)                                                                              \
    bool NAME(sgk_ctx* ctx, int d, int kp1, int q, int S, const PencilArgs& a, const double* B, const double* w, \
              const double* two_scale, const ReactionDev& rx, double scale);
SGK_PENCIL_DECLARE(pencil_f64_d2)
SGK_PENCIL_DECLARE(pencil_f64_d2_jac)
SGK_PENCIL_DECLARE(pencil_f64_d34)
SGK_PENCIL_DECLARE(pencil_f64_d34_jac)
SGK_PENCIL_DECLARE(pencil_f32_d2)
SGK_PENCIL_DECLARE(pencil_f32_d2_jac)
SGK_PENCIL_DECLARE(pencil_f32_d34)
SGK_PENCIL_DECLARE(pencil_f32_d34_jac)
SGK_PENCIL_DECLARE(pencil_df_d2)
SGK_PENCIL_DECLARE(pencil_df_d34)

namespace {

// shared memory of one line in a shape's F passes, in FP64 or double-float,
// and in its Jacobian passes, in FP64 or FP32
template <int D, int K, int S>
size_t line_bytes(int H, bool jac, bool fp64) {
    using namespace sgk_pen;
    if (jac)
        return fp64 ? PencilShape<double, D, K, S, true>::bytes(H) : PencilShape<float, D, K, S, true>::bytes(H);
    return fp64 ? PencilShape<double, D, K, S, false>::bytes(H) : PencilShape<df2, D, K, S, false>::bytes(H);
}

// Lowest levels at which a shape is fused, in FP64 and in mixed mode (1 where
// it is not listed).  A thread takes one cell, so on a coarse grid the pass
// lasts as long as one thread's points while most of the machine idles; the
// general cell pass spreads a cell's points over threads.  Microseconds of F /
// J at the level below the limit and at it, fused against general, FP64:
//   (3,4,7,2)  level 5  2870/3665, 2036/3161 (level 6 has 13 warps a
//              scheduler instead of two)
//   (3,4,7,1)  4   274/ 346,  177/ 251;  5   701/ 864,  882/1254
//   (3,3,5,2)  4   345/ 396,  254/ 357;  5   627/ 826,  853/1227
//   (4,3,5,1)  3   432/ 515,  282/ 381;  4  1805/2382, 2688/4108
//   (4,2,3,2)  3   312/ 350,  208/ 269;  4   847/ 921,  985/1532
//   (2,4,7,2)  2   132/ 148,   94/ 136;  3   155/ 182,  178/ 209
// In mixed mode the FP32 Jacobian products, which are most of the passes, gain
// earlier: (3,4,7,2) F 928 and J 129 us at level 3, general 227 and 180; 941
// and 157 at level 4, general 390 and 296.
struct Lowest {
    int d, kp1, q, S, fp64, mixed;
};
constexpr Lowest LOWEST[] = {{2, 4, 7, 1, 2, 1}, {2, 4, 7, 2, 3, 1}, {3, 2, 3, 2, 2, 1}, {3, 3, 4, 1, 2, 1},
                             {3, 3, 5, 2, 5, 2}, {3, 4, 7, 1, 5, 2}, {3, 4, 7, 2, 6, 4}, {4, 3, 5, 1, 4, 3},
                             {4, 2, 3, 2, 4, 1}};
int lowest_level(int d, int kp1, int q, int S, bool fp64) {
    for (const Lowest& l : LOWEST)
        if (l.d == d && l.kp1 == kp1 && l.q == q && l.S == S) return fp64 ? l.fp64 : l.mixed;
    return 1;
}

// h^{-d/2}, the scale between the pass's basis and the orthonormal one
double basis_scale(int d, int N) { return std::ldexp((d * N) % 2 ? 1.4142135623730951 : 1.0, d * N / 2); }

// The exponents have places in the tables, and the coefficients of the scaled
// basis, c s^{degree + 1}, stand far enough inside the range of FP64 or, in
// mixed mode, of FP32 (c itself may be within it and they not: 1e32 u^3 on
// 64^2 cells).
bool reaction_fits(const ReactionDev& rx, int S, int d, int N, bool fp64) {
    const double s = basis_scale(d, N);
    for (int m = 0; m < rx.nmono; ++m) {
        double v = std::fabs(rx.coef[m]) * s;
        for (int r = 0; r < S; ++r) {
            if (rx.exps[m][r] >= sgk_pen::PDEG) return false;
            v *= std::pow(s, rx.exps[m][r]);
        }
        if (!(v <= (fp64 ? 0x1p1000 : 0x1p100))) return false;
    }
    return true;
}

}  // namespace

bool pencil_df_supported(int d, int kp1, int q, int S, int N, size_t smem_optin) {
    if (N == 0) return false;
    const int H = kp1 << N;
#define SGK_PENCIL_OK(DD, KK, QQ, SS) \
    if (d == DD && kp1 == KK && q == QQ && S == SS) return line_bytes<DD, KK, SS>(H, false, false) <= smem_optin;
    SGK_PENCIL_DF_D2(SGK_PENCIL_OK)
    SGK_PENCIL_DF_D34(SGK_PENCIL_OK)
#undef SGK_PENCIL_OK
    return false;
}

bool pencil_supported(int d, int kp1, int q, int S, int N, const ReactionDev& rx, bool fp64, size_t smem_optin) {
    if (N < lowest_level(d, kp1, q, S, fp64) || !reaction_fits(rx, S, d, N, fp64)) return false;  // level 0: nothing to pair
    const int H = kp1 << N;
    const bool df = !fp64 && pencil_df_supported(d, kp1, q, S, N, smem_optin);
#define SGK_PENCIL_OK(DD, KK, QQ, SS)                                                        \
    if (d == DD && kp1 == KK && q == QQ && S == SS)                                          \
        return (df || line_bytes<DD, KK, SS>(H, false, true) <= smem_optin) &&               \
               line_bytes<DD, KK, SS>(H, true, fp64) <= smem_optin;
    SGK_PENCIL_D2(SGK_PENCIL_OK)
    SGK_PENCIL_D34(SGK_PENCIL_OK)
#undef SGK_PENCIL_OK
    return false;
}

template <typename T>
void pencil_launch(sgk_ctx* ctx, const PencilArgs& a, int d, int kp1, int q, int S, bool jac, const double* B,
                   const double* w, const double* two_scale, const ReactionDev& rx) {
    const double scale = basis_scale(d, a.N);
    KTimer kt(ctx, KC_CELL);
    bool ok = false;
    if constexpr (std::is_same<T, dfloat>::value) {
        // double-float serves the F passes only (Jacobian products stay FP32)
        SGK_REQUIRE(!jac, SGK_EUNSUPPORTED, "no double-float Jacobian pencil");
        ok = (d == 2 ? pencil_df_d2 : pencil_df_d34)(ctx, d, kp1, q, S, a, B, w, two_scale, rx, scale);
    } else if constexpr (std::is_same<T, double>::value) {
        ok = (jac ? (d == 2 ? pencil_f64_d2_jac : pencil_f64_d34_jac)
                  : (d == 2 ? pencil_f64_d2 : pencil_f64_d34))(ctx, d, kp1, q, S, a, B, w, two_scale, rx, scale);
    } else {
        ok = (jac ? (d == 2 ? pencil_f32_d2_jac : pencil_f32_d34_jac)
                  : (d == 2 ? pencil_f32_d2 : pencil_f32_d34))(ctx, d, kp1, q, S, a, B, w, two_scale, rx, scale);
    }
    SGK_REQUIRE(ok, SGK_EUNSUPPORTED, "no fused pencil kernel for this shape");
    check_launch("pencil_kernel");
    count_launch(ctx);
}

template void pencil_launch<double>(sgk_ctx*, const PencilArgs&, int, int, int, int, bool, const double*,
                                    const double*, const double*, const ReactionDev&);
template void pencil_launch<float>(sgk_ctx*, const PencilArgs&, int, int, int, int, bool, const double*,
                                   const double*, const double*, const ReactionDev&);
template void pencil_launch<dfloat>(sgk_ctx*, const PencilArgs&, int, int, int, int, bool, const double*,
                                    const double*, const double*, const ReactionDev&);
