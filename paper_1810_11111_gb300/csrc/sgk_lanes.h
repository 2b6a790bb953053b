// Element types of the reaction passes.
//
//   double, float, dfloat  one value per thread;
//   df2     two values per thread in double-float arithmetic: a packed pair of
//           high parts and one of low parts (sgk_dfloat.h says what a
//           double-float number is and how its sums and products are formed;
//           each lane here goes through the same error-free steps).
//
// The packed type issues fma/add/mul/sub.rn.f32x2.  Measured on the part: a
// packed FMA has the latency of a scalar one (4.4 clocks) and does twice the
// work, at the same 128 lanes per clock and SM; so chains of dependent
// operations, which the TwoSum sequences are, fill the FP32 pipe with half
// the warps (eight warps per SM with one chain each: 88% of its rate, scalar
// FMAs 45%).  FP64 issues one warp instruction per 64 clocks and scheduler
// whatever the chains: there only the operation count matters.  Plain FP32
// passes are bound by their memory phases and want warps, not lanes: packed,
// the Jacobian pass measured 78 us at d = 3, level 6, degree 2 and 439 us at
// degree 3, scalar 74 and 282.
//
// A constant c is stored with the forms its products need (Cst): the
// packed instructions take no negated operands.
#pragma once
#include "sgk_dfloat.h"
#include "sgk_internal.h"

struct f2 {
    unsigned long long v;
};
struct __align__(16) df2 {
    f2 hi, lo;
};

template <typename T>
struct Cst;
template <>
struct Cst<double> {
    double c;
};
template <>
struct Cst<float> {
    float c;
};
template <>
struct Cst<dfloat> {
    float h, l;
};
template <>
struct Cst<df2> {
    float2 ch, nch, cl;  // high part, its negative, low part
};

inline void cst_set(Cst<double>& k, double x) { k.c = x; }
inline void cst_set(Cst<float>& k, double x) { k.c = (float)x; }
inline void cst_set(Cst<dfloat>& k, double x) {
    k.h = (float)x;
    k.l = (float)(x - (double)k.h);
}
inline void cst_set(Cst<df2>& k, double x) {
    const float h = (float)x, l = (float)(x - (double)h);
    k.ch = make_float2(h, h);
    k.nch = make_float2(-h, -h);
    k.cl = make_float2(l, l);
}

// Lanes per thread, the element in device memory, the words of one shared
// memory slot.
template <typename T>
struct LaneTraits;
template <>
struct LaneTraits<double> {
    static constexpr int LANES = 1;
    using Elem = double;
};
template <>
struct LaneTraits<float> {
    static constexpr int LANES = 1;
    using Elem = float;
};
template <>
struct LaneTraits<df2> {
    static constexpr int LANES = 2;
    using Elem = dfloat;
};

#ifdef __CUDACC__
namespace lanes {

__device__ __forceinline__ f2 pack(float a, float b) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ f2 from(const float2& a) { return pack(a.x, a.y); }
__device__ __forceinline__ f2 swap(f2 a) {
    f2 r;
    asm("{.reg .b32 x, y;\n\tmov.b64 {x, y}, %1;\n\tmov.b64 %0, {y, x};}" : "=l"(r.v) : "l"(a.v));
    return r;
}
__device__ __forceinline__ f2 neg(f2 a) {
    f2 r;
    r.v = a.v ^ 0x8000000080000000ull;
    return r;
}
__device__ __forceinline__ f2 add(f2 a, f2 b) {
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ f2 sub(f2 a, f2 b) {
    f2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ f2 mul(f2 a, f2 b) {
    f2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ f2 fma(f2 a, f2 b, f2 c) {
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}

template <typename T>
__device__ __forceinline__ T zero();
template <>
__device__ __forceinline__ double zero<double>() {
    return 0.0;
}
template <>
__device__ __forceinline__ df2 zero<df2>() {
    return df2{f2{0ull}, f2{0ull}};
}

// ---- double
__device__ __forceinline__ double add(double a, double b) { return a + b; }
__device__ __forceinline__ double sub(double a, double b) { return a - b; }
__device__ __forceinline__ double mul(double a, double b) { return a * b; }
__device__ __forceinline__ double mulc(const Cst<double>& k, double x) { return k.c * x; }
__device__ __forceinline__ double maddc(const Cst<double>& k, double x, double a) { return ::fma(k.c, x, a); }
__device__ __forceinline__ double nmaddc(const Cst<double>& k, double x, double a) { return ::fma(-k.c, x, a); }
__device__ __forceinline__ double cvalue(const Cst<double>& k) { return k.c; }
// a + s b, s = +1 or -1 by lane (first: lane 0, second: lane 1)
__device__ __forceinline__ double add_signed(double a, double b, bool n0, bool) { return n0 ? a - b : a + b; }

// ---- float, dfloat
template <>
__device__ __forceinline__ float zero<float>() {
    return 0.f;
}
template <>
__device__ __forceinline__ dfloat zero<dfloat>() {
    return dfloat(0.f, 0.f);
}
__device__ __forceinline__ float add(float a, float b) { return a + b; }
__device__ __forceinline__ float sub(float a, float b) { return a - b; }
__device__ __forceinline__ float mul(float a, float b) { return a * b; }
__device__ __forceinline__ float nmaddc(const Cst<float>& k, float x, float a) { return fmaf(-k.c, x, a); }
__device__ __forceinline__ float cvalue(const Cst<float>& k) { return k.c; }
__device__ __forceinline__ float mulc(const Cst<float>& k, float x) { return k.c * x; }
__device__ __forceinline__ float maddc(const Cst<float>& k, float x, float a) { return fmaf(k.c, x, a); }
__device__ __forceinline__ float add_signed(float a, float b, bool n0, bool) { return n0 ? a - b : a + b; }
__device__ __forceinline__ dfloat add(dfloat a, dfloat b) { return a + b; }
__device__ __forceinline__ dfloat sub(dfloat a, dfloat b) { return a - b; }
__device__ __forceinline__ dfloat mulc(const Cst<dfloat>& k, dfloat x) { return dfloat(k.h, k.l) * x; }
__device__ __forceinline__ dfloat maddc(const Cst<dfloat>& k, dfloat x, dfloat a) { return a + dfloat(k.h, k.l) * x; }
__device__ __forceinline__ dfloat add_signed(dfloat a, dfloat b, bool n0, bool) {
    return a + dfloat(n0 ? -b.hi : b.hi, n0 ? -b.lo : b.lo);
}

__device__ __forceinline__ f2 signs(bool n0, bool n1) { return pack(n0 ? -1.f : 1.f, n1 ? -1.f : 1.f); }

// ---- df2: hi + lo.  A product's rounded part and its residual are formed
// with opposite signs (see Cst): p = a.hi b.hi, ne = -(a.hi b.hi - p + cross
// terms); a sum is TwoSum of the high parts with the low parts added to its
// error.
__device__ __forceinline__ df2 add(df2 a, df2 b) {
    const f2 s = add(a.hi, b.hi);
    const f2 bb = sub(s, a.hi);
    const f2 err = add(sub(a.hi, sub(s, bb)), sub(b.hi, bb));
    return df2{s, add(err, add(a.lo, b.lo))};
}
__device__ __forceinline__ df2 sub(df2 a, df2 b) {
    const f2 s = sub(a.hi, b.hi);
    const f2 bb = sub(s, a.hi);
    const f2 err = sub(sub(a.hi, sub(s, bb)), add(b.hi, bb));
    return df2{s, add(err, sub(a.lo, b.lo))};
}
__device__ __forceinline__ df2 mul(df2 a, df2 b) {
    const f2 p = mul(a.hi, b.hi);
    f2 e = fma(a.hi, b.hi, neg(p));
    e = fma(a.hi, b.lo, e);
    e = fma(a.lo, b.hi, e);
    return df2{p, e};
}
// p and the negated residual of c x
__device__ __forceinline__ void prodc(const Cst<df2>& k, df2 x, f2& np, f2& e) {
    np = mul(from(k.nch), x.hi);          // -(ch xh) rounded
    e = fma(from(k.ch), x.hi, np);        // ch xh - p, exact
    e = fma(from(k.cl), x.hi, e);
    e = fma(from(k.ch), x.lo, e);
}
__device__ __forceinline__ df2 mulc(const Cst<df2>& k, df2 x) {
    f2 p = mul(from(k.ch), x.hi);
    f2 ne = fma(from(k.nch), x.hi, p);    // p - ch xh, exact
    // e = -ne + cross terms
    f2 e = neg(ne);
    e = fma(from(k.cl), x.hi, e);
    e = fma(from(k.ch), x.lo, e);
    return df2{p, e};
}
__device__ __forceinline__ df2 maddc(const Cst<df2>& k, df2 x, df2 a) {
    f2 np, e;
    prodc(k, x, np, e);
    const f2 s = sub(a.hi, np);  // a + p
    const f2 bb = sub(s, a.hi);
    const f2 err = sub(sub(a.hi, sub(s, bb)), add(np, bb));
    return df2{s, add(err, add(a.lo, e))};
}
__device__ __forceinline__ df2 cvalue(const Cst<df2>& k) { return df2{from(k.ch), from(k.cl)}; }
__device__ __forceinline__ df2 add_signed(df2 a, df2 b, bool n0, bool n1) {
    const f2 s = signs(n0, n1);
    return add(a, df2{mul(b.hi, s), mul(b.lo, s)});
}
__device__ __forceinline__ df2 swap_lanes(df2 a) { return df2{swap(a.hi), swap(a.lo)}; }

// ---- shared memory slots
// through volatile accesses: re-read and written at every use (held across
// the quadrature loops they would fill the registers)
__device__ __forceinline__ double vread(const double* p) { return *reinterpret_cast<const volatile double*>(p); }
__device__ __forceinline__ float vread(const float* p) { return *reinterpret_cast<const volatile float*>(p); }
__device__ __forceinline__ void vwrite(float* p, float v) { *reinterpret_cast<volatile float*>(p) = v; }
__device__ __forceinline__ df2 vread(const df2* p) {
    df2 r;
    asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];"
                 : "=l"(r.hi.v), "=l"(r.lo.v)
                 : "r"((unsigned)__cvta_generic_to_shared(p))
                 : "memory");
    return r;
}
__device__ __forceinline__ void vwrite(double* p, double v) { *reinterpret_cast<volatile double*>(p) = v; }
__device__ __forceinline__ void vwrite(df2* p, df2 v) {
    asm volatile("st.shared.v2.b64 [%0], {%1, %2};" ::"r"((unsigned)__cvta_generic_to_shared(p)), "l"(v.hi.v),
                 "l"(v.lo.v)
                 : "memory");
}

// one lane of a slot from device memory (asynchronous), and back
__device__ __forceinline__ void slot_load(double* slot, int, const double* src) { async_copy(slot, src); }
__device__ __forceinline__ void slot_load(float* slot, int, const float* src) { async_copy(slot, src); }
__device__ __forceinline__ float slot_value(const float* slot, int) { return *slot; }
__device__ __forceinline__ void slot_load(df2* slot, int lane, const dfloat* src) {
    float* w = reinterpret_cast<float*>(slot) + lane;
    async_copy(w, &src->hi);
    async_copy(w + 2, &src->lo);
}
__device__ __forceinline__ double slot_value(const double* slot, int) { return *slot; }
__device__ __forceinline__ dfloat slot_value(const df2* slot, int lane) {
    const float* w = reinterpret_cast<const float*>(slot) + lane;
    return dfloat(w[0], w[2]);
}

}  // namespace lanes
#endif
