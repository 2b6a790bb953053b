// Persistent Arnoldi kernel (see arnoldi.cu): device code and launch
// templates.  Each arnoldi_d<D>.cu instantiates arn_launch_k<D> for one
// dimension, so that the variants compile in parallel.
#pragma once
#include <algorithm>

#include "sgk_gmv.h"
#include "sgk_krylov.h"

namespace sgk_arn {

constexpr int PT = 512;                        // threads per CTA, one CTA per SM
constexpr int PNW = PT / 32;                   // warps per CTA
constexpr unsigned BAR_SPIN_LIMIT = 1u << 21;  // polls (an L2 round trip each, ~0.2-0.5 us): about a second

struct ArnArgs {
    int64_t n;
    int M;
    int E;    // slice length per CTA (ceil(n / gridDim.x))
    int smem_vz;   // this CTA's slices of V and Z live in shared memory (and V also in HBM)
    int smem_loc;  // the located rows of every output of the slice live in shared memory
    int list_cap;  // > 0: the slice's pre-located gather entries (at most list_cap) live in shared memory
    const int* eoff;   // pre-located gathers (see sgk_op::gmv_eoff), or null
    const int2* ent;
    // double-float matvec (mixed precision; needs the gather lists and the
    // shared V/Z slices): operator values as (hi, lo) pairs; the gathered
    // vectors (w0, w1) and Z then hold (hi, lo) pairs instead of doubles
    const float2* cvk2;
    int df;
    // eo1: one list per output over all terms of an operator with mixed
    // derivatives (offset of output g; entry q: index of x ei[q], value
    // ev[q]), read from L2 in order, with the whole gathered vector (8 n
    // bytes) staged in shared memory before every matvec; else null
    const int* eo1;
    const unsigned short* ei;
    const double* ev;
    const double* v;
    double* V;  // column c at V + c n
    double* w0;
    double* w1;
    double* Z;     // raw matvec outputs A v_c, column c at Z + c n (own slices only)
    double* H;     // (M + 1) x M row-major
    double* pbuf;  // gridDim.x per-CTA partials of a norm (gamma, explicit fallback)
    unsigned long long* acc;  // FX_SETS rotating sets of FX_COLS fixed-point accumulators (FX_LIMBS words each)
    // fixed-point scales: a partial p of an inner product enters as
    // trunc(p 2^sh); _h for the columns of V^T w (|p| <= ||A||), _n for
    // ||w'||^2 (|p| <= ||A||^2)
    int sh_h, sh_n;
    // a ||w''||^2 above this is no breakdown whatever H holds (its entries
    // are bounded by ||A||): 1e-24 times a bound on ||H||_F^2
    double no_brk;
    unsigned* bar;  // [0] barrier arrivals (zero at launch), [1] error flag
    unsigned bar_extra;  // added to every barrier target: 0, or 1 to make the waits run out (failure test)
    KrylovScalars* ks;
    const int64_t* bounds;  // slice b = [bounds[b], bounds[b+1]) (work-balanced), or null: equal slices of E
};

constexpr int FX_COLS = SGK_MAX_KRYLOV + 2;  // columns of one accumulator set
constexpr int FX_LIMBS = 4;                   // words of a column, see fx_add
// copies of every accumulator: CTA b adds into copy b % FX_COPIES, so that
// the CTAs arriving together do not serialise on the same words
constexpr int FX_COPIES = 8;
constexpr int FX_SET = FX_COPIES * FX_COLS * FX_LIMBS;  // words of one set
constexpr int FX_SETS = 6;                              // two phases a step, three steps in rotation

// Bytes of the staged entry offsets of a slice of E outputs (D per output
// and one end), rounded up to 16.
__host__ __device__ inline size_t arn_eoff_bytes(int E, int d) { return ((sizeof(int) * ((size_t)E * d + 1)) + 15) / 16 * 16; }

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ unsigned ld_relaxed(const unsigned* p) {
    unsigned v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void red_release_add(unsigned* p, unsigned v) {
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// All CTAs arrive; returns false if the wait ran out or another CTA failed.
// Thread 0 arrives with a release add (cumulative over the CTA's writes,
// which the CTA barrier before it orders) and polls with acquire loads,
// whose acquire the CTA barrier after it passes on to every thread; the
// error flag is looked at every 256 polls.
__device__ __forceinline__ bool grid_barrier(unsigned* bar, unsigned target, int* s_ok) {
    __syncthreads();
    if (threadIdx.x == 0) {
        red_release_add(bar, 1u);
        int ok = 1;
        for (unsigned it = 0;; ++it) {
            if (ld_acquire(bar) >= target) break;
            if ((it & 255u) == 255u && (it >= BAR_SPIN_LIMIT || ld_relaxed(bar + 1) != 0u)) {
                ok = 0;
                break;
            }
        }
        if (!ok) atomicExch(bar + 1, 1u);
        *s_ok = ok;
    }
    __syncthreads();
    return *s_ok != 0;
}

// Gather of one output from the staged x by a warp: entries q0 .. qe in
// device memory, lane l takes q0 + l, q0 + l + 32, ... in one chain, eight
// loads in flight; returned in every lane.
__device__ __forceinline__ double gather_row(const unsigned short* __restrict__ ei, const double* __restrict__ ev,
                                             const double* xs, int q0, int qe, int lane, int ncorr, const double* hc,
                                             const double* zc, int64_t zld) {
    constexpr int U = 8;
    double b = 0.0;
    int q = q0 + lane;
    for (; q + (U - 1) * 32 < qe; q += U * 32) {
        double v[U];
        unsigned short i[U];
#pragma unroll
        for (int k = 0; k < U; ++k) {
            v[k] = ev[q + 32 * k];
            i[k] = ei[q + 32 * k];
        }
#pragma unroll
        for (int k = 0; k < U; ++k) b += v[k] * xs[i[k]];
    }
#pragma unroll 4
    for (; q < qe; q += 32) b += ev[q] * xs[ei[q]];
    for (int c = lane; c < ncorr; c += 32) b -= hc[c] * zc[c * zld];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) b += __shfl_xor_sync(0xffffffffu, b, o);
    return b;
}

// asynchronous copy of n 8-byte elements into shared memory by the CTA (16
// bytes at a time, past L1, when the source is aligned)
__device__ __forceinline__ void stage_vector(void* dst, const void* src, int64_t n) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    const char* s = static_cast<const char*>(src);
    if ((reinterpret_cast<uintptr_t>(src) & 15) == 0) {
        for (int i = threadIdx.x; i < (int)(n >> 1); i += PT)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d + 16 * i), "l"(s + 16 * (size_t)i) : "memory");
        if ((n & 1) && threadIdx.x == 0)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d + 8 * (unsigned)(n - 1)),
                         "l"(s + 8 * (size_t)(n - 1))
                         : "memory");
    } else {
        for (int i = threadIdx.x; i < (int)n; i += PT)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d + 8 * i), "l"(s + 8 * (size_t)i) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}
__device__ __forceinline__ void stage_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

__device__ __forceinline__ double warp_sum(double a) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    return a;
}

// out[c] = sum over CTAs b of P[c nb + b], c < ncols (the partials are
// stored column by column, so a column is one contiguous run), identical in every
// CTA; used for the norms of v and of an explicitly normalised w''.  Each thread sums a fixed subset of rows of one column (all its loads
// issued at once), the subset sums go through shared memory and one thread
// per column adds them in a fixed order: FP64 additions with every lane
// busy, no shuffle trees.  P was written by other CTAs during this launch:
// L2 loads.
__device__ __forceinline__ void colsum(const double* P, int nb, int ncols, double* out, double* tmp) {
    // RS row slots per column; ncols * RS <= max(PT, 4 ncols)
    const int RS = ncols <= PT / 32 ? 32 : (ncols <= PT / 16 ? 16 : (ncols <= PT / 8 ? 8 : 4));
    for (int base = 0; base < ncols * RS; base += PT) {
        const int t = base + threadIdx.x;
        if (t < ncols * RS) {
            const int c = t / RS, k0 = t - (t / RS) * RS;
            double v[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int k = k0 + RS * q;
                v[q] = k < nb ? __ldcg(P + (int64_t)c * nb + k) : 0.0;
            }
            // the trip count depends on nb and RS only: uniform, so the
            // additions past the last row slot are not issued
            double acc = v[0];
#pragma unroll
            for (int q = 1; q < 8; ++q)
                if (RS * q < nb) acc += v[q];
            for (int k = k0 + 8 * RS; k < nb; k += RS) acc += __ldcg(P + (int64_t)c * nb + k);
            tmp[t] = acc;
        }
    }
    __syncthreads();
    if ((int)threadIdx.x < ncols) {
        const double* tc = tmp + threadIdx.x * RS;
        double a0 = 0.0, a1 = 0.0;
        for (int k = 0; k < RS; k += 2) {
            a0 += tc[k];
            a1 += tc[k + 1];
        }
        out[threadIdx.x] = a0 + a1;
    }
}

// Exact sums across CTAs.  A CTA's partial p of an inner product is taken as
// the 128-bit integer P = trunc(p 2^sh) (two's complement; sh from a bound on
// |p| such that |P| < 2^110), formed and added by integer operations (the FP64
// pipe issues one warp instruction per 64 clocks).  Integer addition is
// associative: the total is exact whatever the order of arrival, and every
// CTA reads back the same value, in every run.
struct Fix {
    unsigned long long lo, hi;
    bool bad;  // not finite or outside the range
};
__device__ __forceinline__ Fix fx_fixed(double p, int sh) {
    const unsigned long long bits = (unsigned long long)__double_as_longlong(p);
    int e = (int)((bits >> 52) & 0x7ff);
    unsigned long long m = bits & 0xfffffffffffffull;
    Fix f;
    f.bad = e == 0x7ff;
    if (e) m |= 1ull << 52;
    else e = 1;
    const int s = e - 1075 + sh;  // P = m 2^s
    f.bad = f.bad || s > 61;
    if (s >= 0) {
        f.lo = m << (s & 63);
        f.hi = s ? m >> ((64 - s) & 63) : 0ull;
    } else {
        f.lo = s > -64 ? m >> (-s & 63) : 0ull;
        f.hi = 0ull;
    }
    if (f.bad) f.lo = f.hi = 0ull;
    if ((long long)bits < 0) {
        f.lo = ~f.lo + 1ull;
        f.hi = ~f.hi + (f.lo == 0ull ? 1ull : 0ull);
    }
    return f;
}
__device__ __forceinline__ void fx_sum(Fix& f, unsigned long long lo, unsigned long long hi) {
    f.lo += lo;
    f.hi += hi + (f.lo < lo ? 1ull : 0ull);
}
// x rounded to 53 significant bits (ties to even); true when that carries out
__device__ __forceinline__ bool fx_round53(unsigned long long& x) {
    const int drop = 11 - __clzll((long long)x);
    if (drop <= 0) return false;
    const unsigned long long keep = x >> drop, rest = x - (keep << drop), half = 1ull << (drop - 1);
    const unsigned long long up = keep + (rest > half || (rest == half && (keep & 1ull)) ? 1ull : 0ull);
    x = up << drop;
    return (up >> (64 - drop)) != 0ull;
}
// P 2^-sh in FP64: the words are rounded to 53 bits one by one, then their
// sum (two conversions and an FMA, by integer operations)
__device__ __forceinline__ double fx_value(Fix f, int sh) {
    const bool neg = (long long)f.hi < 0;
    if (neg) {
        f.lo = ~f.lo + 1ull;
        f.hi = ~f.hi + (f.lo == 0ull ? 1ull : 0ull);
    }
    if (f.bad) return __longlong_as_double(0x7ff8000000000000ll);
    if ((f.lo | f.hi) == 0ull) return 0.0;
    fx_round53(f.hi);  // below 2^58: no carry
    if (fx_round53(f.lo)) ++f.hi;
    // leading bit to bit 127
    if (f.hi == 0ull) {
        f.hi = f.lo;
        f.lo = 0ull;
        sh += 64;
    }
    const int lz = __clzll((long long)f.hi);
    if (lz) f.hi = (f.hi << lz) | (f.lo >> (64 - lz));
    f.lo <<= lz;
    const int ex = 127 - lz - sh;  // value = 1.xxx 2^ex
    unsigned long long m = f.hi >> 11;
    const unsigned rem = (unsigned)(f.hi & 0x7ffull) | (f.lo ? 1u : 0u);
    m += rem > 0x400u || (rem == 0x400u && (m & 1ull)) ? 1ull : 0ull;  // to nearest, ties to even
    const unsigned long long bits = ((unsigned long long)(ex + 1022) << 52) + m;
    return __longlong_as_double((long long)(bits | (neg ? 1ull << 63 : 0ull)));
}
// df_from_double(x), by integer operations where the pair is normal
__device__ __forceinline__ float2 fx_pair(double x) {
    const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
    const int e = (int)((bits >> 52) & 0x7ff);
    if (e < 949 || e > 1149) return df_to_float2(df_from_double(x));
    // |x| = m 2^(e - 1075): the leading 24 bits to nearest (ties to even), and
    // the rest, which the conversion rounds likewise
    const unsigned long long m = (bits & 0xfffffffffffffull) | (1ull << 52);
    unsigned q = (unsigned)(m >> 29);
    const unsigned rest = (unsigned)m & 0x1fffffffu;
    q += rest > 0x10000000u || (rest == 0x10000000u && (q & 1u)) ? 1u : 0u;
    const int l = (int)((long long)m - ((long long)q << 29));
    const int sign = (long long)bits < 0 ? (int)0x80000000 : 0;
    return make_float2((float)q * __int_as_float(((e - 919) << 23) | sign),
                       (float)l * __int_as_float(((e - 948) << 23) | sign));
}
// Adds a CTA's sum into its copy of a column: P in three words of 56, 56 and
// 16 bits, whose sums over 255 CTAs fit 64; the fourth word counts invalid
// partials.
constexpr unsigned long long FX_M56 = (1ull << 56) - 1;
__device__ __forceinline__ void fx_add(unsigned long long* a, const Fix& f) {
    if (f.bad) {
        atomicAdd(a + 3, 1ull);
        return;
    }
    atomicAdd(a, f.lo & FX_M56);
    atomicAdd(a + 1, ((f.lo >> 56) | (f.hi << 8)) & FX_M56);
    atomicAdd(a + 2, (unsigned long long)((long long)f.hi >> 48));
}

// out[c] (and its pair in outdf when that is not null) = the sum of column c
// < nt (the last one scaled by sh_last), after the barrier that follows the
// additions; by the whole CTA: one thread per column and copy loads the
// copy's four words (two 16-byte L2 loads: other CTAs added them), the copies
// are added by shuffles.  (One thread per column loading all 32 words takes
// 1 900 clocks.  Words that count their own arrivals, polled by their readers
// in place of the barrier, took 6 000 to 11 000 clocks a phase against 5 000:
// the polls hold up the additions they wait for.)
__device__ __forceinline__ void fx_columns(const unsigned long long* set, int nt, int sh, int sh_last, double* out,
                                           float2* outdf) {
    static_assert(FX_COPIES == 8, "eight lanes per column");
    const int k = threadIdx.x & 7;
    for (int base = 0; base < nt; base += PT / 8) {
        const int c = base + (int)(threadIdx.x >> 3);
        ulonglong2 u = make_ulonglong2(0ull, 0ull), v = u;
        if (c < nt) {
            const ulonglong2* p = reinterpret_cast<const ulonglong2*>(set + ((size_t)k * FX_COLS + c) * FX_LIMBS);
            u = __ldcg(p);
            v = __ldcg(p + 1);
        }
        const bool bad = __any_sync(0xffu << (threadIdx.x & 24), v.y != 0ull);
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) {
            u.x += __shfl_xor_sync(0xffffffffu, u.x, o);
            u.y += __shfl_xor_sync(0xffffffffu, u.y, o);
            v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
        }
        if (c < nt && k == 0) {
            // u.x + u.y 2^56 + v.x 2^112 modulo 2^128
            Fix f{u.x, 0ull, bad};
            fx_sum(f, u.y << 56, (u.y >> 8) + (v.x << 48));
            out[c] = fx_value(f, c == nt - 1 ? sh_last : sh);
            if (outdf) outdf[c] = fx_pair(out[c]);
        }
    }
}

// The inner products of the staged slice with its basis columns, sum_{u < ne}
// Vl[c vld + u] ws[u] for c < ncols and with norm also sum ws[u]^2 as column
// ncols: emit(c, sum) by one thread per column.  CH lanes per column (a power
// of two, the most with nt CH <= PT, at most 32) sum strided elements in two
// chains; the CH partials of a column are added in a fixed tree, quarters by
// four threads, then the four by shuffles (129 columns: two and two).  FP64
// additions all of them, in an order that is kept to the bit (see arnoldi.cu);
// adding the lanes' products as integers by shuffles took fewer clocks and
// moved the results of solves that amplify roundings.  An FP64 instruction
// takes 64 clocks, so additions of lanes without an element are left out, and
// a slice of up to four elements (the smallest problems) takes one thread per
// column (432 x 30: 443 us per exponential, 467 without).  tmp holds PT
// doubles.
template <typename Emit>
__device__ __forceinline__ void slice_dots(const double* Vl, int64_t vld, int ncols, const double* ws, int ne,
                                           bool norm, double* tmp, Emit&& emit) {
    static_assert(2 * (SGK_MAX_KRYLOV + 1) <= PT, "two lanes a column");
    const int nt = ncols + (norm ? 1 : 0);
    int CH = 32;
    while (CH > 2 && nt * CH > PT) CH >>= 1;
    const int t = threadIdx.x;
    if (ne <= 4 && CH > 2) {
        // lanes 0..3 with one product each, in the tree's order
        for (int c = t; c < nt; c += PT) {
            const double* vc = c < ncols ? Vl + c * vld : ws;
            double p[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) p[u] = u < ne ? __dmul_rn(vc[u], ws[u]) : 0.0;
            if (ne > 1) p[0] = __dadd_rn(p[0], p[1]);
            if (ne > 2 && CH <= 8) p[0] = __dadd_rn(p[0], __dadd_rn(p[2], p[3]));
            if (ne > 2 && CH > 8) p[0] = __dadd_rn(__dadd_rn(p[0], p[2]), p[3]);
            emit(c, p[0]);
        }
        return;
    }
    if (t < nt * CH) {
        const int c = t / CH, k = t - (t / CH) * CH;
        const double* vc = c < ncols ? Vl + c * vld : ws;
        double a = 0.0, b = 0.0;
        int u = k;
        // long slices lie in L2: several loads in flight
        for (; u + 7 * CH < ne; u += 8 * CH) {
            double v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = vc[u + i * CH];
#pragma unroll
            for (int i = 0; i < 8; i += 2) {
                a += v[i] * ws[u + i * CH];
                b += v[i + 1] * ws[u + (i + 1) * CH];
            }
        }
        for (; u + CH < ne; u += 2 * CH) {
            a += vc[u] * ws[u];
            b += vc[u + CH] * ws[u + CH];
        }
        if (u < ne) a += vc[u] * ws[u];
        tmp[t] = ne > CH ? a + b : a;
    }
    __syncthreads();
    // whole warps: column t / Q, part t % Q
    const int Q = CH < 4 ? CH : 4, per = CH / Q;
    if ((t & ~31) < nt * Q) {
        const int col = min(t, nt * Q - 1);
        const double* p = tmp + col * per;
        const int live = min(per, ne - (col & (Q - 1)) * per);
        double a = p[0];
        for (int i = 1; i < live; ++i) a += p[i];
        if (ne > per) a += __shfl_xor_sync(0xffffffffu, a, 1);
        if (Q == 4 && ne > 2 * per) a += __shfl_xor_sync(0xffffffffu, a, 2);
        if (t < nt * Q && (t & (Q - 1)) == 0) emit(t / Q, a);
    }
}

// sum_{c < ncols} Vl[c vld + u] h[c] for the elements u < ne of the slice, in
// two parts with a CTA barrier between them: combine_begin calls use(u, sum)
// for the elements below the number it returns (all or none), combine_end for
// the others.  The FP64 pipe of a scheduler takes 64 clocks a warp
// instruction, so an element per thread, four chains each, costs 64 ncols
// clocks for every four warps of elements begun.  Slices of one to three warps
// split their columns over the four schedulers instead, 16 ncols clocks a
// warp, where that saves more than the sums in tmp (PT doubles) behind the
// barrier, some 300 clocks.  Per exponential, FP64, never split against this:
// 432 x 30 457 -> 443 us, 1 024 x 30 493 -> 478, 5 504 x 25 432 -> 424, 11 520 x
// 40 839 -> 820; splitting the part beyond four warps of longer slices as well
// made 20 480 x 40 1130 us out of 1087.  The same chains and sums either way,
// so the slicing changes no bit.
template <typename Use>
__device__ __forceinline__ int combine_begin(const double* Vl, int64_t vld, int ncols, const double* h, int ne,
                                             double* tmp, Use&& use) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int warps = (ne + 31) >> 5;
    const int whole = warps < 4 && (4 - warps) * ncols >= 20 ? 0 : ne;
    for (int u = threadIdx.x; u < whole; u += PT) {
        const double* vi = Vl + u;
        double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
        int c = 0;
#pragma unroll 2
        for (; c + 3 < ncols; c += 4) {
            a0 += vi[c * vld] * h[c];
            a1 += vi[(c + 1) * vld] * h[c + 1];
            a2 += vi[(c + 2) * vld] * h[c + 2];
            a3 += vi[(c + 3) * vld] * h[c + 3];
        }
        for (; c < ncols; ++c) a0 += vi[c * vld] * h[c];
        use(u, (a0 + a1) + (a2 + a3));
    }
    const int part = wid & 3, blk = (wid >> 2) * 32 + lane, u = whole + blk;
    if (u < ne) {
        double a = 0.0;
        const int full = ncols & ~3;
        for (int c = part; c < full; c += 4) a += Vl[c * vld + u] * h[c];
        if (part == 0)
            for (int c = full; c < ncols; ++c) a += Vl[c * vld + u] * h[c];
        tmp[part * (PT / 4) + blk] = a;
    }
    return whole;
}
template <typename Use>
__device__ __forceinline__ void combine_end(int whole, int ne, const double* tmp, Use&& use) {
    if ((int)threadIdx.x < ne - whole) {
        const double* p = tmp + threadIdx.x;
        use(whole + (int)threadIdx.x, (p[0] + p[PT / 4]) + (p[2 * (PT / 4)] + p[3 * (PT / 4)]));
    }
}
template <typename Use>
__device__ __forceinline__ void slice_combine(const double* Vl, int64_t vld, int ncols, const double* h, int ne,
                                              double* tmp, Use&& use) {
    const int whole = combine_begin(Vl, vld, ncols, h, ne, tmp, use);
    if (whole < ne) {
        __syncthreads();
        combine_end(whole, ne, tmp, use);
    }
}

// sum of x^2 over the staged slice, written by thread 0 to *out
__device__ __forceinline__ void slice_norm2(const double* ws, int ne, double* red, double* out) {
    double a = 0.0;
    for (int u = threadIdx.x; u < ne; u += PT) a += ws[u] * ws[u];
    a = warp_sum(a);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = a;
    __syncthreads();
    if (threadIdx.x < 32) {
        const double t = warp_sum(threadIdx.x < PNW ? red[threadIdx.x] : 0.0);
        if (threadIdx.x == 0) *out = t;
    }
}

// The Arnoldi process of one exponential on a grid of nb CTAs of which this
// CTA is number b (slice b).  Every CTA of the grid calls it with the same
// arguments; a failed barrier or a breakdown returns from it in every CTA.
template <int D, int KP1, int G, bool DF>
__device__ __forceinline__ void arnoldi_body(const GmvArgs<double, D>& ga, const ArnArgs& a, const int nb,
                                             const int b) {
    // dynamic shared memory: [with eo1, x: n, 16-byte multiple][w slices: 2 E][Vs: (M+1) Es][Zs: (M+1) Es]
    // [located rows, or gather offsets and entries]
    extern __shared__ __align__(16) double smem_dyn[];
    __shared__ double h1[SGK_MAX_KRYLOV + 2];
    __shared__ double h2[SGK_MAX_KRYLOV + 2];
    __shared__ double red[PNW];
    __shared__ double s_scal[4], s_beta;
    // column-sum and combination staging: <= max(PT, 4 (SGK_MAX_KRYLOV + 2))
    __shared__ double ctmp[PT > 4 * (SGK_MAX_KRYLOV + 2) ? PT : 4 * (SGK_MAX_KRYLOV + 2)];
    __shared__ int s_ok, s_flag;
    // double-float matvec: the correction's coefficients and the step's scale
    __shared__ float2 h2df[DF ? SGK_MAX_KRYLOV + 2 : 1];
    __shared__ float2 s_scaldf;
    const int64_t n = a.n;
    const int E = a.E;  // longest slice
    const int64_t lo = a.bounds ? a.bounds[b] : std::min<int64_t>(n, (int64_t)b * E);
    const int ne = (int)((a.bounds ? a.bounds[b + 1] : std::min<int64_t>(n, lo + E)) - lo);
    // the staged slice of w, two buffers alternating by step: the update of
    // step j (v_{j+1} from w') runs during the matvec of step j + 1
    double* const xstage = smem_dyn;
    double* const smem = smem_dyn + (a.eo1 ? (n + 1) / 2 * 2 : 0);
    double* const wsb0 = smem;
    double* const wsb1 = smem + E;
    // shared columns of V and Z have an odd stride: the lanes of one output
    // read different columns of Z at the same row without bank conflicts
    const int Es = E | 1;
    double* const Vs = a.smem_vz ? smem + 2 * E : nullptr;
    double* const Zs = a.smem_vz ? smem + 2 * E + (size_t)(a.M + 1) * Es : nullptr;
    unsigned char* const tail =
        reinterpret_cast<unsigned char*>(smem + 2 * E + (a.smem_vz ? 2 * (size_t)(a.M + 1) * Es : 0));
    GmvLoc<D, int>* const sloc = a.smem_loc ? reinterpret_cast<GmvLoc<D, int>*>(tail) : nullptr;
    // pre-located gathers of the slice: offsets rebased to the slice's first
    // entry, then the entries
    int* const seoff = a.list_cap > 0 || a.eo1 ? reinterpret_cast<int*>(tail) : nullptr;
    int2* const sent = a.list_cap > 0 ? reinterpret_cast<int2*>(tail + arn_eoff_bytes(E, D)) : nullptr;
    // this slice's basis and raw-output columns: shared copies or HBM
    const double* const Vl = a.smem_vz ? Vs : a.V + lo;
    const int64_t vld = a.smem_vz ? Es : n;
    double* const Zl = a.smem_vz ? Zs : a.Z + lo;
    const int64_t zld = a.smem_vz ? Es : n;
    float2* const Zdf = reinterpret_cast<float2*>(Zl);  // Z as (hi, lo) pairs (double-float matvec)
    double* const P2 = a.pbuf;  // norms
    unsigned epoch = 0;
    const bool alone = nb == 1 && a.bar_extra == 0u;  // one CTA: nothing to wait for or to add up
    auto barrier = [&]() {
        if (alone) {
            __syncthreads();
            return true;
        }
        ++epoch;
        const bool ok = grid_barrier(a.bar, epoch * (unsigned)nb + a.bar_extra, &s_ok);
        if (!ok) stage_wait();  // the CTA leaves: none of its copies may land later
        return ok;
    };
    // Fixed-point reductions: the two phases of step j add into sets
    // 2 (j % 3) and 2 (j % 3) + 1, each read after a barrier.  After step j's
    // first barrier every CTA has left step j - 1, and CTA 0 clears that
    // step's sets for step j + 2; its arrival at step j's second barrier, which
    // every CTA waits for, orders the clearing before that use.
    auto fx_set = [&](int j, int phase) { return a.acc + (size_t)(2 * (j % 3) + phase) * FX_SET; };
    // inner products of the slice into a phase (or straight to out)
    auto dots = [&](int j, int phase, double* out, float2* outdf) {
        const int nc = j + 1;
        unsigned long long* set = fx_set(j, phase) + (size_t)(b % FX_COPIES) * FX_COLS * FX_LIMBS;
        slice_dots(Vl, vld, nc, (j & 1) ? wsb1 : wsb0, ne, phase == 1, ctmp, [&](int c, double p) {
            const int sh = c < nc ? a.sh_h : a.sh_n;
            const Fix f = fx_fixed(p, sh);
            if (alone) {
                out[c] = fx_value(f, sh);
                if (outdf) outdf[c] = fx_pair(out[c]);
            } else {
                fx_add(set + (size_t)c * FX_LIMBS, f);
            }
        });
    };
    // and their sums over the CTAs
    auto collect = [&](int j, int phase, double* out, float2* outdf) {
        if (!barrier()) return false;
        if (!alone) {
            fx_columns(fx_set(j, phase), j + 1 + phase, a.sh_h, phase ? a.sh_n : a.sh_h, out, outdf);
            __syncthreads();
        }
        return true;
    };
    const int r = threadIdx.x & (G - 1);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    // the warps that form the step's scalars: those with the least to gather
    constexpr int WNORM = PNW - 1, WCOL = PNW - 2;
    KrylovScalars* ks = a.ks;
    if (sloc)
        for (int u = threadIdx.x; u < ne; u += PT) gmv_locate<double, D, KP1>(ga, lo + u, sloc[u]);
    if (a.eo1) {
        for (int i = threadIdx.x; i <= ne; i += PT) seoff[i] = a.eo1[lo + i];
    } else if (seoff) {
        const int e0 = a.eoff[lo * D], ecount = a.eoff[(lo + ne) * D] - e0;
        if (ecount > a.list_cap) {  // the host sized the list for every slice; fail rather than overrun
            if (threadIdx.x == 0) atomicExch(a.bar + 1, 1u);
            return;
        }
        for (int i = threadIdx.x; i <= ne * D; i += PT) seoff[i] = a.eoff[lo * D + i] - e0;
        for (int i = threadIdx.x; i < ecount; i += PT) sent[i] = a.ent[e0 + i];
    }
    if (!DF && a.eo1) stage_vector(xstage, a.v, n);  // the first gathers read v

    // the accumulator sets start cleared (before the first barrier)
    auto clear_set = [&](unsigned long long* set, int cols) {
        for (int i = threadIdx.x; i < FX_COPIES * cols * FX_LIMBS; i += PT)
            set[(size_t)(i / (cols * FX_LIMBS)) * FX_COLS * FX_LIMBS + i % (cols * FX_LIMBS)] = 0ull;
    };
    if (b == 0 && !alone)
        for (int i = 0; i < FX_SETS; ++i) clear_set(a.acc + (size_t)i * FX_SET, a.M + 1);
    // gamma = ||v||
    for (int u = threadIdx.x; u < ne; u += PT) wsb0[u] = a.v[lo + u];
    __syncthreads();
    slice_norm2(wsb0, ne, red, P2 + b);
    if (!barrier()) return;
    colsum(P2, nb, 1, s_scal, ctmp);
    __syncthreads();
    // scalar FP64 work (square roots, reciprocals, the Frobenius norm of H)
    // stays on warp 0 and is broadcast through shared memory: FP64 issue is
    // about two operations per clock per SM on this part
    if (threadIdx.x == 0) {
        const double gamma = sqrt(s_scal[0]);
        s_scal[1] = gamma > 0.0 ? 1.0 / gamma : 0.0;
        if (DF) s_scaldf = df_to_float2(df_from_double(s_scal[1]));
        if (b == 0) {
            ks->gamma = gamma;
            ks->inv_gamma = s_scal[1];
            ks->fro2 = 0.0;
            ks->stop = gamma > 0.0 ? 0 : 1;
            ks->m_eff = 0;
            ks->breakdown = 0;
        }
    }
    __syncthreads();
    if (!(s_scal[1] > 0.0)) {  // gamma = 0: the same decision in every CTA
        stage_wait();
        return;
    }
    double scale = s_scal[1];
    for (int u = threadIdx.x; u < ne; u += PT) {
        const double y = wsb0[u] * scale;
        a.V[lo + u] = y;
        if (Vs) Vs[u] = y;
        // with the double-float matvec the first gathers read the pairs of
        // v / gamma from w1 (free until the second step writes it): pairs of
        // FP32 numbers have FP32's exponent range, so the pairs of an
        // unnormalised v would lose their low parts below about 1e-30 and
        // their values below about 1e-38
        if (DF) reinterpret_cast<float2*>(a.w1)[lo + u] = df_to_float2(df_from_double(y));
    }
    if (DF) {
        // one more barrier publishes the pairs; the first product is then
        // A v_0 itself (scale 1)
        if (!barrier()) return;
        scale = 1.0;
        if (threadIdx.x == 0) s_scaldf = df_to_float2(df_from_double(1.0));
        __syncthreads();
    }
    // the next matvec gathers x (written by all CTAs) and forms
    // A v_j = scale (A x - corr), corr = sum_c h2_c A v_c over the previous
    // step's columns: with the norm taken by Pythagoras, x is w' (complete at
    // the second phase) and A v_j = (A w' - A V h2) / beta, A V being the
    // stored raw matvec outputs of the slice; after an explicit norm x is w''
    const double* x = a.v;
    const float2* xdf = reinterpret_cast<const float2*>(a.w1);
    int ncorr = 0;                 // columns of the correction (0: none)
    // ||H||_F^2 without the last subdiagonal (warp WCOL), and that one's square
    // (every thread)
    double fro2 = 0.0, sub2 = 0.0;
    // the pending update of the previous step: v_{pj+1} on the slice from
    // that step's staged w (w' - V h2, or w'' after an explicit norm) times
    // its scale, into column pj + 1 of V (global and shared).  The sums over
    // the columns need no scale: they are taken before the barrier behind the
    // gathers, where warps wait for those with long rows, and the rest after it
    int pj = -1;
    bool pexpl = false;
    auto pending_begin = [&]() {
        double* const wp = (pj & 1) ? wsb1 : wsb0;
        return pj < 0 || pexpl ? ne : combine_begin(Vl, vld, pj + 1, h2, ne, ctmp, [&](int u, double sum) { wp[u] -= sum; });
    };
    auto pending_end = [&](int whole) {
        if (pj < 0) return;
        const double* const wp = (pj & 1) ? wsb1 : wsb0;
        double* vg = a.V + (int64_t)(pj + 1) * n + lo;
        double* vs = Vs ? Vs + (int64_t)(pj + 1) * Es : nullptr;
        const double pscale = s_scal[1];
        auto put = [&](int u, double sum) {
            const double y = (wp[u] - sum) * pscale;
            vg[u] = y;
            if (vs) vs[u] = y;
        };
        for (int u = threadIdx.x; u < whole; u += PT) put(u, 0.0);
        combine_end(whole, ne, ctmp, put);
    };
    if (threadIdx.x == 0) s_scal[1] = scale;
    for (int j = 0; j < a.M; ++j) {
        double* w = (j & 1) ? a.w1 : a.w0;
        double* const ws = (j & 1) ? wsb1 : wsb0;
        const int nc = j + 1;
        // A v_j on this slice before its scale, which one warp may still be
        // forming: raw sums into the staged slice (a double, or a pair)
        if (!DF && a.eo1) {
            stage_wait();
            __syncthreads();
            // a warp per output: the rows are long and uneven (hundreds of
            // entries, thousands at low levels)
            for (int u = wid; u < ne; u += PNW) {
                const double acc = gather_row(a.ei, a.ev, xstage, seoff[u], seoff[u + 1], lane, ncorr, h2, Zl + u, zld);
                if (lane == 0) ws[u] = acc;
            }
        }
        for (int base = 0; base < (a.eo1 ? 0 : ne); base += PT / G) {
            const int u = base + (int)threadIdx.x / G;
            const bool live = u < ne;
            const int uu = live ? u : 0;
            // the correction's columns are dealt over the virtual lanes like
            // the matrix rows (sum independent of G)
            if constexpr (DF) {
                const df64 ad = gmv_accumulate_list_df<D, G>(seoff + uu * D, sent, a.cvk2, xdf, r, live, ncorr, h2df,
                                                             Zdf + uu, zld);
                if (live && r == 0) reinterpret_cast<float2*>(ws)[u] = df_to_float2(ad);
            } else {
                double acc;
                if (seoff) {
                    acc = gmv_accumulate_list<D, G>(seoff + uu * D, sent, ga.cvk, x, r, live, ncorr, h2, Zl + uu, zld);
                } else if (sloc) {
                    acc = gmv_accumulate<double, D, G, 2, true>(ga, x, sloc[uu], r, live, ncorr, h2, Zl + uu, zld);
                } else {
                    GmvLoc<D, int> l1;
                    if (live) gmv_locate<double, D, KP1>(ga, lo + u, l1);
                    acc = gmv_accumulate<double, D, G, 2, true>(ga, x, l1, r, live, ncorr, h2, Zl + uu, zld);
                }
                if (live && r == 0) ws[u] = acc;
            }
        }
        const int whole = pending_begin();
        __syncthreads();
        // the scale is there: A v_j staged and kept in Z, by the upper half of
        // the CTA, which the pending update's last sums leave idle
        for (int u = (int)threadIdx.x - PT / 2; u < ne; u += PT / 2) {
            if (u < 0) break;
            if constexpr (DF) {
                const df64 ad = df_mul(df_from_float2(reinterpret_cast<const float2*>(ws)[u]), df_from_float2(s_scaldf));
                ws[u] = df_to_double(ad);
                Zdf[(int64_t)j * zld + u] = df_to_float2(ad);
            } else {
                const double acc = ws[u] * s_scal[1];
                ws[u] = acc;
                Zl[(int64_t)j * zld + u] = acc;
            }
        }
        pending_end(whole);
        __syncthreads();
        dots(j, 0, h1, nullptr);
        if (!collect(j, 0, h1, nullptr)) return;
        if (b == 0 && j > 0 && !alone) {
            clear_set(fx_set(j + 2, 0), nc);
            clear_set(fx_set(j + 2, 1), nc + 1);
        }
        // w' = w - V h1, published for the next matvec
        slice_combine(Vl, vld, nc, h1, ne, ctmp, [&](int u, double sum) {
            const double y = ws[u] - sum;
            ws[u] = y;
            if (DF) reinterpret_cast<float2*>(w)[lo + u] = df_to_float2(df_from_double(y));
            else w[lo + u] = y;
        });
        __syncthreads();
        // second pass: V^T w' and ||w'||^2 in one reduction
        dots(j, 1, h2, DF ? h2df : nullptr);
        if (!collect(j, 1, h2, DF ? h2df : nullptr)) return;
        // the next gathers' vector, copied while the scalars are formed (again
        // after an explicit norm, which changes it)
        if (!DF && a.eo1 && j + 1 < a.M) stage_vector(xstage, w, n);
        // ||w''||^2 = ||w'||^2 - ||h2||^2 (V orthonormal, w'' = w' - V h2).
        // As a rule h2 is rounding and its square below half a unit in the
        // last place of ||w'||^2, which is then the norm as it stands, and far
        // above a breakdown; integer comparisons of exponents tell, alike in
        // every warp, and the next gathers start at once while one warp forms
        // 1 / beta (scalar FP64 work is latency, 64 clocks an operation).
        auto inverse_norm = [&](double b2) {  // one warp
            const bool ok = b2 > 0.0 && b2 < 1.7976931348623157e308;
            const double inv = ok ? rsqrt(b2) : 0.0;
            if (lane == 0) {
                s_scal[1] = inv;
                s_scal[3] = ok ? b2 : 0.0;
                if (DF) s_scaldf = df_to_float2(df_from_double(inv));
                s_beta = b2 * inv;
                if (b == 0) a.H[(int64_t)(j + 1) * a.M + j] = s_beta;
            }
        };
        auto column_of_h = [&]() {  // one warp: ||h1 + h2||^2, CTA 0 stores the column
            double part = 0.0;
            for (int i = lane; i < nc; i += 32) {
                const double hv = h1[i] + h2[i];
                part += hv * hv;
                if (b == 0) a.H[(int64_t)i * a.M + j] = hv;
            }
            fro2 += sub2 + warp_sum(part);
        };
        unsigned hm = 0u;
        for (int i = lane; i < nc; i += 32)
            hm = max(hm, (unsigned)(__double_as_longlong(h2[i]) >> 32) & 0x7fffffffu);
        hm = __reduce_max_sync(0xffffffffu, hm);
        const long long wb = __double_as_longlong(h2[nc]);
        const int eh = (int)(hm >> 20), ew = (int)(wb >> 52);
        // h2_i^2 < 2^(2 (eh - 1022)), nc <= 2^7 of them, against 2^(ew - 1023 - 55)
        const bool plain = wb > __double_as_longlong(a.no_brk) && ew < 0x7ff && eh < 0x7ff &&
                           2 * (eh - 1022) + 7 <= ew - 1023 - 55;
        bool explicit_norm = false;
        if (plain) {
            if (wid == WNORM) inverse_norm(h2[nc]);
            else if (wid == WCOL) column_of_h();
            sub2 = h2[nc];
        } else {
            // near breakdown: when the second pass removed more than 1e-3 of
            // ||w'||^2 the norm is summed explicitly
            if (wid == WNORM) {
                double hh = 0.0;
                for (int i = lane; i < nc; i += 32) hh += h2[i] * h2[i];
                hh = warp_sum(hh);
                const double wn2 = h2[nc], b2 = wn2 - hh;
                if (lane == 0) s_flag = !(hh <= 1e-3 * wn2) || !(b2 > 0.0);
                inverse_norm(b2);
            } else if (wid == WCOL) {
                column_of_h();
                // the square of 1e-12 ||H||_F; no value of beta passes a NaN
                if (lane == 0) s_scal[2] = fro2 == fro2 ? 1e-24 * fro2 : 1.7976931348623157e308;
            }
            __syncthreads();
            explicit_norm = s_flag != 0;
            if (explicit_norm) {
                // w'' in place (published), its norm through a barrier
                if (!DF && a.eo1) {  // the first copy must not land over the second
                    stage_wait();
                    __syncthreads();
                }
                slice_combine(Vl, vld, nc, h2, ne, ctmp, [&](int u, double sum) {
                    const double y = ws[u] - sum;
                    ws[u] = y;
                    if (DF) reinterpret_cast<float2*>(w)[lo + u] = df_to_float2(df_from_double(y));
                    else w[lo + u] = y;
                });
                __syncthreads();
                slice_norm2(ws, ne, red, P2 + b);
                if (!barrier()) return;
                colsum(P2, nb, 1, s_scal, ctmp);
                __syncthreads();
                if (wid == WNORM) inverse_norm(s_scal[0]);
                if (!DF && a.eo1 && j + 1 < a.M) stage_vector(xstage, w, n);
                __syncthreads();
            }
            sub2 = s_scal[3];
            // breakdown: beta not above 1e-12 ||H||_F, the same decision in
            // every thread of every CTA (squares, which order like their bit
            // patterns: neither is negative or a NaN)
            if (!(__double_as_longlong(sub2) > __double_as_longlong(s_scal[2]))) {
                if (b == 0 && threadIdx.x == 0) {
                    ks->m_eff = j + 1;
                    ks->stop = 1;
                    ks->breakdown = 1;
                }
                stage_wait();
                return;
            }
        }
        if (b == 0 && threadIdx.x == 0) ks->m_eff = j + 1;
        // v_{j+1} is formed after the next step's gathers (which read w',
        // published, and need no column of V); the inner products after it
        // read column j + 1
        pj = j;
        pexpl = explicit_norm;
        ncorr = explicit_norm ? 0 : nc;
        x = w;
        xdf = reinterpret_cast<const float2*>(w);
    }
    const int whole = pending_begin();
    __syncthreads();
    pending_end(whole);  // the last column, v_M
}

template <int D, int KP1, int G, bool DF>
__global__ void __launch_bounds__(PT, 1) arnoldi_kernel(const GmvArgs<double, D> ga, const ArnArgs a) {
    arnoldi_body<D, KP1, G, DF>(ga, a, gridDim.x, blockIdx.x);
}

// Many independent Arnoldi processes in one cooperative launch.  CTA c runs
// the work items item_off[c] .. item_off[c+1]-1 in order; item (i, b) makes
// it slice b of instance i's grid of nb[i] CTAs.  The host builds the lists
// from one global order of the instances (each instance's slices take the
// same position in every list that holds them), and every CTA is resident,
// so no CTA waits on an instance that cannot start: an instance's barriers
// only involve the CTAs of its own items.
template <int D>
struct ArnMulti {
    const int* item_off;  // gridDim.x + 1
    const int2* items;    // (instance, slice)
    const GmvArgs<double, D>* ga;
    const ArnArgs* aa;
    const int* nb;
};

template <int D, int KP1, int G, bool DF>
__global__ void __launch_bounds__(PT, 1) arnoldi_multi_kernel(const ArnMulti<D> m) {
    __shared__ ArnArgs s_a;
    __shared__ GmvArgs<double, D> s_ga;
    __shared__ int s_nb;
    const int first = m.item_off[blockIdx.x], last = m.item_off[blockIdx.x + 1];
    for (int it = first; it < last; ++it) {
        const int2 w = m.items[it];
        __syncthreads();  // the previous item is done with shared memory
        {
            const int* src = reinterpret_cast<const int*>(m.aa + w.x);
            int* dst = reinterpret_cast<int*>(&s_a);
            for (int i = threadIdx.x; i < (int)(sizeof(ArnArgs) / sizeof(int)); i += PT) dst[i] = src[i];
            const int* gsrc = reinterpret_cast<const int*>(m.ga + w.x);
            int* gdst = reinterpret_cast<int*>(&s_ga);
            for (int i = threadIdx.x; i < (int)(sizeof(GmvArgs<double, D>) / sizeof(int)); i += PT) gdst[i] = gsrc[i];
            if (threadIdx.x == 0) s_nb = m.nb[w.x];
        }
        __syncthreads();
        arnoldi_body<D, KP1, G, DF>(s_ga, s_a, s_nb, w.y);
    }
}

// Launch arguments of one Arnoldi process (arnoldi_prepare).
struct ArnPrep {
    ArnArgs a;
    size_t smem = 0;
    int nb = 0, G = 0, d = 0, kp1 = 0;
};

// Device copies of the matvec arguments of a list of operators (d = D).
template <int D>
void arn_multi_upload_ga(const std::vector<const sgk_op*>& ops, DevBuf<unsigned char>& buf, cudaStream_t st) {
    std::vector<GmvArgs<double, D>> v;
    v.reserve(ops.size());
    for (const sgk_op* op : ops) v.push_back(make_gmv_args<double, D>(op));
    buf.alloc(v.size() * sizeof(GmvArgs<double, D>));
    buf.upload(reinterpret_cast<const unsigned char*>(v.data()), buf.n, st);
}

template <int D, int KP1, int G>
void arn_multi_launch(cudaStream_t st, bool df, const ArnMulti<D>& m, int grid, size_t smem, size_t smem_optin,
                      int num_sms) {
    auto kern = df ? arnoldi_multi_kernel<D, KP1, G, true> : arnoldi_multi_kernel<D, KP1, G, false>;
    allow_max_dynamic_smem(smem_optin, kern);
    int occ = 0;
    SGK_CUDA_CHECK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, PT, smem));
    SGK_REQUIRE(occ >= 1 && grid <= occ * num_sms, SGK_EUNSUPPORTED, "batched Arnoldi grid does not fit");
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(PT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    SGK_CUDA_CHECK(cudaLaunchKernelEx(&cfg, kern, m));
}

// Batched launch for d = D: degree (k + 1 = kp1) and lanes per output (4 or
// 8) select the kernel; ga points at the device GmvArgs<double, D> array.
template <int D>
void arn_multi_launch_k(cudaStream_t st, int kp1, int G, bool df, const int* item_off, const int2* items,
                        const void* ga, const ArnArgs* aa, const int* nb, int grid, size_t smem, size_t smem_optin,
                        int num_sms) {
    ArnMulti<D> m;
    m.item_off = item_off;
    m.items = items;
    m.ga = static_cast<const GmvArgs<double, D>*>(ga);
    m.aa = aa;
    m.nb = nb;
#define SGK_ARN_MULTI(K, GG)                                                            \
    if (kp1 == K && G == GG) {                                                          \
        arn_multi_launch<D, K, GG>(st, df, m, grid, smem, smem_optin, num_sms);         \
        return;                                                                         \
    }
    SGK_ARN_MULTI(2, 4) SGK_ARN_MULTI(2, 8) SGK_ARN_MULTI(3, 4) SGK_ARN_MULTI(3, 8) SGK_ARN_MULTI(4, 4)
    SGK_ARN_MULTI(4, 8)
#undef SGK_ARN_MULTI
    throw SgkError{SGK_EUNSUPPORTED, "batched Arnoldi: no kernel for this degree and lane count"};
}

template <int D, int KP1, int G>
void arn_launch(sgk_ctx* ctx, const sgk_op* op, const ArnArgs& a, int nb, size_t smem) {
    auto kern = a.df ? arnoldi_kernel<D, KP1, G, true> : arnoldi_kernel<D, KP1, G, false>;
    const GmvArgs<double, D> ga = make_gmv_args<double, D>(op);
    allow_max_dynamic_smem(ctx->smem_optin, kern);
    int occ = 0;
    SGK_CUDA_CHECK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, PT, smem));
    SGK_REQUIRE(occ >= 1 && nb <= occ * ctx->num_sms, SGK_EUNSUPPORTED, "persistent Arnoldi grid does not fit");
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(nb);
    cfg.blockDim = dim3(PT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = ctx->stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    SGK_CUDA_CHECK(cudaLaunchKernelEx(&cfg, kern, ga, a));
}

template <int D, int KP1>
void arn_launch_g(sgk_ctx* ctx, const sgk_op* op, const ArnArgs& a, int nb, size_t smem, int G) {
    switch (G) {
        case 1: arn_launch<D, KP1, 1>(ctx, op, a, nb, smem); break;
        case 2: arn_launch<D, KP1, 2>(ctx, op, a, nb, smem); break;
        case 4: arn_launch<D, KP1, 4>(ctx, op, a, nb, smem); break;
        default: arn_launch<D, KP1, 8>(ctx, op, a, nb, smem); break;
    }
}

template <int D>
void arn_launch_k(sgk_ctx* ctx, const sgk_op* op, const ArnArgs& a, int nb, size_t smem, int G) {
    switch (op->idx->k + 1) {
        case 2: arn_launch_g<D, 2>(ctx, op, a, nb, smem, G); break;
        case 3: arn_launch_g<D, 3>(ctx, op, a, nb, smem, G); break;
        case 4: arn_launch_g<D, 4>(ctx, op, a, nb, smem, G); break;
        default: throw SgkError{SGK_EUNSUPPORTED, "persistent Arnoldi: degree must be 1..3"};
    }
}

}  // namespace sgk_arn
