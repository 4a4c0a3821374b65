// chem_kernel.cuh -- batched backward-Euler chemistry step (sm_103a).
//
// One warp holds 32/G cell slots; the G lanes of a slot cooperate on one
// cell.  All slots of a warp execute the same instruction stream: one Newton
// iteration of Eq. 29 for every slot per trip of the warp loop, so a slot
// whose cell finishes picks up the next cell from a global work counter
// between iterations, without stalling the other slots.  Per-cell state,
// rates, the Jacobian and its LU live in shared memory; HBM only sees the
// cell state (SoA) on load and store.
//
// FP64 is the binding pipe on this part: 2 DFMA/clk/SM against 128 FFMA, and a
// partly masked FP64 instruction or an FP64<->FP32 conversion costs a full
// FP64 slot.  So:
//   - each phase is one loop over a flat, uniform work list (reactions, D
//     entries, Jacobian entries ordered by gather length and interleaved by
//     pass, fixed-size chunks of the species lists);
//   - coefficients are stored in the type they are used in, and the mixed
//     path converts between FP64 and FP32 on the integer pipe;
//   - pivot searches, range choices and finiteness tests compare integer
//     keys; reciprocals refine rcp.approx; exp is a short table-driven
//     evaluation, once per reaction (K_f) and once per species (the split
//     exponentials the equilibrium constants are multiplied from), and the
//     temperature recovery a multiplied-out polynomial.
// Both paths eliminate the energy unknown through the conservation of total
// energy, so the elimination runs on the ns species unknowns.  The mixed
// path (JT = float) keeps the FP64 residual, rates, sources and
// temperature, and moves everything that only feeds the Jacobian to FP32;
// it writes the Jacobian's rank-two part and the identity densely, four
// rows per store, then adds the sparse reaction sums, and its LU is in
// registers (24 to 36 unknowns) or organised by columns.  It is bound by
// latency and by the FP64 pipe (57 % busy), so its slot layout is cut to what
// it reads (20 warps per SM at 36 species), and its FP32 arithmetic keeps its
// order to the bit: another rounding of the Jacobian changes the substep
// schedules of some 4 % of the cells.
//   Code size: with 20 warps at different phases, the instructions of one
// Newton iteration have to stay in the SM's instruction caches.  The
// compiler's unrolling of the many short runtime-count loops made the mixed
// kernel 114 KB, and instruction fetch its first stall; every loop below is
// therefore kept rolled (#pragma unroll 1) unless it says otherwise, and
// the few unrolled bodies are written out by hand.
#pragma once

#include <cuda_runtime.h>
#include <math_constants.h>

#include <type_traits>

#include "chem_fp64.cuh"
#include "chem_internal.h"

namespace chem {

constexpr unsigned kFull = 0xffffffffu;

enum SlotState : int {
    kFree = 0,        // needs a cell
    kInitT = 1,       // needs the temperature of its input state
    kNewtonT = 2,     // needs the temperature of the current Newton iterate
    kNewtonReady = 3, // runs a Newton iteration this trip
    kCheckT = 4,      // needs the temperature of a converged iterate
    kRejected = 5,    // its substep attempt failed
    kDead = 6         // no more cells
};
// What a slot's settled state asks for, done in one place per pass (each
// copy of that code would take its share of the instruction caches).
enum SlotAction : int {
    kNoAction = 0,
    kStartSubstep = 1,
    kFailSubstep = 2,
    kEmitCell = 3
};

// The sum of a warp's doubles by integer additions: the terms become 58-bit
// fixed-point numbers at the largest one's exponent, rounded, which
// redux.sync adds in three pieces, and the sum is rounded to a double once.
// No FP64 operation, where a tree of shuffles takes five.  Against the exact
// sum of 32 terms the largest error is 1.3e-16 of the sum of magnitudes, the
// tree's 4.7e-16.  The FP64 path's seven sums an iteration: 16,384 cells of
// 36 species 92.3 -> 90.6 ms.  (The mixed path has four, and gains nothing:
// 94.0 against 94.2 ms for 65,536 cells.)  Returns false (and no sum) where
// an exponent is at the ends of the range: a term below 2^-895 as the
// largest, infinities, NaN.
__device__ __forceinline__ bool warp_sum(double v, double &sum) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const unsigned hi = (unsigned)(b >> 32), e = (hi >> 20) & 0x7ffu;
    const unsigned em = __reduce_max_sync(kFull, e);
    if (em - 128u >= 0x7f0u - 128u) return false;
    unsigned long long f = ((b & 0xfffffffffffffULL) | 0x10000000000000ULL) << 6;
    f = ((f >> min(em - e, 63u)) + 1) >> 1;
    if (e == 0) f = 0;   // zero (or negligible)
    const long long F = (int)hi < 0 ? -(long long)f : (long long)f;
    const unsigned l = __reduce_add_sync(kFull, (unsigned)F & 0xffffffu);
    const unsigned m = __reduce_add_sync(kFull, (unsigned)(F >> 24) & 0xffffffu);
    const int h = __reduce_add_sync(kFull, (int)(F >> 48));
    const long long S = ((long long)h << 48) + ((long long)m << 24) + (long long)l;
    const unsigned long long a = (unsigned long long)(S < 0 ? -S : S);
    const int lz = __clzll((long long)a);
    const unsigned long long n = a << lz;
    // (the mantissa's leading bit adds one to the exponent)
    unsigned long long r = ((unsigned long long)(em + 5 - lz) << 52) + (n >> 11) + ((n >> 10) & 1);
    if (S < 0) r |= 0x8000000000000000ULL;
    sum = S == 0 ? 0.0 : __longlong_as_double((long long)r);
    return true;
}

template <int G>
struct Grp {
    template <typename V>
    __device__ __forceinline__ static V sum(V v) {
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
        return v;
    }
    template <bool INT>
    __device__ __forceinline__ static double sum(double v, const Fp64Ops &op) {
        double r;
        if (INT && G == 32 && warp_sum(v, r)) return r;
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) v = op.add(v, __shfl_xor_sync(kFull, v, o));
        return v;
    }
    __device__ __forceinline__ static int any(int v) {
        if constexpr (G == 32) {
            return __any_sync(kFull, v);
        } else {
#pragma unroll
            for (int o = G / 2; o > 0; o >>= 1) v |= __shfl_xor_sync(kFull, v, o);
            return v;
        }
    }
    // maximum of non-negative doubles on the integer pipe (their bit
    // patterns order the same way; a NaN, whose bits are larger than any
    // number's, wins): for a whole warp the high words by redux.sync, then
    // the low words of the lanes holding the high maximum
    __device__ __forceinline__ static double max_nonneg(double v) {
        unsigned long long b = (unsigned long long)__double_as_longlong(v);
        if constexpr (G == 32) {
            const unsigned hi = (unsigned)(b >> 32);
            const unsigned mhi = __reduce_max_sync(kFull, hi);
            const unsigned mlo = __reduce_max_sync(kFull, hi == mhi ? (unsigned)b : 0u);
            return __longlong_as_double((long long)(((unsigned long long)mhi << 32) | mlo));
        } else {
#pragma unroll
            for (int o = G / 2; o > 0; o >>= 1) {
                const unsigned long long b2 = __shfl_xor_sync(kFull, b, o);
                b = b2 > b ? b2 : b;
            }
            return __longlong_as_double((long long)b);
        }
    }
    // largest key, lowest index on ties
    template <typename K>
    __device__ __forceinline__ static void argmax(K &k, int &i) {
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) {
            const K k2 = __shfl_xor_sync(kFull, k, o);
            const int i2 = __shfl_xor_sync(kFull, i, o);
            if (k2 > k || (k2 == k && i2 < i)) {
                k = k2;
                i = i2;
            }
        }
    }
};

template <typename JT> __device__ __forceinline__ JT to_jt(double v);
template <> __device__ __forceinline__ double to_jt<double>(double v) { return v; }
template <> __device__ __forceinline__ float to_jt<float>(double v) { return d2f_rz(v); }
__device__ __forceinline__ double to_f64(double v) { return v; }
__device__ __forceinline__ double to_f64(float v) { return f2d_alu(v); }

// Argmax over a whole warp (one cell per warp) with redux.sync: the largest
// key, the lowest index on ties, as the shuffle tree gives it.  FP64 keys
// take the high word, then the low word among the lanes holding the high
// maximum; FP32 keys fit one word.
__device__ __forceinline__ void warp_argmax(unsigned long long &k, int &i) {
    const unsigned hi = (unsigned)(k >> 32), lo = (unsigned)k;
    const unsigned mhi = __reduce_max_sync(kFull, hi);
    const unsigned mlo = __reduce_max_sync(kFull, hi == mhi ? lo : 0u);
    i = (int)__reduce_min_sync(kFull, (hi == mhi && lo == mlo) ? (unsigned)i : 0xffffffffu);
    k = ((unsigned long long)mhi << 32) | mlo;
}
__device__ __forceinline__ void warp_argmax(unsigned &k, int &i) {
    const unsigned m = __reduce_max_sync(kFull, k);
    i = (int)__reduce_min_sync(kFull, k == m ? (unsigned)i : 0xffffffffu);
    k = m;
}

// |v| as an ordered integer key (NaN maps to 0 so it is never the pivot).
__device__ __forceinline__ unsigned long long abs_key(double v) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffULL;
    return b > 0x7ff0000000000000ULL ? 0ULL : b;
}
__device__ __forceinline__ unsigned abs_key(float v) {
    const unsigned b = __float_as_uint(v) & 0x7fffffffu;
    return b > 0x7f800000u ? 0u : b;
}
__device__ __forceinline__ bool key_is_inf(unsigned long long k) { return k >= 0x7ff0000000000000ULL; }
__device__ __forceinline__ bool key_is_inf(unsigned k) { return k >= 0x7f800000u; }
// the pivot key of a matrix type: 64 bits for FP64, 32 for FP32
template <typename JT>
using PivotKey = decltype(abs_key(JT(0)));

// FP32 reciprocal of the pivot: the hardware approximation (within an ulp or
// two), enough for an elimination whose result Newton refines in FP64.
__device__ __forceinline__ float frcp(float a) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
    return r;
}

// The library exp for the arguments the table path does not take; kept out
// of line so its code is not repeated at every call site.
static __device__ __noinline__ double exp_outside(double x) { return exp(x); }

// A small signed integer (|v| < 2^22) as a float without a conversion
// instruction: add it to the bit pattern of 1.5 * 2^23, whose ulp is 1.
__device__ __forceinline__ float small_int_to_float(int v) {
    return __int_as_float(0x4B400000 + v) - 12582912.0f;
}
// The coefficient of a packed list word (a signed power of two stored as
// the sign and exponent bits of its double, over the reaction index in bits
// 0..19) as a double and as a float, by integer operations only: the
// float's exponent is the double's less 1023 - 127.
__device__ __forceinline__ double word_nu_double(unsigned wv) {
    return __hiloint2double((int)(wv & 0xfff00000u), 0);
}
__device__ __forceinline__ float word_nu_float(unsigned wv) {
    const unsigned hi = wv & 0xfff00000u;
    return __int_as_float((int)((hi & 0x80000000u) | (((hi & 0x7ff00000u) - 0x38000000u) << 3)));
}

// A positive integer below 2^20 as a double from integer operations only
// (biased exponent of its top bit, the bits below it), exact.
__device__ __forceinline__ double small_pos_int_to_double(int v) {
    const int e = 31 - __clz(v);
    const unsigned hi = ((unsigned)(1023 + e) << 20) | (((unsigned)v << (20 - e)) & 0xfffffu);
    return __hiloint2double((int)hi, 0);
}

// exp by the table-driven reduction of P. T. P. Tang, ACM TOMS 15(2), 1989:
// x = (256 k + j) ln2/256 + r with |r| about ln2/512, exp(x) = 2^k 2^(j/256)
// e^r, 2^(j/256) from a 256-entry table and e^r - 1 = r (1 + r (1/2 + r t)).
//   The FP64 pipe bounds the step, so only what needs 53 bits is left to it:
// five operations.
//   The integer n = 256 k + j is rounded in FP32 (near a half it may be the
// next one, which only moves r past ln2/512, to 0.0014) and becomes a double
// on the integer pipe.
//   r is x less n times ln2/256 rounded to 53 bits: exact, a multiple of
// 2^-61 below 2^-9.  What the constant lacks, d = -n 9.06e-20 of at most
// 2e-14, is FP32's and comes as d (1 + r) with the last multiplication.
//   t = 1/6 + r/24 is FP32 from r rounded, its error of 2^-27 standing behind
// r^3 < 2^-28; its constant is two units above 1/6, which stands for the next
// term's r^2/120.
//   Against extended precision on [-64, 64] the largest error is 1.24 ulp and
// the root mean square 0.418 ulp; with all of it in FP64 (eight operations, t
// without the next term) they were 1.32 and 0.421.  exp_near: y 2^(n >> 8) =
// exp(x) for |x| <= 1024.
__device__ __forceinline__ double exp_near(double x, const double *tab, const Fp64Ops &op, int &n) {
    const double2 c0 = ld_const2(tab + kConstExp);
    const float z = fmaf(near_float(x), 369.32993f, 12582912.f);   // x * 256/ln2 + 1.5 * 2^23
    n = __float_as_int(z) - 0x4b400000;
    const float nf = z - 12582912.f;
    const double r = fma(f2d_int(nf), c0.x, x);
    const float rf = near_float(r), d = nf * -0x1.abc9e4p-64f;
    double p = fma(r, f2d_pos(fmaf(rf, 0x1.555556p-5f, 0x1.555558p-3f)), c0.y);
    p = fma(r, p, op.one);
    p = fma(p, r, f2d_int(fmaf(d, rf, d)));   // e^r - 1
    const double s = __ldg(tab + (n & (kExpTab - 1)));
    return fma(s, p, s);
}
// |x| >= 512, infinities and NaN (decided on the exponent bits, no FP64
// compare) fall back to the library exp.
__device__ __forceinline__ double fexp(double x, const double *tab, const Fp64Ops &op) {
    const unsigned hi = (unsigned)((unsigned long long)__double_as_longlong(x) >> 32);
    if (((hi >> 20) & 0x7ffu) > 0x407u) return exp_outside(x);
    int n;
    const double y = exp_near(x, tab, op, n);   // |n| < 2^18
    const long long k = (long long)(n >> 8);
    return __longlong_as_double(__double_as_longlong(y) + (k << 52));
}

// exp(x) = y 2^k with y in [0.99, 2.01]: the reduction of fexp without its
// final scaling, so that products of many exponentials can be formed
// without overflow.  From |x| = 1024 on the reduction is in FP64 throughout:
// exact up to its two roundings for any |x| < 2^22 (the products with
// ln2/256 are fused, and the table index fits an int); beyond that (and for
// infinities) k saturates at +-2^24 with y = 1, and a NaN x gives a NaN y.
struct SplitExp {
    double y;
    int k;
};
static __device__ __noinline__ SplitExp split_exp_far(double x, const double *tab) {
    const unsigned hi = (unsigned)((unsigned long long)__double_as_longlong(x) >> 32);
    const unsigned ex = (hi >> 20) & 0x7ffu;
    if (ex >= 0x415u) {
        const bool nan = ex == 0x7ffu && ((hi & 0xfffffu) | (unsigned)__double_as_longlong(x));
        return SplitExp{nan ? x : 1.0, (hi >> 31) ? -(1 << 24) : (1 << 24)};
    }
    const double t = fma(x, 369.3299304675746, 6755399441055744.0);   // + 1.5 * 2^52: rounded to an integer
    const int n = (int)(unsigned)__double_as_longlong(t);
    const double nd = t - 6755399441055744.0;
    double r = fma(nd, -0x1.62e42fefa0000p-9, x);   // ln2/256 in two parts
    r = fma(nd, -0x1.cf79abc9e3b3ap-48, r);
    const double p = r * fma(r, fma(r, fma(r, 1.0 / 24.0, 1.0 / 6.0), 0.5), 1.0);
    const double s = __ldg(tab + (n & (kExpTab - 1)));
    return SplitExp{fma(s, p, s), n >> 8};
}
__device__ __forceinline__ void split_exp(double x, const double *tab, const Fp64Ops &op, double &y, int &k) {
    const unsigned hi = (unsigned)((unsigned long long)__double_as_longlong(x) >> 32);
    if (((hi >> 20) & 0x7ffu) > 0x408u) {
        const SplitExp f = split_exp_far(x, tab);
        y = f.y;
        k = f.k;
        return;
    }
    int n;
    y = exp_near(x, tab, op, n);
    k = n >> 8;
}
// v 2^k on the exponent bits for a normal v; zero, subnormal, infinite and
// NaN v come back unchanged, a result below the normal range is a signed
// zero and one above it an infinity.
__device__ __forceinline__ double scale_pow2(double v, int k) {
    const long long b = __double_as_longlong(v);
    const int e = (int)((b >> 52) & 0x7ff);
    if (e == 0 || e == 0x7ff) return v;
    const int ne = e + k;
    const long long sgn = b & (long long)0x8000000000000000ULL;
    if (ne <= 0) return __longlong_as_double(sgn);
    if (ne >= 0x7ff) return __longlong_as_double(sgn | 0x7ff0000000000000LL);
    return __longlong_as_double(b + ((long long)k << 52));
}

// ln x for x >= 2 by the table-driven reduction of P. T. P. Tang, ACM TOMS
// 16(4), 1990: x = 2^k y with y in [1, 2), F = 1 + j/128 the table point
// nearest to y (j = 0..128), f = y - F (exact, |f| <= 2^-8), u = f (1/F),
// and ln x = k ln2 + ln F + ln(1 + u) with ln(1 + u) by its series to u^6
// (truncation below 2^-56 / 7), within 1.5 ulp.  The terms from u^4 on are
// formed in FP32 (their error of 2^-26 stands behind u^4 < 2^-32, the result
// is at least 0.69): eight FP64 operations.  {1/F, ln F} come from a table;
// k becomes a double on the integer pipe.  (Below 2
// the result can be small next to k ln2 + ln F, and the table's rounding
// then leaves an absolute error near 1e-16.  The kernels take it of T in
// [200, 6000] K.)
__device__ __forceinline__ double flog(double x, const double2 *tab, const double *exp_tab, const Fp64Ops &op) {
    const long long b = __double_as_longlong(x);
    const int k = (int)(b >> 52) - 1023;
    const double y = __longlong_as_double((b & 0x000fffffffffffffLL) | 0x3ff0000000000000LL);
    const int j = (int)((b >> 45) & 0x7f) + (int)((b >> 44) & 1);
    const double F = __longlong_as_double(0x3ff0000000000000LL + ((long long)j << 45));
    const double2 t = __ldg(tab + j);
    const double2 c1 = ld_const2(exp_tab + kConstLog), c2 = ld_const2(exp_tab + kConstLog + 2);
    const double u = op.mul(op.sub(y, F), t.x);
    const float uf = near_float(u), w = fmaf(uf, fmaf(uf, 1.f / 6.f, -0.2f), 0.25f);
    double p = fma(-u, f2d_pos(w), c1.x);   // 1/3 - u (1/4 - u/5 + u^2/6)
    p = fma(u, p, c1.y);                    // -1/2
    p = fma(u, p, op.one);
    const double kd = f2d_alu(small_int_to_float(k));
    return fma(u, p, fma(kd, c2.x, t.y));   // ln 2
}

// NASA-7 entropy from the thermo coefficients of one species and range
// (layout in chem_internal.h)
__device__ __forceinline__ double nasa_s(const CoefRow<double> &th, double T, double lnT, const Fp64Ops &op) {
    return op.add(fma(th[0], lnT, op.mul(T, fma(T, fma(T, fma(T, th[12], th[11]), th[10]), th[1]))), th[13]);
}
// Sums over a cell's species with one species per lane (wide warps, below),
// in the order of G0 lanes per cell: lane l of those sums the terms l, l + G0,
// ... one after another, then the partial sums meet in a tree.  Terms i >= cnt
// (at most 32 lanes) are not there; `first` is added to lane 0's partial sum.
// Every lane gets the result.
template <int G0>
__device__ __forceinline__ double wide_dot(double a, double b, int cnt, const Fp64Ops &op, double first = 0.0,
                                           bool has_first = false) {
    const int l = threadIdx.x & (G0 - 1);
    double p = 0.0;
#pragma unroll 1
    for (int i = l; i - l < cnt; i += G0) {
        const double x = __shfl_sync(kFull, a, i), y = __shfl_sync(kFull, b, i);
        if (i < cnt) p = fma(x, y, p);
    }
    if (has_first && l == 0) p = op.add(p, first);
#pragma unroll
    for (int o = G0 / 2; o > 0; o >>= 1) p = op.add(p, __shfl_xor_sync(kFull, p, o));
    return p;
}
template <int G0>
__device__ __forceinline__ float wide_dotf(float a, float b, int cnt, float first = 0.f, bool has_first = false) {
    const int l = threadIdx.x & (G0 - 1);
    float p = 0.f;
#pragma unroll 1
    for (int i = l; i - l < cnt; i += G0) {
        const float x = __shfl_sync(kFull, a, i), y = __shfl_sync(kFull, b, i);
        if (i < cnt) p = fmaf(x, y, p);
    }
    if (has_first && l == 0) p += first;
#pragma unroll
    for (int o = G0 / 2; o > 0; o >>= 1) p += __shfl_xor_sync(kFull, p, o);
    return p;
}

// Temperature recovery from (rho_s, e) for every slot whose `need` is set:
// Newton on sum_s rho_s e_s^sens(T) = e, safeguarded by bisection on
// [kTlo, kThi] (Eq. 3 with the kinetic energy left to the flux stage).  A
// Newton step of at most kTstep T ends it: with the derivative good to 1e-7
// (c_v changes by less than a millionth at a t_mid that is no kink) the
// temperature is then good to 1e-15, and another pass would only confirm that.
// A step from near a kink, which may cross it with the other side's
// derivative, ends it at kTtol T.  Uniform across the warp.
//   `cold` slots have no guess, and no energy steps down at a t_mid, or up by
// a thousandth of it: where no density is negative either (so that e(T) is
// increasing and has one root) three Newton steps in FP32 find one, from which
// two FP64 passes suffice instead of six.
//   A diverging substep's densities, some negative and large, often have no
// temperature, and halving the bracket down to one of its ends takes up to 48
// passes to find that out: 36 species, mixed, 4 % of the recoveries took two
// thirds of the passes.  So once a Newton step leaves the bracket, the
// residual is held against the most that it can change over the bracket,
// `slope` = sum |rho_s| max c_v,s times the bracket's width and, however
// narrow it is, times the kelvins step_K that the energies' steps at t_mid
// are worth: a larger one keeps its sign, and the passes would have ended at
// the bracket's end, as this does.  (A hundredth of the width and of a kelvin
// on top keep later Newton steps from ending inside the bracket first: none
// could be below 0.01 K.)
//   The energies come from the multiplied-out polynomials (five DFMA per
// species, no 1/T); with F32 the derivative sum c_v is formed in FP32, which
// changes the Newton steps by a relative 1e-7 and not the root.  Without, a
// slot whose last step was below a millionth of T and near no kink keeps its
// derivative (it has changed by no more than that, and the step after is below
// 1e-12 T), and a pass of such slots forms the energies alone: 2^19 cells of 9
// species 26.8 -> 26.3 ms.
template <int G, int G0, bool F32>
__device__ __forceinline__ void recover_T(const DeviceMech &m, const double *tab, const double *x, int sl, bool need,
                                          bool cold, double guess, double &T_out, bool &ok) {
    const int ns = m.ns;
    const Fp64Ops op = fp64_ops(tab);
    double lo = kTlo, hi = kThi, T = guess;
    if (!(bits_gt(T, lo) && bits_lt(T, hi))) T = 1500.0;
    bool done = !need;
    ok = false;
    float slope = CUDART_INF_F;
    const double e = x[ns];
    if (__any_sync(kFull, cold)) {
        float Tf = 1500.f;
        int neg = 0;
#pragma unroll 1
        for (int it = 0; it < 3; ++it) {
            const long long Tb = __double_as_longlong(f2d_alu(Tf));
            float f = 0.f, fp = 0.f, wr = 0.f;
#pragma unroll 1
            for (int s = sl; s < ns; s += G) {
                const auto d = coef_row(m.tpoly_f, ns, s, thermo_range(m, s, Tb));
                const float r = d2f_rz(x[s]);
                neg |= r < 0.f;
                const float es = fmaf(fmaf(fmaf(fmaf(fmaf(d[10], Tf, d[9]), Tf, d[8]), Tf, d[7]), Tf, d[6]), Tf, d[5]);
                const float cv = fmaf(fmaf(fmaf(fmaf(d[4], Tf, d[3]), Tf, d[2]), Tf, d[1]), Tf, d[0]);
                if constexpr (G == G0) {
                    f = fmaf(r, es, f);
                    fp = fmaf(r, cv, fp);
                } else {
                    wr = r;
                    f = es;
                    fp = cv;
                }
            }
            if constexpr (G == G0) {
                f = Grp<G>::sum(f);
                fp = Grp<G>::sum(fp);
            } else {
                f = wide_dotf<G0>(wr, f, ns);
                fp = wide_dotf<G0>(wr, fp, ns);
            }
            f -= d2f_rz(e);
            Tf -= __fdividef(f, fp);
            Tf = fminf(fmaxf(Tf, (float)kTlo), (float)kThi);   // (a NaN goes to the lower end)
        }
        neg = Grp<G>::any(neg);
        const double Ts = f2d_alu(Tf);
        if (cold && !neg && bits_gt(Ts, lo) && bits_lt(Ts, hi)) T = Ts;
    }
    bool near = false;   // (FP64) the last step was small: the derivative is kept
    double rfp = 0.0;
#pragma unroll 1
    for (int it = 1; it <= kTmaxIter; ++it) {
        if (!__any_sync(kFull, !done)) break;
        const bool slopes = F32 || __any_sync(kFull, !done && !near);
        // (FP64: in front of the sums, 2^20 cells of 9 species 51.8 ms, behind
        // them 52.2; mixed behind them, 2^18 of 36 species 354.1 and 358.7 ms)
        bool kink = !F32 && near_kink(m, T);
        const long long Tb = __double_as_longlong(T);
        const float Tf = F32 ? d2f_rz(T) : 0.f;
        double f = 0.0, fp = 0.0, xs = 0.0;
        float fpf = 0.f, xf = 0.f;
#pragma unroll 1
        for (int s = sl; s < ns; s += G) {
            const int rg = thermo_range(m, s, Tb);
            const auto c = coef_row(m.tpoly, ns, s, rg);
            const double es = fma(fma(fma(fma(fma(c[5], T, c[4]), T, c[3]), T, c[2]), T, c[1]), T, c[0]);
            xs = x[s];
            if constexpr (G == G0)
                f = fma(xs, es, f);
            else
                f = es;
            if (F32) {
                const auto d = coef_row(m.tpoly_f, ns, s, rg);
                const float cv = fmaf(fmaf(fmaf(fmaf(d[4], Tf, d[3]), Tf, d[2]), Tf, d[1]), Tf, d[0]);
                xf = d2f_rz(xs);
                if constexpr (G == G0)
                    fpf = fmaf(xf, cv, fpf);
                else
                    fpf = cv;
            } else if (slopes) {
                const double cv = fma(fma(fma(fma(c[10], T, c[9]), T, c[8]), T, c[7]), T, c[6]);
                if constexpr (G == G0)
                    fp = fma(xs, cv, fp);
                else
                    fp = cv;
            }
        }
        if constexpr (G == G0)
            f = Grp<G>::template sum<!F32>(f, op);
        else
            f = wide_dot<G0>(xs, f, ns, op);
        f = op.sub(f, e);
        if (F32) {
            if constexpr (G == G0)
                fpf = Grp<G>::sum(fpf);
            else
                fpf = wide_dotf<G0>(xf, fpf, ns);
            rfp = f2d_alu(__frcp_rn(fpf));
        } else if (slopes) {
            if constexpr (G == G0)
                fp = Grp<G>::template sum<!F32>(fp, op);
            else
                fp = wide_dot<G0>(xs, fp, ns, op);
            // (whatever the warp's other slots need, for the same bits)
            if (!near) rfp = frcp1(fp, op);
        }
        bool left = false;
        if (!done) {
            const long long fb = __double_as_longlong(f);
            if ((fb << 1) == 0) {
                done = true;
                ok = true;
            } else {
                if (fb > 0)
                    hi = T;
                else
                    lo = T;
                // (comparisons of non-negative doubles on their bit patterns)
                double Tn = fma(-f, rfp, T), dT = op.sub(Tn, T);
                const bool inside = bits_gt(Tn, lo) && bits_lt(Tn, hi);
                if (F32) kink = inside && near_kink(m, T);
                const double tol = (inside && !kink ? kTstep : kTtol) * T;
                // (a step below half an ulp leaves T at an end of the bracket:
                // it ends the recovery, bisecting would start it all over)
                if (!inside && bits_gt(fabs(dT), tol)) {
                    Tn = 0.5 * (lo + hi);
                    dT = op.sub(Tn, T);
                    left = true;
                }
                if (!F32) near = inside && !kink && !bits_gt(fabs(dT), 1e-6 * T);
                T = Tn;
                if (!bits_gt(fabs(dT), tol)) {
                    done = true;
                    ok = bits_gt(T, kTlo * (1.0 + 1e-9)) && bits_lt(T, kThi * (1.0 - 1e-9));
                }
            }
        }
        if (__any_sync(kFull, left)) {
            if (__any_sync(kFull, left && slope == CUDART_INF_F)) {
                slope = 0.f;
#pragma unroll 1
                for (int s = sl; s < ns; s += G) slope = fmaf(fabsf(d2f_rz(x[s])), __ldg(m.cv_max + s), slope);
                slope = Grp<G>::sum(slope);
            }
            // (infinities and NaN compare false)
            if (left && fabsf(d2f_rz(f)) > slope * fmaf(1.01f, d2f_rz(hi) - d2f_rz(lo), m.step_K)) done = true;
        }
    }
    if (need) T_out = T;
}

// FP32 trailing update a_ik -= a_ij (a_jk / a_jj) of elimination step j
// (i > j, k > j, the right-hand side column n included) on the column-major
// matrix A[k*ld + i], ld a multiple of 4.  A lane owns a column, keeps
// a_jk / a_jj in a register and walks its rows four at a time with 16-byte
// loads and stores; the a_ij of the pivot column are 16-byte broadcast
// reads.  When fewer columns than lanes remain, the rows of each column are
// split over 2, 4, ... lanes at multiples of four rows.  The multipliers are
// never stored: the right-hand side is eliminated with the matrix, and back
// substitution reads U only.  Each element gets fma(-a_ij, a_jk / a_jj, a_ik)
// whichever lane computes it.
template <int G>
__device__ __forceinline__ void lu_update_colmajor(float *A, int ld, int n, int j, int sl, float inv) {
    const int C = n - j, r0 = j + 1;
    if (r0 >= n) return;
    int kc = sl, i0 = r0, i1 = n;
    if (C < G) {
        const int lg = C > 1 ? 32 - __clz(C - 1) : 0;   // columns rounded up to 2^lg
        const int lgB = (__ffs(G) - 1) - lg;              // lanes per column, log2
        kc = sl & ((1 << lg) - 1);
        if (kc >= C) return;
        const int part = sl >> lg, base = r0 & ~3;
        const int rows = ((((n - base) + (1 << lgB) - 1) >> lgB) + 3) & ~3;
        i0 = max(r0, base + part * rows);
        i1 = min(n, base + (part + 1) * rows);
    }
    const float *cj = A + j * ld;
#pragma unroll 1
    for (int k = j + 1 + kc; k <= n; k += G) {
        float *ck = A + k * ld;
        const float ajk = ck[j] * inv;
        int i = i0;
#pragma unroll 1
        for (; i < i1 && (i & 3); ++i) ck[i] = fmaf(-cj[i], ajk, ck[i]);
#pragma unroll 1
        for (; i + 4 <= i1; i += 4) {
            const float4 l = *reinterpret_cast<const float4 *>(cj + i);
            float4 v = *reinterpret_cast<const float4 *>(ck + i);
            v.x = fmaf(-l.x, ajk, v.x);
            v.y = fmaf(-l.y, ajk, v.y);
            v.z = fmaf(-l.z, ajk, v.z);
            v.w = fmaf(-l.w, ajk, v.w);
            *reinterpret_cast<float4 *>(ck + i) = v;
        }
#pragma unroll 1
        for (; i < i1; ++i) ck[i] = fmaf(-cj[i], ajk, ck[i]);
    }
}

// FP32 elimination of [A | rhs] and back substitution with the matrix in
// registers (one cell per warp, kLuRegMinN <= N <= kLuRegN unknowns).  Lane l
// holds row l, one column per register; the rows past 32 (at most four) are
// spread over eight lanes each.  Rows never move: id0 (and id1 of the lane's
// row past 32) carries the index the row would have after the swaps, and is
// negative once the row has been a pivot.  Step j: two redux find the pivot
// (largest |a_ij|, then the lowest index), its owner writes the row's columns
// j .. N to shared memory (row j of U, from A's start on), and every lane
// reads them back and updates its rows with fma(-a_ij, a_jk / a_jj, a_ik): the
// pivots and roundings of lu_update_colmajor.  The results move one register
// down, so that column j is always in register 0 and the loop body is one
// copy of the code.  The solution goes to A[N ld ...].
//   Bound by latency: 36 unknowns take 25,900 cycles with one warp on the SM
// and 41,600 with 20, in shared memory 43,800 and 57,500 before back
// substitution.  A branch costs a warp some thirty cycles here, so the body is
// straight-line: registers past the live columns are carried along
// (what they hold is never used), rows of U may run past their end into the
// next row's place, and only whole groups of eight columns are skipped.
constexpr int kLuRegMinN = 24, kLuRegN = 36;
// floats of U's rows of length 1 .. L (columns j .. N, rounded up to 4)
__device__ __forceinline__ int lu_u_size(int L) {
    const int q = L >> 2, r = L & 3;
    return (8 * q + 4 * r) * (q + 1);
}
__device__ __forceinline__ bool lu_registers(float *A, int ld, int N, int lane) {
    constexpr int NC = 40, NE = 5;
    float a[NC], x[NE];
    const int xr = 32 + (lane >> 3), xc = lane & 7;   // the lane's row past 32, its columns 8 q + xc
    const bool extra = N > 32;
    const int li = min(lane, N - 1);
#pragma unroll
    for (int k = 0; k < NC; ++k) a[k] = A[min(k, N) * ld + li];
    int id0 = lane < N ? lane << 8 | lane : -1, id1 = xr < N ? xr << 8 | xr : -1;
#pragma unroll
    for (int q = 0; q < NE; ++q) x[q] = A[min(8 * q + xc, N) * ld + min(xr, N - 1)];
    __syncwarp();   // every entry is in a register before U's rows are stored
    unsigned worst = 0x7f7fffffu, most = 0u;   // smallest and largest pivot key
    float *u = A;   // row j of U: columns j .. N
#pragma unroll 1
    for (int j = 0; j < N; ++j) {
        const int cols = N + 1 - j, xo = xc - (j & 7);   // xo: offset in u of the lane's slot 0
        const float m0 = a[0], m1 = __shfl_sync(kFull, x[0], (lane & ~7) | (j & 7));
        const unsigned k0 = abs_key(m0), k1 = abs_key(m1);
        const unsigned best = __reduce_max_sync(kFull, max(id0 >= 0 ? k0 : 0u, id1 >= 0 ? k1 : 0u));
        // (the index of a row that is done is above any as an unsigned number)
        const unsigned cand = __reduce_min_sync(kFull, min(k0 == best ? (unsigned)id0 : 0xffffffffu,
                                                           k1 == best ? (unsigned)id1 : 0xffffffffu));
        worst = min(worst, best);
        most = max(most, best);
        const bool p0 = id0 == (int)cand, p1 = id1 == (int)cand;
        if (p0) {
#pragma unroll
            for (int c = 0; c < NC; c += 8) {
                if (c >= cols) break;
                *reinterpret_cast<float4 *>(u + c) = make_float4(a[c], a[c + 1], a[c + 2], a[c + 3]);
                *reinterpret_cast<float4 *>(u + c + 4) = make_float4(a[c + 4], a[c + 5], a[c + 6], a[c + 7]);
            }
        }
#pragma unroll
        for (int q = 0; q < NE; ++q)
            if (p1 && 8 * q + xo >= 0) u[8 * q + xo] = x[q];
        // the row at index j takes the pivot's index
        const int cp = (int)(cand & 0xffffff00u);
        id0 = p0 ? -1 : id0 >> 8 == j ? cp | (id0 & 0xff) : id0;
        id1 = p1 ? -1 : id1 >> 8 == j ? cp | (id1 & 0xff) : id1;
        __syncwarp();
        const float inv = frcp(u[0]);
        if (extra) {
#pragma unroll
            for (int q = 0; q < NE; ++q) x[q] = fmaf(-m1, u[max(8 * q + xo, 0)] * inv, x[q]);
            if ((j & 7) == 7) {
#pragma unroll
                for (int q = 0; q + 1 < NE; ++q) x[q] = x[q + 1];
            }
        }
#pragma unroll
        for (int c = 0; c < NC; c += 8) {
            if (c >= cols) break;
            const float4 v = *reinterpret_cast<const float4 *>(u + c), w = *reinterpret_cast<const float4 *>(u + c + 4);
            if (c > 0) a[c - 1] = fmaf(-m0, v.x * inv, a[c]);
            a[c] = fmaf(-m0, v.y * inv, a[c + 1]);
            a[c + 1] = fmaf(-m0, v.z * inv, a[c + 2]);
            a[c + 2] = fmaf(-m0, v.w * inv, a[c + 3]);
            a[c + 3] = fmaf(-m0, w.x * inv, a[c + 4]);
            a[c + 4] = fmaf(-m0, w.y * inv, a[c + 5]);
            a[c + 5] = fmaf(-m0, w.z * inv, a[c + 6]);
            a[c + 6] = fmaf(-m0, w.w * inv, a[c + 7]);
        }
        u += (cols + 3) & ~3;
    }
    // back substitution: lane l solves rows l and l + 32; each solved entry
    // reaches the lanes by a shuffle
    const int n1 = lu_u_size(N + 1), l1 = min(lane + 32, N - 1);
    const float *u0 = A + (n1 - lu_u_size(N + 1 - li) - li), *u1 = A + (n1 - lu_u_size(N + 1 - l1) - l1);
    float y0 = u0[N], y1 = u1[N];
    const float d0 = frcp(u0[li]), d1 = frcp(u1[l1]);
#pragma unroll 1
    for (int j = N - 1; j >= 32; --j) {
        const float v0 = u0[j], v1 = u1[j];
        const float dj = __shfl_sync(kFull, y1 * d1, j & 31);
        y0 = fmaf(-v0, dj, y0);
        y1 = lane + 32 < j ? fmaf(-v1, dj, y1) : lane + 32 == j ? dj : y1;
    }
#pragma unroll 2
    for (int j = min(N, 32) - 1; j >= 0; --j) {
        const float v0 = u0[j];
        const float dj = __shfl_sync(kFull, y0 * d0, j);
        y0 = lane < j ? fmaf(-v0, dj, y0) : lane == j ? dj : y0;
    }
    __syncwarp();
    if (lane < N) A[N * ld + lane] = y0;
    if (lane + 32 < N) A[N * ld + lane + 32] = y1;
    __syncwarp();
    return worst == 0u || key_is_inf(most);
}

// The elimination by columns and the back substitution of one cell per warp
// for the sizes lu_registers does not take.  Out of line, so that it takes no
// place in the instruction caches beside the code that runs.
static __device__ __noinline__ bool lu_columns(unsigned A_shared, int ld, int N) {
    float *A = static_cast<float *>(__cvta_shared_to_generic(A_shared));
    const int lane = threadIdx.x & 31;
    bool sing = false;
#pragma unroll 1
    for (int j = 0; j < N; ++j) {
        unsigned best = 0;
        int bi = N;
#pragma unroll 1
        for (int i = j + lane; i < N; i += 32) {
            const unsigned kk = abs_key(A[j * ld + i]);
            if (bi == N || kk > best) {
                best = kk;
                bi = i;
            }
        }
        warp_argmax(best, bi);
        if (best == 0 || key_is_inf(best)) sing = true;
        if (bi != j && bi < N) {
#pragma unroll 1
            for (int k = j + lane; k <= N; k += 32) {
                const float t = A[k * ld + j];
                A[k * ld + j] = A[k * ld + bi];
                A[k * ld + bi] = t;
            }
        }
        __syncwarp();
        const float inv = frcp(A[j * ld + j]);
        lu_update_colmajor<32>(A, ld, N, j, lane, inv);
        __syncwarp();
        // the reciprocal replaces the pivot once every lane has read it
        if (lane == 0) A[j * ld + j] = inv;
    }
    __syncwarp();
    // lane l keeps rows l and l + 32 of the right-hand side in registers, and
    // each solved entry reaches the lanes by a shuffle
    float y0 = lane < N ? A[N * ld + lane] : 0.f, y1 = lane + 32 < N ? A[N * ld + lane + 32] : 0.f;
#pragma unroll 1
    for (int j = N - 1; j >= 0; --j) {
        const float yj = __shfl_sync(kFull, j < 32 ? y0 : y1, j & 31);
        const float dj = yj * A[j * ld + j];
        if (lane == (j & 31)) {
            if (j < 32)
                y0 = dj;
            else
                y1 = dj;
        }
        if (lane < j) y0 = fmaf(-A[j * ld + lane], dj, y0);
        if (lane + 32 < j) y1 = fmaf(-A[j * ld + lane + 32], dj, y1);
    }
    __syncwarp();
    if (lane < N) A[N * ld + lane] = y0;
    if (lane + 32 < N) A[N * ld + lane + 32] = y1;
    __syncwarp();
    return sing;
}

template <typename JT>
struct SlotMem {
    double *x, *x0, *c, *hRT, *es, *em, *emi, *Q, *part;
    int *ek;
    JT *D, *dTdr, *w, *u, *A, *dQdT, *qtb, *A1, *A2, *rhs;
    JT *cJ, *hJ, *esJ;   // FP32 path: c, h/RT and the energies e_s in the Jacobian type
    // layout and sizes in chem_internal.h (slot_bytes_for, slot_stride); the FP64 path has
    // no FP32 copies (cJ = c, hJ = hRT), the FP32 path no FP64 hRT, es or
    // dTdr.  The species values of the rates (c, the split exponentials em,
    // emi, ek, and h/RT) share the union with the matrix: they are written
    // again every iteration, sentinel included.
    __device__ __forceinline__ void carve(char *base, const DeviceMech &m) {
        const int ns = m.ns, n = ns + 1, nr = m.nr;
        constexpr int jt = (int)sizeof(JT);
        double *p = reinterpret_cast<double *>(base);
        x = p;
        x0 = x + n;
        es = jt == 8 ? x0 + n : nullptr;
        char *q = base + slot_dbl_bytes(ns, jt);
        JT *t = reinterpret_cast<JT *>(q);
        const int ss = small_stride(ns, jt);
        w = t;
        u = w + ss;
        rhs = u + ss;
        if (jt == 8) {
            dTdr = rhs + ss;
            esJ = reinterpret_cast<JT *>(es);
        } else {
            dTdr = nullptr;
            esJ = rhs + ss;
        }
        q += slot_small_bytes(ns, jt);
        // D region: Q and the gather partials until the D entries replace them
        Q = reinterpret_cast<double *>(q);
        part = Q + nr;
        D = reinterpret_cast<JT *>(q);
        q += slot_dreg_bytes(nr, m.nD, m.n_items, jt);
        // union: species values and per-reaction values, then (after the D
        // entries) the matrix
        A = reinterpret_cast<JT *>(q);
        c = reinterpret_cast<double *>(q);
        em = c + ns + 1;
        emi = em + ns + 1;
        hRT = jt == 8 ? emi + ns + 1 : nullptr;
        ek = reinterpret_cast<int *>(emi + (jt == 8 ? 2 : 1) * (ns + 1));
        if (jt == 8) {
            cJ = reinterpret_cast<JT *>(c);
            hJ = reinterpret_cast<JT *>(hRT);
        } else {
            cJ = reinterpret_cast<JT *>(ek + ns + 1);
            hJ = cJ + ns + 1;
        }
        dQdT = reinterpret_cast<JT *>(q + slot_union_species_bytes(ns, jt));
        A1 = dQdT + nr;
        A2 = A1 + nr;
        qtb = A2 + nr;
    }
};

// Sources, Jacobian and one Newton update of Eq. 29 for every slot of the
// warp.  Inputs per slot: x, x0, T, h.  Outputs: x <- x + delta, the scaled
// norm, and a flag for a singular pivot or a non-finite update.
//   G0: the lanes per cell whose order of summation is kept (G, or fewer in a
// wide warp, where a species has a lane of its own).
template <int G, int G0, typename JT>
__device__ void newton_iteration(const DeviceMech &m, const double *tab, SlotMem<JT> &sm, int sl,
                                 double T, double h, double atol_rho, double atol_e, double rtol,
                                 double &norm, bool &bad, double &T_pred) {
    const int ns = m.ns, nr = m.nr;
    constexpr bool f32 = sizeof(JT) == 4;
    // the linear system solved: the species block, with the energy unknown
    // eliminated (phase 5)
    // the matrix: FP64 row-major with rows of N + 1 (the right-hand side
    // last), FP32 column-major with columns of ldc rows (a multiple of 4, for
    // the 16-byte accesses of its elimination; the right-hand side is column N)
    const int N = ns, ldA = N + 1, ldc = (N + 3) & ~3;
    auto ix = [&](int i, int k) -> int { return f32 ? k * ldc + i : i * ldA + k; };
    const Fp64Ops op = fp64_ops(tab);
    // sums and products in the Jacobian type
    auto jadd = [&](JT a, JT b) -> JT {
        if constexpr (f32)
            return a + b;
        else
            return op.add(a, b);
    };
    auto jmul = [&](JT a, JT b) -> JT {
        if constexpr (f32)
            return a * b;
        else
            return op.mul(a, b);
    };
    const double invT = frcp(T, op);
    const double lnT = flog(T, m.log_tab, tab, op);   // T in [200, 6000] K: normal
    const double lnPaRT = op.sub(kLnPaOverR, lnT);

    // 1. concentrations and thermodynamics (species); the heat capacity only
    //    feeds dT/drho, dT/de and the next temperature guess, so the FP32
    //    path forms it in FP32
    const long long Tb = __double_as_longlong(T);
    const float Tf = f32 ? d2f_rz(T) : 0.f;
    double ctot = 0.0, rhocv = 0.0, xs = 0.0;
    float rhocvf = 0.f, xf = 0.f;
#pragma unroll 1
    for (int s = sl; s < ns; s += G) {
        const double *spr = m.sp + s * kSpStride;
        xs = sm.x[s];
        const double ci = op.mul(xs, __ldg(spr + 1));
        sm.c[s] = ci;
        ctot = G == G0 ? op.add(ctot, ci) : ci;
        const int rg = thermo_range(m, s, Tb);
        const auto th = coef_row(m.thermo, ns, s, rg);
        const double hRT = fma(th[9], invT, fma(T, fma(T, fma(T, fma(T, th[8], th[7]), th[6]), th[5]), th[0]));
        const double sR = nasa_s(th, T, lnT, op);
        const double RM = __ldg(spr + 2);
        // exp(g_s/RT - ln(P_a/RT)) split into mantissa and power of two,
        // for the equilibrium constants (phase 2)
        double ey;
        int eK;
        split_exp(op.sub(op.sub(hRT, sR), lnPaRT), tab, op, ey, eK);
        sm.em[s] = ey;
        sm.emi[s] = frcp(ey, op);
        sm.ek[s] = eK;
        if (f32) {
            // the species energy with its formation part, e_s = (R/M) T (h/RT
            // - 1): the Jacobian's temperature column (-e_s dT/de) and the
            // linearised temperature guess need no more, so FP32
            const JT hJs = to_jt<JT>(hRT);
            sm.esJ[s] = (JT)__ldg(m.spf + s * kSpStride + 2) * Tf * (hJs - (JT)1);
            const auto d = coef_row(m.tpoly_f, ns, s, rg);
            const float cv = fmaf(fmaf(fmaf(fmaf(d[4], Tf, d[3]), Tf, d[2]), Tf, d[1]), Tf, d[0]);
            xf = d2f_rz(xs);
            rhocvf = G == G0 ? fmaf(xf, cv, rhocvf) : cv;
            sm.cJ[s] = to_jt<JT>(ci);
            sm.hJ[s] = hJs;
        } else {
            const double hm1 = op.sub(hRT, op.one);
            const double es = fma(op.mul(RM, T), hm1, -__ldg(spr + 3));
            const auto c = coef_row(m.tpoly, ns, s, rg);
            const double cv = fma(fma(fma(fma(c[10], T, c[9]), T, c[8]), T, c[7]), T, c[6]);
            rhocv = G == G0 ? fma(xs, cv, rhocv) : cv;
            sm.hRT[s] = hm1;
            sm.es[s] = es;
        }
    }
    if (sl == 0) {
        // sentinel species: concentration 1, no Gibbs or enthalpy contribution
        sm.c[ns] = 1.0;
        sm.em[ns] = 1.0;
        sm.emi[ns] = 1.0;
        sm.ek[ns] = 0;
        if (f32) {
            sm.cJ[ns] = (JT)1;
            sm.hJ[ns] = (JT)0;
        } else {
            sm.hRT[ns] = 0.0;
        }
    }
    if constexpr (G == G0)
        ctot = Grp<G>::template sum<!f32>(ctot, op);
    else
        ctot = wide_dot<G0>(ctot, op.one, ns, op);
    double dTde;
    float dTdef = 0.f;
    if (f32) {
        if constexpr (G == G0)
            rhocvf = Grp<G>::sum(rhocvf);
        else
            rhocvf = wide_dotf<G0>(xf, rhocvf, ns);
        dTdef = __frcp_rn(rhocvf);
        dTde = f2d_alu(dTdef);
        // dT/drho_k = -e_k^sens dT/de is formed where the Jacobian needs it
    } else {
        if constexpr (G == G0)
            rhocv = Grp<G>::template sum<!f32>(rhocv, op);
        else
            rhocv = wide_dot<G0>(xs, rhocv, ns, op);
        dTde = frcp(rhocv, op);
#pragma unroll 1
        for (int s = sl; s < ns; s += G) sm.dTdr[s] = (JT)op.mul(-op.add(sm.es[s], __ldg(m.sp + s * kSpStride + 3)), dTde);
    }
    __syncwarp();

    // 2. rates per reaction: Eq. 23 forward rate, Eq. 24 equilibrium
    //    constant, Eq. 25 progress rate, and their temperature derivatives
    const JT iT = to_jt<JT>(invT);
    // (the next reaction's parameters are loaded while this one is
    // evaluated: the loop is kept rolled, so nothing else would overlap them)
    static_assert(kRxnDStride == 4, "a reaction's FP64 parameters are two double2");
    double2 nAb = make_double2(0.0, 0.0), nEd = make_double2(0.0, 0.0);
    int2 nf = make_int2(0, 0);
    auto load_rxn = [&](int r) {
        if (r < nr) {
            const double2 *rd = reinterpret_cast<const double2 *>(m.rxn_d + (size_t)r * kRxnDStride);
            nAb = __ldg(rd);
            nEd = __ldg(rd + 1);
            nf = __ldg(reinterpret_cast<const int2 *>(m.rxn_f) + r);
        }
    };
    load_rxn(sl);
#pragma unroll 1
    for (int r = sl; r < nr; r += G) {
        const double lnA = nAb.x, beta = nAb.y, EaR = nEd.x;
        const int fr = nf.x, fpw = nf.y;
        load_rxn(r + G);
        const int a0 = fr & 0xff, a1 = (fr >> 8) & 0xff, a2 = (fr >> 16) & 0xff;
        const int b0 = fpw & 0xff, b1 = (fpw >> 8) & 0xff, b2 = (fpw >> 16) & 0xff;
        // third factor slots: the sentinel's factors are exactly 1 (0 for the
        // enthalpies), so a pass none of whose reactions has a third factor on
        // either side skips them, with bit-identical results (the 36-species
        // mechanism has at most two per side); the vote makes the branch
        // uniform, so the skipped FP64 products cost no pipe slot
        const bool s3 = __any_sync(__activemask(), (a2 != ns) | (b2 != ns));
        double Pf = op.mul(sm.c[a0], sm.c[a1]);
        double Pb = op.mul(sm.c[b0], sm.c[b1]);
        const double kf = fexp(fma(-EaR, invT, fma(beta, lnT, lnA)), tab, op);
        // K_b = K_f / K_c with 1/K_c = (RT/P_a)^dnu exp(dG/RT) (Eq. 24) as
        // the product over the factor slots of the species' exp(g/RT) (RT/P_a)
        // (products) and their inverses (reactants), the sentinel giving 1:
        // mantissas multiplied in FP64, powers of two added as integers, so no
        // exponential per reaction and no overflow in the partial products
        int K2 = (sm.ek[b0] + sm.ek[b1]) - (sm.ek[a0] + sm.ek[a1]);
        double Pm;
        if (s3) {
            Pf = op.mul(Pf, sm.c[a2]);
            Pb = op.mul(Pb, sm.c[b2]);
            K2 = (sm.ek[b0] + sm.ek[b1] + sm.ek[b2]) - (sm.ek[a0] + sm.ek[a1] + sm.ek[a2]);
            Pm = op.mul(op.mul(op.mul(sm.em[b0], sm.em[b1]), sm.em[b2]),
                        op.mul(op.mul(sm.emi[a0], sm.emi[a1]), sm.emi[a2]));
        } else {
            Pm = op.mul(op.mul(sm.em[b0], sm.em[b1]), op.mul(sm.emi[a0], sm.emi[a1]));
        }
        const double kb = scale_pow2(op.mul(kf, Pm), K2);
        double CM = 1.0;
        const bool tb = (fr >> 24) & 1;
        if (tb) {
            CM = ctot;
            const int e0 = __ldg(m.eff_ptr + r), e1 = __ldg(m.eff_ptr + r + 1);
#pragma unroll 1
            for (int e = e0; e < e1; ++e) CM = fma(__ldg(m.eff_c + e), sm.c[__ldg(m.eff_sp + e)], CM);
        }
        const double rev = op.mul(kb, Pb);
        const double q = fma(kf, Pf, -rev);
        sm.Q[r] = f32 || tb ? op.mul(CM, q) : q;   // in the D region until phase 4
        if (f32) {
            // Jacobian-only quantities in FP32 from FP32 copies
            const float4 rf = __ldg(reinterpret_cast<const float4 *>(m.rxn_df) + r);
            // (products formed in FP32 from converted factors: the FP64
            // pipe keeps to the rates the residual needs)
            const JT CMf = to_jt<JT>(CM);
            const JT A1v = CMf * to_jt<JT>(kf), A2v = CMf * to_jt<JT>(kb);
            sm.A1[r] = A1v;
            sm.A2[r] = A2v;
            if (r < m.ntb) sm.qtb[r] = to_jt<JT>(q);
            const JT shf = s3 ? (sm.hJ[b0] + sm.hJ[b1] + sm.hJ[b2]) - (sm.hJ[a0] + sm.hJ[a1] + sm.hJ[a2])
                              : (sm.hJ[b0] + sm.hJ[b1]) - (sm.hJ[a0] + sm.hJ[a1]);
            const JT dlnkf = fmaf(rf.y * iT, iT, __fmul_rn(rf.x, iT));
            const JT dlnKc = (shf - (JT)rf.z) * iT;
            // concentration products again in FP32 (a conversion costs an
            // FP64-pipe slot, three FP32 products do not)
            JT PfJ = sm.cJ[a0] * sm.cJ[a1], PbJ = sm.cJ[b0] * sm.cJ[b1];
            if (s3) {
                PfJ *= sm.cJ[a2];
                PbJ *= sm.cJ[b2];
            }
            sm.dQdT[r] = A1v * PfJ * dlnkf - A2v * PbJ * (dlnkf - dlnKc);
        } else {
            // Jacobian-only quantities, scaled by -h here where it costs
            // nothing: -h C_M k_f, -h C_M k_b, -h q_tb, and -h T dQ/dT (the
            // species' sums take the 1/T)
            //   T dln k_f/dT = beta + E/RT,
            //   T dln k_b/dT = that less sum nu (h/RT - 1),
            // so that T dQ/dT = C_M (q (beta + E/RT) + reverse rate times the
            // sum): three operations fewer than from both rates
            const double hb = op.add(sm.hRT[b0], sm.hRT[b1]), ha = op.add(sm.hRT[a0], sm.hRT[a1]);
            const double sh = s3 ? op.sub(op.add(hb, sm.hRT[b2]), op.add(ha, sm.hRT[a2])) : op.sub(hb, ha);
            const double CMh = tb ? op.mul(CM, -h) : -h;
            if (r < m.ntb) sm.qtb[r] = (JT)op.mul(q, -h);
            sm.A1[r] = (JT)op.mul(CMh, kf);
            sm.A2[r] = (JT)op.mul(CMh, kb);
            sm.dQdT[r] = (JT)op.mul(CMh, fma(q, fma(EaR, invT, beta), op.mul(rev, sh)));
        }
    }
    __syncwarp();

    // 3. species sources (Eq. 26) and the rank-1 vectors of the Jacobian, as
    //    fixed-size chunks of each species' reaction list, then per species
    //    (an item's partial sums: sum nu Q in FP64, then sum nu dQ/dT and
    //    sum nu q_tb in the Jacobian type, packed into the next 16 bytes)
    const GatherLayout &gl = m.gl[layout_index(G)];
    const unsigned *gl_j_w = G == G0 ? gl.j_w : m.j_w_wide[layout_index(G0)];
    //   The table's words come from L2 as often as from L1, so an item's
    //   words are loaded four at a time (16 bytes), the next item's
    //   descriptor with them, and the operands of four terms at a time; the
    //   sums keep the order of the list.
    auto item_at = [&](int it) -> int2 { return it < m.n_items ? __ldg(gl.it_meta + it) : make_int2(0, 0); };
    auto item_words = [&](int e, int rem) -> uint4 {
        return rem > 0 ? __ldg(reinterpret_cast<const uint4 *>(gl.sp_w + e)) : make_uint4(0u, 0u, 0u, 0u);
    };
    static_assert(kChunk == 8, "an item is two groups of four terms");
    int2 im = item_at(sl);
    uint4 iwords = item_words(im.x, im.y >> 16);
#pragma unroll 1
    for (int it = sl; it < m.n_items; it += G) {
        const int e1 = im.x + 4 * G, id = im.y & 0xffff;
        int rem = im.y >> 16;
        im = item_at(it + G);
        double sq = 0.0;
        JT sdq = 0, squ = 0;
#pragma unroll 1
        for (int half = 0; half < 2; ++half) {
            const uint4 wc = iwords;
            iwords = half == 0 ? item_words(e1, rem - 4) : item_words(im.x, im.y >> 16);
            const unsigned wv[4] = {wc.x, wc.y, wc.z, wc.w};
            double Qv[4];
            JT dq[4], qt[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                // (a missing term's word is 0: reaction 0 is read and not used)
                const int r = (int)(wv[q] & 0xfffffu);
                Qv[q] = sm.Q[r];
                dq[q] = sm.dQdT[r];
                qt[q] = r < m.ntb ? sm.qtb[r] : (JT)0;
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                if (q < rem) {
                    const double nu = word_nu_double(wv[q]);   // nu_rs != 0 in a list
                    const JT nuj = f32 ? (JT)word_nu_float(wv[q]) : (JT)nu;
                    sq = fma(nu, Qv[q], sq);
                    sdq += nuj * dq[q];
                    if ((int)(wv[q] & 0xfffffu) < m.ntb) squ += nuj * qt[q];
                }
            }
            rem -= 4;
        }
        constexpr int iw = (int)(item_bytes((int)sizeof(JT)) / 8);   // doubles per item
        sm.part[iw * id] = sq;
        JT *pj = reinterpret_cast<JT *>(sm.part + iw * id + 1);
        pj[0] = sdq;
        pj[1] = squ;
    }
    __syncwarp();
    double dEt = 0.0, wef = 0.0;
#pragma unroll 1
    for (int s = sl; s < ns; s += G) {
        double sq = 0.0;
        JT sdq = 0, squ = 0;
        const int i0 = __ldg(m.sp_item_ptr + s), i1 = __ldg(m.sp_item_ptr + s + 1);
        constexpr int iw = (int)(item_bytes((int)sizeof(JT)) / 8);
#pragma unroll 1
        for (int it = i0; it < i1; ++it) {
            sq = op.add(sq, sm.part[iw * it]);
            const JT *pj = reinterpret_cast<const JT *>(sm.part + iw * it + 1);
            sdq = jadd(sdq, pj[0]);
            squ = jadd(squ, pj[1]);
        }
        const double M = __ldg(m.sp + s * kSpStride);
        const double ef = __ldg(m.sp + s * kSpStride + 3);
        const JT MJ = f32 ? (JT)__ldg(m.spf + s * kSpStride) : (JT)M;
        const double wds = op.mul(M, sq);
        // right-hand side -F_s = -(x_s - x0_s - h wdot_s), FP64 until stored
        const double dx = op.sub(sm.x[s], sm.x0[s]);
        sm.rhs[s] = to_jt<JT>(-fma(-h, wds, dx));
        // (FP64: -h w and -h u, from sums over -h T dQ/dT and -h q_tb)
        const JT ws = jmul(f32 ? MJ : (JT)op.mul(M, invT), sdq), us = jmul(MJ, squ);
        sm.w[s] = ws;
        sm.u[s] = us;
        wef = ef;
        dEt = G == G0 ? fma(ef, dx, dEt) : dx;
    }
    // the total-energy residual R_E = F_e + sum_s e_f,s F_s = (x_e - x0_e) +
    // sum_s e_f,s (x_s - x0_s), in which the sources cancel (Omega_e =
    // -sum_s e_f,s wdot_s); it replaces the energy equation (phase 5)
    if constexpr (G == G0)
        dEt = Grp<G>::template sum<!f32>(dEt, op);
    else
        dEt = wide_dot<G0>(wef, dEt, ns, op);
    const double RE = op.add(dEt, op.sub(sm.x[ns], sm.x0[ns]));
    __syncwarp();

    // 4. D entries: d Q_r / d rho_k without the all-ones third-body part,
    //    grouped so that each group is one uniform loop body (FP32: one
    //    branch-free body that selects the sides by their orders, two
    //    entries per trip so their loads overlap; its entries are M_k dQ_r /
    //    drho_k, with integer orders, and the gather applies the 1/M_k)
    if (f32) {
        const JT *__restrict__ A1v = sm.A1;
        const JT *__restrict__ A2v = sm.A2;
        const JT *__restrict__ cJv = sm.cJ;
        const JT *__restrict__ qv = sm.qtb;
        JT *__restrict__ Dw = sm.D;
        // (descriptors and efficiencies are loaded one trip ahead)
        struct DEntry {
            int2 pk;
            float ce;
        };
        auto entry_at = [&](int j) -> DEntry {
            DEntry d{make_int2(0, 0), 0.f};
            if (j < m.nD) {
                d.pk = __ldg(m.d_pk + j);
                d.ce = __ldg(m.d_cef + j);
            }
            return d;
        };
        auto dval = [&](const DEntry &en) -> JT {
            const int2 pk = en.pk;
            const int r = pk.x & 0xffff, vf = (pk.x >> 16) & 15, vb = (pk.x >> 20) & 15, i1 = pk.y;
            const JT fwd = (JT)small_int_to_float(vf) * A1v[r] * (cJv[i1 & 0xff] * cJv[(i1 >> 8) & 0xff]);
            const JT bwd = (JT)small_int_to_float(vb) * A2v[r] * (cJv[(i1 >> 16) & 0xff] * cJv[(i1 >> 24) & 0xff]);
            JT d = (vf ? fwd : (JT)0) - (vb ? bwd : (JT)0);
            if (r < m.ntb) d = fma((JT)en.ce, qv[r], d);
            return d;
        };
        DEntry e0 = entry_at(sl), e1 = entry_at(sl + G);
#pragma unroll 1
        for (int j = sl; j < m.nD; j += 2 * G) {
            const DEntry c0 = e0, c1 = e1;
            e0 = entry_at(j + 2 * G);
            e1 = entry_at(j + 3 * G);
            // (past the end: the descriptor 0 reads reaction 0, and is dropped)
            const JT v0 = dval(c0), v1 = dval(c1);
            Dw[j] = v0;
            if (j + G < m.nD) Dw[j + G] = v1;
        }
    } else {
    int2 npk = sl < m.nD ? __ldg(m.d_pk64 + sl) : make_int2(0, 0);
    double nce = sl < m.nD ? __ldg(m.d_ce + sl) : 0.0;
#pragma unroll 1
    for (int j = sl; j < m.nD; j += G) {
        // the FP64 D entries are M_k dQ_r/drho_k as well: integer orders from
        // the descriptor (exact doubles by integer operations), alpha - 1
        // from an 8-byte table, and the gather applies the 1/M_k
        // (in an order of their own: first those of order 1 with one
        // remaining factor, then with two: one and two multiplications
        // instead of three)
        const int2 pk = npk;
        const double ce = nce;
        if (j + G < m.nD) {
            npk = __ldg(m.d_pk64 + j + G);
            nce = __ldg(m.d_ce + j + G);
        }
        const int r = pk.x & 0xffff, vf = (pk.x >> 16) & 15, vb = (pk.x >> 20) & 15, i1 = pk.y;
        const int fa = i1 & 0xff, fb = (i1 >> 8) & 0xff, ba = (i1 >> 16) & 0xff, bb = (i1 >> 24) & 0xff;
        // (one side's factors, selected without a branch; the reactant side
        // where a species is on both)
        // (-h M_k dQ_r/drho_k, from -h C_M k)
        double dd;
        if (j < m.nD_2) {
            const bool f = j < m.nD_F1 || (j >= m.nD_1 && j < m.nD_F2);
            double A = f ? sm.A1[r] : sm.A2[r];
            if (j >= m.nD_1) A = op.mul(A, sm.c[f ? fb : bb]);
            dd = op.mul(A, sm.c[f ? fa : ba]);
            if (!f) dd = -dd;
        } else {
            const bool f = vf > 0;
            const double v = small_pos_int_to_double(f ? vf : max(vb, 1));
            const double A = op.mul(v, f ? sm.A1[r] : sm.A2[r]), cc = op.mul(sm.c[f ? fa : ba], sm.c[f ? fb : bb]);
            dd = op.mul(A, cc);
            if (!f) dd = vb > 0 ? -dd : 0.0;
            if (f && vb > 0)
                dd = fma(A, cc, -op.mul(op.mul(small_pos_int_to_double(vb), sm.A2[r]), op.mul(sm.c[ba], sm.c[bb])));
        }
        sm.D[j] = r < m.ntb ? (JT)fma(ce, (double)sm.qtb[r], dd) : (JT)dd;
    }
    }
    __syncwarp();
    // the per-reaction arrays are dead from here on; the matrix takes their place

    // 5. right-hand side into the matrix, with the energy unknown
    //    eliminated.  The energy row of I - hJ is [e_f, 1] - sum_s e_f,s
    //    (row s) (J_ek = -sum_s e_f,s J_sk), so with the species equations
    //    it reduces to the conservation law de = -R_E - e_f . drho;
    //    substituted into the species rows, whose energy-column entry is
    //    a_s = -h w_s dT/de, it leaves
    //      sum_k (A_sk - a_s e_f,k) drho_k = -F_s + a_s R_E,
    //    the same solution as the full system of Eq. 29 in exact
    //    arithmetic, with one unknown fewer and no energy row to form
    const JT mh = to_jt<JT>(-h);
    {
        const JT cRE = f32 ? mh * (JT)dTdef * d2f_rz(RE) : (JT)op.mul(dTde, RE);   // (FP64: w carries the -h)
#pragma unroll 1
        for (int i = sl; i < N; i += G) sm.A[ix(i, N)] = fma(sm.w[i], cRE, sm.rhs[i]);
    }

    // 6. the reduced system's -h J'_sk = -h (J_sk - w_s e_f,k dT/de), plus
    //    the identity.  J_sk = w_s dT/drho_k + (u_s + M_s sum_r nu_rs D_rk) / M_k
    //    (the D entries carry the factor M_k): a rank-two part, in which
    //    the reduced system's column factor dT/drho_k - e_f,k dT/de stands
    //    for dT/drho_k, plus the gathered sums (longest gather lists
    //    first, so the lanes of a pass run lists of nearly equal length;
    //    four terms in flight per trip, two accumulators)
    const JT *__restrict__ Dv = sm.D;
    if constexpr (f32) {
        // 6a. the rank-two part and the identity, dense: a lane writes
        //     rows 4g..4g+3 of column k with one 16-byte store, from
        //     16-byte reads of w and u (the padding rows of a column take
        //     values that nothing reads).  Task t = k ldc/4 + g steps by G,
        //     the carry taken without a division.
        const int NG = ldc >> 2;
        const unsigned rc = __ldg(m.div16 + NG);
        int k = (int)(((unsigned)sl * rc) >> 16), g = sl - k * NG;
        const int dk = (int)(((unsigned)G * rc) >> 16), dg = G - dk * NG;
        const float cTe = -(mh * dTdef);
#pragma unroll 1
        while (k < N) {
            const float cT = cTe * sm.esJ[k], cU = mh * __ldg(m.spf + k * kSpStride + 1);
            const float4 wv = *reinterpret_cast<const float4 *>(sm.w + 4 * g);
            const float4 uv = *reinterpret_cast<const float4 *>(sm.u + 4 * g);
            const int dd = k - 4 * g;   // the diagonal's row within the four
            float4 a;
            a.x = fmaf(wv.x, cT, uv.x * cU) + (dd == 0 ? 1.f : 0.f);
            a.y = fmaf(wv.y, cT, uv.y * cU) + (dd == 1 ? 1.f : 0.f);
            a.z = fmaf(wv.z, cT, uv.z * cU) + (dd == 2 ? 1.f : 0.f);
            a.w = fmaf(wv.w, cT, uv.w * cU) + (dd == 3 ? 1.f : 0.f);
            *reinterpret_cast<float4 *>(sm.A + k * ldc + 4 * g) = a;
            k += dk;
            g += dg;
            if (g >= NG) {
                g -= NG;
                ++k;
            }
        }
        __syncwarp();
        // 6b. the gathered sums of the entries that have reaction terms,
        //     added as -h (M_s / M_k) sum_r nu_rs D_rk
        //     (the word's top nine bits are those of the float coefficient)
        auto coef = [](unsigned wv) -> float { return __int_as_float((int)(wv & 0xff800000u)); };
        //     Most lists have fewer than four terms, and the table's words
        //     often come from L2: a list's metadata is loaded two entries
        //     ahead, its words one chunk of four ahead.  A branch costs a warp
        //     some thirty cycles, so the lanes of a pass run the chunks of its
        //     longest list (lane 0's) together, a missing term being a zero
        //     times D entry 0 (the table is padded, all reads are in it).
        //     Terms in a whole chunk alternate between two accumulators, those
        //     of a partial one follow the first.
        const int nnz = m.nJ_nz;
        auto meta_at = [&](int p) -> int4 { return p < nnz ? __ldg(gl.j_meta32 + p) : make_int4(0, 0, 0, 0); };
        auto words_at = [&](int e) -> uint4 {
            const unsigned *wp = gl_j_w + e;
            return make_uint4(__ldg(wp), __ldg(wp + G), __ldg(wp + 2 * G), __ldg(wp + 3 * G));
        };
        int4 me = meta_at(sl), mn = meta_at(sl + G);
        uint4 wn = words_at(me.x);
#pragma unroll 1
        for (int p = sl; p - sl < nnz; p += G) {
            float *ap = reinterpret_cast<float *>(sm.A) + me.z;
            const float av = *ap, fac = mh * __int_as_float(me.w);
            int e = me.x, rem = me.y, chunks = (__shfl_sync(kFull, rem, 0) + 3) >> 2;
            uint4 w = wn;
            me = mn;
            mn = meta_at(p + 2 * G);
            float a0 = 0.f, a1 = 0.f;
#pragma unroll 1
            do {
                const unsigned x0 = rem > 0 ? w.x : 0u, x1 = rem > 1 ? w.y : 0u, x2 = rem > 2 ? w.z : 0u,
                               x3 = rem > 3 ? w.w : 0u;
                const bool whole = rem > 3;
                const float v0 = Dv[x0 & 0x7fffffu], v1 = Dv[x1 & 0x7fffffu], v2 = Dv[x2 & 0x7fffffu],
                            v3 = Dv[x3 & 0x7fffffu];
                rem -= 4;
                e += 4 * G;
                --chunks;
                w = words_at(chunks > 0 ? e : me.x);
                a0 = fmaf(coef(x0), v0, a0);
                const float b = fmaf(coef(x1), v1, whole ? a1 : a0);
                a0 = fmaf(coef(x2), v2, whole ? a0 : b);
                a1 = whole ? fmaf(coef(x3), v3, b) : a1;
            } while (chunks > 0);
            wn = w;
            if (p < nnz) *ap = fmaf(fac, a0 + a1, av);
        }
        __syncwarp();
    } else {
        // (loads ahead as in the FP32 pass; w, u and the D entries carry the
        // -h, the initial values the identity and u: two FP64 operations per
        // entry beside its terms)
        struct Terms {
            int4 d;
            double2 c0, c1;
        };
        auto terms_at = [&](int e, int rem) -> Terms {
            Terms t{make_int4(0, 0, 0, 0), make_double2(0.0, 0.0), make_double2(0.0, 0.0)};
            if (rem > 0) {
                t.d = __ldg(reinterpret_cast<const int4 *>(gl.j_d + e));
                t.c0 = __ldg(reinterpret_cast<const double2 *>(gl.j_c + e));
                t.c1 = __ldg(reinterpret_cast<const double2 *>(gl.j_c + e) + 1);
            }
            return t;
        };
        auto meta_at = [&](int p) -> int2 { return p < m.nJ ? __ldg(gl.j_meta + p) : make_int2(0, 0); };
        int2 me = meta_at(sl), mn = meta_at(sl + G);
        Terms tn = terms_at(me.x, me.y >> 16);
#pragma unroll 1
        for (int p = sl; p < m.nJ; p += G) {
            const int len = me.y >> 16, s = (me.y >> 8) & 0xff, k = me.y & 0xff;
            int e = me.x, rem = len;
            Terms t = tn;
            me = mn;
            mn = meta_at(p + 2 * G);
            tn = terms_at(me.x, me.y >> 16);
            const double invMk = __ldg(m.sp + k * kSpStride + 1);
            // -h w_s dT/drho_k plus the identity; the sum starts from -h u_s
            // (one accumulator: a warp's FP64 operations do not overlap)
            const double J = fma((double)sm.w[s], (double)sm.dTdr[k], s == k ? op.one : op.nz);
            double ua = sm.u[s];
            if (len > 0) {
#pragma unroll 1
                for (;;) {
                    const double v0 = Dv[t.d.x], v1 = Dv[t.d.y], v2 = Dv[t.d.z], v3 = Dv[t.d.w];
                    const Terms tc = t;
                    const int rc = rem;
                    rem -= 4;
                    e += 4 * G;
                    t = terms_at(e, rem);
                    ua = fma(tc.c0.x, v0, ua);
                    if (rc > 1) ua = fma(tc.c0.y, v1, ua);
                    if (rc > 2) ua = fma(tc.c1.x, v2, ua);
                    if (rc > 3) ua = fma(tc.c1.y, v3, ua);
                    if (rem <= 0) break;
                }
            }
            // (D entries scaled by M_k; the FP64 lists' coefficients are nu_rs M_s)
            sm.A[ix(s, k)] = (JT)fma(invMk, ua, J);
        }
        __syncwarp();
    }

    // 7. Gaussian elimination with row partial pivoting on [A | -F]
    //    (Sec. 3.2), ties to the lowest row; the pivot's reciprocal replaces
    //    the diagonal
    bool sing = false;
    if constexpr (f32 && G == 32) {
        if (G == G0 && N >= kLuRegMinN && N <= kLuRegN)
            sing = lu_registers(reinterpret_cast<float *>(sm.A), ldc, N, sl);
        else
            sing = lu_columns((unsigned)__cvta_generic_to_shared(sm.A), ldc, N);
    } else {
#pragma unroll 1
    for (int j = 0; j < N; ++j) {
        PivotKey<JT> best = 0;
        int bi = N;
#pragma unroll 1
        for (int i = j + sl; i < N; i += G) {
            const PivotKey<JT> kk = abs_key(sm.A[ix(i, j)]);
            if (bi == N || kk > best) {
                best = kk;
                bi = i;
            }
        }
        if constexpr (G == 32)
            warp_argmax(best, bi);
        else
            Grp<G>::argmax(best, bi);
        if (best == 0 || key_is_inf(best)) sing = true;
        if (bi != j && bi < N) {
#pragma unroll 1
            for (int k = j + sl; k <= N; k += G) {
                const JT t = sm.A[ix(j, k)];
                sm.A[ix(j, k)] = sm.A[ix(bi, k)];
                sm.A[ix(bi, k)] = t;
            }
        }
        __syncwarp();
        // (the FP64 pivot takes the full-precision reciprocal: a 1e-14 error
        // in every multiplier reaches the trace species of ill-conditioned
        // cells at 1e-10)
        JT inv;
        if constexpr (f32)
            inv = frcp(sm.A[ix(j, j)]);
        else
            inv = frcp(sm.A[ix(j, j)], op);
        if (!f32) {
#pragma unroll 1
            for (int i = j + 1 + sl; i < N; i += G) sm.A[i * ldA + j] = jmul(sm.A[i * ldA + j], inv);
            __syncwarp();
            if (sl == 0) sm.A[j * ldA + j] = inv;
        }
        if (f32) {
            // FP32: bound by issue and latency, not by the pipe; the update
            // reads column j unscaled and never A[j][j]
            lu_update_colmajor<G>(reinterpret_cast<float *>(sm.A), ldc, N, j, sl, (float)inv);
        } else {
            // FP64: a flat walk over the trailing elements keeps every lane of
            // every FP64 instruction busy (a masked lane costs a full slot)
            // (sl / cols and G / cols by a reciprocal multiply: both numerators
            // are below 64, and an integer division would take conversions on
            // the FP64 pipe)
            const int cols = N - j;
            const int tot = (N - j - 1) * cols;
            const unsigned rc = __ldg(m.div16 + cols);
            int e = sl;
            const int q0 = (int)(((unsigned)sl * rc) >> 16), dq = (int)(((unsigned)G * rc) >> 16);
            int i = j + 1 + q0, k = j + 1 + (sl - q0 * cols);
            const int di = dq, dk = G - dq * cols;
            // (two elements per trip, so that their loads overlap)
            auto next = [&]() {
                i += di;
                k += dk;
                if (k > N) {
                    k -= cols;
                    ++i;
                }
            };
            const JT *rj = sm.A + j * ldA;
#pragma unroll 1
            for (; e + G < tot; e += 2 * G) {
                JT *p0 = sm.A + i * ldA;
                const int k0 = k;
                next();
                JT *p1 = sm.A + i * ldA;
                const int k1 = k;
                next();
                const JT l0 = p0[j], u0 = rj[k0], v0 = p0[k0], l1 = p1[j], u1 = rj[k1], v1 = p1[k1];
                p0[k0] = fma(-l0, u0, v0);
                p1[k1] = fma(-l1, u1, v1);
            }
            if (e < tot) {
                JT *p0 = sm.A + i * ldA;
                p0[k] = fma(-p0[j], rj[k], p0[k]);
            }
        }
        __syncwarp();
        // FP32: the reciprocal replaces the pivot once every lane has read it
        if (f32 && sl == 0) sm.A[ix(j, j)] = inv;
    }
    __syncwarp();
    // back substitution, U delta = y
#pragma unroll 1
        for (int j = N - 1; j >= 0; --j) {
            const JT dj = jmul(sm.A[ix(j, N)], sm.A[ix(j, j)]);
            __syncwarp();
            if (sl == 0) sm.A[ix(j, N)] = dj;
#pragma unroll 1
            for (int i = sl; i < j; i += G) sm.A[ix(i, N)] -= sm.A[ix(i, j)] * dj;
            __syncwarp();
        }
    }

    // 8. update, convergence norm, and the linearised temperature of the
    //    new iterate (dT = (de - sum_s e_s^sens drho_s) / (rho cv)) as the
    //    next recovery's starting guess.  The norm's ratios are FP64 on both
    //    paths (they decide acceptance and the divergence abort) and their
    //    maximum is taken on the bit patterns; a zero scale counts a nonzero
    //    update as infinitely large.
    auto ratio = [&](double d, double den) -> double {
        if (__double_as_longlong(den) > 0) return op.mul(fabs(d), frcp1(den, op));
        return (__double_as_longlong(d) << 1) != 0 ? CUDART_INF : 0.0;
    };
    double nrm = 0.0, des = 0.0, se = 0.0, dw = 0.0;
    float desf = 0.f, sef = 0.f, dwf = 0.f;
    int nonfinite = 0;
#pragma unroll 1
    for (int i = sl; i < N; i += G) {
        float df = 0.f;
        double d;
        if (f32) {
            df = (float)sm.A[ix(i, N)];
            d = f2d_alu(df);
            // (e_s with its formation part: see below)
            const float es = (float)sm.esJ[i], ef = __ldg(m.spf + i * kSpStride + 3);
            dwf = df;
            desf = G == G0 ? fmaf(-es, df, desf) : -es;
            sef = G == G0 ? fmaf(ef, df, sef) : ef;
        } else {
            d = (double)sm.A[ix(i, N)];
            const double es = sm.es[i], ef = __ldg(m.sp + i * kSpStride + 3);
            dw = d;
            des = G == G0 ? fma(-es, d, des) : -es;
            se = G == G0 ? fma(ef, d, se) : ef;
        }
        const double xi = op.add(sm.x[i], d);
        sm.x[i] = xi;
        if (!finite_bits(xi)) nonfinite = 1;
        const double ri = ratio(d, fma(rtol, fabs(xi), atol_rho));
        if (bits_gt(ri, nrm)) nrm = ri;
    }
    {
        // the eliminated energy unknown: de = -R_E - e_f . drho
        if constexpr (G == G0) {
            sef = Grp<G>::sum(sef);
            se = f32 ? 0.0 : Grp<G>::template sum<!f32>(se, op);
        } else {
            sef = f32 ? wide_dotf<G0>(sef, dwf, N) : 0.f;
            se = f32 ? 0.0 : wide_dot<G0>(se, dw, N, op);
        }
        const double de = op.sub(-RE, f32 ? f2d_alu(sef) : se);
        if (sl == 0) {
            const double xe = op.add(sm.x[ns], de);
            sm.x[ns] = xe;
            if (!finite_bits(xe)) nonfinite = 1;
            const double ri = ratio(de, fma(rtol, fabs(xe), atol_e));
            if (bits_gt(ri, nrm)) nrm = ri;
        }
        // dT = (de - sum_s e_s^sens drho_s) / (rho cv), where de = -R_E -
        // e_f . drho: the FP32 path's e_s carry e_f, so it adds -R_E
        if constexpr (G == G0) {
            if (sl == 0) {
                if (f32)
                    desf += d2f_rz(-RE);
                else
                    des = op.add(des, de);
            }
            des = f32 ? f2d_alu(Grp<G>::sum(desf)) : Grp<G>::template sum<!f32>(des, op);
        } else {
            des = f32 ? f2d_alu(wide_dotf<G0>(desf, dwf, N, d2f_rz(-RE), true))
                      : wide_dot<G0>(des, dw, N, op, de, true);
        }
    }
    nrm = Grp<G>::max_nonneg(nrm);
    nonfinite = Grp<G>::any(nonfinite);
    __syncwarp();
    norm = nrm;
    bad = sing || nonfinite;
    T_pred = fma(des, dTde, T);
}

// ---- request-server queue (ServeQueue in chem_internal.h) -----------------
__device__ __forceinline__ unsigned long long globaltimer_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ unsigned long long ld_acquire_sys(const unsigned long long *p) {
    unsigned long long v;
    asm volatile("ld.acquire.sys.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
template <typename T>
__device__ __forceinline__ T ld_vol(const T *p) {
    return *reinterpret_cast<const volatile T *>(p);
}
// A relaxed load from L2 (not L1, which may hold another launch's or an
// earlier chunk's copy): for device values that are either immutable while
// they are read (a live chunk's descriptor copy) or only hints (`next`, the
// budget copy, the poll time).  Unlike volatile loads, several of these can
// be in flight at once.
template <typename T>
__device__ __forceinline__ T ld_cg(const T *p) {
    static_assert(sizeof(T) == 8 || sizeof(T) == 4, "8- or 4-byte values");
    T r;
    if constexpr (sizeof(T) == 8) {
        const long long v = __ldcg(reinterpret_cast<const long long *>(p));
        memcpy(&r, &v, 8);
    } else {
        const int v = __ldcg(reinterpret_cast<const int *>(p));
        memcpy(&r, &v, 4);
    }
    return r;
}
__device__ __forceinline__ long long ld_acquire_gpu(const long long *p) {
    long long v;
    asm volatile("ld.acquire.gpu.global.s64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
// Refreshes the device copies of the host's `tail` and of this launch's
// budget, and tells the host where the hand-out of cells stands (`front`:
// the first virtual cell of the current chunk; the cursor only grows, and
// every claim attempt and every idle poll comes here, so the host sees the
// claims catch up with what it published): at most one warp per launch
// every kServePollNs.
__device__ __forceinline__ void serve_refresh(const ServeQueue &q) {
    const unsigned long long now = globaltimer_ns();
    const unsigned long long last = ld_cg(q.dpoll);
    if (now - last < (unsigned long long)kServePollNs || atomicCAS(q.dpoll, last, now) != last) return;
    const unsigned long long t = ld_acquire_sys(q.tail);
    const int bud = ld_vol(q.budget);
    __threadfence();   // what the host wrote before `tail`, before the copy of `tail`
    atomicMax(q.dtail, t);
    *reinterpret_cast<volatile int *>(q.dbudget) = bud;
    *reinterpret_cast<volatile unsigned long long *>(q.front) = ld_cg(q.chunk) << kServeChunkLog;
}
// Copies the host descriptor of chunk c (ring entry ce) into the device ring;
// called after a claim from the chunk succeeded, so the chunk is live and
// its entry stable.  The sequence number is written last.
__device__ __forceinline__ void serve_mirror(const ServeQueue &q, int ce, long long c) {
    const ServeDesc *hd = q.desc + ce;
    ServeDesc *md = q.mdesc + ce;
    md->start = ld_vol(&hd->start);
    md->n_cells = ld_vol(&hd->n_cells);
    md->ld = ld_vol(&hd->ld);
    md->rho = ld_vol(&hd->rho);
    md->e = ld_vol(&hd->e);
    md->T_out = ld_vol(&hd->T_out);
    md->status = ld_vol(&hd->status);
    md->dt = ld_vol(&hd->dt);
    __threadfence();
    *reinterpret_cast<volatile long long *>(&md->seq) = c;
}
// Claims up to k consecutive cells of the current chunk for a warp's free
// slots: returns how many (0 when none is published or the launch's block
// budget excludes this block), the first one's virtual number in v0 and the
// chunk's ring entry in e.  The chunk's size comes from the device copy of
// its descriptor when one is there, else from host memory (the entry is
// read after `tail` shows the chunk published and holds it until all of its
// cells are done), and the first claim makes the copy.  Bounded by the
// guard; a pass claims, finds the chunk exhausted and moves on, or starts
// the entry's counter.
__device__ __forceinline__ int serve_claim(const ServeQueue &q, int k, long long &v0, int &e) {
    serve_refresh(q);
    if ((int)blockIdx.x >= ld_cg(q.dbudget)) return 0;
    long long c = (long long)ld_cg(q.chunk);
    const unsigned long long tail = (unsigned long long)ld_acquire_gpu(reinterpret_cast<const long long *>(q.dtail));
    // chunks published: the last one's real cells end at `tail`
    const long long nch = (long long)((tail + (1ULL << kServeChunkLog) - 1) >> kServeChunkLog);
#pragma unroll 1
    for (int guard = 0; guard < 64 && c < nch; ++guard) {
        const int ce = (int)(c % q.cap);
        const bool mirrored = ld_acquire_gpu(&q.mdesc[ce].seq) == c;
        long long nc;
        if (mirrored) {
            nc = ld_cg(&q.mdesc[ce].n_cells);
        } else {
            const ServeDesc *d = q.desc + ce;
            if (ld_vol(&d->seq) != c) {
                // a stale chunk number (finished, its entry reused since)
                // moves on; an entry out of order is an error
                const long long c2 = (long long)ld_cg(q.chunk);
                if (c2 != c) {
                    c = c2;
                    continue;
                }
                atomicExch(q.error, 1);
                return 0;
            }
            nc = ld_vol(&d->n_cells);
        }
        // the entry's counter: the first claim of this lap of the ring
        // starts it (the counter is never reset otherwise, so claims that
        // arrive after a chunk is handed out only find it exhausted)
        const long long lap = c / q.cap;
        constexpr unsigned long long kCount = (1ULL << kClaimLapShift) - 1;
        unsigned long long r = ld_cg(q.claimed + ce);
        if ((long long)(r >> kClaimLapShift) < lap) {
            atomicCAS(q.claimed + ce, r, (unsigned long long)lap << kClaimLapShift);
            continue;
        }
        if ((long long)(r >> kClaimLapShift) > lap) {
            // the entry has moved on: a stale chunk number
            const long long c2 = (long long)ld_cg(q.chunk);
            if (c2 != c) {
                c = c2;
                continue;
            }
            atomicExch(q.error, 1);
            return 0;
        }
        if ((long long)(r & kCount) < nc) {
            r = atomicAdd(q.claimed + ce, (unsigned long long)k);
            const long long off = (long long)(r & kCount);
            if ((long long)(r >> kClaimLapShift) != lap) {
                // only a claim through a chunk number older than a whole
                // ring of chunks gets here
                atomicExch(q.error, 1);
                return 0;
            }
            if (off < nc) {
                if (!mirrored) serve_mirror(q, ce, c);
                const long long cnt = min((long long)k, nc - off);
                v0 = (c << kServeChunkLog) + off;
                e = ce;
                return (int)cnt;
            }
        }
        // the chunk is handed out: on to the next
        atomicMax(q.chunk, (unsigned long long)(c + 1));
        ++c;
    }
    return 0;
}
// Counts a finished cell of ring entry e (lane 0 of its slot); the slot that
// finishes the request's last cell resets the entry's counters for the next
// request and publishes the completion record to the host.
__device__ __forceinline__ void serve_cell_done(const ServeQueue &q, int e) {
    __threadfence();   // the cell's results before its count
    atomicMax(q.t_last + e, globaltimer_ns());
    __threadfence();
    const unsigned long long prev = atomicAdd(q.done + e, 1ULL);
    const ServeDesc *d = q.mdesc + e;
    if ((long long)prev + 1 == ld_cg(&d->n_cells)) {
        const unsigned long long tf = atomicExch(q.t_first + e, ~0ULL);
        const unsigned long long tl = atomicExch(q.t_last + e, 0ULL);
        atomicExch(q.done + e, 0ULL);
        __threadfence_system();
        volatile ServeDone *f = q.fin + e;
        f->t_first = tf;
        f->t_last = tl;
        __threadfence_system();
        f->seq = ld_cg(&d->seq);
    }
}

// Wide warps (be_kernel) serve at most this many lanes per cell.
constexpr int kWideMaxG = 8;

// A slot's cell and where its integration stands.
struct SlotVars {
    int state;
    long long cell;
    // request-server mode: the slot's ring entry and its request's dt
    int qe;
    double sdt;
    double T, T0, Tin, h, norm_prev, atol_rho, atol_e;
    int k, level, attempts, iters, subs, fails;
    long long t_units;
};
// (kept in a slot's matrix on the way to a wide warp, FP32 at five species)
static_assert(sizeof(SlotVars) <= 6 * 8 * 4, "slot variables");
__device__ __forceinline__ SlotVars free_slot(double dt) {
    SlotVars v;
    v.state = kFree;
    v.cell = -1;
    v.qe = -1;
    v.sdt = dt;
    v.T = v.T0 = 1500.0;
    v.Tin = CUDART_NAN;
    v.h = 0.0;
    v.norm_prev = CUDART_INF;
    v.atol_rho = v.atol_e = 0.0;
    v.k = v.level = v.attempts = v.iters = v.subs = v.fails = 0;
    v.t_units = 0;
    return v;
}

// Steps the warp's slots, G lanes each, until no cell is left for any of them
// (or, with few slots left and b.wide, until the rest is better stepped by
// wide warps).  Q: request-server mode, cells claimed from b.queue (each
// slot's request descriptor in host memory; its dt, buffers and completion
// accounting).  G0: see newton_iteration.
template <int G, int G0, typename JT, bool Q>
__device__ __forceinline__ void step_cells(const DeviceMech &m, const StepOptions &o, const StepBatch &b,
                                           SlotMem<JT> &sm, SlotVars &v) {
    constexpr int S = 32 / G;
    const int lane = threadIdx.x & 31;
    const int slot = lane / G;
    const int sl = lane - slot * G;
    const int ns = m.ns, n = ns + 1;
    const double *tab = m.exp_tab;   // 2 KB, stays in L1
    int &state = v.state, &qe = v.qe, &k = v.k, &level = v.level, &attempts = v.attempts, &iters = v.iters,
        &subs = v.subs, &fails = v.fails;
    long long &cell = v.cell, &t_units = v.t_units;
    double &sdt = v.sdt, &T = v.T, &T0 = v.T0, &Tin = v.Tin, &h = v.h, &norm_prev = v.norm_prev,
           &atol_rho = v.atol_rho, &atol_e = v.atol_e;
    unsigned long long idle_since = 0;
    (void)S;
    (void)idle_since;
    (void)qe;
    const long long total = 1LL << o.max_halvings;

    // per-cell outputs (lane 0 of the slot); in request-server mode the
    // request's own buffers, and the cell counted done
    auto emit = [&](int code, double Tv) {
        if (sl == 0) {
            if constexpr (Q) {
                const ServeDesc *d = b.queue.mdesc + qe;
                int *st = ld_cg(&d->status);
                double *to = ld_cg(&d->T_out);
                if (st) st[cell] = code;
                if (to) to[cell] = Tv;
                serve_cell_done(b.queue, qe);
            } else {
                if (b.status) b.status[cell] = code;
                if (b.T_out) b.T_out[cell] = Tv;
                if (b.newton_iters) b.newton_iters[cell] = iters;
                if (b.substeps) b.substeps[cell] = subs;
                if (b.failures) b.failures[cell] = fails;
            }
        }
    };
#pragma unroll 1
    for (;;) {
        // refill free slots and settle every pending temperature recovery
        bool q_dry = false;   // request-server mode: a claim this trip found no cell
#pragma unroll 1
        for (int pass = 0; pass < 2; ++pass) {
            long long got = -1;
            bool loading;
            const double *rho_in = b.rho, *e_in = b.e;
            long long ld_in = b.ld;
            if constexpr (Q) {
                // the warp's free slots take consecutive cells of one chunk,
                // claimed by lane 0, which reads the chunk's descriptor once
                const unsigned lead = __ballot_sync(kFull, state == kFree && sl == 0);
                int cnt = 0, e = -1;
                long long v0 = 0;
                double cdt = 0.0;   // the chunk's dt (a slot's own sdt changes only when it loads)
                if (lane == 0 && lead && !q_dry) {
                    cnt = serve_claim(b.queue, __popc(lead), v0, e);
                    if (cnt > 0) {
                        const ServeDesc *d = b.queue.mdesc + e;
                        rho_in = ld_cg(&d->rho);
                        e_in = ld_cg(&d->e);
                        ld_in = ld_cg(&d->ld);
                        cdt = ld_cg(&d->dt);
                        atomicMin(b.queue.t_first + e, globaltimer_ns());
                    }
                }
                cnt = __shfl_sync(kFull, cnt, 0);
                if (lead && cnt == 0) q_dry = true;
                loading = false;
                if (cnt > 0) {
                    e = __shfl_sync(kFull, e, 0);
                    v0 = __shfl_sync(kFull, v0, 0);
                    rho_in = reinterpret_cast<const double *>(
                        __shfl_sync(kFull, reinterpret_cast<unsigned long long>(rho_in), 0));
                    e_in = reinterpret_cast<const double *>(
                        __shfl_sync(kFull, reinterpret_cast<unsigned long long>(e_in), 0));
                    ld_in = __shfl_sync(kFull, ld_in, 0);
                    cdt = __shfl_sync(kFull, cdt, 0);
                    // this slot's rank among the warp's free slots
                    const int rank = __popc(lead & ((1u << (slot * G)) - 1u));
                    loading = state == kFree && rank < cnt;
                    if (loading) {
                        qe = e;
                        sdt = cdt;
                        cell = (v0 & ((1LL << kServeChunkLog) - 1)) + rank;
                    }
                }
            } else {
                if (state == kFree && sl == 0) got = (long long)atomicAdd(b.work_counter, 1ULL);
                got = __shfl_sync(kFull, got, slot * G);
                loading = state == kFree && got < b.n_cells;
                if (state == kFree && !loading) state = kDead;
                if (loading) cell = got;
            }
            int act = state == kRejected ? kFailSubstep : kNoAction, code = kCellOk;
            bool advanced = false;   // the cell reached dt: its state is written
            // (with no cell to load, the sums' FP64 additions would be a twentieth of
            // all of an iteration's)
            if (__any_sync(kFull, loading)) {
                int nonfin = 0;
                double rt = 0.0, es = 0.0;
                if (loading) {
                    iters = subs = fails = 0;
                    Tin = CUDART_NAN;
                    if (!Q && b.schedule && sl == 0) {
#pragma unroll 1
                        for (int w = 0; w < kSchedWords; ++w) b.schedule[cell * kSchedWords + w] = 0u;
                    }
#pragma unroll 1
                    for (int i = sl; i < n; i += G) {
                        const double v = i < ns ? rho_in[(size_t)i * ld_in + cell] : e_in[cell];
                        sm.x0[i] = v;
                        sm.x[i] = v;
                        if (!isfinite(v)) nonfin = 1;
                        const double ev = fabs(i < ns ? v * __ldg(m.sp + i * kSpStride + 3) : v);
                        if (i < ns) rt = G == G0 ? rt + v : v;
                        es = G == G0 ? es + ev : ev;
                    }
                }
                nonfin = Grp<G>::any(nonfin);
                if constexpr (G == G0) {
                    rt = Grp<G>::sum(rt);
                    es = Grp<G>::sum(es);
                } else {
                    const Fp64Ops op = fp64_ops(tab);
                    rt = wide_dot<G0>(rt, op.one, ns, op);
                    es = wide_dot<G0>(es, op.one, n, op);
                }
                if (loading) {
                    atol_rho = o.atol_rel * rt;
                    atol_e = o.atol_rel * es;
                    T = (!Q && b.T_in) ? b.T_in[cell] : 1500.0;
                    if (nonfin || !(rt > 0.0)) {
                        act = kEmitCell;
                        code = kCellBadInput;
                    } else {
                        state = kInitT;
                    }
                }
            }
            __syncwarp();
            const bool needT = state == kInitT || state == kNewtonT || state == kCheckT;
            if (!__any_sync(kFull, needT || act != kNoAction)) break;
            double Tr = T;
            bool ok = false;
            recover_T<G, G0, sizeof(JT) == 4>(m, tab, sm.x, sl, needT, state == kInitT && (Q || !b.T_in) && m.fp32_start, T,
                                              Tr, ok);
            int neg = 0;
            if (__any_sync(kFull, state == kCheckT)) {
#pragma unroll 1
                for (int i = sl; i < ns; i += G)
                    if (bits_lt(sm.x[i], 0.0) && bits_gt(fabs(sm.x[i]), atol_rho)) neg = 1;   // x < -atol
                neg = Grp<G>::any(neg);
            }
            __syncwarp();
            if (state == kInitT) {
                if (!ok) {
                    act = kEmitCell;
                    code = kCellTFailed;
                } else {
                    T = T0 = Tin = Tr;
                    t_units = 0;
                    level = 0;
                    attempts = 0;
                    act = sdt == 0.0 ? kEmitCell : kStartSubstep;
                }
            } else if (state == kNewtonT) {
                if (!ok) {
                    act = kFailSubstep;
                } else {
                    T = Tr;
                    state = kNewtonReady;
                }
            } else if (state == kCheckT) {
                if (!ok || neg) {
                    act = kFailSubstep;
                } else {
                    T = Tr;
                    // accept the substep (and record it: attempt attempts - 1
                    // < 32 kSchedWords, the budget being capped when recording)
                    if (!Q && b.schedule && sl == 0) {
                        const int a = attempts - 1;
                        b.schedule[cell * kSchedWords + (a >> 5)] |= 1u << (a & 31);
                    }
                    if (!Q && b.substep_states && subs < kSubstepStates) {
                        double *rec = b.substep_states + ((size_t)cell * kSubstepStates + subs) * n;
#pragma unroll 1
                        for (int i = sl; i < n; i += G) rec[i] = sm.x[i];
                    }
#pragma unroll 1
                    for (int i = sl; i < n; i += G) sm.x0[i] = sm.x[i];
                    T0 = T;
                    t_units += total >> level;
                    ++subs;
                    if (level > 0) --level;
                    advanced = t_units == total;
                    act = advanced ? kEmitCell : kStartSubstep;
                }
            }
            if (act == kFailSubstep) {
                ++fails;
                ++level;
                act = kStartSubstep;
                if (level > o.max_halvings) {
                    act = kEmitCell;
                    code = kCellNewtonFailed;
                }
            }
            if (act == kStartSubstep) {
                if (attempts >= o.max_attempts) {
                    act = kEmitCell;
                    code = kCellTooManySteps;
                } else {
                    while ((total >> level) > total - t_units) ++level;
                    h = sdt * __hiloint2double((1023 - level) << 20, 0);   // sdt 2^-level, level <= 40
                    ++attempts;
#pragma unroll 1
                    for (int i = sl; i < n; i += G) sm.x[i] = sm.x0[i];
                    T = T0;
                    k = 0;
                    norm_prev = CUDART_INF;
                    state = kNewtonReady;
                }
            }
            if (act == kEmitCell) {
                if (advanced) {
                    double *rho_out = b.rho, *e_out = b.e;
                    long long ld_out = b.ld;
                    if constexpr (Q) {
                        const ServeDesc *d = b.queue.mdesc + qe;
                        rho_out = ld_cg(&d->rho);
                        e_out = ld_cg(&d->e);
                        ld_out = ld_cg(&d->ld);
                    }
#pragma unroll 1
                    for (int i = sl; i < n; i += G) {
                        if (i < ns)
                            rho_out[(size_t)i * ld_out + cell] = sm.x[i];
                        else
                            e_out[cell] = sm.x[i];
                    }
                    if constexpr (Q) {
                        // every lane's results before lane 0 counts the cell done
                        // (the slot's G lanes are converged here)
                        __syncwarp(G == 32 ? kFull : (((1u << G) - 1u) << (slot * G)));
                    }
                }
                emit(code, code == kCellOk ? T : Tin);
                state = kFree;
            }
            __syncwarp();
        }
        if constexpr (G == G0 && !Q && G <= kWideMaxG) {
            // (a slot is dead once the cells have run out)
            if (b.wide && __popc(__ballot_sync(kFull, state != kDead && sl == 0)) <= S / 4) return;
        }
        if (!__any_sync(kFull, state == kNewtonReady)) {
            if (__all_sync(kFull, state == kDead)) break;
            if constexpr (Q) {
                // no published cell for any slot of the warp: poll for more
                // (bounded by the linger time, then the warp leaves)
                if (__all_sync(kFull, state == kFree)) {
                    const unsigned long long now = globaltimer_ns();
                    if (idle_since == 0) idle_since = now;
                    if (lane == 0) serve_refresh(b.queue);
                    __syncwarp();
                    // one decision for the whole warp
                    if (__any_sync(kFull, (int)blockIdx.x >= ld_cg(b.queue.dbudget) ||
                                              now - idle_since > (unsigned long long)b.queue.linger_ns))
                        break;
                    __nanosleep(20000);
                }
            }
            continue;
        }
        if constexpr (Q) idle_since = 0;
        // one Newton iteration of Eq. 29 for every slot
        double norm = 0.0, T_pred = T;
        bool bad = false;
        newton_iteration<G, G0, JT>(m, tab, sm, sl, T, h, atol_rho, atol_e, o.rtol, norm, bad, T_pred);
        if (state == kNewtonReady) {
            // start the next temperature recovery from the linear prediction
            if (bits_gt(T_pred, kTlo) && bits_lt(T_pred, kThi)) T = T_pred;
            ++iters;
            if (o.point_implicit || !bits_gt(norm, 1.0) ||
                (o.conv_kappa > 0.0 && k >= 1 && bits_lt(norm, norm_prev) &&
                 norm * norm <= o.conv_kappa * (norm_prev - norm))) {
                // (the contraction-rate stop theta / (1 - theta) norm <= kappa,
                // theta = norm / norm_prev < 1, multiplied out: no division)
                state = kCheckT;
            } else if (o.div_check && k >= 2 && !bits_lt(norm, norm_prev)) {
                state = kRejected;
            } else {
                norm_prev = norm;
                ++k;
                state = k >= o.max_newton ? kRejected : kNewtonT;
            }
            if (bad) state = kRejected;
        }
        __syncwarp();
    }
}

// At most 10 warps per block and 96 registers per thread: 20 warps fit on an
// SM when shared memory allows it (2 blocks of 10; the mixed path at 36
// species, 11.5 KB per cell).
//   Wide warps: with several cells per warp, an iteration is a serial chain
// that takes a warp as long for one cell as for all (4 lanes per cell, 9
// species, alone on its SM: 89,000 cycles mixed, 152,000 FP64), and the last
// cells of a launch and the cells of a small one leave most of it idle.  A
// warp with a quarter of its cells left and no more to come therefore steps
// them one after another with all its lanes, a species to a lane, each in
// the slot's shared memory; with b.one_cell it starts so, one cell at a time.
// Sums and lists keep the order of G lanes per cell, so that a cell's result
// does not depend on where it ends.  9 species, dt 1e-6, before and after:
// 1,000 cells 1.82 -> 0.72 ms (FP64), 0.96 -> 0.47 ms (mixed); 16,000 cells
// 3.59 -> 2.04 and 1.97 -> 1.13 ms; 262,144 cells 16.2 -> 15.2 and 7.0 -> 6.4
// ms.  At an eighth of the cells left 16,000 cells take 2.37 and 1.16 ms, at
// three eighths 2.15 and 1.14, at five 2.02 and 1.17 (262,144 mixed: 6.5,
// 6.5, 6.7).
template <int G, typename JT, bool Q = false>
__global__ void __launch_bounds__(kMaxBlockThreads, 2) be_kernel(DeviceMech m, StepOptions o, StepBatch b) {
    extern __shared__ __align__(16) char smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, slot = lane / G;
    const int per_warp = !Q && G <= kWideMaxG && b.one_cell ? 1 : 32 / G;
    const long long sbytes = slot_stride(m, (int)sizeof(JT), G);
    char *warp_mem = smem + (size_t)warp * per_warp * sbytes;
    SlotMem<JT> sm;
    // (carved before the barrier: 2 % less time than behind it at 36 species, mixed)
    if constexpr (Q || G > kWideMaxG) sm.carve(warp_mem + slot * sbytes, m);
    __syncthreads();
    if (!Q && b.chain_next) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if constexpr (Q || G > kWideMaxG) {
        SlotVars v = free_slot(b.dt);
        step_cells<G, G, JT, Q>(m, o, b, sm, v);
    } else {
        unsigned left = 1;
        {
            SlotVars v = free_slot(b.dt);
            sm.carve(warp_mem + (b.one_cell ? 0 : slot) * sbytes, m);
            if (!b.one_cell) {
                step_cells<G, G, JT, false>(m, o, b, sm, v);
                left = __ballot_sync(kFull, v.state != kDead && lane % G == 0);
            }
            // (the matrix is not in use here; b.wide implies it is large enough)
            if (v.state != kDead && lane == (b.one_cell ? 0 : slot * G)) *reinterpret_cast<SlotVars *>(sm.A) = v;
            __syncwarp();
        }
#pragma unroll 1
        while (left) {
            const int src = __ffs(left) - 1;
            left &= left - 1;
            sm.carve(warp_mem + src / G * sbytes, m);
            SlotVars w = *reinterpret_cast<const SlotVars *>(sm.A);
            __syncwarp();
            step_cells<32, G, JT, false>(m, o, b, sm, w);
        }
    }
    // (a chain's launches end in order: what follows the last one in its
    // stream finds all of them done)
    if (!Q && b.chain_prev) asm volatile("griddepcontrol.wait;" ::: "memory");
}

}  // namespace chem
