// chem_fp64.cuh -- FP64 arithmetic of the kernels on a part whose FP64 pipe is
// its scarcest unit: register-only fused multiply-adds, conversions and
// comparisons on the integer pipe, reciprocals.
#pragma once

#include <cuda_runtime.h>

#include "chem_internal.h"

namespace chem {

// The FP64 pipe takes a warp's fused multiply-add with three register
// operands every 16 cycles, but an addition, a multiplication or anything
// with a constant operand only every 19 (measured, 4 to 20 warps on an SM).
// So sums and products are written as fused multiply-adds with a 1 and a -0
// in registers (the same results, signed zeros included), and constants come
// from a table in global memory.  The loads are volatile: the compiler must
// not see the values, nor keep all of them in registers.
struct Fp64Ops {
    double one, nz;   // 1 and -0
    __device__ __forceinline__ double add(double a, double b) const { return __fma_rn(a, one, b); }
    __device__ __forceinline__ double sub(double a, double b) const { return __fma_rn(-b, one, a); }
    __device__ __forceinline__ double mul(double a, double b) const { return __fma_rn(a, b, nz); }
};
__device__ __forceinline__ double2 ld_const2(const double *p) {
    double2 v;
    asm volatile("ld.global.nc.v2.f64 {%0, %1}, [%2];"
                 : "=d"(v.x), "=d"(v.y)
                 : "l"(__cvta_generic_to_global(p)));
    return v;
}
// (tab: the exp table, which the constants follow)
__device__ __forceinline__ Fp64Ops fp64_ops(const double *tab) {
    const double2 v = ld_const2(tab + kConstOne);
    return Fp64Ops{v.x, v.y};
}

// Conversions between FP64 and FP32 on the integer pipe: on this part a
// conversion instruction occupies the FP64 pipe as long as a DFMA does.
// FP64 -> FP32 rounds toward zero; magnitudes below the smallest normal
// float give a signed zero, above the largest an infinity; NaN stays NaN.
__device__ __forceinline__ float d2f_rz(double x) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const unsigned hi = (unsigned)(b >> 32), lo = (unsigned)b;
    const unsigned sign = hi & 0x80000000u;
    const int e = (int)((hi >> 20) & 0x7ffu) - 896;
    const unsigned man = ((hi & 0xfffffu) << 3) | (lo >> 29);
    unsigned f = sign | ((unsigned)e << 23) | man;
    if (e <= 0) f = sign;
    if (e >= 255) f = sign | 0x7f800000u | ((e == 1151 && ((hi & 0xfffffu) | lo)) ? 0x400000u : 0u);
    return __uint_as_float(f);
}
// FP32 -> FP64, exact for normal floats and infinities (NaN stays NaN,
// subnormal floats give a signed zero).
__device__ __forceinline__ double f2d_alu(float v) {
    const unsigned u = __float_as_uint(v);
    const unsigned sign = u & 0x80000000u, e = (u >> 23) & 0xffu, man = u & 0x7fffffu;
    unsigned hi = sign | ((e + 896u) << 20) | (man >> 3);
    unsigned lo = man << 29;
    if (e == 0) {
        hi = sign;
        lo = 0u;
    }
    if (e == 255u) hi = sign | 0x7ff00000u | (man >> 3);
    return __hiloint2double((int)hi, (int)lo);
}
// The same for values whose range is known, in a third of the instructions:
// a double of magnitude below 2^128 (one below the smallest normal float
// gives one of its order), an integer below 2^24 (not -0), a positive normal
// float.
__device__ __forceinline__ float near_float(double x) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const unsigned hi = (unsigned)(b >> 32);
    const int e = max((int)(hi & 0x7fffffffu) - 0x38000000, 0);
    return __uint_as_float((hi & 0x80000000u) | __funnelshift_l((unsigned)b, (unsigned)e, 3));
}
__device__ __forceinline__ double f2d_int(float v) {
    const unsigned u = __float_as_uint(v);
    const unsigned hi = (u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u);
    return __hiloint2double(u ? (int)hi : 0, (int)(u << 29));
}
__device__ __forceinline__ double f2d_pos(float v) {
    const unsigned u = __float_as_uint(v);
    return __hiloint2double((int)((u >> 3) + 0x38000000u), (int)(u << 29));
}
// Order of doubles by their bit patterns (integer pipe): exact for a >= 0
// against b > 0; a negative a counts as smaller, a NaN a as larger.
__device__ __forceinline__ bool bits_gt(double a, double b) {
    return __double_as_longlong(a) > __double_as_longlong(b);
}
__device__ __forceinline__ bool bits_lt(double a, double b) {
    return __double_as_longlong(a) < __double_as_longlong(b);
}
__device__ __forceinline__ bool finite_bits(double v) {
    return ((unsigned)((unsigned long long)__double_as_longlong(v) >> 52) & 0x7ffu) != 0x7ffu;
}

// Reciprocal: the hardware approximation r refined with its residual
// e = 1 - a r as r (1 + e + e^2), whose error is e^3 (the approximation is
// good to about 2^-23, so below FP64 rounding): three FP64 operations.
__device__ __forceinline__ double frcp(double a, const Fp64Ops &op) {
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(a));
    const double e = fma(-a, r, op.one);
    return fma(r, fma(e, e, e), r);
}
// One Newton step only (relative error about 1e-14): for reciprocals that
// scale a convergence ratio or the temperature recovery's Newton step, never
// a rate, an energy or the elimination.
__device__ __forceinline__ double frcp1(double a, const Fp64Ops &op) {
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(a));
    const double e = fma(-a, r, op.one);
    return fma(r, e, r);
}
// range of species s at T (1: T > T_mid, the high range)
__device__ __forceinline__ int thermo_range(const DeviceMech &m, int s, long long Tbits) {
    return Tbits > __ldg(reinterpret_cast<const long long *>(m.tmid) + s) ? 1 : 0;
}
// whether a small step of the temperature recovery from T may cross a t_mid
// at which an energy or a heat capacity changes: the derivative is then
// another range's, off by as much as the heat capacity changes
__device__ __forceinline__ bool near_kink(const DeviceMech &m, double T) {
    return bits_gt(T, m.kink_lo) & bits_lt(T, m.kink_hi);
}

}  // namespace chem
