// chem_fields.cu -- whole-field conversions: the chemistry state from (T, P,
// Y) (Dalton, Eq. 5, and Eq. 3), and the temperature of given states.
//
// One thread per cell.  Both kernels are bound by the FP64 pipe, so the
// energies come from the multiplied-out polynomials (five fused multiply-adds
// per species instead of nine operations on h/RT) and sums and products are
// register-only fused multiply-adds (chem_fp64.cuh).  A block keeps its
// cells' rows (Y, or rho) in shared memory, [species][thread], and the
// polynomial coefficients species-major beside them: the temperature's
// iterations read neither again from L2.
#include <cuda_runtime.h>

#include "../../include/chem.h"
#include "chem_fp64.cuh"
#include "chem_handle.h"

namespace chem {

constexpr int kFieldThreads = 128;   // cells per block; 32 when a call has few
constexpr int kEnergyCoefs = 12;     // per species and range: c0..c5, d0..d4, 0 (kTpolyStride)
constexpr int kEnergyCoefsF = 12;    // the same in FP32

// Copies the energy polynomials to shared memory as [species][range][12].
__device__ __forceinline__ void stage_tpoly(const DeviceMech &m, double *tab) {
    static_assert(kEnergyCoefs == kTpolyStride, "the table's own coefficients");
    const int ns = m.ns;
    for (int e = threadIdx.x; e < ns * 2 * kEnergyCoefs; e += blockDim.x) {
        const int s = e / (2 * kEnergyCoefs), q = e - s * 2 * kEnergyCoefs, rg = q / kEnergyCoefs,
                  c = q - rg * kEnergyCoefs;
        tab[e] = __ldg(m.tpoly + (size_t)(2 * c + rg) * ns + s);
    }
}

// Bound by the FP64 pipe (five operations per species) and by memory alike.
// 524,365 cells of 36 species: 0.43 ms with h/RT and two reads of Y, 0.29 ms so.
__global__ void __launch_bounds__(kFieldThreads) state_from_tpy_kernel(DeviceMech m, long long n, long long ld,
                                                                       const double *T, const double *P,
                                                                       const double *Y, double *rho, double *e) {
    extern __shared__ __align__(16) double sm_f[];
    const int ns = m.ns, bs = blockDim.x;
    double *tab = sm_f, *y = sm_f + ns * 2 * kEnergyCoefs + threadIdx.x;   // y[s * bs]
    const Fp64Ops op = fp64_ops(m.exp_tab);
    const long long i = blockIdx.x * (long long)bs + threadIdx.x;
    const bool live = i < n;
    stage_tpoly(m, tab);
    const double Ti = live ? T[i] : 1000.0;
    double invW = 0.0;
#pragma unroll 4
    for (int s = 0; s < ns; ++s) {
        const double v = live ? Y[(size_t)s * ld + i] : 0.0;
        y[s * bs] = v;
        invW = fma(v, __ldg(m.sp + s * kSpStride + 1), invW);
    }
    __syncthreads();   // the table
    if (!live) return;
    const double rt = P[i] / (kR * Ti * invW);
    const long long Tb = __double_as_longlong(Ti);
    double ei = 0.0;
#pragma unroll 2
    for (int s = 0; s < ns; ++s) {
        const double rs = op.mul(rt, y[s * bs]);
        rho[(size_t)s * ld + i] = rs;
        const double2 *c =
            reinterpret_cast<const double2 *>(tab + (2 * s + thermo_range(m, s, Tb)) * kEnergyCoefs);
        const double2 c01 = c[0], c23 = c[1], c45 = c[2];
        const double es = fma(fma(fma(fma(fma(c45.y, Ti, c45.x), Ti, c23.y), Ti, c23.x), Ti, c01.y), Ti, c01.x);
        ei = fma(rs, es, ei);
    }
    e[i] = ei;
}

// Temperature of (rho, e): Newton on sum_s rho_s e_s^sens(T) = e safeguarded by
// bisection on [kTlo, kThi], ended as in the step.  Without a guess, and where
// no density is negative and no energy steps down at a t_mid or far up (so
// that e(T) is increasing and has one root), Newton runs in FP32 first, at a
// sixty-fourth of the cost: from 1500 K the FP64 iterations were six or seven,
// from there they are two.
// Bound by the FP64 pipe: after a step below a millionth of T that is near no
// kink the derivative is kept (it has changed by as much, and the next step is
// below 1e-12 T), so that the last iteration evaluates the energies alone.
// 524,365 cells of 36 species: 6.4 ms with c_p/R and h/RT re-read from L2 and
// the FP64 iterations from 1500 K, 0.81 ms without, 0.70 ms with one
// derivative.
__global__ void __launch_bounds__(kFieldThreads) temperature_kernel(DeviceMech m, long long n, long long ld,
                                                                    const double *rho, const double *e,
                                                                    const double *Tg, double *Tout) {
    extern __shared__ __align__(16) double sm_f[];
    const int ns = m.ns, bs = blockDim.x;
    double *tab = sm_f, *x = sm_f + ns * 2 * kEnergyCoefs + threadIdx.x;   // x[s * bs]
    float *tabf = reinterpret_cast<float *>(sm_f + ns * 2 * kEnergyCoefs + (size_t)ns * bs);
    const Fp64Ops op = fp64_ops(m.exp_tab);
    const long long i = blockIdx.x * (long long)bs + threadIdx.x;
    const bool live = i < n;
    stage_tpoly(m, tab);
    bool nonneg = true;
#pragma unroll 4
    for (int s = 0; s < ns; ++s) {
        const double v = live ? rho[(size_t)s * ld + i] : 0.0;
        x[s * bs] = v;
        nonneg = nonneg && __double_as_longlong(v) >= 0;
    }
    __syncthreads();   // the table
    for (int q = threadIdx.x; q < ns * 2 * kEnergyCoefs; q += bs) tabf[q] = (float)tab[q];
    __syncthreads();
    if (!live) return;
    double lo = kTlo, hi = kThi, T = Tg ? Tg[i] : 1500.0;
    if (!(T > lo && T < hi)) T = 1500.0;
    const double ei = e[i];
    if (!Tg && nonneg && m.fp32_start) {
        const float ef = d2f_rz(ei);
        float Tf = 1500.f;
#pragma unroll 1
        for (int it = 0; it < 4; ++it) {
            const long long Tb = __double_as_longlong(f2d_alu(Tf));
            float f = -ef, fp = 0.f;
#pragma unroll 1
            for (int s = 0; s < ns; ++s) {
                const float4 *c =
                    reinterpret_cast<const float4 *>(tabf + (2 * s + thermo_range(m, s, Tb)) * kEnergyCoefsF);
                const float4 a = c[0], b = c[1], d = c[2];   // c0..c3 | c4 c5 d0 d1 | d2 d3 d4 0
                const float r = d2f_rz(x[s * bs]);
                f = fmaf(r, fmaf(fmaf(fmaf(fmaf(fmaf(b.y, Tf, b.x), Tf, a.w), Tf, a.z), Tf, a.y), Tf, a.x), f);
                fp = fmaf(r, fmaf(fmaf(fmaf(fmaf(d.z, Tf, d.y), Tf, d.x), Tf, b.w), Tf, b.z), fp);
            }
            Tf -= __fdividef(f, fp);
            // (a NaN goes to the lower end as well, which is no start)
            Tf = fminf(fmaxf(Tf, (float)kTlo), (float)kThi);
        }
        const double Ts = f2d_alu(Tf);
        if (Ts > lo && Ts < hi) T = Ts;
    }
    bool ok = false, near = false;
    double slope = 0.0;   // 1 / (df/dT)
#pragma unroll 1
    for (int it = 1; it <= kTmaxIter; ++it) {
        const long long Tb = __double_as_longlong(T);
        const bool kink = near_kink(m, T);
        double f = 0.0;
        if (near) {
#pragma unroll 2
            for (int s = 0; s < ns; ++s) {
                const double2 *c =
                    reinterpret_cast<const double2 *>(tab + (2 * s + thermo_range(m, s, Tb)) * kEnergyCoefs);
                const double2 c01 = c[0], c23 = c[1], c45 = c[2];
                f = fma(x[s * bs], fma(fma(fma(fma(fma(c45.y, T, c45.x), T, c23.y), T, c23.x), T, c01.y), T, c01.x), f);
            }
        } else {
            double fp = 0.0;
#pragma unroll 2
            for (int s = 0; s < ns; ++s) {
                const double2 *c =
                    reinterpret_cast<const double2 *>(tab + (2 * s + thermo_range(m, s, Tb)) * kEnergyCoefs);
                const double2 c01 = c[0], c23 = c[1], c45 = c[2], d01 = c[3], d23 = c[4], d4 = c[5];
                const double r = x[s * bs];
                f = fma(r, fma(fma(fma(fma(fma(c45.y, T, c45.x), T, c23.y), T, c23.x), T, c01.y), T, c01.x), f);
                fp = fma(r, fma(fma(fma(fma(d4.x, T, d23.y), T, d23.x), T, d01.y), T, d01.x), fp);
            }
            slope = 1.0 / fp;
        }
        f = op.sub(f, ei);
        if (f == 0.0) {
            ok = true;
            break;
        }
        if (f > 0.0)
            hi = T;
        else
            lo = T;
        double Tn = fma(-f, slope, T), dT = Tn - T;
        const bool inside = Tn > lo && Tn < hi;
        const double tol = (inside && !kink ? kTstep : kTtol) * T;
        // (a step below half an ulp leaves T at an end of the bracket)
        if (!inside && !(fabs(dT) <= tol)) {
            Tn = 0.5 * (lo + hi);
            dT = Tn - T;
        }
        near = inside && !kink && fabs(dT) <= 1e-6 * T;
        T = Tn;
        if (fabs(dT) <= tol) {
            ok = !(T <= kTlo * (1.0 + 1e-9) || T >= kThi * (1.0 - 1e-9));
            break;
        }
    }
    Tout[i] = ok ? T : NAN;
}

// Threads per block: 128 once they fill the SMs, else 32, so that a small
// field spreads over more of them.
static int field_threads(const Handle *h, long long n) { return n >= (long long)kFieldThreads * h->num_sms ? kFieldThreads : 32; }

}  // namespace chem

using namespace chem;

extern "C" int chem_state_from_tpy(chem_handle_t hh, int64_t n, int64_t ld, const double *T, const double *P,
                                   const double *Y, double *rho_s, double *e, void *stream) {
    Handle *h = hh;
    if (!h || !T || !P || !Y || !rho_s || !e) return fail(CHEM_E_INVALID_ARG, "NULL argument");
    if (n < 0 || (ld != 0 && ld < n)) return fail(CHEM_E_INVALID_ARG, "sizes");
    if (n == 0) return CHEM_OK;
    if (ld == 0) ld = n;
    const int bs = field_threads(h, n);
    const size_t smem = ((size_t)h->ns * 2 * kEnergyCoefs + (size_t)h->ns * bs) * sizeof(double);
    cudaError_t ce = cudaFuncSetAttribute(state_from_tpy_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)h->max_smem_optin);
    if (ce != cudaSuccess) return cuda_fail(ce, "cudaFuncSetAttribute");
    state_from_tpy_kernel<<<(unsigned)((n + bs - 1) / bs), bs, smem, (cudaStream_t)stream>>>(h->mech, n, ld, T, P, Y,
                                                                                            rho_s, e);
    ce = cudaGetLastError();
    if (ce != cudaSuccess) return cuda_fail(ce, "state_from_tpy launch");
    h->launches.fetch_add(1);
    return CHEM_OK;
}

extern "C" int chem_temperature(chem_handle_t hh, int64_t n, int64_t ld, const double *rho_s, const double *e,
                                const double *T_guess, double *T_out, void *stream) {
    Handle *h = hh;
    if (!h || !rho_s || !e || !T_out) return fail(CHEM_E_INVALID_ARG, "NULL argument");
    if (n < 0 || (ld != 0 && ld < n)) return fail(CHEM_E_INVALID_ARG, "sizes");
    if (n == 0) return CHEM_OK;
    if (ld == 0) ld = n;
    const int bs = field_threads(h, n);
    const size_t smem = ((size_t)h->ns * 2 * kEnergyCoefs + (size_t)h->ns * bs) * sizeof(double) +
                        (size_t)h->ns * 2 * kEnergyCoefsF * sizeof(float);
    cudaError_t ce = cudaFuncSetAttribute(temperature_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)h->max_smem_optin);
    if (ce != cudaSuccess) return cuda_fail(ce, "cudaFuncSetAttribute");
    temperature_kernel<<<(unsigned)((n + bs - 1) / bs), bs, smem, (cudaStream_t)stream>>>(h->mech, n, ld, rho_s, e,
                                                                                         T_guess, T_out);
    ce = cudaGetLastError();
    if (ce != cudaSuccess) return cuda_fail(ce, "temperature launch");
    h->launches.fetch_add(1);
    return CHEM_OK;
}
