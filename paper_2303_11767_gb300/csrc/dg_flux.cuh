// dg_flux.cuh -- pointwise physics shared by the stage kernels: the fluxes
// of the shallow water system on the sphere (paper Eq. sph3) and the Rusanov
// flux (Eq. rusanov), with h stored relative to a reference depth.
#pragma once

#include <cuda_runtime.h>

#include "dg_internal.h"

namespace dgk {

// Programmatic dependent launch: a stage kernel lets the next kernel of the
// stream start its prologue as soon as all of its own CTAs are running, and
// waits for the previous kernel's results before its first dependent read.
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Launch `kernel` on `s` with the programmatic-serialization attribute.
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                              Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

template <typename T>
__device__ __forceinline__ T rcp(T x);
// FP64: correctly rounded, as wave_sqrt below.  (The FP64 pipe, 2 lanes per SM,
// bounds the FP64 stage; approximations with one third-order correction, within
// one ulp, made it only 4 to 5 % faster: 180x90 degree 3 104.0 against 108.9 us,
// and two more operations that round them correctly took 109.7.)
template <>
__device__ __forceinline__ double rcp<double>(double x) { return 1.0 / x; }
// FP32: the SFU reciprocal alone (<= 1 ulp; __fdividef(1, x) scales its
// argument around it, for depths that do not occur)
template <>
__device__ __forceinline__ float rcp<float>(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ double wave_sqrt(double x) { return sqrt(x); }
// The wave speed |u| + sqrt(gh).  FP32: the root is x * rsqrt(x) on the SFU, its
// product part of the sum; it only feeds the Rusanov dissipation
__device__ __forceinline__ double wave_speed(double u, double gh) { return fabs(u) + wave_sqrt(gh); }
__device__ __forceinline__ float wave_speed(float u, float gh)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(gh));
    return fma(gh, y, fabsf(u));
}

// Finiteness of many values with one test at the end: chk = fma(x, 0, chk)
// for each x stays 0 while every x is finite and becomes NaN (for good) at
// the first Inf or NaN (Inf * 0 = NaN); one FMA per value instead of a
// compare and a predicated OR.  The rounding intrinsics keep the compiler
// from dropping the product.
__device__ __forceinline__ float nf_acc(float x, float chk) { return __fmaf_rn(x, 0.0f, chk); }
__device__ __forceinline__ double nf_acc(double x, double chk) { return __fma_rn(x, 0.0, chk); }

// The same for FP64 with integer operations on the exponent, off the FP64
// pipe: the largest magnitude word seen.
__device__ __forceinline__ unsigned nf_acc_bits(double x, unsigned m) { return max(m, (unsigned)__double2hiint(x) & 0x7fffffffu); }
__device__ __forceinline__ bool nf_bits(unsigned m) { return m >= 0x7ff00000u; }

// h <= 0 makes u = hu/h meaningless; a NaN depth is reported as non-finite.
template <typename T>
__device__ __forceinline__ void check_depth(T h, unsigned &st)
{
    if (!(h > T(0))) st |= (h != h) ? DG_STATUS_NONFINITE : DG_STATUS_NONPHYSICAL;
}

// (FP64: the compares only where the exponent is not that of a positive number)
template <>
__device__ __forceinline__ void check_depth<double>(double h, unsigned &st)
{
    if ((unsigned)(__double2hiint(h) - 1) >= 0x7fefffffu && !(h > 0.0))
        st |= (h != h) ? DG_STATUS_NONFINITE : DG_STATUS_NONPHYSICAL;
}

// Every multiply-add below is an explicit fma, and every sum that a product
// enters an explicit addition: these functions are inlined at several call
// sites (an edge's flux is evaluated by whichever tile or band owns it), and
// left to the compiler's contraction the same edge could round differently at
// two sites.

// P = g h' (href + h'/2); FP64 with the constants folded, one operation less
template <typename T>
__device__ __forceinline__ T pressure(T hp, T href, T g) { return (hp * g) * fma(T(0.5), hp, href); }
template <>
__device__ __forceinline__ double pressure<double>(double hp, double href, double g) { return hp * fma(0.5 * g, hp, g * href); }

// out = c/2 ((fl + fr) - a (R - L)), a the larger of the speeds (both >= 0)
template <typename T>
__device__ __forceinline__ void rusanov_out(const T *L, const T *R, const T *fl, const T *fr, T al, T ar, T aglob, T c, T *out)
{
    if constexpr (sizeof(T) == 8) {
        // non-negative doubles order like their bits; the factor 1/2 sits in c
        const double a = aglob > 0.0 ? aglob : __longlong_as_double(max(__double_as_longlong(al), __double_as_longlong(ar)));
        const double hc = 0.5 * c;
#pragma unroll
        for (int f = 0; f < 3; ++f) out[f] = hc * fma(-a, R[f] - L[f], __dadd_rn(fl[f], fr[f]));
    } else {
        const T a = aglob > T(0) ? aglob : fmax(al, ar);   // global mode: the stage's largest |u| + c
        const T hc = T(0.5) * c;
#pragma unroll
        for (int f = 0; f < 3; ++f) out[f] = hc * fma(-a, R[f] - L[f], __fadd_rn(fl[f], fr[f]));
    }
}

// Physical lambda-flux (hu, hu u + P, hu v) of a state q = (h', hu, hv) with
// h = href + h' and the pressure P = g h' (href + h'/2) (the constant part
// g href^2/2 is carried by the rho table), and the wave speed |u| + sqrt(g h).
template <typename T>
__device__ __forceinline__ void lam_flux(const T *q, T href, T g, T *f, T &speed, unsigned &st)
{
    const T h = href + q[0];
    check_depth(h, st);
    const T u = q[1] * rcp(h);
    const T P = pressure(q[0], href, g);
    f[0] = q[1];
    f[1] = fma(q[1], u, P);
    f[2] = q[2] * u;
    speed = wave_speed(u, g * h);
}

template <typename T>
__device__ __forceinline__ void th_flux(const T *q, T href, T g, T *f, T &speed, unsigned &st)
{
    const T h = href + q[0];
    check_depth(h, st);
    const T v = q[2] * rcp(h);
    const T P = pressure(q[0], href, g);
    f[0] = q[2];
    f[1] = q[1] * v;
    f[2] = fma(q[2], v, P);
    speed = wave_speed(v, g * h);
}

// Rusanov flux through a lambda-face, left state L (west), right state R
// (east): F* = (F(L) + F(R))/2 - alpha/2 (R - L) with alpha the larger
// one-sided |u| + c; the cos(theta) of U = cos(theta) q cancels against the
// 1/cos(theta) of the eigenvalue of dF/dU.  Scaled by cF = 2/(R dlambda).
template <typename T>
__device__ __forceinline__ void rusanov_lam(const T *L, const T *R, T href, T g, T cF, T *out, unsigned &st,
                                            T aglob = T(0))
{
    T fl[3], fr[3], al, ar;
    lam_flux(L, href, g, fl, al, st);
    lam_flux(R, href, g, fr, ar, st);
    rusanov_out(L, R, fl, fr, al, ar, aglob, cF, out);
}

// Rusanov flux through a theta-face, lower state S, upper state N, times the
// edge cos(theta) ce (flux and jump of U both carry it); scaled by cG.
template <typename T>
__device__ __forceinline__ void rusanov_th(const T *S, const T *Nq, T href, T g, T cGce, T *out, unsigned &st,
                                           T aglob = T(0))
{
    T fs[3], fn[3], as, an;
    th_flux(S, href, g, fs, as, st);
    th_flux(Nq, href, g, fn, an, st);
    rusanov_out(S, Nq, fs, fn, as, an, aglob, cGce, out);
}

}  // namespace dgk
