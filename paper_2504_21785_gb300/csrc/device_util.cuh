// Device helpers shared by the reconstruction kernels.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

namespace fgr {

// Box window of a Gaussian centred at c on one grid axis (see fgr.h):
//   m_lo = ceil(((c - rs) - lo) / h),  m_hi = floor(((c + rs) - lo) / h),
// clipped to [0, n) (empty when m_lo > m_hi).  Evaluated with explicit
// round-to-nearest operations so that no contraction changes the decision.
__device__ __forceinline__ void window_bounds(double c, double rs, double lo, double h, int64_t n,
                                              int64_t *mlo, int64_t *mhi) {
    double a = __ddiv_rn(__dsub_rn(__dsub_rn(c, rs), lo), h);
    double b = __ddiv_rn(__dsub_rn(__dadd_rn(c, rs), lo), h);
    a = ceil(a);
    b = floor(b);
    a = fmin(fmax(a, 0.0), (double)n);
    b = fmin(fmax(b, -1.0), (double)(n - 1));
    *mlo = (int64_t)a;
    *mhi = (int64_t)b;
}

// q = x / step with floor(q) equal to floor of the correctly rounded quotient:
// x * (1/step) differs from it by a few ulps, so it decides the floor unless it
// lies within 1e-9 (relative) of an integer, where the division is done.
__device__ __forceinline__ double quotient_for_floor(double x, double step, double inv_step) {
    const double r = x * inv_step;
    const double n = rint(r);
    if (fabs(r - n) <= 1e-9 * fmax(1.0, fabs(r))) return __ddiv_rn(x, step);
    return r;
}

// floor(fl(x / step)) as an int, mostly without FP64 arithmetic: the FP32
// product (float)x * (float)inv_step has a relative error below 2e-7, so when
// it lies more than 1e-6 (relative) away from an integer its floor is the
// floor of the exact quotient; otherwise (and for |x/step| >= 1e6) the FP64
// path above decides.
__device__ __forceinline__ int floor_div_int(double x, double step, double inv_step) {
    const float rf = (float)x * (float)inv_step;
    const float fl = floorf(rf);
    const float fr = rf - fl;
    const float tol = 1e-6f * fmaxf(1.f, fabsf(rf));
    if (fabsf(rf) < 1e6f && fr > tol && fr < 1.f - tol) return (int)fl;
    const double r = floor(quotient_for_floor(x, step, inv_step));
    return (int)fmin(fmax(r, -1e9), 1e9);
}

// x as h + l in FP32 by integer operations on its bits (FP64 instructions and
// conversions run at 1/64 of the FP32 rate): h is x truncated to 24 bits, l the
// next 23 bits, |x - h - l| < 2^-46 |x|.  False (h = l = 0) unless x is zero or
// 2^-100 <= |x| < 2^126.
__device__ __forceinline__ bool split_double(double x, float &h, float &l) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const unsigned mag = hi & 0x7fffffffu, sgn = hi & 0x80000000u;
    const bool in_range = (mag >> 20) - 923u < 226u;
    const unsigned hb = __funnelshift_l(lo, mag, 3) - 0xc0000000u;         // exponent - 896
    const unsigned lb = ((mag & 0x7ff00000u) << 3) - 0xcb800000u;          // exponent - 919: 2^-23 h's last bit
    const float lf = __uint_as_float(lb | ((lo & 0x1fffffffu) >> 6)) - __uint_as_float(lb);
    h = in_range ? __uint_as_float(hb | sgn) : 0.f;
    l = in_range ? __uint_as_float(__float_as_uint(lf) ^ sgn) : 0.f;
    return in_range || (mag | lo) == 0u;
}

// Grid coordinate x_m = lo + m*h without contraction.
__device__ __forceinline__ double grid_x(double lo, double h, int64_t m) {
    return __dadd_rn(lo, __dmul_rn((double)m, h));
}

// Round to nearest integer for |x| < 2^22 with two FP32 additions on the FMA pipe.
__device__ __forceinline__ float rint_fast(float x) {
    const float magic = 12582912.0f;  // 1.5 * 2^23
    return __fsub_rn(__fadd_rn(x, magic), magic);
}

// Two FP32 operations per instruction (sm_100 and later).  The FMA pipe does no
// more of them per clock (75.7 against 76.0 TFLOP/s measured), but they take
// half the issue slots, which bind the kernels that use them.
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    float2 d;
    asm("{\n\t.reg .b64 a, b, c, d;\n\t"
        "mov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\tmov.b64 c, {%6, %7};\n\t"
        "fma.rn.f32x2 d, a, b, c;\n\t"
        "mov.b64 {%0, %1}, d;\n\t}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return d;
}

__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
    float2 d;
    asm("{\n\t.reg .b64 a, b, d;\n\t"
        "mov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\t"
        "mul.rn.f32x2 d, a, b;\n\t"
        "mov.b64 {%0, %1}, d;\n\t}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}

__device__ __forceinline__ float2 both(float x) { return make_float2(x, x); }

// 2^x on the special-function unit (relative error about 2^-22).
__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ void atomic_add_c(float2 *p, float re, float im) {
    atomicAdd(p, make_float2(re, im));
}

__device__ __forceinline__ void atomic_add_c(double2 *p, double re, double im) {
    atomicAdd(&p->x, re);
    atomicAdd(&p->y, im);
}

}  // namespace fgr
