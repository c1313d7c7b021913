// Arithmetic of the defect-correction update r -= A_0 e (FP64 r, FP32 e), shared
// by the update kernels and the resident solve of small grids.
#pragma once
#include <cuda_runtime.h>

namespace sg {

__device__ __forceinline__ void two_sum(float a, float b, float& s, float& err) {
    s = a + b;
    const float bb = s - a;
    err = (a - (s - bb)) + (b - bb);
}

// float -> double from the IEEE fields (subnormal floats, below 1.2e-38, become 0).
__device__ __forceinline__ double f2d_bits(float x) {
    const unsigned u = __float_as_uint(x);
    const unsigned sgn = u & 0x80000000u, ex = (u >> 23) & 0xffu, m = u & 0x7fffffu;
    unsigned hi, lo;
    if (ex == 0u) { hi = sgn; lo = 0u; }
    else if (ex == 255u) { hi = sgn | 0x7ff00000u | (m >> 3); lo = m << 29; }
    else { hi = sgn | ((ex + 896u) << 20) | (m >> 3); lo = m << 29; }
    return __hiloint2double((int)hi, (int)lo);
}

// double -> float by truncating the significand (within one FP32 ulp; values
// below 2^-126 become 0, beyond the FP32 range +-inf).
__device__ __forceinline__ float d2f_bits(double x) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const unsigned sgn = hi & 0x80000000u, ex = (hi >> 20) & 0x7ffu, mh = hi & 0xfffffu;
    if (ex <= 896u) return __uint_as_float(sgn);
    if (ex >= 1151u) return __uint_as_float(sgn | 0x7f800000u | ((ex == 2047u && (mh | lo)) ? 0x400000u : 0u));
    return __uint_as_float(sgn | ((ex - 896u) << 23) | (mh << 3) | (lo >> 29));
}

// r -= (A_0 e) for one cell, A_0 the homogeneous operator, formed without
// rounding: the FP32 neighbour sum is split by TwoSum into a value and its
// exact error (products by -6 and -2 are exact up to one FMA term), and both
// enter r through FP64 FMAs.  TWOD: without the z axis (its 1 / h^2 is zero).
template <bool UNIFORM, bool TWOD = false>
__device__ __forceinline__ double update_r(double ihx2, double ihy2, double ihz2, float c, float xm, float xp,
                                           float ym, float yp, float zm, float zp, double r) {
    if (UNIFORM) {
        // sum of the six neighbours minus 6 c, compensated
        const float p = -6.0f * c;
        const float perr = fmaf(-6.0f, c, -p);          // -6 c = p + perr exactly
        float s = xm, comp = perr, t;
        two_sum(s, xp, s, t); comp += t;
        two_sum(s, ym, s, t); comp += t;
        two_sum(s, yp, s, t); comp += t;
        two_sum(s, zm, s, t); comp += t;
        two_sum(s, zp, s, t); comp += t;
        two_sum(s, p, s, t); comp += t;
        const double nih2 = -ihx2;
        r = fma(nih2, f2d_bits(s), r);
        r = fma(nih2, f2d_bits(comp), r);
    } else {
        // per-axis second differences (-2 c is exact), compensated
        const float m2 = -2.0f * c;
        const float a[3][2] = {{xm, xp}, {ym, yp}, {zm, zp}};
        const double ih[3] = {ihx2, ihy2, ihz2};
#pragma unroll
        for (int d = 0; d < (TWOD ? 2 : 3); ++d) {
            float s, comp, t;
            two_sum(a[d][0], a[d][1], s, comp);
            two_sum(s, m2, s, t);
            comp += t;
            r = fma(-ih[d], f2d_bits(s), r);
            r = fma(-ih[d], f2d_bits(comp), r);
        }
    }
    return r;
}

}  // namespace sg
