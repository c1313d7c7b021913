// What the plane-streaming super-step kernels share: asynchronous strip copies
// with reflected or periodic halos, packed FP32 pairs, the arithmetic of one strip
// of a stage and its coefficients.
#pragma once
#include "sg_internal.cuh"

#include <algorithm>
#include <cmath>

namespace sg {

namespace {

__device__ __forceinline__ void cpa4(float* smem, const float* gmem) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cpa16(float* smem, const float* gmem) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cpa_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cpa_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }
__device__ __forceinline__ void cpa_wait_prev() { asm volatile("cp.async.wait_group 1;\n" ::: "memory"); }

// Index of cell v of an axis of n cells in the stored array and its sign:
// periodic image, or odd reflection about both walls (period 2n).
__host__ __device__ __forceinline__ int map_axis(int v, int n, bool periodic, int* sign) {
    if (v >= 0 && v < n) {                  // inside the box: no integer division
        *sign = 1;
        return v;
    }
    if (periodic) {
        *sign = 1;
        const int m = v % n;
        return m < 0 ? m + n : m;
    }
    int m = v % (2 * n);
    if (m < 0) m += 2 * n;
    if (m < n) {
        *sign = 1;
        return m;
    }
    *sign = -1;
    return 2 * n - 1 - m;
}

// Coefficients, all FP32 (the kernel never converts from FP64).
struct LeanCoef {
    float ax[4], ay[4], az[4], b[4];    // stage j >= 2: Y_j = ax sx + ay sy + az sz + b c + W_j
    float ihx2, ihy2, ihz2, m2s;        // stage 1: Lf = ihx2 sx + ihy2 sy + ihz2 sz + m2s c - f
    float m1t;                          //          Y1 = c + m1t Lf
    float k2y0, k2z, k2f;               //          W2 = k2y0 c + k2z Lf + k2f f
    float k3c, k3l, k3f;                //          W3 = nu_3 Y1 + c0_3 c + gamma~_3 tau Lf - mu~_3 tau f
                                        //             = k3c c + k3l Lf + k3f f  (Y1 = c + m1t Lf)
    float kz[4];                        // Y0 = 0: Y1 = kz[1] f, W_j = kz[j] f
    float zx, zy, zz, zb;               // Y0 = 0: Y2 = zx sx(f) + zy sy(f) + zz sz(f) + zb f
};

// The first stage's coefficients as pairs of equal floats (operands of packed FP32).
struct FirstCoef {
    float2 ihx, ihy, ihz, m2s, m1t, k2y0, k2z, k2f, k3c, k3l, k3f;
};
__host__ __device__ __forceinline__ FirstCoef first_coef(const LeanCoef& k) {
    auto two = [](float v) { return make_float2(v, v); };
    return {two(k.ihx2), two(k.ihy2), two(k.ihz2), two(k.m2s), two(k.m1t), two(k.k2y0),
            two(k.k2z),  two(k.k2f),  two(k.k3c),  two(k.k3l), two(k.k3f)};
}

// Source of one 4-cell strip of a staged plane.
struct LoadDesc {
    int dst;        // offset in the plane (floats); -1: this thread loads nothing
    int row;        // source row offset (y index * nx)
    int x01, x23;   // source x of the four cells, 16 bits each
    int flags;      // bit 4: one 16-byte copy; bits 0-3: cells negated by the x/y reflection
};

// Cells gx .. gx + 3 of row gy, copied to offset dst of the plane.
__device__ __forceinline__ LoadDesc make_desc(int dst, int gx, int gy, const LevelGeom& g, bool vec_ok) {
    LoadDesc d;
    d.dst = dst;
    int sy;
    const int yy = map_axis(gy, g.ny, g.per[1] != 0, &sy);
    d.row = yy * g.nx;
    int xs[4], mask = 0;
    bool contiguous = true;
    for (int e = 0; e < 4; ++e) {
        int sx;
        xs[e] = map_axis(gx + e, g.nx, g.per[0] != 0, &sx);
        if (sx * sy < 0) mask |= 1 << e;
        if (sx < 0 || xs[e] != xs[0] + e) contiguous = false;
    }
    d.x01 = xs[0] | (xs[1] << 16);
    d.x23 = xs[2] | (xs[3] << 16);
    const bool vec = vec_ok && contiguous && (xs[0] & 3) == 0;
    d.flags = mask | (vec ? 16 : 0);
    return d;
}

__device__ __forceinline__ void issue(const LoadDesc& d, float* plane_dst, const float* plane_src) {
    if (d.dst < 0) return;
    const float* s = plane_src + d.row;
    if (d.flags & 16) {
        cpa16(plane_dst + d.dst, s + (d.x01 & 0xffff));
    } else {
        cpa4(plane_dst + d.dst + 0, s + (d.x01 & 0xffff));
        cpa4(plane_dst + d.dst + 1, s + (d.x01 >> 16));
        cpa4(plane_dst + d.dst + 2, s + (d.x23 & 0xffff));
        cpa4(plane_dst + d.dst + 3, s + (d.x23 >> 16));
    }
}

// After the thread's copies arrived: negate the cells whose reflection sign
// (x, y and the plane's z sign) is negative.
__device__ __forceinline__ void fixup(const LoadDesc& d, float* plane_dst, int zsign) {
    if (d.dst < 0) return;
    const int m = zsign < 0 ? (~d.flags & 15) : (d.flags & 15);
    if (m == 0) return;
    float4* p = reinterpret_cast<float4*>(plane_dst + d.dst);
    float4 v = *p;
    if (m & 1) v.x = -v.x;
    if (m & 2) v.y = -v.y;
    if (m & 4) v.z = -v.z;
    if (m & 8) v.w = -v.w;
    *p = v;
}

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ void st4(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }

// Packed FP32 pairs (Blackwell f32x2 instructions): each call is two
// independent FP32 operations with the rounding of the scalar ones.
__device__ __forceinline__ unsigned long long pk(float2 v) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(v.x), "f"(v.y));
    return r;
}
__device__ __forceinline__ float2 upk(unsigned long long r) {
    float2 v;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(v.x), "=f"(v.y) : "l"(r));
    return v;
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(pk(a)), "l"(pk(b)), "l"(pk(c)));
    return upk(d);
}
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(pk(a)), "l"(pk(b)));
    return upk(d);
}
__device__ __forceinline__ float2 lo2(float4 v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ float2 hi2(float4 v) { return make_float2(v.z, v.w); }
__device__ __forceinline__ float2 dup2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float4 cat4(float2 a, float2 b) { return make_float4(a.x, a.y, b.x, b.y); }

// One strip of stage j >= 2: Y_j = ax sx + ay sy + az sz + b c + W_j.
__device__ __forceinline__ float4 later_strip(float4 c, float4 n, float4 s, float4 d, float4 u, float l, float r,
                                              float2 ax, float2 ay, float2 az, float2 bb, float4 w) {
    const float2 sx01 = make_float2(l + c.y, c.x + c.z), sx23 = make_float2(c.y + c.w, c.z + r);
    const float2 v01 = fma2(ax, sx01, fma2(ay, add2(lo2(n), lo2(s)), fma2(az, add2(lo2(d), lo2(u)), fma2(bb, lo2(c), lo2(w)))));
    const float2 v23 = fma2(ax, sx23, fma2(ay, add2(hi2(n), hi2(s)), fma2(az, add2(hi2(d), hi2(u)), fma2(bb, hi2(c), hi2(w)))));
    return cat4(v01, v23);
}

__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
    unsigned long long d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(pk(a)), "l"(pk(b)));
    return upk(d);
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
    unsigned long long d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(pk(a)), "l"(pk(b)));
    return upk(d);
}

// One strip of stage 1: Lf = L Y0 - f, Y1 = c + mu~_1 tau Lf and the combined
// fields W_2 (and W_3 for s = 3), in packed FP32 pairs (cells 0, 1 and 2, 3 of
// the strip): a thread runs two strips of a row pair, so four independent
// pairs hide the latency of the chain Lf -> Y1 -> W_j.
template <int S, typename K>
__device__ __forceinline__ void first_strip(const K& k, float4 c, float4 n, float4 s, float4 d, float4 u,
                                            float l, float r, float4 f, float4& y1, float4& w2, float4& w3) {
    const float2 sx01 = make_float2(l + c.y, c.x + c.z), sx23 = make_float2(c.y + c.w, c.z + r);
    const float2 lf01 = sub2(fma2(k.ihx, sx01, fma2(k.ihy, add2(lo2(n), lo2(s)), fma2(k.ihz, add2(lo2(d), lo2(u)),
                                                                                    mul2(k.m2s, lo2(c))))), lo2(f));
    const float2 lf23 = sub2(fma2(k.ihx, sx23, fma2(k.ihy, add2(hi2(n), hi2(s)), fma2(k.ihz, add2(hi2(d), hi2(u)),
                                                                                    mul2(k.m2s, hi2(c))))), hi2(f));
    y1 = cat4(fma2(k.m1t, lf01, lo2(c)), fma2(k.m1t, lf23, hi2(c)));
    w2 = cat4(fma2(k.k2y0, lo2(c), fma2(k.k2z, lf01, mul2(k.k2f, lo2(f)))),
              fma2(k.k2y0, hi2(c), fma2(k.k2z, lf23, mul2(k.k2f, hi2(f)))));
    if (S == 3) {
        w3 = cat4(fma2(k.k3c, lo2(c), fma2(k.k3l, lf01, mul2(k.k3f, lo2(f)))),
                  fma2(k.k3c, hi2(c), fma2(k.k3l, lf23, mul2(k.k3f, hi2(f)))));
    } else {
        w3 = make_float4(0.f, 0.f, 0.f, 0.f);
    }
}

__device__ __forceinline__ float4 scale4(float k, float4 v) { return make_float4(k * v.x, k * v.y, k * v.z, k * v.w); }

__device__ __forceinline__ void store_out(float* dst, float4 v, bool vec, int n) {
    if (vec) {
        st4(dst, v);
    } else {
        dst[0] = v.x;
        if (n > 1) dst[1] = v.y;
        if (n > 2) dst[2] = v.z;
        if (n > 3) dst[3] = v.w;
    }
}

// The spacing of the FP32 numbers at x.
inline double spacing_f32(double x) { return x == 0.0 ? 0.0 : std::ldexp(1.0, std::ilogb(x) - 23); }

// FP32 coefficients a of the axes' neighbour sums, near a0, and b = m - 2 (ax + ay + az)
// of the cell itself (m: an FP32 number) without rounding: an error of b acts on the cell,
// one of ax on a second difference only.  The sum of the a is taken on the grid on which b
// is an FP32 number; the axis that the difference moves least takes it.
inline void sum_exact(double m, const double a0[3], float* a[3], float* b) {
    const double sum = a0[0] + a0[1] + a0[2];
    // (1 + 1e-6: also where rounding takes b past a power of two)
    const double q = 0.5 * std::max(spacing_f32(m), spacing_f32((m - 2.0 * sum) * (1.0 + 1e-6)));
    const double on_grid = q > 0.0 ? q * std::nearbyint(sum / q) : sum;
    for (int d = 0; d < 3; ++d) *a[d] = float(a0[d]);
    int best = -1;
    double best_v = 0.0, best_r = 0.0;
    for (int d = 0; d < 3; ++d) {
        const double v = on_grid - double(*a[(d + 1) % 3]) - double(*a[(d + 2) % 3]);
        const double r = std::fabs(v - a0[d]) / std::fabs(a0[d]);
        if (a0[d] == 0.0 || double(float(v)) != v || !(best < 0 || r < best_r)) continue;
        best = d;
        best_v = v;
        best_r = r;
    }
    if (best >= 0) *a[best] = float(best_v);
    *b = float(m - 2.0 * (double(*a[0]) + double(*a[1]) + double(*a[2])));
}

// The weights of the cell's own values add up without rounding too: b + 2 (ax + ay + az) =
// mu_j, and 1 - mu_j for Y0.  (All coefficients rounded one by one, a super-step of s = 3 of
// a smooth 30 x 62 x 46 field in cells of three widths was off by 2.0e-7; by 1.0e-7 so, as
// stage by stage.)
inline LeanCoef make_lean_coef(const LevelGeom& g, int order, int s, const FusedCoef& cf) {
    LeanCoef k{};
    const double hx = g.ihx2f, hy = g.ihy2f, hz = g.ihz2f;
    const double tau = cf.tau;
    double mu[4] = {};
    for (int j = 2; j <= s; ++j) {
        const double mt = cf.mut_tau[j];
        const double a0[3] = {mt * hx, mt * hy, mt * hz};
        const double b0 = double(cf.mu[j]) - 2.0 * (a0[0] + a0[1] + a0[2]);
        const double q = spacing_f32(b0 * (1.0 + 1e-6));
        mu[j] = q > 0.0 ? q * std::nearbyint(cf.mu[j] / q) : double(cf.mu[j]);
        float* a[3] = {&k.ax[j], &k.ay[j], &k.az[j]};
        sum_exact(mu[j], a0, a, &k.b[j]);
    }
    const double h0[3] = {hx, hy, hz};
    float* h[3] = {&k.ihx2, &k.ihy2, &k.ihz2};
    sum_exact(0.0, h0, h, &k.m2s);
    k.m1t = float(double(cf.mut1) * tau);
    const double gt_2 = order == 2 ? cf.gt[2] : 0.0;
    k.k2y0 = float(1.0 - mu[2]);                    // nu_2 + c0_2
    k.k2z = float(gt_2 * tau);
    k.k2f = float(-double(cf.mut_tau[2]));
    if (s >= 3) {
        const double gt_3 = order == 2 ? cf.gt[3] : 0.0;
        const double nu3 = cf.nu[3];
        k.k3c = float(1.0 - mu[3]);                 // nu_3 + c0_3
        k.k3l = float(nu3 * double(cf.mut1) * tau + gt_3 * tau);
        k.k3f = float(-double(cf.mut_tau[3]));
    }
    // Y0 = 0: Z0 = -tau f, Y1 = -mu~_1 tau f
    const double y1 = -double(cf.mut1) * tau;
    k.kz[1] = float(y1);
    const double kz2 = -gt_2 * tau - double(cf.mut_tau[2]);
    k.kz[2] = float(kz2);
    // Y2 = mu~_2 tau (hx sx + hy sy + hz sz) Y1 + b_2 Y1 + kz2 f with Y1 = y1 f
    {
        const double mt = cf.mut_tau[2];
        k.zx = float(mt * hx * y1);
        k.zy = float(mt * hy * y1);
        k.zz = float(mt * hz * y1);
        k.zb = float((double(cf.mu[2]) - 2.0 * mt * (hx + hy + hz)) * y1 + kz2);
    }
    if (s >= 3) {
        const double gt_3 = order == 2 ? cf.gt[3] : 0.0;
        k.kz[3] = float(double(cf.nu[3]) * y1 - gt_3 * tau - double(cf.mut_tau[3]));
    }
    return k;
}

}  // namespace

}  // namespace sg
