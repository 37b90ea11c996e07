// lattice_sites.cuh -- FP64 per-site helpers shared by the diagnostic passes
// over the current field (observables, volume render): site loads widened to
// double, first differences and the charge determinant.
#pragma once

#include "skyrme_device.cuh"

namespace skyrme {

// The exact FP64 value of an FP32 number, on the integer pipe: the conversion
// instruction runs on the FP64 pipe (16 cycles of an SM per warp), which
// bounds these passes, and a site needs 52 conversions.  Normal numbers are
// re-biased and shifted, zeros keep their sign, infinities and NaN their
// fraction; denormals are normalised.
__device__ __forceinline__ double widen(float f)
{
    const unsigned b = __float_as_uint(f), a = b & 0x7fffffffu;
    unsigned hi = (a >> 3) + (a >= 0x7f800000u ? 0x70000000u : 0x38000000u), lo = a << 29;
    if (a < 0x00800000u) {  // zero or denormal: a 2^-149
        const int s = __clz((int)a);  // 9 .. 31 (a != 0)
        const unsigned frac = a << (s + 1 & 31);
        hi = a ? ((unsigned)(31 - s - 149 + 1023) << 20) + (s == 31 ? 0u : frac >> 12) : 0u;
        lo = a && s != 31 ? frac << 20 : 0u;
    }
    return __hiloint2double((int)(hi | (b & 0x80000000u)), (int)lo);
}

__device__ __forceinline__ void load_site(const float4 *p, size_t i, double v[4])
{
    const float4 q = __ldg(p + i);
    v[0] = widen(q.x), v[1] = widen(q.y), v[2] = widen(q.z), v[3] = widen(q.w);
}
__device__ __forceinline__ void load_site(const dvec4 *p, size_t i, double v[4])
{
    const dvec4 q = load4<double>(p + i);
    v[0] = q.x, v[1] = q.y, v[2] = q.z, v[3] = q.w;
}

// First differences u[k][A] = 12h d_k phi^A (k = x, y, z) of the site at
// linear index c: 8 (p1 - m1) - (p2 - m2), the 4th-order central stencil
// without its 1/(12h), which the callers apply to their sums.
template <typename V>
__device__ __forceinline__ void site_first_differences(const V *phi, size_t c, size_t sx, size_t sy,
                                                       double u[3][4])
{
    const size_t st[3] = {sx, sy, 1};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        double m2v[4], m1v[4], p1v[4], p2v[4];
        load_site(phi, c - 2 * st[k], m2v);
        load_site(phi, c - st[k], m1v);
        load_site(phi, c + st[k], p1v);
        load_site(phi, c + 2 * st[k], p2v);
#pragma unroll
        for (int A = 0; A < 4; ++A) u[k][A] = ::fma(8.0, p1v[A] - m1v[A], m2v[A] - p2v[A]);
    }
}

// a b - c d, the product c d rounded
__device__ __forceinline__ double minor2(double a, double b, double c, double d)
{
    return ::fma(a, b, -(c * d));
}

// det[phi, u_x, u_y, u_z] by the 2x2 minors of its first and last two rows;
// the baryon density is -(12h)^-3 det / (2 pi^2).  Multiply-adds are written
// out: they are wanted in files compiled without contraction too.
__device__ __forceinline__ double charge_determinant(const double p[4], const double u[3][4])
{
    const double s0 = minor2(p[0], u[0][1], u[0][0], p[1]), s1 = minor2(p[0], u[0][2], u[0][0], p[2]);
    const double s2 = minor2(p[0], u[0][3], u[0][0], p[3]), s3 = minor2(p[1], u[0][2], u[0][1], p[2]);
    const double s4 = minor2(p[1], u[0][3], u[0][1], p[3]), s5 = minor2(p[2], u[0][3], u[0][2], p[3]);
    const double q5 = minor2(u[1][2], u[2][3], u[2][2], u[1][3]), q4 = minor2(u[1][1], u[2][3], u[2][1], u[1][3]);
    const double q3 = minor2(u[1][1], u[2][2], u[2][1], u[1][2]), q2 = minor2(u[1][0], u[2][3], u[2][0], u[1][3]);
    const double q1 = minor2(u[1][0], u[2][2], u[2][0], u[1][2]), q0 = minor2(u[1][0], u[2][1], u[2][0], u[1][1]);
    return ::fma(s5, q0, ::fma(-s4, q1, ::fma(s3, q2, ::fma(s2, q3, ::fma(-s1, q4, s0 * q5)))));
}

}  // namespace skyrme
