// init_fields.cu -- initial fields of Section 4 built on the device:
// rational-map Skyrmions (Section 4.1, Table 1 degrees 1 to 4), the product
// ansatz of isorotated 1-Skyrmions (Section 4.2, Eq. "Product ansatz",
// optionally symmetrised by renormalising U_1..U_K + U_K..U_1), and a
// smoothed-noise start (vacuum plus Gaussian-smoothed N(0,1) noise inside a
// ball, each component scaled to unit standard deviation over the ball).
//
// The noise uses the SplitMix64 generator (Steele, Lea and Flood 2014) in
// counter form with Box-Muller normals; the two velocity buffers serve as
// temporaries and are zeroed afterwards.
#include <cuda_runtime.h>
#include <math.h>

#include "lattice_sites.cuh"
#include "packed_f32.cuh"
#include "skyrme_device.cuh"
#include "skyrme_internal.h"

namespace skyrme {

constexpr int kMaxConstituents = 64;
constexpr int kMaxHalfWidth = 96;  // smoothing taps on each side

// One isorotated hedgehog of the product ansatz.  Conjugation by the
// orientation A rotates the vector part (the columns of `rot`) and multiplies
// the scalar part by |A|^2.
struct Constituent {
    double pos[3], rot[3][3], norm;
};
struct ProductArgs {
    int K;
    double scale, inv_scale;
    const double2 *table;  // the profile table (null: none), of intervals from `base`
    int base;
    Constituent c[kMaxConstituents];
};

struct SmoothArgs {
    int half;
    double w[2 * kMaxHalfWidth + 1];
};

__device__ __forceinline__ double coord(int i, int n, double h) { return ((double)i - 0.5 * (double)(n - 1)) * h; }

__device__ __forceinline__ bool interior(int x, int y, int z, int n0, int n1, int n2)
{
    return x >= 2 && x <= n0 - 3 && y >= 2 && y <= n1 - 3 && z >= 2 && z <= n2 - 3;
}

// (a0, a)(b0, b) = (a0 b0 - a.b, a0 b + b0 a - a x b) for U = a0 + i a.tau
__host__ __device__ __forceinline__ void su2_mul(const double a[4], const double b[4], double r[4])
{
    const double r0 = a[0] * b[0] - (a[1] * b[1] + a[2] * b[2] + a[3] * b[3]);
    const double r1 = a[0] * b[1] + b[0] * a[1] - (a[2] * b[3] - a[3] * b[2]);
    const double r2 = a[0] * b[2] + b[0] * a[2] - (a[3] * b[1] - a[1] * b[3]);
    const double r3 = a[0] * b[3] + b[0] * a[3] - (a[1] * b[2] - a[2] * b[1]);
    r[0] = r0; r[1] = r1; r[2] = r2; r[3] = r3;
}

template <typename T>
__device__ __forceinline__ void put(vec4_t<T> *p, const double v[4])
{
    store4<T>(p, make4<T>((T)v[0], (T)v[1], (T)v[2], (T)v[3]));
}

// Riemann-sphere direction of R(z) = P/Q in homogeneous form; z = Z1/Z0 with
// (Z1, Z0) = (x + i y, r + z3) for z3 >= 0 and the equivalent (r - z3, x - i y)
// otherwise.
__device__ void rm_direction(int B, double x, double y, double z3, double r, double nh[3])
{
    double z1r, z1i, z0r, z0i;
    if (z3 >= 0.0) { z1r = x; z1i = y; z0r = r + z3; z0i = 0.0; }
    else { z1r = r - z3; z1i = 0.0; z0r = x; z0i = -y; }
    double pr, pi, qr, qi;
    if (B == 1) { pr = z1r; pi = z1i; qr = z0r; qi = z0i; }
    else if (B == 2) {  // R = z^2
        pr = z1r * z1r - z1i * z1i; pi = 2 * z1r * z1i;
        qr = z0r * z0r - z0i * z0i; qi = 2 * z0r * z0i;
    } else if (B == 3) {
        // R = (sqrt3 i z^2 - 1) / (z (z^2 - sqrt3 i)):
        // P = z0 (sqrt3 i z1^2 - z0^2), Q = z1 (z1^2 - sqrt3 i z0^2)
        const double c = sqrt(3.0);
        const double a2r = z1r * z1r - z1i * z1i, a2i = 2 * z1r * z1i;
        const double b2r = z0r * z0r - z0i * z0i, b2i = 2 * z0r * z0i;
        const double ar = -c * a2i - b2r, ai = c * a2r - b2i;
        const double cr = a2r + c * b2i, ci = a2i - c * b2r;
        pr = z0r * ar - z0i * ai; pi = z0r * ai + z0i * ar;
        qr = z1r * cr - z1i * ci; qi = z1r * ci + z1i * cr;
    } else {
        // z1^2, z0^2, z1^4, z0^4, z1^2 z0^2
        const double a2r = z1r * z1r - z1i * z1i, a2i = 2 * z1r * z1i;
        const double b2r = z0r * z0r - z0i * z0i, b2i = 2 * z0r * z0i;
        const double a4r = a2r * a2r - a2i * a2i, a4i = 2 * a2r * a2i;
        const double b4r = b2r * b2r - b2i * b2i, b4i = 2 * b2r * b2i;
        const double mr = a2r * b2r - a2i * b2i, mi = a2r * b2i + a2i * b2r;
        const double k = 2.0 * sqrt(3.0);
        // P = z1^4 + i k z1^2 z0^2 + z0^4 ; Q = z1^4 - i k z1^2 z0^2 + z0^4
        pr = a4r - k * mi + b4r; pi = a4i + k * mr + b4i;
        qr = a4r + k * mi + b4r; qi = a4i - k * mr + b4i;
    }
    const double den = pr * pr + pi * pi + qr * qr + qi * qi;
    if (den == 0.0) { nh[0] = nh[1] = nh[2] = 0.0; return; }
    nh[0] = 2.0 * (pr * qr + pi * qi) / den;
    nh[1] = 2.0 * (pi * qr - pr * qi) / den;
    nh[2] = (qr * qr + qi * qi - pr * pr - pi * pi) / den;
}

template <typename T> __global__ void k_fill_vacuum(vec4_t<T> *phi, size_t total)
{
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total;
         i += (size_t)gridDim.x * blockDim.x)
        store4<T>(phi + i, make4<T>(T(1), T(0), T(0), T(0)));
}

template <typename T>
__global__ void k_seed_rm(vec4_t<T> *phi, int n0, int n1, int n2, double h, int B, double scale)
{
    const size_t total = (size_t)n0 * n1 * n2;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total;
         i += (size_t)gridDim.x * blockDim.x) {
        const int z = (int)(i % n2), y = (int)((i / n2) % n1), x = (int)(i / ((size_t)n2 * n1));
        const double cx = coord(x, n0, h), cy = coord(y, n1, h), cz = coord(z, n2, h);
        const double r = sqrt(cx * cx + cy * cy + cz * cz);
        const double f = M_PI * exp(-r / scale);
        double nh[3];
        rm_direction(B, cx, cy, cz, r, nh);
        const double sf = sin(f);
        const double v[4] = {cos(f), sf * nh[0], sf * nh[1], sf * nh[2]};
        put<T>(phi + i, v);
    }
}

// A hedgehog's profile as functions of q = r^2, with rho = r / scale:
//   C(q) = cos(pi exp(-rho)),  S(q) = sin(pi exp(-rho)) / r.
// Evaluated directly they take about 60 FP64 instructions (reciprocal square
// root, exponential, sine and cosine).  A large seed instead tabulates their
// Taylor polynomials of degree 10 on intervals of q, 32 to an octave (the
// upper bits of q are the interval), from q / scale^2 of about 2^-12 to 2^10;
// 21 instructions.  The offset from an interval's centre is at most 1/64 of q,
// so the truncation is below 1e-17 of the value for rho < 20 and 3e-15 of it
// at rho = 30, where the value is 1e-13.
constexpr int kProfileTerms = 11;
constexpr int kProfileIntervals = 22 * 32;
constexpr size_t kProfileTableBytes = (size_t)kProfileIntervals * kProfileTerms * sizeof(double2);

// First interval: of q = 2^(e - 12), e the exponent of scale^2.
static int profile_base(double scale) { return (ilogb(scale * scale) - 12 + 1023) * 32; }

// Taylor coefficients, to degree N - 1, of C and S about q (in powers of q' - q).
template <int N> __device__ __forceinline__ void profile_series(double q, double scale, double (&C)[N], double (&Q)[N])
{
    // rho to twice the precision, so that exp(-rho) is good to its own rounding
    const double is = 1.0 / scale, is_lo = ::fma(-is, scale, 1.0) * is;
    const double r = sqrt(q), r_lo = ::fma(-r, r, q) / (2.0 * r);
    const double a = r * is, a_lo = ::fma(r, is, -a) + ::fma(r, is_lo, r_lo * is);
    // series in tau = (q' - q) / q: b of sqrt(1 + tau), E of exp(-rho), S and C
    // of sine and cosine of f = pi E, Q of S / r
    double b[N], E[N], S[N];
    b[0] = 1.0;
    E[0] = exp(-a);
    E[0] -= E[0] * a_lo;
    sincospi(E[0], &S[0], &C[0]);
#pragma unroll
    for (int k = 1; k < N; ++k) {
        b[k] = b[k - 1] * (0.5 - (k - 1)) / k;
        double e = 0.0;
#pragma unroll
        for (int j = 1; j <= k; ++j) e -= j * (a * b[j]) * E[k - j];
        E[k] = e / k;
    }
#pragma unroll
    for (int k = 1; k < N; ++k) {
        double sk = 0.0, ck = 0.0;
#pragma unroll
        for (int j = 1; j <= k; ++j) {
            const double jf = j * M_PI * E[j];
            sk += jf * C[k - j];
            ck -= jf * S[k - j];
        }
        S[k] = sk / k;
        C[k] = ck / k;
    }
    double qk = 1.0;
#pragma unroll
    for (int k = 0; k < N; ++k) {
        double v = S[k] / r;
#pragma unroll
        for (int j = 1; j <= k; ++j) v -= b[j] * Q[k - j];
        Q[k] = v;
    }
#pragma unroll
    for (int k = 0; k < N; ++k) {
        C[k] *= qk;
        Q[k] *= qk;
        qk /= q;
    }
}

__global__ void k_profile_table(double2 *table, int base, double scale)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= kProfileIntervals) return;
    constexpr int N = kProfileTerms;
    double C[N], S[N];
    profile_series<N>(__hiloint2double(((base + i) << 15) | (1 << 14), 0), scale, C, S);  // the interval's centre
#pragma unroll
    for (int k = 0; k < N; ++k) table[i * N + k] = make_double2(C[k], S[k]);
}

// A scale whose reciprocal and products are far from the ends of the range.
static bool ordinary_scale(double scale) { return scale > 1e-100 && scale < 1e100; }

// C and S at q = r^2, directly.  inv_scale: 0 unless the scale is an ordinary one.
__device__ __forceinline__ void profile_direct(double q, double scale, double inv_scale, double &c, double &s)
{
    double inv, rho;
    // (the test is on the integer pipe: 2^-600 <= q < 2^600)
    if ((unsigned)__double2hiint(q) - 0x1a700000u < 0x4b000000u && inv_scale != 0.0) {
        inv = rsqrt(q);
        double r = q * inv;
        r = ::fma(0.5 * inv, ::fma(-r, r, q), r);
        rho = r * inv_scale;
        rho = ::fma(::fma(-rho, scale, r), inv_scale, rho);
    } else {  // r = 0, or a step of the above could overflow
        const double r = sqrt(q);
        inv = r > 0.0 ? 1.0 / r : 0.0;
        rho = r / scale;
    }
    sincospi(exp(-rho), &s, &c);
    s *= inv;
}

// The ansatz at one site in FP64.
template <bool SYM, bool TAB>
__device__ __forceinline__ void product_site(const ProductArgs &a, double cx, double cy, double cz, double out[4])
{
    // forward product U_1 U_2 ... U_K; the reverse product is
    // accumulated by left multiplication: U_K ... U_1
    double fwd[4], rev[4];
    for (int k = 0; k < a.K; ++k) {
        const Constituent &c = a.c[k];
        double dx = cx - c.pos[0], dy = cy - c.pos[1], dz = cz - c.pos[2];
        const double q = dx * dx + dy * dy + dz * dz;
        double cf, sf;
        const int j = (__double2hiint(q) >> 15) - a.base;
        if (TAB && j >= 0 && j < kProfileIntervals) {
            const double2 *t = a.table + j * kProfileTerms;
            const double d = q - __hiloint2double(((a.base + j) << 15) | (1 << 14), 0);
            double2 v = __ldg(t + kProfileTerms - 1);
            cf = v.x, sf = v.y;
#pragma unroll
            for (int m = kProfileTerms - 2; m >= 0; --m) {
                v = __ldg(t + m);
                cf = ::fma(cf, d, v.x);
                sf = ::fma(sf, d, v.y);
            }
        } else {
            profile_direct(q, a.scale, a.inv_scale, cf, sf);
            // r^2 overflows: sf = 0, and the rotation's sums may overflow too
            if (__double2hiint(q) == 0x7ff00000) dx = dy = dz = 0.0;
        }
        const double u[4] = {cf * c.norm, sf * (c.rot[0][0] * dx + c.rot[0][1] * dy + c.rot[0][2] * dz),
                             sf * (c.rot[1][0] * dx + c.rot[1][1] * dy + c.rot[1][2] * dz),
                             sf * (c.rot[2][0] * dx + c.rot[2][1] * dy + c.rot[2][2] * dz)};
        if (k == 0) {
#pragma unroll
            for (int m = 0; m < 4; ++m) fwd[m] = rev[m] = u[m];
        } else {
            su2_mul(fwd, u, fwd);
            if (SYM) su2_mul(u, rev, rev);
        }
    }
    if (SYM) {
        const double t[4] = {fwd[0] + rev[0], fwd[1] + rev[1], fwd[2] + rev[2], fwd[3] + rev[3]};
        const double n2s = t[0] * t[0] + t[1] * t[1] + t[2] * t[2] + t[3] * t[3];
        const bool small = n2s < 1e-24;
        const double rn = rsqrt(n2s);
#pragma unroll
        for (int m = 0; m < 4; ++m) out[m] = small ? fwd[m] : t[m] * rn;
    } else {
#pragma unroll
        for (int m = 0; m < 4; ++m) out[m] = fwd[m];
    }
}

// The product ansatz over the whole state: the field into both buffers, its
// outer layers the vacuum, zero velocities.
//
// Bound by the FP64 pipe (2 lanes per SM and cycle).  Per site and constituent
// it took 185 instructions with the conjugation as two SU(2) products, sine
// and cosine of pi exp(-r) apart, and four divisions.  The conjugation is now
// a 3x3 rotation and the profile comes from one reciprocal square root and one
// sincospi (no range reduction, and the product with pi is not rounded first),
// or from the table (TAB).
// 256^3, 8 constituents, symmetrised: 44.6 ms before, 25.4 with the direct
// profile (101 instructions), 17.6 with the table (74; 92% of the pipe).  Against
// 113-bit arithmetic the field's rms error fell from 2.0e-16 to 1.7e-16.
template <typename T, bool SYM, bool TAB>
__global__ void __launch_bounds__(256) k_seed_product(vec4_t<T> *phi0, vec4_t<T> *phi1, vec4_t<T> *vel0,
                                                      vec4_t<T> *vel1, int n0, int n1, int n2, double h,
                                                      const __grid_constant__ ProductArgs a)
{
    // Blocks take 256 sites in memory order, whatever the planes' size (a block to a
    // part of one plane left most lanes idle in small planes: 300 x 6 x 6 with 64
    // constituents 1740 us, now 525).  32-bit indices: fewer than 4e9 sites, and
    // 3e5 more in the last pass.
    const unsigned total = (unsigned)n0 * n1 * n2;
    for (unsigned s = blockIdx.x * 256 + threadIdx.x; s < total; s += gridDim.x * 256) {
        const unsigned row = s / (unsigned)n2;
        const int z = (int)(s - row * (unsigned)n2), x = (int)(row / (unsigned)n1), y = (int)(row - (unsigned)x * n1);
        double out[4] = {1.0, 0.0, 0.0, 0.0};
        if (interior(x, y, z, n0, n1, n2)) {
            const double cx = coord(x, n0, h), cy = coord(y, n1, h), cz = coord(z, n2, h);
            product_site<SYM, TAB>(a, cx, cy, cz, out);
        }
        put<T>(phi0 + s, out);
        put<T>(phi1 + s, out);
        const vec4_t<T> zero = make4<T>(T(0), T(0), T(0), T(0));
        store4<T>(vel0 + s, zero);
        store4<T>(vel1 + s, zero);
    }
}

// ---- the ansatz of a large FP32 state, in double-floats
//
// The field of an FP32 state is rounded to 24 bits at the end, and the FP32
// pipe issues 64 times the FP64 pipe's instructions.  k_seed_product_f32
// evaluates the ansatz in unevaluated sums hi + lo of two floats (error-free
// products by FMA, Knuth's and Dekker's sums), with a margin for the error beside
// it, and stores hi where no value within the margin rounds to another float.
// The margin is measured, not proven (kPairEps); should an error ever exceed it,
// the value stored is at most one ulp from the rounding of the exact one.  The
// sites where the margin does not decide (one in 150 with eight constituents),
// and those where a profile is outside the table, are collected per warp and
// evaluated in FP64, 32 at a time.
//
// Positions are in units of the profile's scale.  A warp takes 32 sites along
// z; the rotated offsets R_k (x - x_k) of its middle come from FP64 once per
// warp, a lane's own are off by (lane - 16) R_k e_z h.  The profile comes from
// a table of Taylor polynomials of degree 6 in q, 256 intervals to an octave
// (450 KB; the part in use lies in L1), the first three coefficients in
// double-floats: below 2^-46 of the value for rho < 16, 2^-42 up to 32.
// U_1 ... U_k and the conjugate of U_k ... U_1 are the two halves of the
// packed FP32 instructions: the second is the product of the conjugates.
//
// Bound by issue and the FP32 pipe (59% and 62% busy with 16 warps per SM; 336
// warp instructions per 32 sites and constituent, 240 of them FP32, most of those
// packed; 20 and 24 warps with fewer registers were 3% slower).  FP64 and
// double-float, symmetrised: 256^3 with 8 constituents 17.6 and 2.02 ms (2.35 with
// products and their rounding errors formed before they are summed), with one
// 2.07 and 0.51 ms (268 MB written four times: 0.16 ms); 151^3 with 4 constituents
// 1.84 and 0.30 ms; 128^3 with 64 constituents 17.5 and 2.8 ms.
constexpr int kPairOctaves = 22, kPairPerOctave = 256;  // q / scale^2 from 2^-12 to 2^10
constexpr int kPairIntervals = kPairOctaves * kPairPerOctave;
constexpr int kPairBase = (127 - 12) * kPairPerOctave;
constexpr int kPairVecs = 5;  // float4 per interval: (C, S) pairs hi, lo of degrees 0 to 2, then 3 to 6
constexpr size_t kPairTableBytes = (size_t)kPairIntervals * kPairVecs * sizeof(float4);
// The margins err[] below: a scalar component's error goes with the number of
// products and with the vector errors that each product hands it, a vector
// component's with P, the sum of the constituents' pion sizes; how these grow was
// taken from the arithmetic, their factors from comparisons with FP64.  Over
// lattice spacings of 0.001 to 2.7 scales (pairs_apply) and 1 to 64 constituents,
// spread out, in one place, alike and with one dominating, the largest error met
// was 0.20 of them (0.56 without the P^2 term, with 64 constituents at 0.02).
constexpr float kPairEps = 0x1p-40f, kPairCross = 1.f / 64;

__global__ void k_pair_table(float4 *table)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= kPairIntervals) return;
    constexpr int N = 7;
    double C[N], S[N];
    profile_series<N>((double)__int_as_float(((kPairBase + i) << 15) | (1 << 14)), 1.0, C, S);
    float4 *t = table + i * kPairVecs;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        // C itself passes through 0: its hi part is kept as 3 + hi, exactly
        const double off = k == 0 ? 3.0 : 0.0;
        const float c = (float)(C[k] + off), v = (float)S[k];
        t[k] = make_float4(c, v, (float)(C[k] - ((double)c - off)), (float)(S[k] - (double)v));
    }
    t[3] = make_float4((float)C[3], (float)S[3], (float)C[4], (float)S[4]);
    t[4] = make_float4((float)C[5], (float)S[5], (float)C[6], (float)S[6]);
}

// -x off the FP32 pipe
__device__ __forceinline__ float neg(float x) { return __int_as_float(__float_as_int(x) ^ (int)0x80000000); }
// (ch + cl) + (xh + xl)(d + dl), two quantities.  |ch| is above |xh d|, so that
// ch - (the rounded sum) is exact and the rounding error one more FMA.
__device__ __forceinline__ void horner(float2 ch, float2 cl, float2 &xh, float2 &xl, float2 d, float2 dl)
{
    const float2 s = __ffma2_rn(xh, d, ch);
    float2 e = __ffma2_rn(xh, d, __ffma2_rn(s, bc(-1.f), ch));
    e = __ffma2_rn(xl, d, e);
    e = __ffma2_rn(xh, dl, e);
    xl = __fadd2_rn(cl, e);
    xh = s;
}
// sum_j x_j y_j of pairs of double-floats.  The products are added to `shift`,
// above twice their partial sums: what a sum kept of a product is then exact in
// one subtraction, and what it dropped one more FMA.
struct Pairs4 {
    float2 h[4], l[4];
};
__device__ __forceinline__ void dot_pairs(const float2 (&xh)[4], const float2 (&xl)[4], const float2 (&y)[4],
                                          const float2 (&yl)[4], float2 shift, float2 &h, float2 &l)
{
    const float2 m1 = bc(-1.f);
    float2 s = shift, n;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float2 t = __ffma2_rn(xh[j], y[j], s);
        const float2 e = __ffma2_rn(xh[j], y[j], __ffma2_rn(t, m1, s));
        n = j == 0 ? e : __fadd2_rn(n, e);
        s = t;
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) n = __ffma2_rn(xl[j], y[j], __ffma2_rn(xh[j], yl[j], n));
    s = __ffma2_rn(shift, m1, s);
    h = __fadd2_rn(s, n);
    l = __ffma2_rn(__ffma2_rn(s, m1, h), m1, n);
}
// x y of two quantities' quaternions, y given with its negative
__device__ __forceinline__ void mul_pairs(Pairs4 &x, const Pairs4 &y, const Pairs4 &n, float2 shift0, float2 shift)
{
    Pairs4 r;
    const auto row = [&](int i, float2 y0, float2 y1, float2 y2, float2 y3, float2 l0, float2 l1, float2 l2, float2 l3) {
        const float2 yy[4] = {y0, y1, y2, y3}, ll[4] = {l0, l1, l2, l3};
        dot_pairs(x.h, x.l, yy, ll, i == 0 ? shift0 : shift, r.h[i], r.l[i]);
    };
    row(0, y.h[0], n.h[1], n.h[2], n.h[3], y.l[0], n.l[1], n.l[2], n.l[3]);
    row(1, y.h[1], y.h[0], n.h[3], y.h[2], y.l[1], y.l[0], n.l[3], y.l[2]);
    row(2, y.h[2], y.h[3], y.h[0], n.h[1], y.l[2], y.l[3], y.l[0], n.l[1]);
    row(3, y.h[3], n.h[2], y.h[1], y.h[0], y.l[3], n.l[2], y.l[1], y.l[0]);
    x = r;
}

// The ansatz at a lane's site: val[] its components hi + lo, err[] margins for
// their errors.  ob[3 k + i]: component i
// of the rotated offset of constituent k from the warp's middle (hi, lo) and
// its increment along z (hi, lo); zl: the lane's site from the middle.  False
// where a profile is outside the table.
template <bool SYM>
__device__ __forceinline__ bool product_pairs(const float4 *ob, int K, const float4 *__restrict__ table, float zl,
                                              float hs, DF (&val)[4], float (&err)[4])
{
    Pairs4 x;  // U_1 ... U_k and the conjugate of U_k ... U_1, which is conj(U_1) ... conj(U_k)
    float P = 0.f;
    for (int k = 0; k < K; ++k) {
        float ph[3], pl[3], qh = 0.f, ql = 0.f;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const float4 o = ob[3 * k + i];
            const float w = __fmul_rn(o.z, zl);
            const float we = __fmaf_rn(o.w, zl, __fmaf_rn(o.z, zl, -w));
            two_sum(o.x, w, ph[i], pl[i]);
            pl[i] = __fadd_rn(pl[i], __fadd_rn(o.y, we));
            const float t = __fmul_rn(ph[i], ph[i]);
            const float te = __fmaf_rn(__fadd_rn(pl[i], pl[i]), ph[i], __fmaf_rn(ph[i], ph[i], -t));
            if (i == 0) {
                qh = t, ql = te;
            } else {
                float e;
                two_sum(qh, t, qh, e);
                ql = __fadd_rn(ql, __fadd_rn(e, te));
            }
        }
        const DF q = quick_two_sum(qh, ql);
        const int bits = __float_as_int(q.hi), j = (bits >> 15) - kPairBase;
        if ((unsigned)j >= (unsigned)kPairIntervals) return false;
        const float4 *t = table + j * kPairVecs;
        const float4 t0 = __ldg(t), t1 = __ldg(t + 1), t2 = __ldg(t + 2), t3 = __ldg(t + 3), t4 = __ldg(t + 4);
        // q from the interval's centre (the subtraction is exact)
        const DF dq = quick_two_sum(__fsub_rn(q.hi, __int_as_float((bits & ~0x7fff) | 0x4000)), q.lo);
        const float2 d = bc(dq.hi), dl = bc(dq.lo);
        float2 xh = __ffma2_rn(make_float2(t4.z, t4.w), d, make_float2(t4.x, t4.y));
        xh = __ffma2_rn(xh, d, make_float2(t3.z, t3.w));
        xh = __ffma2_rn(xh, d, make_float2(t3.x, t3.y));
        float2 xl = __ffma2_rn(xh, d, make_float2(t2.z, t2.w));
        xh = make_float2(t2.x, t2.y);
        horner(make_float2(t1.x, t1.y), make_float2(t1.z, t1.w), xh, xl, d, dl);
        horner(make_float2(t0.x, t0.y), make_float2(t0.z, t0.w), xh, xl, d, dl);
        xh.x -= 3.f;
        // U_k and its conjugate
        Pairs4 y, n;
        y.h[0] = bc(xh.x), y.l[0] = bc(xl.x);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const float u = __fmul_rn(xh.y, ph[i]);
            const float ul = __fmaf_rn(xl.y, ph[i], __fmaf_rn(xh.y, pl[i], __fmaf_rn(xh.y, ph[i], -u)));
            y.h[i + 1] = make_float2(u, neg(u)), n.h[i + 1] = make_float2(neg(u), u);
            y.l[i + 1] = make_float2(ul, neg(ul)), n.l[i + 1] = make_float2(neg(ul), ul);
            P = __fadd_rn(P, fabsf(u));
        }
        P = __fmaf_rn(0.25f * hs, xh.y, P);  // the offsets' own rounding (they reach 16 sites from the lane's)
        if (k == 0) {
            x = y;
        } else {
            // the vector components' partial sums stay below 2 P, the scalar's below 1
            const float big = __int_as_float(((__float_as_int(P) & 0x7f800000) + (2 << 23)) | 0x400000);
            mul_pairs(x, y, n, bc(3.f), bc(big));
        }
    }
    // the scalar's margin grows with P^2 too: each product hands it the vector's error
    const float eps = kPairEps * __fmaf_rn(4.f, hs, 1.f), e0 = eps * (1.f + (float)K + kPairCross * P * P),
                e1 = eps * __fmaf_rn(0.0625f, (float)K, 1.f) * P;
    if (!SYM) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            val[i] = quick_two_sum(x.h[i].x, x.l[i].x);
            err[i] = i == 0 ? e0 : e1;
        }
        return true;
    }
    // t = U_1 ... U_K + U_K ... U_1, divided by its norm
    DF t[4], q = {0.f, 0.f};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float sg = i == 0 ? 1.f : -1.f;
        float s, e;
        two_sum(x.h[i].x, sg * x.h[i].y, s, e);
        t[i] = quick_two_sum(s, __fadd_rn(e, __fmaf_rn(sg, x.l[i].y, x.l[i].x)));
        q = df_add(q, df_mul(t[i], t[i]));
    }
    if (!(q.hi > 0x1p-20f)) return false;
    // 1 / sqrt(q): y0 and one step, q y0^2 = 1 - g
    const float y0 = rsqrtf(q.hi), a = __fmul_rn(y0, y0), ae = __fmaf_rn(y0, y0, -a);
    const float b = __fmul_rn(q.hi, a);
    const float be = __fmaf_rn(q.lo, a, __fmaf_rn(q.hi, ae, __fmaf_rn(q.hi, a, -b)));
    const float g = __fsub_rn(__fsub_rn(1.f, b), be);
    const DF y = {y0, __fmul_rn(__fmul_rn(y0, g), __fmaf_rn(0.375f, g, 0.5f))};
    // (2 y0 >= 1: |t| <= 2)  A component's error, and what the others' do to it through the norm
    const float y2 = 4.f * (y0 * y0);
#pragma unroll
    for (int i = 0; i < 4; ++i) val[i] = df_mul(t[i], y);
    const float v0 = fabsf(val[0].hi), vs = fabsf(val[1].hi) + fabsf(val[2].hi) + fabsf(val[3].hi);
    err[0] = y2 * __fmaf_rn(v0 * vs, e1, e0);
#pragma unroll
    for (int i = 1; i < 4; ++i) err[i] = y2 * __fmaf_rn(fabsf(val[i].hi), __fmaf_rn(vs, e1, v0 * e0), e1);
    return true;
}

// An integer as a double, by one FP64 addition.
__device__ __forceinline__ double to_double(int i)
{
    return __hiloint2double(0x43300000, i ^ (int)0x80000000) - (0x1p52 + 0x1p31);
}

// The sites the margin left open, in FP64.
template <bool SYM>
__device__ __noinline__ void product_open(const ProductArgs &a, float4 *phi0, float4 *phi1, unsigned s, int n0, int n1,
                                          int n2, double h)
{
    const unsigned row = s / (unsigned)n2;
    const int z = (int)(s - row * (unsigned)n2), y = (int)(row % (unsigned)n1), x = (int)(row / (unsigned)n1);
    double out[4];
    product_site<SYM, false>(a, coord(x, n0, h), coord(y, n1, h), coord(z, n2, h), out);
    put<float>(phi0 + s, out);
    put<float>(phi1 + s, out);
}

constexpr int kPairWarps = 8;
template <bool SYM>
__global__ void __launch_bounds__(32 * kPairWarps, 2)
    k_seed_product_f32(float4 *phi0, float4 *phi1, float4 *vel0, float4 *vel1, int n0, int n1, int n2, double h,
                       const __grid_constant__ ProductArgs a, const float4 *table, unsigned table_sites)
{
    __shared__ double s_row[3 * kMaxConstituents][4];  // change per half step in x, y, z; offset of the centre
    __shared__ float2 s_dz[3 * kMaxConstituents];      // change per step in z
    __shared__ float4 s_ob[kPairWarps][3 * kMaxConstituents];
    __shared__ unsigned s_open[kPairWarps][64];
    __shared__ int s_left[kPairWarps];
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32, K3 = 3 * a.K;
    const double hs = h * a.inv_scale;
    for (int i = threadIdx.x; i < K3; i += blockDim.x) {
        const Constituent &c = a.c[i / 3];
        const double *r = c.rot[i % 3];
        for (int j = 0; j < 3; ++j) s_row[i][j] = 0.5 * (r[j] * hs);
        const double dz = r[2] * hs;
        s_dz[i] = make_float2((float)dz, (float)(dz - (double)(float)dz));
        s_row[i][3] = -(r[0] * c.pos[0] + r[1] * c.pos[1] + r[2] * c.pos[2]) * a.inv_scale;
    }
    __syncthreads();
    const unsigned segs = ((unsigned)n2 + 31) / 32, items = (unsigned)n0 * n1 * segs;
    int open = 0;
    for (unsigned it = blockIdx.x * kPairWarps + warp; it < items; it += gridDim.x * kPairWarps) {
        // (the segments are rotated by a hash of the row, or a warp could get the same one,
        // with more or fewer open sites than the others', every time)
        const unsigned row = it / segs;
        const int zc = (int)((it - row * segs + (row * 0x9E3779B9u >> 16)) % segs) * 32 + 16, z = zc - 16 + lane;
        const int y = (int)(row % (unsigned)n1), x = (int)(row / (unsigned)n1);
        const unsigned s = row * (unsigned)n2 + z;
        float4 out = make_float4(1.f, 0.f, 0.f, 0.f);
        bool sure = true;
        if (x >= 2 && x <= n0 - 3 && y >= 2 && y <= n1 - 3) {
            const double xi = to_double(2 * x - (n0 - 1)), yi = to_double(2 * y - (n1 - 1)),
                         zi = to_double(2 * zc - (n2 - 1));
            for (int i = lane; i < K3; i += 32) {
                const double *r = s_row[i], o = ::fma(r[0], xi, ::fma(r[1], yi, ::fma(r[2], zi, r[3])));
                const float oh = (float)o;
                const float2 dz = s_dz[i];
                s_ob[warp][i] = make_float4(oh, (float)(o - widen(oh)), dz.x, dz.y);
            }
            __syncwarp();
            if (z >= 2 && z <= n2 - 3) {
                DF v[4];
                float err[4];
                sure = product_pairs<SYM>(s_ob[warp], a.K, table, (float)(lane - 16), (float)hs, v, err);
                if (sure) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        sure = sure && __fadd_rn(v[i].hi, __fadd_rn(v[i].lo, err[i])) == v[i].hi &&
                               __fadd_rn(v[i].hi, __fsub_rn(v[i].lo, err[i])) == v[i].hi;
                    }
                    out = make_float4(v[0].hi, v[1].hi, v[2].hi, v[3].hi);
                }
            }
            __syncwarp();
        }
        if (z < n2) {
            const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
            if (sure) {
                phi0[s] = out;
                phi1[s] = out;
            }
            vel0[s] = zero;
            if (s >= table_sites) vel1[s] = zero;  // (the table is in its first sites)
        }
        const unsigned m = __ballot_sync(0xffffffffu, !sure);
        if (m) {
            if (!sure) s_open[warp][open + __popc(m & ((1u << lane) - 1))] = s;
            open += __popc(m);
            __syncwarp();
            if (open >= 32) {
                open -= 32;
                product_open<SYM>(a, phi0, phi1, s_open[warp][open + lane], n0, n1, n2, h);
                __syncwarp();
            }
        }
    }
    // the sites left over, packed over the block's warps
    if (lane == 0) s_left[warp] = open;
    __syncthreads();
    int i = threadIdx.x, w = 0;
    while (w < kPairWarps && i >= s_left[w]) i -= s_left[w++];
    if (w < kPairWarps) product_open<SYM>(a, phi0, phi1, s_open[w][i], n0, n1, n2, h);
}

// ------------------------------------------------------------------ noise
__device__ __forceinline__ uint64_t splitmix64_at(uint64_t seed, uint64_t i)
{
    uint64_t z = seed + (i + 1ull) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

__device__ __forceinline__ double normal_at(uint64_t seed, uint64_t k)
{
    const double scale = 1.0 / 9007199254740992.0;  // 2^-53
    const double u1 = ((double)(splitmix64_at(seed, 2 * k) >> 11) + 1.0) * scale;
    const double u2 = (double)(splitmix64_at(seed, 2 * k + 1) >> 11) * scale;
    return sqrt(-2.0 * log(u1)) * cos(2.0 * M_PI * u2);
}

template <typename T>
__global__ void k_noise(vec4_t<T> *out, int n0, int n1, int n2, double h, double radius,
                        uint64_t seed)
{
    const size_t total = (size_t)n0 * n1 * n2;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total;
         i += (size_t)gridDim.x * blockDim.x) {
        const int z = (int)(i % n2), y = (int)((i / n2) % n1), x = (int)(i / ((size_t)n2 * n1));
        const double cx = coord(x, n0, h), cy = coord(y, n1, h), cz = coord(z, n2, h);
        double v[4] = {0, 0, 0, 0};
        if (cx * cx + cy * cy + cz * cz <= radius * radius)
            for (int c = 0; c < 4; ++c) v[c] = normal_at(seed, 4ull * i + (uint64_t)c);
        put<T>(out + i, v);
    }
}

// One separable Gaussian pass along `axis`; zero outside the lattice.
template <typename T>
__global__ void k_smooth(const vec4_t<T> *src, vec4_t<T> *dst, int n0, int n1, int n2, int axis,
                         SmoothArgs w)
{
    const size_t total = (size_t)n0 * n1 * n2;
    const int nax = axis == 0 ? n0 : (axis == 1 ? n1 : n2);
    const size_t stride = axis == 0 ? (size_t)n1 * n2 : (axis == 1 ? (size_t)n2 : 1);
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total;
         i += (size_t)gridDim.x * blockDim.x) {
        const int z = (int)(i % n2), y = (int)((i / n2) % n1), x = (int)(i / ((size_t)n2 * n1));
        const int c = axis == 0 ? x : (axis == 1 ? y : z);
        double acc[4] = {0, 0, 0, 0};
        for (int k = -w.half; k <= w.half; ++k) {
            const int cc = c + k;
            if (cc < 0 || cc >= nax) continue;
            const vec4_t<T> s = load4<T>(src + (size_t)((long long)i + (long long)k * (long long)stride));
            const double wk = w.w[k + w.half];
            acc[0] += wk * (double)s.x;
            acc[1] += wk * (double)s.y;
            acc[2] += wk * (double)s.z;
            acc[3] += wk * (double)s.w;
        }
        put<T>(dst + i, acc);
    }
}

// Moments over the ball: pass 0 sums the values (and the count), pass 1 the
// squared deviations from the mean.  Per-block partials, fixed-order finish.
template <typename T>
__global__ void k_ball_moments(const vec4_t<T> *src, int n0, int n1, int n2, double h,
                               double radius, int pass, double *parts, double *stats,
                               unsigned int *counter)
{
    const size_t total = (size_t)n0 * n1 * n2;
    double v[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    double mean[4] = {0, 0, 0, 0};
    if (pass == 1)
        for (int c = 0; c < 4; ++c) mean[c] = stats[c];
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total;
         i += (size_t)gridDim.x * blockDim.x) {
        const int z = (int)(i % n2), y = (int)((i / n2) % n1), x = (int)(i / ((size_t)n2 * n1));
        const double cx = coord(x, n0, h), cy = coord(y, n1, h), cz = coord(z, n2, h);
        if (cx * cx + cy * cy + cz * cz > radius * radius) continue;
        const vec4_t<T> s = load4<T>(src + i);
        const double a[4] = {(double)s.x, (double)s.y, (double)s.z, (double)s.w};
        for (int c = 0; c < 4; ++c) {
            const double d = a[c] - mean[c];
            v[c] += pass == 0 ? a[c] : d * d;
        }
        v[4] += 1.0;
    }
    __shared__ double red[8 * 8];
    __shared__ int s_last;
    double out[8];
    block_reduce<8, -1>(v, red, out);
    if (threadIdx.x == 0) {
        for (int q = 0; q < 8; ++q) parts[(size_t)blockIdx.x * 8 + q] = out[q];
        __threadfence();
        s_last = (atomicAdd(counter, 1u) == gridDim.x - 1);
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    if (threadIdx.x == 0) {
        double tot[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        for (unsigned int b = 0; b < gridDim.x; ++b)
            for (int q = 0; q < 8; ++q) tot[q] += __ldcg(parts + (size_t)b * 8 + q);
        const double cnt = tot[4];
        for (int c = 0; c < 4; ++c) {
            if (pass == 0) stats[c] = cnt > 0 ? tot[c] / cnt : 0.0;
            else stats[4 + c] = cnt > 0 ? sqrt(tot[c] / cnt) : 0.0;
        }
        *counter = 0;
    }
}

template <typename T>
__global__ void k_noise_finish(vec4_t<T> *phi, const vec4_t<T> *noise, size_t total,
                               const double *stats)
{
    double sd[4];
    for (int c = 0; c < 4; ++c) sd[c] = stats[4 + c] > 0.0 ? stats[4 + c] : 1.0;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total;
         i += (size_t)gridDim.x * blockDim.x) {
        const vec4_t<T> s = load4<T>(noise + i);
        const double t[4] = {1.0 + (double)s.x / sd[0], (double)s.y / sd[1], (double)s.z / sd[2],
                             (double)s.w / sd[3]};
        const double nrm = sqrt(t[0] * t[0] + t[1] * t[1] + t[2] * t[2] + t[3] * t[3]);
        double o[4] = {1, 0, 0, 0};
        if (nrm >= 1e-12)
            for (int c = 0; c < 4; ++c) o[c] = t[c] / nrm;
        put<T>(phi + i, o);
    }
}

static int grid_for(size_t total)
{
    size_t b = (total + 255) / 256;
    if (b > 152 * 8) b = 152 * 8;
    return (int)(b < 1 ? 1 : b);
}

// Whether the double-float kernel takes the ansatz: unit orientations, rows that
// fill a warp, 32-bit indices, a spacing at which the error was measured (coarser
// ones than 2.7 scales fail the last condition), offsets small enough for their
// rounding, and a lattice that lies largely inside the table (32 scales from a constituent):
// outside, the attempt costs 7% on top of the FP64 evaluation.  At 128^3 with 4
// constituents, FP64 and double-float: 1.69 and 1.82 ms with nearly every site
// outside, 1.73 and 1.74 ms with a box of +-64 scales (the estimate is then 0.08).
static bool pairs_apply(const skyrme_lattice &lat, const ProductArgs &pa)
{
    const double total = (double)lat.n[0] * lat.n[1] * lat.n[2];
    if (pa.inv_scale == 0.0 || lat.n[2] < 24 || total >= 4.2e9 || total * sizeof(float4) < (double)kPairTableBytes) return false;
    const double hs = lat.h * pa.inv_scale;
    if (!(hs >= 0.001 && hs <= 2.75)) return false;
    double inside = 1.0;
    for (int j = 0; j < 3; ++j) {
        double reach = 0.0;
        for (int k = 0; k < pa.K; ++k) reach = fmax(reach, fabs(pa.c[k].pos[j]));
        reach = (reach + 0.5 * lat.n[j] * lat.h) * pa.inv_scale;
        if (!(reach <= 256.0)) return false;
        inside *= fmin(1.0, 28.0 / reach);
    }
    for (int k = 0; k < pa.K; ++k)
        if (!(fabs(pa.c[k].norm - 1.0) <= 0x1p-48)) return false;
    return inside >= 0.3;
}

static cudaError_t launch_product_f32(const skyrme_lattice &lat, const ProductArgs &pa, bool sym, const FlowArgs &a,
                                      cudaStream_t s)
{
    // the table lies in the first sites of the second velocity buffer, which
    // are zeroed afterwards
    float4 *phi0 = static_cast<float4 *>(a.phi[0]), *phi1 = static_cast<float4 *>(a.phi[1]);
    float4 *v0 = static_cast<float4 *>(a.vel[0]), *v1 = static_cast<float4 *>(a.vel[1]);
    k_pair_table<<<(kPairIntervals + 31) / 32, 32, 0, s>>>(v1);
    auto kernel = sym ? k_seed_product_f32<true> : k_seed_product_f32<false>;
    kernel<<<2 * 152, 32 * kPairWarps, 0, s>>>(phi0, phi1, v0, v1, lat.n[0], lat.n[1], lat.n[2], lat.h, pa, v1,
                                               (unsigned)(kPairTableBytes / sizeof(float4)));
    const cudaError_t e = cudaMemsetAsync(v1, 0, kPairTableBytes, s);
    return e != cudaSuccess ? e : cudaGetLastError();
}

template <typename T>
static cudaError_t seed_impl(const skyrme_lattice &lat, const skyrme_seed &sd, const FlowArgs &a,
                             size_t scratch_bytes, cudaStream_t s)
{
    vec4_t<T> *phi0 = static_cast<vec4_t<T> *>(a.phi[0]);
    const int n0 = lat.n[0], n1 = lat.n[1], n2 = lat.n[2];
    const size_t total = (size_t)n0 * n1 * n2;
    const int g = grid_for(total);
    switch (sd.kind) {
    case SKYRME_SEED_VACUUM:
        k_fill_vacuum<T><<<g, 256, 0, s>>>(phi0, total);
        break;
    case SKYRME_SEED_RATIONAL_MAP:
        k_seed_rm<T><<<g, 256, 0, s>>>(phi0, n0, n1, n2, lat.h, sd.B, sd.profile_scale);
        break;
    case SKYRME_SEED_PRODUCT: {
        ProductArgs pa;
        pa.K = sd.B;
        pa.scale = sd.profile_scale;
        pa.inv_scale = ordinary_scale(sd.profile_scale) ? 1.0 / sd.profile_scale : 0.0;
        pa.table = nullptr;
        pa.base = 0;
        for (int k = 0; k < sd.B; ++k) {
            Constituent &c = pa.c[k];
            const double *q = sd.quaternions + 4 * k;
            const double A[4] = {q[0], q[1], q[2], q[3]}, Ad[4] = {q[0], -q[1], -q[2], -q[3]};
            double t[4], r[4];
            for (int j = 0; j < 3; ++j) {  // A (0, e_j) A^dagger
                c.pos[j] = sd.positions[3 * k + j];
                const double e[4] = {0.0, j == 0 ? 1.0 : 0.0, j == 1 ? 1.0 : 0.0, j == 2 ? 1.0 : 0.0};
                su2_mul(A, e, t);
                su2_mul(t, Ad, r);
                for (int i = 0; i < 3; ++i) c.rot[i][j] = r[i + 1];
            }
            su2_mul(A, Ad, r);
            c.norm = r[0];
        }
        // The double-float kernel takes 60 us at least (its table, the FP64
        // remainder): 64^3 with one constituent 66 us against 79, 32^3 with eight
        // 91 against 93, 50^3 with one 60 against 60.
        const double work = (double)total * sd.B;
        if (sizeof(T) == 4 && work >= 2.5e5 && pairs_apply(lat, pa)) return launch_product_f32(lat, pa, sd.symmetrise, a, s);
        // The table costs a launch of 26 us and saves 30 instructions per site
        // and constituent (48 us per million of them); it needs the scratch
        // behind the control block and an ordinary scale.
        if (work >= 1e6 && scratch_bytes >= kProfileTableBytes && ordinary_scale(sd.profile_scale)) {
            pa.base = profile_base(sd.profile_scale);
            double2 *table = reinterpret_cast<double2 *>(a.step_parts);
            k_profile_table<<<(kProfileIntervals + 31) / 32, 32, 0, s>>>(table, pa.base, pa.scale);
            pa.table = table;
        }
        vec4_t<T> *phi1 = static_cast<vec4_t<T> *>(a.phi[1]);
        vec4_t<T> *v0 = static_cast<vec4_t<T> *>(a.vel[0]), *v1 = static_cast<vec4_t<T> *>(a.vel[1]);
        auto kernel = pa.table ? (sd.symmetrise ? k_seed_product<T, true, true> : k_seed_product<T, false, true>)
                               : (sd.symmetrise ? k_seed_product<T, true, false> : k_seed_product<T, false, false>);
        kernel<<<g, 256, 0, s>>>(phi0, phi1, v0, v1, n0, n1, n2, lat.h, pa);
        break;
    }
    case SKYRME_SEED_NOISE: {
        vec4_t<T> *t0 = static_cast<vec4_t<T> *>(a.vel[0]);
        vec4_t<T> *t1 = static_cast<vec4_t<T> *>(a.vel[1]);
        SmoothArgs w;
        w.half = (int)ceil(4.0 * sd.sigma / lat.h);
        double wsum = 0.0;
        for (int k = -w.half; k <= w.half; ++k) {
            w.w[k + w.half] = exp(-(k * lat.h) * (k * lat.h) / (2.0 * sd.sigma * sd.sigma));
            wsum += w.w[k + w.half];
        }
        for (int k = 0; k <= 2 * w.half; ++k) w.w[k] /= wsum;
        k_noise<T><<<g, 256, 0, s>>>(t0, n0, n1, n2, lat.h, sd.radius, sd.seed);
        k_smooth<T><<<g, 256, 0, s>>>(t0, t1, n0, n1, n2, 0, w);
        k_smooth<T><<<g, 256, 0, s>>>(t1, t0, n0, n1, n2, 1, w);
        k_smooth<T><<<g, 256, 0, s>>>(t0, t1, n0, n1, n2, 2, w);
        Ctrl *c = static_cast<Ctrl *>(a.ctrl);
        double *stats = c->energy;  // 8 doubles: mean[4], sd[4]
        unsigned int *ctr = &c->edone;
        k_ball_moments<T><<<g, 256, 0, s>>>(t1, n0, n1, n2, lat.h, sd.radius, 0, a.energy_parts,
                                            stats, ctr);
        k_ball_moments<T><<<g, 256, 0, s>>>(t1, n0, n1, n2, lat.h, sd.radius, 1, a.energy_parts,
                                            stats, ctr);
        k_noise_finish<T><<<g, 256, 0, s>>>(phi0, t1, total, stats);
        break;
    }
    default:
        return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_seed(const skyrme_lattice &lat, const skyrme_seed &seed, const FlowArgs &a,
                        cudaStream_t s)
{
    const ScratchLayout L = scratch_layout(lat);
    const size_t bytes = L.total - L.step_off;  // both record regions, one behind the other
    if (lat.precision == 64) return seed_impl<double>(lat, seed, a, bytes, s);
    return seed_impl<float>(lat, seed, a, bytes, s);
}

int max_constituents() { return kMaxConstituents; }
int max_smoothing_half_width() { return kMaxHalfWidth; }

}  // namespace skyrme
