// render.cu -- headless volume render of the baryon density (Section 6.2,
// ray tracing).  The picture goes to a caller-owned device RGBA buffer in
// place of a GL pixel buffer.
//
//   1. k_render_volume: one FP64 record per site, {B0, pion / |pion|}, in the
//      caller's volume buffer.  B0 uses the flow's lattice derivatives at
//      interior sites and is 0 on the boundary layers.  Max B0 is an atomic
//      max on the bit pattern, since positive doubles order like their bits.
//   2. k_render_normalise: B0 / max B0, or 0 everywhere when max B0 <= 0; for
//      a whole render it also marks the bricks of sites that reach the level
//      set.
//   3. k_render_rays: one thread per pixel.
//      - A perspective ray crosses the lattice box in fixed steps.
//      - Each step takes trilinear samples of all four components.
//      - The transfer input is (b - levelset) scale; negative inputs are
//        skipped.
//      - The colour is input^2 (pion, 1/input).
//      - Compositing is front to back and stops once alpha exceeds 0.95.
//      - The result is multiplied by brightness and clamped to [0, 1].
// The ray arithmetic is FP64, compiled without multiply-add contraction.
// That way the skip and stop decisions round the same way as a plain C
// restatement compiled with contraction off.  Only the output is FP32.
//
// All three kernels are bound by the FP64 pipe (2 lanes per SM and cycle), so
// what they save is FP64 instructions:
//   - the field is widened on the integer pipe (load_site) and the density
//     takes first differences with explicit multiply-adds;
//   - the three divisions by |pion| share one reciprocal (divide_by below);
//   - most samples of a picture lie where B0 is below the level set and count
//     for nothing.  The ray finds the next sample that may count in FP32 and
//     on the integer pipe, by tests that leave no doubt (k_render_rays), and
//     only those samples take the FP64 arithmetic, which is that of the plain
//     march, operation for operation.
// Measured on a 128^3 FP32 field, 1024 x 768 pixels, step 0.005 (before ->
// now): volume 886 -> 400 us (98 FP64 instructions per site, 88% of the pipe),
// normalisation 65 -> 35, rays 17000 -> 165.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>

#include "lattice_sites.cuh"
#include "skyrme_device.cuh"
#include "skyrme_internal.h"

namespace skyrme {

constexpr double kRenderEye = 4.0;     // eye on the view-space z axis
constexpr double kRenderFocal = 2.0;   // image plane distance (vertical half-extent 1)
constexpr double kRenderAlphaStop = 0.95;
constexpr size_t kBrickOffset = 256;  // scratch: max B0 first, the brick tables here

// The correctly rounded quotient a / b from r, the correctly rounded 1 / b
// (Markstein, IBM J. Res. Dev. 34 (1990) 111): the first correction brings the
// quotient within one unit in the last place, from which the second rounds
// correctly.  5 operations instead of a division's.  The theorem needs exact
// residuals a - q b and normal operands, so values near the ends of the range
// take the division.  b > 0.
__device__ __forceinline__ double divide_by(double a, double b, double r)
{
    const unsigned m = (unsigned)__double2hiint(a) & 0x7fffffffu;
    if ((m | (unsigned)__double2loint(a)) == 0u) return a;  // a zero keeps its sign
    if (m - 0x20000000u >= 0x3fe00000u) return a / b;       // |a| outside 2^-511 .. 2^511
    double q = __dmul_rn(a, r);
    q = ::fma(::fma(-q, b, a), r, q);
    return ::fma(::fma(-q, b, a), r, q);
}
// whether 1/b and the quotients are far from the ends of the range
__device__ __forceinline__ bool divisor_in_range(double b)
{
    const unsigned e = (unsigned)__double2hiint(b) & 0x7ff00000u;
    return e - 0x30000000u < 0x20000000u;  // 2^-255 <= b < 2^257
}

// Bricks of S = 2^shift sites per axis, a bit each.  A bit is set when a site
// that a sample in the brick, or up to one cell beside it, interpolates may
// reach the level set (or is not finite): sites S j - 1 .. S j + S + 1 for
// brick j.
struct Bricks {
    unsigned *bits;  // null: none
    int shift;
    int nb[3];
    __device__ __forceinline__ int index(int bx, int by, int bz) const { return (bx * nb[1] + by) * nb[2] + bz; }
};
// Two levels: coarse bricks carry a ray through empty space, fine ones close
// to the surface, where testing a cell costs eight gathers.
struct BrickLevels {
    Bricks fine, coarse;
};

// Mark every brick that lists site c.
__device__ __forceinline__ void mark_bricks(const Bricks &br, const int (&c)[3])
{
    int j0[3], j1[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        j0[a] = max(c[a] - 2, 0) >> br.shift;
        j1[a] = min((c[a] + 1) >> br.shift, br.nb[a] - 1);
    }
    for (int jx = j0[0]; jx <= j1[0]; ++jx)
        for (int jy = j0[1]; jy <= j1[1]; ++jy)
            for (int jz = j0[2]; jz <= j1[2]; ++jz) {
                const int i = br.index(jx, jy, jz);
                const unsigned m = 1u << (i & 31);
                // most neighbours find the bit set already
                if (!(__ldcg(br.bits + (i >> 5)) & m)) atomicOr(br.bits + (i >> 5), m);
            }
}

// Whether the brick that holds lattice coordinates g is empty; then e is the
// distance to its nearest far face along the ray (in the unit that gives g
// the slope gd per unit, igd = |1 / gd|).
__device__ __forceinline__ bool empty_brick(const Bricks &br, const float (&g)[3], const float (&gd)[3],
                                            const float (&igd)[3], float &e)
{
    int b[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) b[a] = min(max((int)floorf(g[a]) >> br.shift, 0), br.nb[a] - 1);
    const int i = br.index(b[0], b[1], b[2]);
    if ((br.bits[i >> 5] >> (i & 31)) & 1u) return false;
    e = 1e30f;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float face = (float)((b[a] + (gd[a] > 0.0f ? 1 : 0)) << br.shift);
        e = fminf(e, (gd[a] > 0.0f ? face - g[a] : g[a] - face) * igd[a]);
    }
    return true;
}

template <typename V>
__global__ void __launch_bounds__(256) k_render_volume(const V *phi0, const V *phi1, const Ctrl *ctrl,
                                                       int n0, int n1, int n2, double bscale,
                                                       dvec4 *vol, unsigned long long *bmax_bits)
{
    const V *phi = __ldcg(&ctrl->cur) ? phi1 : phi0;
    const unsigned plane = (unsigned)n1 * n2;
    const size_t sx = plane, sy = (size_t)n2;
    const unsigned pblocks = (plane + 255) / 256, items = pblocks * n0;
    double local_max = 0.0;
    for (unsigned it = blockIdx.x; it < items; it += gridDim.x) {
        const unsigned x = it / pblocks, i = (it - x * pblocks) * 256 + threadIdx.x;
        if (i >= plane) continue;
        const int y = (int)(i / (unsigned)n2), z = (int)(i - (unsigned)y * n2);
        const size_t s = (size_t)x * sx + i;
        double ph[4];
        load_site(phi, s, ph);
        double b = 0.0;
        if ((int)x >= 2 && (int)x <= n0 - 3 && y >= 2 && y <= n1 - 3 && z >= 2 && z <= n2 - 3) {
            double u[3][4];
            site_first_differences(phi, s, sx, sy, u);
            b = bscale * charge_determinant(ph, u);
        }
        const double np = sqrt(ph[1] * ph[1] + ph[2] * ph[2] + ph[3] * ph[3]);
        dvec4 out;
        out.x = b;
        if (divisor_in_range(np)) {
            const double r = 1.0 / np;
            out.y = divide_by(ph[1], np, r);
            out.z = divide_by(ph[2], np, r);
            out.w = divide_by(ph[3], np, r);
        } else if (np > 0.0) {
            out.y = ph[1] / np;
            out.z = ph[2] / np;
            out.w = ph[3] / np;
        } else {
            out.y = out.z = out.w = 0.0;
        }
        store4<double>(vol + s, out);
        local_max = fmax(local_max, b);
    }
    for (int o = 16; o > 0; o >>= 1) local_max = fmax(local_max, __shfl_xor_sync(0xffffffffu, local_max, o));
    if ((threadIdx.x & 31) == 0 && local_max > 0.0)
        atomicMax(bmax_bits, (unsigned long long)__double_as_longlong(local_max));
}

// The order of doubles against a positive threshold's high word: a value whose
// key is below the threshold's key is finite and below the threshold.  (Not
// finite, either sign: the largest key.)
__device__ __forceinline__ int density_key(double v)
{
    const int hi = __double2hiint(v);
    return ((unsigned)hi & 0x7ff00000u) == 0x7ff00000u ? 0x7fffffff : hi;
}

// threshold_key: of a value just below the level set (see launch_render_rays)
__global__ void __launch_bounds__(256) k_render_normalise(dvec4 *vol, int n0, int n1, int n2,
                                                          const unsigned long long *bmax_bits,
                                                          BrickLevels br, int threshold_key)
{
    const double bmax = __longlong_as_double((long long)*bmax_bits);
    const bool share = divisor_in_range(bmax);
    const double r = share ? 1.0 / bmax : 0.0;
    const unsigned plane = (unsigned)n1 * n2, pblocks = (plane + 255) / 256, items = pblocks * n0;
    for (unsigned it = blockIdx.x; it < items; it += gridDim.x) {
        const unsigned x = it / pblocks, i = (it - x * pblocks) * 256 + threadIdx.x;
        if (i >= plane) continue;
        dvec4 *v = vol + (size_t)x * plane + i;
        const double b = v->x;
        const double q = share ? divide_by(b, bmax, r) : (bmax > 0.0 ? b / bmax : 0.0);
        v->x = q;
        if (br.fine.bits && density_key(q) >= threshold_key) {
            const int y = (int)(i / (unsigned)n2), z = (int)(i - (unsigned)y * n2);
            const int c[3] = {(int)x, y, z};
            mark_bricks(br.fine, c);
            mark_bricks(br.coarse, c);
        }
    }
}

struct RayParams {
    int width, height;
    int n[3];
    int max_samples;  // per ray, a bound the valid parameters never reach
    double view[9];
    // the same for every pixel (FP64 once on the host, and FP32 copies)
    double aspect, half[3], s, box[3], eye[3];  // box[i] = half[i] / s, eye in box space
    float viewf[9], aspectf, halff[3], sf, boxf[3], eyef[3];
    float miss;         // every channel of a pixel without a sample
    double levelset, scale, brightness, step;
    int threshold_key;  // density_key of a value just below the level set
    float threshold;    // the same value, rounded down
    BrickLevels bricks;
};

// Cell and offsets of lattice coordinates g, clamped to the lattice.
__device__ __forceinline__ void cell_of(const int n[3], const double g[3], int i0[3], double w[3])
{
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const double t = fmin(fmax(g[a], 0.0), (double)(n[a] - 1));
        i0[a] = min((int)floor(t), n[a] - 2);
        w[a] = t - (double)i0[a];
    }
}

// A ray's sample positions t_0 = t_near, t_{k+1} = fl(t_k + step).  Within one
// binade of t the rounded sum adds the same multiple `inc` of t's ulp every
// time (t is a multiple of the ulp, so the rounding of t + step depends on
// step alone, unless it is a tie), and t + j inc is exact: j steps at once.
struct RayClock {
    double t, inc, top;  // top: the end of t's binade
    int k;               // t = t_k
    bool jump;
    __device__ __forceinline__ void binade(double step)
    {
        const int hi = __double2hiint(t) & 0x7ff00000;
        top = __hiloint2double(hi + 0x00100000, 0);
        inc = (t + step) - t;
        const double half_ulp = __hiloint2double(hi - (53 << 20), 0);
        jump = hi >= (64 << 20) && hi < 0x7fd00000 && fabs(step - inc) != half_ulp;
    }
    __device__ __forceinline__ void advance(int to, double step, float inv_step)
    {
        while (k < to) {
            if (jump) {
                // steps that stay below top by at least one step (FP32 with margin)
                const int room = (int)((float)(top - t) * inv_step * 0.99999f) - 2;
                const int j = min(to - k, room);
                if (j > 0) {
                    t += (double)j * inc;
                    k += j;
                    continue;
                }
            }
            t += step;
            ++k;
            if (t >= top) binade(step);
        }
    }
};

// FP32 value of a double from its high word, truncated to 20 fraction bits
// (relative error below 1e-6); 0 below the FP32 range, infinity above.
__device__ __forceinline__ float high_word_value(int hi)
{
    const unsigned a = (unsigned)hi & 0x7fffffffu;
    const unsigned m = a < 0x38100000u ? 0u : a >= 0x47f00000u ? 0x7f800000u : (a - 0x38000000u) << 3;
    return __uint_as_float(m | ((unsigned)hi & 0x80000000u));
}

// The ray of pixel (ix, iy) in box space: unit direction d and the interval of
// t inside the box (tnear > tfar: none).
__device__ __forceinline__ void pixel_ray(const RayParams &rp, int ix, int iy, double (&d)[3],
                                          double &tnear, double &tfar)
{
    double dv[3] = {(2.0 * (ix + 0.5) / rp.width - 1.0) * rp.aspect, 2.0 * (iy + 0.5) / rp.height - 1.0,
                    -kRenderFocal};
    const double nd = sqrt(dv[0] * dv[0] + dv[1] * dv[1] + dv[2] * dv[2]);
#pragma unroll
    for (int i = 0; i < 3; ++i) dv[i] /= nd;
    // view space -> box space through the row-major rotation
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        d[i] = 0.0;
#pragma unroll
        for (int j = 0; j < 3; ++j) d[i] += rp.view[3 * i + j] * dv[j];
    }
    // slab intersection with |p_i| <= half_i / s
    tnear = -1e300, tfar = 1e300;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const double b = rp.box[i], o = rp.eye[i];
        if (d[i] != 0.0) {
            double t0 = (-b - o) / d[i], t1 = (b - o) / d[i];
            if (t0 > t1) {
                const double tmp = t0;
                t0 = t1;
                t1 = tmp;
            }
            if (t0 > tnear) tnear = t0;
            if (t1 < tfar) tfar = t1;
        } else if (o < -b || o > b) {
            tnear = 1.0;
            tfar = 0.0;
        }
    }
    if (tnear < 0.0) tnear = 0.0;
}

// One sample of the march at t: false when its input is negative; else its
// colour.  `inside`: the cell i0 is known and no clamp applies.
__device__ __forceinline__ bool ray_sample(const RayParams &rp, const dvec4 *__restrict__ vol,
                                           const double (&d)[3], double t, bool inside, int (&i0)[3],
                                           double (&col)[4])
{
    const size_t sy = rp.n[2], sx = (size_t)rp.n[1] * rp.n[2];
    double g[3], w[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) g[i] = (rp.eye[i] + t * d[i]) * rp.s + rp.half[i];
    if (inside) {
#pragma unroll
        for (int a = 0; a < 3; ++a) w[a] = g[a] - (double)i0[a];
    } else {
        cell_of(rp.n, g, i0, w);
    }
    const dvec4 *c0 = vol + ((size_t)i0[0] * sx + (size_t)i0[1] * sy + i0[2]);
    const double x0 = 1.0 - w[0], y0 = 1.0 - w[1], z0 = 1.0 - w[2];
    const double xy[4] = {x0 * y0, w[0] * y0, x0 * w[1], w[0] * w[1]};
    double wt[8], smp[4];
    smp[0] = 0.0;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        wt[c] = xy[c & 3] * ((c & 4) ? w[2] : z0);
        smp[0] += wt[c] * __ldg(&c0[((c & 1) ? sx : 0) + ((c & 2) ? sy : 0) + ((c & 4) ? 1 : 0)].x);
    }
    const double input = (smp[0] - rp.levelset) * rp.scale;
    if (input < 0.0) return false;
    smp[1] = smp[2] = smp[3] = 0.0;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const dvec4 *q = c0 + ((c & 1) ? sx : 0) + ((c & 2) ? sy : 0) + ((c & 4) ? 1 : 0);
        const double2 zw = __ldg(reinterpret_cast<const double2 *>(&q->z));
        smp[1] += wt[c] * __ldg(&q->y);
        smp[2] += wt[c] * zw.x;
        smp[3] += wt[c] * zw.y;
    }
    col[0] = input * input * smp[1];
    col[1] = input * input * smp[2];
    col[2] = input * input * smp[3];
    col[3] = input;
    return true;
}

__device__ __forceinline__ float pixel_value(double sum, double brightness)
{
    double v = sum * brightness;
    v = v < 0.0 ? 0.0 : (v > 1.0 ? 1.0 : v);
    return (float)v;
}

// Whether the ray of pixel (ix, iy) may have a sample that counts: it meets the
// box, and a coarse brick near the level set.  FP32, along the unnormalised ray
// o + t d.  The box is widened by 1e-4, a hundred times the rounding of a point
// on the ray there; the bricks cover a cell more than their sites, against the
// rounding and the quarter cell that each crossing goes on past the face.  The
// LANES lanes of `group` look at an equal part of the ray each (sub: which).
template <int LANES>
__device__ __forceinline__ bool ray_may_count(const RayParams &rp, int ix, int iy, int sub, unsigned group)
{
    const float u = (2.0f * ((float)ix + 0.5f) / (float)rp.width - 1.0f) * rp.aspectf;
    const float v = 2.0f * ((float)iy + 0.5f) / (float)rp.height - 1.0f;
    float d[3], tn = 0.0f, tf = 1e30f;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        d[i] = rp.viewf[3 * i] * u + rp.viewf[3 * i + 1] * v - rp.viewf[3 * i + 2] * (float)kRenderFocal;
        const float b = rp.boxf[i] + 1e-4f, id = 1.0f / d[i];
        const float t0 = (-b - rp.eyef[i]) * id, t1 = (b - rp.eyef[i]) * id;
        tn = fmaxf(tn, fminf(t0, t1));  // fmin, fmax pass over NaN
        tf = fminf(tf, fmaxf(t0, t1));
    }
    if (!(tn <= tf) || !rp.bricks.coarse.bits) return tn <= tf;
    const float quarter = 0.25f / (rp.sf * sqrtf(u * u + v * v + (float)(kRenderFocal * kRenderFocal)));
    float gd[3], igd[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) gd[a] = d[a] * rp.sf, igd[a] = fabsf(1.0f / gd[a]);
    const float part = (tf - tn) * (1.0f / LANES), end = sub == LANES - 1 ? tf : tn + part * (float)(sub + 1);
    bool hit = false;
    for (float t = tn + part * (float)sub; t <= end;) {
        float g[3], e;
#pragma unroll
        for (int a = 0; a < 3; ++a) g[a] = fmaf(t, gd[a], rp.eyef[a] * rp.sf + rp.halff[a]);
        if (!empty_brick(rp.bricks.coarse, g, gd, igd, e)) {
            hit = true;
            break;
        }
        t += fmaxf(e, 0.0f) + quarter;
    }
    return LANES == 1 ? hit : __any_sync(group, hit) != 0;
}

// The plain march, one ray per thread (8 x 4 pixels per warp): where no sample
// can be passed over (a level set or scale that is not positive), and where a
// ray takes so few that the search costs more (few_samples).
__global__ void __launch_bounds__(32) k_render_rays_plain(const __grid_constant__ RayParams rp,
                                                          const dvec4 *__restrict__ vol, float4 *rgba)
{
    const int tiles_x = (rp.width + 7) >> 3, ty0 = blockIdx.x / tiles_x, tx0 = blockIdx.x - ty0 * tiles_x;
    const int ix = 8 * tx0 + (threadIdx.x & 7), iy = 4 * ty0 + (threadIdx.x >> 3);
    if (ix >= rp.width || iy >= rp.height) return;
    if (!ray_may_count<1>(rp, ix, iy, 0, 0u)) {
        rgba[(size_t)iy * rp.width + ix] = make_float4(rp.miss, rp.miss, rp.miss, rp.miss);
        return;
    }
    double d[3], tnear, tfar, sum[4] = {0.0, 0.0, 0.0, 0.0};
    pixel_ray(rp, ix, iy, d, tnear, tfar);
    int k = 0;
    for (double t = tnear; t <= tfar && k < rp.max_samples; t += rp.step, ++k) {
        int i0[3];
        double col[4];
        if (!ray_sample(rp, vol, d, t, false, i0, col)) continue;
        const double keep = 1.0 - sum[3];
#pragma unroll
        for (int c = 0; c < 4; ++c) sum[c] += col[c] * keep;
        if (sum[3] > kRenderAlphaStop) break;
    }
    rgba[(size_t)iy * rp.width + ix] =
        make_float4(pixel_value(sum[0], rp.brightness), pixel_value(sum[1], rp.brightness),
                    pixel_value(sum[2], rp.brightness), pixel_value(sum[3], rp.brightness));
}

// The march with samples passed over, eight lanes per ray.
//
// The plain march takes every sample k = 0, 1, ... while t_k <= t_far.  A
// sample with input < 0 changes nothing, and input is negative whenever the
// eight values it interpolates are below the level set by more than rounding
// (the weights are non-negative and sum to 1).  So, for a positive level set
// and scale:
//   - a ray that meets no coarse brick near the level set has no sample that
//     counts; the lanes look at an eighth of the ray each;
//   - empty bricks are crossed in one go;
//   - else the lanes take eight samples at once, in FP32: one whose cell's
//     eight high words are below the threshold, or whose FP32 interpolation is
//     below the level set by more than its error bound, is passed over;
// and the samples left are computed in FP64 as in the plain march, at the t_k
// that the repeated additions would have given (RayClock), and composited in
// order.  FP32 positions are within `tol` cells of the FP64 ones (each factor
// of (o + t d) s + half rounded: under 30 * 2^-24 s for rays from the eye at 4
// to the box); the bricks allow a whole cell, the cell tests ask for `tol`
// from the faces.
//
// Eight lanes because few rays reach the surface and those are long: with a
// ray per lane 440 warps did all the work, one cell test of gathers (1100
// cycles) after another: 344 us for 1024 x 768 pixels of a 128^3 field, 165
// with eight.
__global__ void __launch_bounds__(128) k_render_rays(const __grid_constant__ RayParams rp,
                                                     const dvec4 *__restrict__ vol, float4 *rgba)
{
    __shared__ double colours[4][32][4];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, sub = lane & 7;
    const unsigned group = 0xffu << (lane & 24);
    const int tiles_x = (rp.width + 3) >> 2, ty0 = blockIdx.x / tiles_x, tx0 = blockIdx.x - ty0 * tiles_x;
    const int ix = 4 * tx0 + 2 * (warp & 1) + ((lane >> 3) & 1), iy = 4 * ty0 + 2 * (warp >> 1) + (lane >> 4);
    if (ix >= rp.width || iy >= rp.height) return;  // whole groups
    float *out = reinterpret_cast<float *>(rgba + ((size_t)iy * rp.width + ix));
    if (!ray_may_count<8>(rp, ix, iy, sub, group)) {
        if (sub < 4) out[sub] = rp.miss;
        return;
    }
    double d[3], tnear, tfar;
    pixel_ray(rp, ix, iy, d, tnear, tfar);
    // FP32 copies for the search: lattice coordinates gf = of + t df
    float of[3], df[3], idf[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        of[i] = (float)(rp.eye[i] * rp.s + rp.half[i]);
        df[i] = (float)(d[i] * rp.s);
        idf[i] = fabsf(1.0f / df[i]);
    }
    const float tnf = (float)tnear, stepf = (float)rp.step, inv_step = 1.0f / stepf;
    const float tend = (float)tfar * 1.000004f + 1e-6f, tol = 4e-6f * rp.sf;
    const size_t sy = rp.n[2], sx = (size_t)rp.n[1] * rp.n[2];
    RayClock clk;
    clk.t = tnear;
    clk.k = 0;
    clk.binade(rp.step);
    double sum = 0.0, alpha = 0.0;  // component sub & 3 (each lane one), and component 3
    bool more = tnear <= tfar;
    int k0 = 0;  // the group's first sample not yet dealt with
    while (more) {
        const float t0 = fmaf((float)k0, stepf, tnf);
        if (k0 >= rp.max_samples || t0 > tend) break;
        if (rp.bricks.coarse.bits) {
            float g[3], e;
#pragma unroll
            for (int a = 0; a < 3; ++a) g[a] = fmaf(t0, df[a], of[a]);
            if (empty_brick(rp.bricks.coarse, g, df, idf, e) || empty_brick(rp.bricks.fine, g, df, idf, e)) {
                k0 += max((int)(fminf(e, 16.0f) * inv_step), 0) + 1;
                continue;
            }
        }
        // ---- eight samples: may mine count?
        const int k = k0 + sub;
        const float tk = fmaf((float)k, stepf, tnf);
        bool mine = k < rp.max_samples && tk <= tend, inside = mine;
        int i0[3];
        float w[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float g = fmaf(tk, df[a], of[a]), f = floorf(g);
            i0[a] = (int)f;
            w[a] = g - f;
            inside = inside && i0[a] >= 0 && i0[a] <= rp.n[a] - 2 && w[a] > tol && w[a] < 1.0f - tol;
        }
        if (inside) {
            const int *c0 = reinterpret_cast<const int *>(vol + ((size_t)i0[0] * sx + (size_t)i0[1] * sy + i0[2])) + 1;
            int hi[8], top = -0x7fffffff - 1;
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                hi[c] = __ldg(c0 + 8 * (((c & 1) ? sx : 0) + ((c & 2) ? sy : 0) + ((c & 4) ? 1 : 0)));
                top = max(top, ((unsigned)hi[c] & 0x7ff00000u) == 0x7ff00000u ? 0x7fffffff : hi[c]);
            }
            float v[8], lo = 3.4e38f, up = -3.4e38f;
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                v[c] = high_word_value(hi[c]);
                lo = fminf(lo, v[c]);
                up = fmaxf(up, v[c]);
            }
            // along x, y, z in turn
#pragma unroll
            for (int c = 0; c < 8; c += 2) v[c] = fmaf(w[0], v[c + 1] - v[c], v[c]);
            v[0] = fmaf(w[1], v[2] - v[0], v[0]);
            v[4] = fmaf(w[1], v[6] - v[4], v[4]);
            const float bf = fmaf(w[2], v[4] - v[0], v[0]);
            const float err = 4.0f * tol * (up - lo) + 8e-6f * fmaxf(fabsf(up), fabsf(lo));
            mine = top >= rp.threshold_key && !(bf + err < rp.threshold);
        }
        unsigned left = __ballot_sync(group, mine);
        k0 += 8;
        if (!left) continue;
        // ---- the candidates in FP64
        bool late = false;
        if (mine) {
            clk.advance(k, rp.step, inv_step);
            late = !(clk.t <= tfar);
            double col[4];
            mine = !late && ray_sample(rp, vol, d, clk.t, inside, i0, col);
            if (mine) {
#pragma unroll
                for (int c = 0; c < 4; ++c) colours[warp][lane][c] = col[c];
            }
        }
        __syncwarp(group);
        left = __ballot_sync(group, mine);
        more = !__any_sync(group, late);
        // front to back: each lane its component, every lane the alpha
        while (left) {
            const int j = __ffs(left) - 1;
            left &= left - 1;
            const double in = colours[warp][j][3], c = colours[warp][j][lane & 3];
            const double keep = 1.0 - alpha;
            sum += c * keep;
            alpha += in * keep;
            if (alpha > kRenderAlphaStop) {
                more = false;
                break;
            }
        }
        __syncwarp(group);
    }
    if (sub < 4) out[sub] = pixel_value(sum, rp.brightness);
}

bool render_params_valid(const skyrme_render_params &p)
{
    if (p.width < 1 || p.height < 1 || (long long)p.width * p.height > SKYRME_RENDER_MAX_PIXELS)
        return false;
    if (!(p.step >= SKYRME_RENDER_MIN_STEP && p.step <= 1.0)) return false;
    if (!isfinite(p.levelset) || !isfinite(p.transfer_scale) || !isfinite(p.brightness)) return false;
    // view: a rotation (orthonormal rows) to 1e-9
    for (int i = 0; i < 9; ++i)
        if (!isfinite(p.view[i])) return false;
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j) {
            double dot = 0.0;
            for (int k = 0; k < 3; ++k) dot += p.view[3 * i + k] * p.view[3 * j + k];
            if (fabs(dot - (i == j ? 1.0 : 0.0)) > 1e-9) return false;
        }
    return true;
}

// Whether samples below the level set may be passed over, and the threshold:
// a value below (1 - 1e-9) levelset interpolates to less than the level set
// whatever the rounding of its weights and sums (relative 1e-15), and
// (b - levelset) scale then comes out negative, not a rounded zero.
static bool render_threshold(const skyrme_render_params &p, double *value, int *key)
{
    if (!(p.levelset > 1e-30 && p.levelset < 1e30 && p.transfer_scale > 1e-200)) return false;
    *value = p.levelset * (1.0 - 1e-9);
    uint64_t bits;
    memcpy(&bits, value, sizeof(bits));
    *key = (int)(bits >> 32);
    return true;
}

// Whether the rays take so few samples that the plain march is the faster one.
// The search sets a ray up in FP64 in eight lanes, which costs a picture that
// fills the chip as much as 25 samples of the march, and 45 where nearly every
// sample counts (a low level set); a march of few rays does not fill it.  Judged
// by the ray through the picture's centre and the pixels that the box covers.
// Search and plain march, us, 1024 x 768 pixels of a 40^3 volume, level set 0.2:
// 5.4 samples 964 and 208, 11 967 and 296, 23 977 and 495, 45 992 and 870, 91 1016
// and 1641 (a whole render's bricks help the search: 45 samples 1.2 times faster);
// 320 x 240 pixels of 400 x 12 x 400 edge on, 8 samples: 27 and 44.
static bool few_samples(const RayParams &rp)
{
    double chord = 1e300, area = 0.0;  // of the box; the area as seen
    for (int i = 0; i < 3; ++i) {
        const double d = fabs(rp.view[3 * i + 2]);
        if (d > 0.0) chord = std::min(chord, 2.0 * rp.box[i] / d);
        area += 4.0 * rp.box[(i + 1) % 3] * rp.box[(i + 2) % 3] * d;
    }
    // a picture is 2 eye / focal high where the box is
    const double high = rp.height * (kRenderFocal / (2.0 * kRenderEye));
    const double hits = std::min(area * high * high, (double)rp.width * rp.height);
    return chord < rp.step * std::min(rp.levelset < 0.01 ? 48.0 : 24.0, 0.1 * sqrt(hits));
}

// Brick tables of a whole render in `bytes` of scratch: the smallest fine
// bricks whose bits fit in 32 KiB (a ray's lookups find them in L1), coarse
// ones four times as wide.  Returns the bytes used (0: none).
static size_t render_bricks(const int n[3], void *scratch, size_t bytes, BrickLevels &out)
{
    auto level = [&](Bricks &br, int shift) {
        size_t total = 1;
        br.shift = shift;
        for (int a = 0; a < 3; ++a) {
            br.nb[a] = ((n[a] - 1) >> shift) + 1;
            total *= br.nb[a];
        }
        return (total + 31) / 32 * 4;  // bytes
    };
    out = BrickLevels{};
    for (int shift = 1; shift <= 10; ++shift) {
        BrickLevels lv = {};
        const size_t fine = level(lv.fine, shift), coarse = level(lv.coarse, shift + 2);
        if (fine > 32768 || fine + coarse > bytes) continue;
        lv.fine.bits = static_cast<unsigned *>(scratch);
        lv.coarse.bits = lv.fine.bits + fine / 4;
        out = lv;
        return fine + coarse;
    }
    return 0;
}

static cudaError_t volume_kernels(const skyrme_lattice &lat, const FlowArgs &a, void *vol,
                                  void *scratch, const BrickLevels &br, size_t brick_bytes,
                                  int threshold_key, cudaStream_t s)
{
    auto *bits = static_cast<unsigned long long *>(scratch);
    // max B0, and the brick tables behind it
    cudaError_t e = cudaMemsetAsync(bits, 0, kBrickOffset + brick_bytes, s);
    if (e != cudaSuccess) return e;
    const double k1 = 1.0 / (12.0 * lat.h), bscale = -0.050660591821168885 * k1 * k1 * k1;
    const long long items = (long long)lat.n[0] * (((long long)lat.n[1] * lat.n[2] + 255) / 256);
    const int blocks = (int)std::min<long long>(items, 152LL * 8);
    dvec4 *v = static_cast<dvec4 *>(vol);
    const Ctrl *ctrl = static_cast<const Ctrl *>(a.ctrl);
    if (lat.precision == 64)
        k_render_volume<dvec4><<<blocks, 256, 0, s>>>(static_cast<const dvec4 *>(a.phi[0]),
                                                     static_cast<const dvec4 *>(a.phi[1]), ctrl,
                                                     lat.n[0], lat.n[1], lat.n[2], bscale, v, bits);
    else
        k_render_volume<float4><<<blocks, 256, 0, s>>>(static_cast<const float4 *>(a.phi[0]),
                                                      static_cast<const float4 *>(a.phi[1]), ctrl,
                                                      lat.n[0], lat.n[1], lat.n[2], bscale, v, bits);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_render_normalise<<<blocks, 256, 0, s>>>(v, lat.n[0], lat.n[1], lat.n[2], bits, br, threshold_key);
    return cudaGetLastError();
}

static cudaError_t ray_kernel(const int n[3], const void *vol, const skyrme_render_params &p,
                              float *rgba, const BrickLevels &br, cudaStream_t s)
{
    RayParams rp;
    rp.width = p.width;
    rp.height = p.height;
    for (int i = 0; i < 3; ++i) rp.n[i] = n[i];
    for (int i = 0; i < 9; ++i) rp.view[i] = p.view[i];
    rp.levelset = p.levelset;
    rp.scale = p.transfer_scale;
    rp.brightness = p.brightness;
    rp.step = p.step;
    // a chord of the box is at most 2 sqrt(3) long
    rp.max_samples = (int)ceil(3.5 / p.step) + 2;
    rp.aspect = (double)p.width / (double)p.height;
    rp.s = 0.0;
    for (int i = 0; i < 3; ++i) {
        rp.half[i] = 0.5 * (double)(n[i] - 1);
        rp.s = std::max(rp.s, rp.half[i]);
    }
    for (int i = 0; i < 3; ++i) {
        rp.box[i] = rp.half[i] / rp.s;
        // view space (0, 0, eye) to box space; the products by 0 and 4 are exact
        rp.eye[i] = (p.view[3 * i] * 0.0 + p.view[3 * i + 1] * 0.0) + p.view[3 * i + 2] * kRenderEye;
        rp.halff[i] = (float)rp.half[i];
        rp.boxf[i] = (float)rp.box[i];
        rp.eyef[i] = (float)rp.eye[i];
    }
    for (int i = 0; i < 9; ++i) rp.viewf[i] = (float)p.view[i];
    rp.aspectf = (float)rp.aspect;
    rp.sf = (float)rp.s;
    // (a negative brightness leaves -0, as the clamp does)
    rp.miss = (float)(0.0 * p.brightness);
    double threshold = 0.0;
    rp.threshold_key = 0;
    const bool skip = render_threshold(p, &threshold, &rp.threshold_key);
    rp.threshold = (float)(threshold * (1.0 - 1e-6));
    rp.bricks = br;
    float4 *out = reinterpret_cast<float4 *>(rgba);
    const dvec4 *v = static_cast<const dvec4 *>(vol);
    if (skip && !few_samples(rp)) {
        const long long tiles = (long long)((p.width + 3) / 4) * ((p.height + 3) / 4);
        k_render_rays<<<(unsigned)tiles, 128, 0, s>>>(rp, v, out);
    } else {
        const long long tiles = (long long)((p.width + 7) / 8) * ((p.height + 3) / 4);
        k_render_rays_plain<<<(unsigned)tiles, 32, 0, s>>>(rp, v, out);
    }
    return cudaGetLastError();
}

cudaError_t launch_render_volume(const skyrme_lattice &lat, const FlowArgs &a, void *vol,
                                 void *scratch, cudaStream_t s)
{
    return volume_kernels(lat, a, vol, scratch, BrickLevels{}, 0, 0, s);
}

cudaError_t launch_render_rays(const int n[3], const void *vol, const skyrme_render_params &p,
                               float *rgba, cudaStream_t s)
{
    return ray_kernel(n, vol, p, rgba, BrickLevels{}, s);
}

cudaError_t launch_render(const skyrme_lattice &lat, const FlowArgs &a,
                          const skyrme_render_params &p, void *vol, void *scratch,
                          size_t scratch_bytes, float *rgba, cudaStream_t s)
{
    BrickLevels br = {};
    double threshold;
    int key = 0;
    size_t brick_bytes = 0;
    if (render_threshold(p, &threshold, &key) && scratch_bytes > kBrickOffset)
        brick_bytes = render_bricks(lat.n, static_cast<char *>(scratch) + kBrickOffset,
                                    scratch_bytes - kBrickOffset, br);
    cudaError_t e = volume_kernels(lat, a, vol, scratch, br, brick_bytes, key, s);
    return e != cudaSuccess ? e : ray_kernel(lat.n, vol, p, rgba, br, s);
}

}  // namespace skyrme
