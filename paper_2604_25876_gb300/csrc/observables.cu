// observables.cu -- Section 5 observables of the current field: centre of
// mass (Eq. "CoM"), RMS radius (Eq. "RMS radius"), quadrupole (Eq. "Q tensor"
// with rho = B0 / 2), the inertia tensors U, V, W (Eqs. "U/V/W inertia
// tensor") and the monopole D-term (Eq. "D-term").
//
// The paper writes these with su(2) currents.  For U = phi^0 + i phi^a tau^a
// they reduce to 4-vector algebra with
//   d_k       the tangent part of the lattice derivative, d_k phi - (phi . d_k phi) phi
//             (the lattice L_k = U^dagger d_k U is taken as its traceless part),
//   A_ij      = d_i . d_j,
//   K_a       = (0, e_a x pi)                      (isorotation about axis a),
//   G_b       = -sum_nl eps_bnl r_n d_l             (rotation about axis b, r = x - X_c),
// as
//   U_ab = 2 sum [K_a.K_b (1 + tr A) - sum_k (K_a.d_k)(K_b.d_k)],
//   V_ab = the same with G_a, G_b,
//   W_ab = -2 sum [K_a.G_b (1 + tr A) - sum_k (K_a.d_k)(G_b.d_k)],
//   T_ij = 2 A_ij (1 + tr A) - 2 (A A)_ij - delta_ij (tr A + (tr^2 A - tr A^2)/2 + e0),
// which is what T = a U a/2 + b V b/2 - a W b means for the kinetic energy of
// the model's Lagrangian.  The baryon density and the energy density are those
// of the flow (Eqs. "B0_components" and "SkyrmeEnergy_phi" with the lattice
// derivatives).
//
// The kernels evaluate these without forming d_k or G_b.  With p_k = phi.d_k phi
// (raw derivatives), Y_ak = K_a.d_k = (pi x D_k)_a (D_k the vector part of
// d_k phi; K_a is orthogonal to phi), B = (1 + tr A) 1 - A, Z = A B and
// H = Y B:
//   A_ij = d_i phi . d_j phi - p_i p_j (2 - |phi|^2),
//   U_ab = 2 sum [(|pi|^2 delta_ab - pi_a pi_b)(1 + tr A) - (Y Y^T)_ab],
//   V_ab = 2 sum (e_a x r) . Z (e_b x r),
//   W_ab = 2 sum e_b . (r x H_a),
//   r_i r_j T_ij - r^2 tr T / 3 = 2 (r . Z r - r^2 tr Z / 3)
// (the isotropic part of T drops out of the D-term).  That is about 280 FP64
// instructions per site instead of 560, and the field is widened to FP64 on
// the integer pipe (52 conversions more): the passes are bound by the FP64
// pipe, 2 lanes per SM and cycle.  Measured on a 151^3 FP32 field: first
// pass 875 -> 487 us, second 3465 -> 1683 us (91% of the pipe).
// All arithmetic is FP64 whatever the field's precision; the sums run in a
// fixed order (persistent CTAs, one partial record each, the last CTA summing
// the records), so repeated calls are bitwise equal.  The centre of mass goes
// from the first pass to the second on the device.
#include <cuda_runtime.h>
#include <math.h>
#include <string.h>

#include <algorithm>

#include "lattice_sites.cuh"
#include "skyrme_device.cuh"
#include "skyrme_internal.h"

namespace skyrme {

constexpr int kObsCtas = 152;
constexpr int kObsThreads = 256;
constexpr int kObsSums = 32;   // doubles per record
constexpr int kObsPlanes = 4;  // x-planes of a thread's run (y, z and their products stay put)

// record layout
enum {
    O_B = 0, O_XB = 1,  // pass 0: det, x det, y det, z det
    // pass 1: energy; r_i r_j det; U; the parts of V; W; the diagonal of the D-term
    O_E = 0, O_M = 1, O_U = 7, O_VD = 13, O_VO = 16, O_S = 19, O_W = 22, O_D = 31,
};
// the totals follow the records: pass 0's, then pass 1's, then X (3 doubles)
constexpr int kObsTotals = kObsCtas * kObsSums;

template <typename T> struct ObsArgs {
    const vec4_t<T> *phi[2];
    Ctrl *ctrl;
    double *parts;
    int n0, n1, n2;
    int blocks, items;  // (y, z) blocks of 256 sites, work items
    int share;          // runs of planes that share an item where a plane's sites fit in a block
    double h, two_m2;
    double K144, k1sq, k1qu;  // 144 h^2, and 1/(12h) to the 2nd and 4th power
};

// Sum of v[q] over the warp's lanes for 32 quantities at once: each exchange
// halves the quantities a lane carries (16 + 8 + 4 + 2 + 1 additions instead
// of 5 per quantity).  Lane q ends with the total of quantity q.
__device__ __forceinline__ double warp_transpose_sum(double (&v)[32])
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int q = 0; q < o; ++q) {
            const double keep = up ? v[q + o] : v[q], send = up ? v[q] : v[q + o];
            v[q] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
    return v[0];
}

template <typename T, int PASS>
__global__ void __launch_bounds__(kObsThreads) k_observables(const __grid_constant__ ObsArgs<T> a)
{
    const int cur = __ldcg(&a.ctrl->cur);
    const vec4_t<T> *phi = cur ? a.phi[1] : a.phi[0];
    const int iy = a.n1 - 4, iz = a.n2 - 4;
    const size_t sx = (size_t)a.n1 * a.n2, sy = (size_t)a.n2;
    double *totals = a.parts + kObsTotals;
    double X[3] = {0.0, 0.0, 0.0};
    if (PASS == 1) {
#pragma unroll
        for (int i = 0; i < 3; ++i) X[i] = __ldcg(totals + 2 * kObsSums + i);
    }
    double acc[kObsSums];
#pragma unroll
    for (int q = 0; q < kObsSums; ++q) acc[q] = 0.0;

    for (int it = blockIdx.x; it < a.items; it += gridDim.x) {
        const int xi = it / a.blocks, sub = a.share > 1 ? (int)threadIdx.x / (iy * iz) : 0;
        const int xc = xi * a.share + sub;
        const int s = (it - xi * a.blocks) * kObsThreads + (int)threadIdx.x - sub * iy * iz;
        if (sub >= a.share || s >= iy * iz) continue;
        const int y = 2 + s / iz, z = 2 + s % iz;
        const double r1 = ((double)y - 0.5 * (a.n1 - 1)) * a.h - X[1];
        const double r2 = ((double)z - 0.5 * (a.n2 - 1)) * a.h - X[2];
        const double m11 = r1 * r1, m22 = r2 * r2, m12 = r1 * r2;
        const int xa = 2 + xc * kObsPlanes, xb = min(xa + kObsPlanes, a.n0 - 2);
        size_t c = (size_t)xa * sx + (size_t)y * sy + z;
        for (int x = xa; x < xb; ++x, c += sx) {
            double ph[4], d[3][4];
            load_site(phi, c, ph);
            site_first_differences(phi, c, sx, sy, d);
            const double det = charge_determinant(ph, d);
            const double r0 = ((double)x - 0.5 * (a.n0 - 1)) * a.h - X[0];
            if (PASS == 0) {
                acc[O_B] += det;
                acc[O_XB] = ::fma(r0, det, acc[O_XB]);
                acc[O_XB + 1] = ::fma(r1, det, acc[O_XB + 1]);
                acc[O_XB + 2] = ::fma(r2, det, acc[O_XB + 2]);
            } else {
                auto dp = [](const double *u, const double *v) {
                    return u[0] * v[0] + u[1] * v[1] + u[2] * v[2] + u[3] * v[3];
                };
                double a00 = dp(d[0], d[0]), a11 = dp(d[1], d[1]), a22 = dp(d[2], d[2]);
                double a01 = dp(d[0], d[1]), a02 = dp(d[0], d[2]), a12 = dp(d[1], d[2]);
                // energy density of the flow (raw lattice derivatives)
                acc[O_E] += ::fma(a.k1sq, a00 + a11 + a22,
                                  ::fma(a.k1qu, a00 * (a11 + a22) + a11 * a22 -
                                                    (a01 * a01 + a02 * a02 + a12 * a12),
                                        a.two_m2 * (1.0 - ph[0])));
                // moments of the charge
                const double m00 = r0 * r0, m01 = r0 * r1, m02 = r0 * r2;
                acc[O_M + 0] = ::fma(m00, det, acc[O_M + 0]);
                acc[O_M + 1] = ::fma(m11, det, acc[O_M + 1]);
                acc[O_M + 2] = ::fma(m22, det, acc[O_M + 2]);
                acc[O_M + 3] = ::fma(m01, det, acc[O_M + 3]);
                acc[O_M + 4] = ::fma(m02, det, acc[O_M + 4]);
                acc[O_M + 5] = ::fma(m12, det, acc[O_M + 5]);
                // A: the products of the tangent derivatives
                const double s1 = ph[1] * ph[1], s2 = ph[2] * ph[2], s3 = ph[3] * ph[3];
                {
                    const double w = 2.0 - (ph[0] * ph[0] + (s1 + s2 + s3));
                    const double p0 = dp(ph, d[0]), p1 = dp(ph, d[1]), p2 = dp(ph, d[2]);
                    const double w0 = -w * p0, w1 = -w * p1, w2 = -w * p2;
                    a00 = ::fma(w0, p0, a00), a11 = ::fma(w1, p1, a11), a22 = ::fma(w2, p2, a22);
                    a01 = ::fma(w0, p1, a01), a02 = ::fma(w0, p2, a02), a12 = ::fma(w1, p2, a12);
                }
                const double one_tr = a.K144 + (a00 + a11 + a22);
                // Y[k][a] = (pi x D_k)_a
                double Y[3][3];
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    Y[k][0] = minor2(ph[2], d[k][3], ph[3], d[k][2]);
                    Y[k][1] = minor2(ph[3], d[k][1], ph[1], d[k][3]);
                    Y[k][2] = minor2(ph[1], d[k][2], ph[2], d[k][1]);
                }
                {
                    const int qi[6] = {0, 1, 2, 0, 0, 1}, qj[6] = {0, 1, 2, 1, 2, 2};
                    const double kk[6] = {s2 + s3, s1 + s3, s1 + s2, -ph[1] * ph[2], -ph[1] * ph[3],
                                          -ph[2] * ph[3]};
#pragma unroll
                    for (int t = 0; t < 6; ++t) {
                        double v = ::fma(kk[t], one_tr, acc[O_U + t]);
#pragma unroll
                        for (int k = 0; k < 3; ++k) v = ::fma(-Y[k][qi[t]], Y[k][qj[t]], v);
                        acc[O_U + t] = v;
                    }
                }
                // B = (1 + tr A) 1 - A
                const double b00 = one_tr - a00, b11 = one_tr - a11, b22 = one_tr - a22;
                // W: H_a = Y_a B (over k), W_ab += e_b . (r x H_a)
#pragma unroll
                for (int g = 0; g < 3; ++g) {
                    const double h0 = Y[0][g] * b00 - Y[1][g] * a01 - Y[2][g] * a02;
                    const double h1 = Y[1][g] * b11 - Y[0][g] * a01 - Y[2][g] * a12;
                    const double h2 = Y[2][g] * b22 - Y[0][g] * a02 - Y[1][g] * a12;
                    acc[O_W + 3 * g + 0] = ::fma(-r2, h1, ::fma(r1, h2, acc[O_W + 3 * g + 0]));
                    acc[O_W + 3 * g + 1] = ::fma(-r0, h2, ::fma(r2, h0, acc[O_W + 3 * g + 1]));
                    acc[O_W + 3 * g + 2] = ::fma(-r1, h0, ::fma(r0, h1, acc[O_W + 3 * g + 2]));
                }
                // Z = A B (symmetric), the tensor of V and of the D-term
                const double z00 = a00 * b00 - a01 * a01 - a02 * a02;
                const double z11 = a11 * b11 - a01 * a01 - a12 * a12;
                const double z22 = a22 * b22 - a02 * a02 - a12 * a12;
                const double z01 = a01 * b11 - a00 * a01 - a02 * a12;
                const double z02 = a02 * b22 - a00 * a02 - a01 * a12;
                const double z12 = a12 * b22 - a01 * a02 - a11 * a12;
                acc[O_VD + 0] = ::fma(m22, z11, ::fma(m11, z22, acc[O_VD + 0]));
                acc[O_VD + 1] = ::fma(m22, z00, ::fma(m00, z22, acc[O_VD + 1]));
                acc[O_VD + 2] = ::fma(m11, z00, ::fma(m00, z11, acc[O_VD + 2]));
                acc[O_VO + 0] = ::fma(m02, z12, ::fma(m12, z02, ::fma(-m22, z01, ::fma(-m01, z22, acc[O_VO + 0]))));
                acc[O_VO + 1] = ::fma(m01, z12, ::fma(m12, z01, ::fma(-m11, z02, ::fma(-m02, z11, acc[O_VO + 1]))));
                acc[O_VO + 2] = ::fma(m01, z02, ::fma(m02, z01, ::fma(-m00, z12, ::fma(-m12, z00, acc[O_VO + 2]))));
                acc[O_S + 0] = ::fma(m01, z01, acc[O_S + 0]);
                acc[O_S + 1] = ::fma(m02, z02, acc[O_S + 1]);
                acc[O_S + 2] = ::fma(m12, z12, acc[O_S + 2]);
                const double third = (m00 + m11 + m22) * (1.0 / 3.0);
                acc[O_D] = ::fma(m00 - third, z00, ::fma(m11 - third, z11, ::fma(m22 - third, z22, acc[O_D])));
            }
        }
    }

    // block sums in a fixed order: each warp by exchanges, then over the warps
    __shared__ double red[kObsThreads / 32][kObsSums];
    __shared__ int s_last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    red[warp][lane] = warp_transpose_sum(acc);
    __syncthreads();
    if (warp == 0) {
        double v = 0.0;
#pragma unroll
        for (int w = 0; w < kObsThreads / 32; ++w) v += red[w][lane];
        a.parts[(size_t)blockIdx.x * kObsSums + lane] = v;
        __threadfence();
        __syncwarp();
        if (lane == 0) s_last = atomicAdd(&a.ctrl->edone, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return;
    // the last CTA: warp w sums the records w, w + 8, ..., lane q quantity q
    __threadfence();
    double v = 0.0;
#pragma unroll 4
    for (int i = warp; i < (int)gridDim.x; i += kObsThreads / 32)
        v += __ldcg(a.parts + (size_t)i * kObsSums + lane);
    red[warp][lane] = v;
    __syncthreads();
    if (warp != 0) return;
    v = 0.0;
#pragma unroll
    for (int w = 0; w < kObsThreads / 32; ++w) v += red[w][lane];
    totals[PASS * kObsSums + lane] = v;
    if (PASS == 0) {
        // X = sum x b / sum b: the factors of the charge density cancel
        const double b = __shfl_sync(0xffffffffu, v, O_B);
        if (lane >= O_XB && lane < O_XB + 3) totals[2 * kObsSums + lane - O_XB] = v / b;
    }
    if (lane == 0) a.ctrl->edone = 0;
}

template <typename T>
static skyrme_status observables_impl(const skyrme_lattice &lat, const FlowArgs &fa,
                                      skyrme_observables_t *out, cudaStream_t s)
{
    ObsArgs<T> a;
    a.phi[0] = static_cast<const vec4_t<T> *>(fa.phi[0]);
    a.phi[1] = static_cast<const vec4_t<T> *>(fa.phi[1]);
    a.ctrl = static_cast<Ctrl *>(fa.ctrl);
    a.parts = fa.energy_parts;
    a.n0 = lat.n[0];
    a.n1 = lat.n[1];
    a.n2 = lat.n[2];
    a.blocks = ((a.n1 - 4) * (a.n2 - 4) + kObsThreads - 1) / kObsThreads;
    // Small planes: items of several runs, where one run each would be more items than
    // CTAs (3000 x 6 x 7 FP32 370 us so, 118 now); no more to an item than that
    // takes, for a CTA's warps share its SM's FP64 pipe (400 x 10 x 10 110 us with one
    // each, 156 with blocks filled).
    const int runs = (a.n0 - 4 + kObsPlanes - 1) / kObsPlanes;
    a.share = std::max(1, std::min(kObsThreads / ((a.n1 - 4) * (a.n2 - 4)), (runs + kObsCtas - 1) / kObsCtas));
    a.items = a.blocks * ((runs + a.share - 1) / a.share);
    a.h = lat.h;
    // the derivatives are carried without their 1/(12h) = k1 (d_k phi = k1 u_k):
    // Y, A, B, H, Z then hold powers 1, 2, 2, 3, 4 of 12h, taken out of the sums
    const double k1 = 1.0 / (12.0 * lat.h), k1sq = k1 * k1;
    a.k1sq = k1sq;
    a.k1qu = k1sq * k1sq;
    a.K144 = 144.0 * lat.h * lat.h;
    a.two_m2 = 2.0 * lat.m * lat.m;
    k_observables<T, 0><<<kObsCtas, kObsThreads, 0, s>>>(a);
    if (cudaGetLastError() != cudaSuccess) return SKYRME_ECUDA;
    k_observables<T, 1><<<kObsCtas, kObsThreads, 0, s>>>(a);
    if (cudaGetLastError() != cudaSuccess) return SKYRME_ECUDA;
    double tot[2 * kObsSums + 3];
    if (cudaMemcpyAsync(tot, a.parts + kObsTotals, sizeof(tot), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return SKYRME_ECUDA;
    const double h3 = lat.h * lat.h * lat.h;
    const double kb = h3 * -0.050660591821168885 * k1 * k1sq;  // b = -det / (2 pi^2)
    const double *t0 = tot, *t1 = tot + kObsSums, *X = tot + 2 * kObsSums;
    out->B = kb * t0[O_B];
    if (!(out->B != 0.0) || !isfinite(out->B)) {
        // no baryon density: no centre of mass to take moments about
        memset(out, 0, sizeof(*out));
        return isfinite(t0[O_B]) ? SKYRME_EINVAL : SKYRME_ENONFINITE;
    }
    for (int i = 0; i < 3; ++i) out->X[i] = X[i];
    out->E = h3 * t1[O_E];
    const double r2b = kb * (t1[O_M] + t1[O_M + 1] + t1[O_M + 2]);
    out->R = sqrt(r2b / out->B);
    const int qi[6] = {0, 1, 2, 0, 0, 1}, qj[6] = {0, 1, 2, 1, 2, 2};
    double trace_off = 0.0;  // sum of r_i r_j Z_ij, i < j
    for (int t = 0; t < 6; ++t) {
        const int i = qi[t], j = qj[t];
        out->Q[i][j] = out->Q[j][i] = 0.5 * (3.0 * kb * t1[O_M + t] - (t < 3 ? r2b : 0.0));
        out->U[i][j] = out->U[j][i] = 2.0 * h3 * k1sq * t1[O_U + t];
        // V_00 = sum r_2^2 Z_11 + r_1^2 Z_22 - 2 r_1 r_2 Z_12 and cyclically
        const double v = t < 3 ? t1[O_VD + t] - 2.0 * t1[O_S + 2 - t] : t1[O_VO + t - 3];
        out->V[i][j] = out->V[j][i] = 2.0 * h3 * a.k1qu * v;
        if (t >= 3) trace_off += t1[O_S + t - 3];
    }
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j) out->W[i][j] = 2.0 * h3 * k1 * k1sq * t1[O_W + 3 * i + j];
    out->D = -2.0 * out->E / 5.0 * h3 * a.k1qu * 2.0 * (t1[O_D] + 2.0 * trace_off);
    if (!isfinite(out->E) || !isfinite(out->D) || !isfinite(out->R)) return SKYRME_ENONFINITE;
    return SKYRME_OK;
}

skyrme_status compute_observables(const skyrme_lattice &lat, const FlowArgs &a,
                                  skyrme_observables_t *out, cudaStream_t s)
{
    return lat.precision == 64 ? observables_impl<double>(lat, a, out, s)
                               : observables_impl<float>(lat, a, out, s);
}

size_t observables_parts_bytes() { return (size_t)(kObsTotals + 2 * kObsSums + 3) * sizeof(double); }

}  // namespace skyrme
