// flow_f64.cu -- the FP64 step of the Newton and arrested Newton flows (gradient
// flows run on the tile kernel of flow_generic.cu) (Section 3: 4th-order
// first, second and mixed derivatives, Euler-Lagrange gradient, tangent
// projection of Eq. "Newton_flow", v += dt F, phi = normalise(phi + dt v);
// Section 2.1 and 7.8 densities).
//
// GB300 issues two FP64 lanes per SM and cycle (a warp instruction takes 16
// cycles of its SM), so the step is bound by the FP64 pipe, and everything
// else is there to keep the pipe busy with few instructions:
//
//  * Every warp is a pipeline of its own: it owns a column of 32 (y, z) sites
//    (2 x 16, or 4 x 8 where that pads the lattice less) and marches along x
//    through its share of the lattice's (column, x-plane) units, plane by
//    plane, with no barrier between warps.  It brings its own haloed planes
//    into shared memory with cp.async, four at the start of a run and then one
//    ahead (an iteration takes thousands of cycles); the extra halo traffic of
//    so small a column is nothing at this rate (3.75 sites read per site, from
//    L2).
//  * u_y and u_z (u_i = 12h d_i phi) are formed once per site, when its plane
//    arrives, and kept in shared memory for the five planes of the mixed
//    derivatives d_xy, d_xz; only u_y's z-halo is formed twice, one component
//    per lane.  The x-stencil's field values stay in registers.
//  * The derivatives carry no 1/h factors, and nothing is scaled per site: the
//    force comes out as F / 2B, B = 1/(1728 h^4), with 2B in the time step, the
//    masses divided by B, and the sums scaled at the end.  About 325 FP64
//    instructions per site, against 364 of the tile kernel that this replaces.
//  * Units per warp decide the time of a small lattice, so the launch takes 8,
//    6 or 4 warps per SM, whichever leaves the busiest SM less to do
//    (plan_warps).
//  * A launch runs several steps of a small lattice (kLaunchSites, kLaunchSteps): every CTA
//    waits for the decision and goes on to the next step, over one more barrier
//    when sites were corrected.  One step per launch and now, us per step in a
//    graph and on a stream: 24 x 26 x 28 26.9 and 29.2 -> 25.1 and 25.2, 48^3
//    73.7 and 76.3 -> 72.1 and 72.2, 90 x 75 x 83 326 and 329 -> 325 and 326.
//  * Launches whose CTAs wait for one another (for the decision, or for the next
//    step) are cooperative: the CTAs of one are resident together, whatever other
//    streams run.  Consecutive launches are not programmatic dependents, whose
//    CTAs start one by one as the last launch's leave: two flows on two streams
//    could then each hold some SMs and wait for CTAs that the other leaves no
//    room for.
//  * Measured (us per iteration, tile kernel and fix-up launch before -> now):
//    48^3 103.6 -> 72, 64^3 187 -> 153, 128^3 1392 -> 1166 (1.635 G
//    site-updates/s, 322 instructions per site at the measured FP64 FMA rate: full),
//    90 x 75 x 83 lightly bound 409 -> 325, 72 x 80 x 100 sextic 520 -> 417.
//  * The arrest decision falls in the last CTA to finish; the launch is
//    cooperative, and every warp corrects its own sites when the decision that
//    the step ran with was wrong (flow_generic.cu has the scheme).
#include <cuda_runtime.h>
#include <math.h>
#include <string.h>

#include <algorithm>

#include "skyrme_device.cuh"
#include "skyrme_internal.h"
#include "tma.cuh"

namespace skyrme {

constexpr int kMaxWarps = 8;    // per CTA, one CTA per SM
constexpr int kMaxShare = 160 * kMaxWarps;  // warps of a launch
constexpr int kPlaneSlots = 4;  // planes x .. x + 2 of the centre, and the next one arriving
constexpr double kLaunchSites = 1 << 22;  // site updates of a launch of several steps,
constexpr int kLaunchSteps = 128;         // and its steps, at most
constexpr int kSums64 = 8;      // e2, e4, potential, det, |F|^2, max |F|^2, e6, (unused)

struct F64Params {
    dvec4 *phi[2];
    dvec4 *vel[2];
    Ctrl *ctrl;
    double *parts;
    double *slab_rec;  // x-slab: the record goes here, the decision is made later
    int n0, n1, n2;
    int nix, nzt;      // interior planes, columns along z
    long long units;   // columns * planes
    int mode, fuse_fix;
    int steps;         // of this launch
    double dt, dt2;    // dt, and 2 dt B
    double K144;       // 144 h^2
    double bm2, bmy2, bmz2, bmw2;  // squared masses / B
    double my2, mz2, mw2, m2x2;    // and for the potential density (2 m^2)
    double c6b;        // c6 / (144 h^2)
    double h3, scale[kSums64];  // of the sums (1/h factors; not h^3)
    int start[kMaxShare + 1];   // first unit of every warp (share_units)
};

template <int TZ> struct ColumnShape {
    static constexpr int TY = 32 / TZ, RY = TY + 4, RZ = TZ + 4, SITES = RY * RZ;
    static constexpr int COPIES = (2 * SITES + 31) / 32;  // 16-byte copies per lane
    static constexpr int HALO = TY * 4 * 4 / 32;          // u_y halo components per lane
};
template <int TZ> struct WarpSmem {
    using S = ColumnShape<TZ>;
    dvec4 plane[kPlaneSlots][S::SITES];
    dvec4 uy[5][S::TY][S::RZ];
    dvec4 uz[5][32];
};
// Dynamic shared memory: this, then one WarpSmem per warp
struct __align__(128) StepSmem64 {
    double red[kMaxWarps][kSums64];
    double tot[kSums64];
    int last, fix;
};

__device__ __forceinline__ dvec4 lds(const dvec4 *p) { return load4<double>(p); }
// A site from L2: L1 may hold what an earlier step of the launch read there
__device__ __forceinline__ dvec4 ldcg4(const dvec4 *p)
{
    const double2 *q = reinterpret_cast<const double2 *>(p), a = __ldcg(q), b = __ldcg(q + 1);
    return dvec4{a.x, a.y, b.x, b.y};
}
__device__ __forceinline__ double dot4(const double (&a)[4], const double (&b)[4])
{
    return a[0] * b[0] + a[1] * b[1] + a[2] * b[2] + a[3] * b[3];
}
__device__ __forceinline__ void vec(double (&v)[4], const dvec4 &d) { v[0] = d.x, v[1] = d.y, v[2] = d.z, v[3] = d.w; }
// u = 8 (p1 - m1) - (p2 - m2) = 12h d phi (applied to u_j: 144h^2 d_ij phi = -12 N_ij)
__device__ __forceinline__ double first(double m2, double m1, double p1, double p2)
{
    return ::fma(8.0, p1 - m1, m2 - p2);
}
__device__ __forceinline__ dvec4 first(const dvec4 &m2, const dvec4 &m1, const dvec4 &p1, const dvec4 &p2)
{
    return dvec4{first(m2.x, m1.x, p1.x, p2.x), first(m2.y, m1.y, p1.y, p2.y),
                 first(m2.z, m1.z, p1.z, p2.z), first(m2.w, m1.w, p1.w, p2.w)};
}
__device__ __forceinline__ void first(double (&o)[4], const dvec4 &m2, const dvec4 &m1, const dvec4 &p1,
                                      const dvec4 &p2)
{
    vec(o, first(m2, m1, p1, p2));
}
// N = (p2 + m2) + 30 c - 16 (p1 + m1) = -12h^2 d^2 phi
__device__ __forceinline__ double second(double m2, double m1, double c, double p1, double p2)
{
    return ::fma(-16.0, p1 + m1, ::fma(30.0, c, p2 + m2));
}
__device__ __forceinline__ void second(double (&o)[4], const dvec4 &m2, const dvec4 &m1, const dvec4 &c,
                                       const dvec4 &p1, const dvec4 &p2)
{
    o[0] = second(m2.x, m1.x, c.x, p1.x, p2.x), o[1] = second(m2.y, m1.y, c.y, p1.y, p2.y);
    o[2] = second(m2.z, m1.z, c.z, p1.z, p2.z), o[3] = second(m2.w, m1.w, c.w, p1.w, p2.w);
}

// F / 2B at a site from its unscaled derivatives (u, N, M = -12 N_ij for ij =
// xy, xz, yz), and its densities {tr A, quartic form, potential (1 - phi^0 for
// the standard model), det, sextic det^2}.  The brace of the Euler-Lagrange
// equation over -B is (site_physics of the tile kernels, regrouped)
//   sum_i [N_ii (144h^2 + tr A - A_ii) + u_i C_i] - 2 sum_{i<j} N_ij A_ij,
//   C_i = sum_{j != i} N_ij.u_j - (sum_{j != i} N_jj).u_i.
template <bool EXT>
__device__ __forceinline__ void step_site(const F64Params &p, const double (&ph)[4], const double (&u)[3][4],
                                          const double (&N)[3][4], const double (&M)[3][4], double (&F)[4],
                                          double (&dens)[5])
{
    const double a00 = dot4(u[0], u[0]), a11 = dot4(u[1], u[1]), a22 = dot4(u[2], u[2]);
    const double a01 = dot4(u[0], u[1]), a02 = dot4(u[0], u[2]), a12 = dot4(u[1], u[2]);
    constexpr double kM = -1.0 / 12.0, kS = 1.0 / 6.0;
    double L12[4], L02[4], L01[4];
#pragma unroll
    for (int A = 0; A < 4; ++A) {
        L12[A] = N[1][A] + N[2][A];
        L02[A] = N[0][A] + N[2][A];
        L01[A] = N[0][A] + N[1][A];
    }
    const double c0 = ::fma(kM, dot4(M[0], u[1]) + dot4(M[1], u[2]), -dot4(L12, u[0]));
    const double c1 = ::fma(kM, dot4(M[0], u[0]) + dot4(M[2], u[2]), -dot4(L02, u[1]));
    const double c2 = ::fma(kM, dot4(M[1], u[0]) + dot4(M[2], u[1]), -dot4(L01, u[2]));
    const double tra = a00 + a11 + a22, K = p.K144 + tra;
    const double k0 = K - a00, k1 = K - a11, k2 = K - a22;
    const double b01 = kS * a01, b02 = kS * a02, b12 = kS * a12;
    double H[4];  // G / 2B
#pragma unroll
    for (int A = 0; A < 4; ++A)
        H[A] = N[0][A] * k0 + N[1][A] * k1 + N[2][A] * k2 + M[0][A] * b01 + M[1][A] * b02 + M[2][A] * b12 +
               u[0][A] * c0 + u[1][A] * c1 + u[2][A] * c2;
    H[0] -= p.bm2;
    // 2x2 minors of the rows (phi, u_x) and (u_y, u_z)
    double s[6], c[6];
    {
        const double(&r1)[4] = u[0], (&r2)[4] = u[1], (&r3)[4] = u[2];
        s[0] = ph[0] * r1[1] - r1[0] * ph[1], s[1] = ph[0] * r1[2] - r1[0] * ph[2];
        s[2] = ph[0] * r1[3] - r1[0] * ph[3], s[3] = ph[1] * r1[2] - r1[1] * ph[2];
        s[4] = ph[1] * r1[3] - r1[1] * ph[3], s[5] = ph[2] * r1[3] - r1[2] * ph[3];
        c[0] = r2[0] * r3[1] - r3[0] * r2[1], c[1] = r2[0] * r3[2] - r3[0] * r2[2];
        c[2] = r2[0] * r3[3] - r3[0] * r2[3], c[3] = r2[1] * r3[2] - r3[1] * r2[2];
        c[4] = r2[1] * r3[3] - r3[1] * r2[3], c[5] = r2[2] * r3[3] - r3[2] * r2[3];
    }
    const double D = s[0] * c[5] - s[1] * c[4] + s[2] * c[3] + s[3] * c[2] - s[4] * c[1] + s[5] * c[0];
    const double w = 1.0 - ph[0];
    dens[0] = tra;
    dens[1] = a00 * (a11 + a22) + a11 * a22 - (a01 * a01 + a02 * a02 + a12 * a12);
    dens[2] = w;
    dens[3] = D;
    dens[4] = 0.0;
    if constexpr (EXT) {
        // Section 7.8 potentials and their gradient
        const double w2 = w * w;
        H[0] -= p.bmy2 * ph[0] + p.bmz2 * w + p.bmw2 * w2 * w;
        dens[2] = p.m2x2 * w + p.my2 * (1.0 - ph[0] * ph[0]) + p.mz2 * w2 + 0.5 * p.mw2 * w2 * w2;
        if (p.c6b != 0.0) {
            // the sextic term: P = dD/dphi and Q_i = dD/du_i, the cofactor rows
            // of [phi; u_x; u_y; u_z]; in F / 2B it is c6 / (144 h^2)
            // [D P / 3 + sum_i (d_i D) Q_i] with the signs of N
            const double(&x)[4] = u[0], (&v)[4] = u[1], (&z)[4] = u[2];
            const double P[4] = {x[1] * c[5] - x[2] * c[4] + x[3] * c[3], -x[0] * c[5] + x[2] * c[2] - x[3] * c[1],
                                 x[0] * c[4] - x[1] * c[2] + x[3] * c[0], -x[0] * c[3] + x[1] * c[1] - x[2] * c[0]};
            const double Q0[4] = {-ph[1] * c[5] + ph[2] * c[4] - ph[3] * c[3], ph[0] * c[5] - ph[2] * c[2] + ph[3] * c[1],
                                  -ph[0] * c[4] + ph[1] * c[2] - ph[3] * c[0], ph[0] * c[3] - ph[1] * c[1] + ph[2] * c[0]};
            const double Q1[4] = {z[1] * s[5] - z[2] * s[4] + z[3] * s[3], -z[0] * s[5] + z[2] * s[2] - z[3] * s[1],
                                  z[0] * s[4] - z[1] * s[2] + z[3] * s[0], -z[0] * s[3] + z[1] * s[1] - z[2] * s[0]};
            const double Q2[4] = {-v[1] * s[5] + v[2] * s[4] - v[3] * s[3], v[0] * s[5] - v[2] * s[2] + v[3] * s[1],
                                  -v[0] * s[4] + v[1] * s[2] - v[3] * s[0], v[0] * s[3] - v[1] * s[1] + v[2] * s[0]};
            const double d0 = ::fma(kM, dot4(Q1, M[0]) + dot4(Q2, M[1]), dot4(Q0, N[0]));
            const double d1 = ::fma(kM, dot4(Q0, M[0]) + dot4(Q2, M[2]), dot4(Q1, N[1]));
            const double d2 = ::fma(kM, dot4(Q0, M[1]) + dot4(Q1, M[2]), dot4(Q2, N[2]));
            const double e = p.c6b * D * (1.0 / 3.0), e0 = p.c6b * d0, e1 = p.c6b * d1, e2 = p.c6b * d2;
#pragma unroll
            for (int A = 0; A < 4; ++A) H[A] += e * P[A] + e0 * Q0[A] + e1 * Q1[A] + e2 * Q2[A];
            dens[4] = D * D;
        }
    }
    const double hp = dot4(H, ph);
#pragma unroll
    for (int A = 0; A < 4; ++A) F[A] = ::fma(hp, ph[A], -H[A]);
}

// A warp's column of the lattice.
struct Column {
    int y0, z0;  // first interior site
};
template <int TZ> __device__ __forceinline__ Column column_at(const F64Params &p, int col)
{
    const int cy = col / p.nzt;
    return Column{2 + cy * ColumnShape<TZ>::TY, 2 + (col - cy * p.nzt) * TZ};
}

// The correction of a mispredicted arrest decision at the sites of units
// [u0, u1), which this warp updated.
template <int TZ>
__device__ __forceinline__ void correct_sites(const F64Params &p, int cur, int fix, int u0, int u1, int ly, int lz)
{
    const dvec4 *vo = cur ? p.vel[1] : p.vel[0], *fo = cur ? p.phi[1] : p.phi[0];
    dvec4 *vn = cur ? p.vel[0] : p.vel[1], *fn = cur ? p.phi[0] : p.phi[1];
    const size_t sx = (size_t)p.n1 * p.n2;
    for (int us = u0; us < u1;) {
        const int col = us / p.nix, x = us - col * p.nix, len = min(u1 - us, p.nix - x);
        us += len;
        const Column c = column_at<TZ>(p, col);
        const int y = c.y0 + ly, z = c.z0 + lz;
        if (y > p.n1 - 3 || z > p.n2 - 3) continue;
        size_t s = (size_t)(2 + x) * sx + (size_t)y * p.n2 + z;
        for (int i = 0; i < len; ++i, s += sx) {
            dvec4 v, f;
            arrest_fix_site(ldcg4(vn + s), ldcg4(vo + s), ldcg4(fo + s), (double)fix, p.dt, v, f);
            store4<double>(vn + s, v);
            store4<double>(fn + s, f);
        }
    }
}

__device__ __forceinline__ void st_release_s32(int *p, int v)
{
    asm volatile("st.release.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ int ld_acquire_s32(const int *p)
{
    int v;
    asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
// Polls until f() or the wait limit; whether f() came true.
template <typename F> __device__ __forceinline__ bool wait_until(F f)
{
    if (f()) return true;
    const unsigned long long t0 = global_ns();
    do {
        if (f()) return true;
    } while (global_ns() - t0 < kWaitLimitNs);
    return false;
}

template <bool EXT, int TZ>
__global__ void __launch_bounds__(32 * kMaxWarps, 1) k_step_f64(const __grid_constant__ F64Params p)
{
    using S = ColumnShape<TZ>;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    StepSmem64 &sm = *reinterpret_cast<StepSmem64 *>(smem_raw);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, warps = blockDim.x >> 5;
    WarpSmem<TZ> &ws = reinterpret_cast<WarpSmem<TZ> *>(smem_raw + sizeof(StepSmem64))[warp];
    const int ly = lane / TZ, lz = lane % TZ;
    int cur = __ldcg(&p.ctrl->cur);
    long long steps0 = tid == 0 ? ld_acquire_s64(&p.ctrl->steps) : 0;
    for (int step = 1;; ++step, cur ^= 1) {
        const int pred = p.mode == MODE_ARRESTED ? __ldcg(&p.ctrl->pred) : 0;
        const dvec4 *phi = cur ? p.phi[1] : p.phi[0], *vin = cur ? p.vel[1] : p.vel[0];
        dvec4 *phi_out = cur ? p.phi[0] : p.phi[1], *vel_out = cur ? p.vel[0] : p.vel[1];
        const bool use_v = !pred;
        const size_t sx = (size_t)p.n1 * p.n2;
        // this warp's units, a contiguous range
        const int wid = blockIdx.x * warps + warp, u0 = p.start[wid], u1 = p.start[wid + 1];
        double acc[kSums64];
#pragma unroll
        for (int q = 0; q < kSums64; ++q) acc[q] = 0.0;
        long long mx = 0;  // bits of max |F / 2B|^2

        for (int us = u0; us < u1;) {
            const int col = us / p.nix, xs = 2 + (us - col * p.nix), xe = 2 + min(u1 - col * p.nix, p.nix);
            us += xe - xs;
            const Column c = column_at<TZ>(p, col);
            const int y = c.y0 + ly, z = c.z0 + lz;
            const bool valid = y <= p.n1 - 3 && z <= p.n2 - 3;
            // this lane's copies of a haloed plane: byte offsets in the plane
            // (sites outside the lattice are not read; only lanes that are not
            // valid would use them)
            int off[S::COPIES];
#pragma unroll
            for (int j = 0; j < S::COPIES; ++j) {
                const int i = lane + 32 * j, site = i >> 1, ry = site / S::RZ, rz = site - ry * S::RZ;
                const int gy = c.y0 - 2 + ry, gz = c.z0 - 2 + rz;
                off[j] = site < S::SITES && gy < p.n1 && gz < p.n2 ? (gy * p.n2 + gz) * 2 + (i & 1) : -1;
            }
            auto fetch = [&](int x) {
                const double2 *src = reinterpret_cast<const double2 *>(phi + (size_t)x * sx);
                const uint32_t dst = smem_u32(&ws.plane[x % kPlaneSlots][0]) + 16 * lane;
#pragma unroll
                for (int j = 0; j < S::COPIES; ++j)
                    if (off[j] >= 0)
                        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 512 * j),
                                     "l"(__cvta_generic_to_global(src + off[j]))
                                     : "memory");
                asm volatile("cp.async.commit_group;" ::: "memory");
            };
            int next = xs - 2;  // the next plane to fetch
            while (next < min(xs + 2, xe + 2)) fetch(next++);
            dvec4 r[5] = {};  // phi at x - 2 .. x + 2 of the centre x = q - 2
            const size_t col_site = (size_t)y * p.n2 + z;
            for (int q = xs - 2; q < xe + 2; ++q) {
                // plane q lands: the planes fetched after it may still be on their way
                switch (next - 1 - q) {
                case 0: asm volatile("cp.async.wait_group 0;" ::: "memory"); break;
                case 1: asm volatile("cp.async.wait_group 1;" ::: "memory"); break;
                case 2: asm volatile("cp.async.wait_group 2;" ::: "memory"); break;
                default: asm volatile("cp.async.wait_group 3;" ::: "memory"); break;
                }
                __syncwarp();
                // the next plane's slot is free when its plane of four before has
                // been a centre, or, at the start of a run, has arrived
                if (next < xe + 2 && q >= (next - 4 < xs ? next - 3 : next - 1)) fetch(next++);
                const int x = q - 2;
                const bool centre = x >= xs;
                dvec4 v = {0.0, 0.0, 0.0, 0.0};
                if (centre && use_v && valid) v = ldcg4(vin + (size_t)x * sx + col_site);
                {
                    // ---- plane q arrives: u_y (with its z-halo) and u_z
                    const dvec4 *P = &ws.plane[q % kPlaneSlots][0];
                    auto at = [&](int ry, int rz) { return lds(P + ry * S::RZ + rz); };
                    const dvec4 c4 = at(ly + 2, lz + 2);
                    r[0] = r[1], r[1] = r[2], r[2] = r[3], r[3] = r[4], r[4] = c4;
                    store4<double>(&ws.uy[q % 5][ly][lz + 2],
                                   first(at(ly, lz + 2), at(ly + 1, lz + 2), at(ly + 3, lz + 2), at(ly + 4, lz + 2)));
                    store4<double>(&ws.uz[q % 5][lane],
                                   first(at(ly + 2, lz), at(ly + 2, lz + 1), at(ly + 2, lz + 3), at(ly + 2, lz + 4)));
#pragma unroll
                    for (int j = 0; j < S::HALO; ++j) {
                        const int i = lane + 32 * j, hy = i >> 4, hc = (i >> 2) & 3, k = i & 3;
                        const int hz = hc < 2 ? hc : TZ + hc;
                        const double *b = reinterpret_cast<const double *>(P + hy * S::RZ + hz) + k;
                        reinterpret_cast<double *>(&ws.uy[q % 5][hy][hz])[k] =
                            first(b[0], b[4 * S::RZ], b[12 * S::RZ], b[16 * S::RZ]);
                    }
                }
                if (!centre) continue;  // (the same for the whole warp)
                // ---- centre x: u_y's halo was written two planes ago
                const dvec4 *P = &ws.plane[x % kPlaneSlots][0];
                auto at = [&](int ry, int rz) { return lds(P + ry * S::RZ + rz); };
                double ph[4], u[3][4], N[3][4], M[3][4], F[4], dens[5];
                vec(ph, r[2]);
                first(u[0], r[0], r[1], r[3], r[4]);
                second(N[0], r[0], r[1], r[2], r[3], r[4]);
                second(N[1], at(ly, lz + 2), at(ly + 1, lz + 2), r[2], at(ly + 3, lz + 2), at(ly + 4, lz + 2));
                second(N[2], at(ly + 2, lz), at(ly + 2, lz + 1), r[2], at(ly + 2, lz + 3), at(ly + 2, lz + 4));
                const int s0 = x % 5, m2 = (x + 3) % 5, m1 = (x + 4) % 5, p1 = (x + 1) % 5, p2 = (x + 2) % 5;
                vec(u[1], lds(&ws.uy[s0][ly][lz + 2]));
                vec(u[2], lds(&ws.uz[s0][lane]));
                first(M[0], lds(&ws.uy[m2][ly][lz + 2]), lds(&ws.uy[m1][ly][lz + 2]), lds(&ws.uy[p1][ly][lz + 2]),
                      lds(&ws.uy[p2][ly][lz + 2]));
                first(M[1], lds(&ws.uz[m2][lane]), lds(&ws.uz[m1][lane]), lds(&ws.uz[p1][lane]), lds(&ws.uz[p2][lane]));
                first(M[2], lds(&ws.uy[s0][ly][lz]), lds(&ws.uy[s0][ly][lz + 1]), lds(&ws.uy[s0][ly][lz + 3]),
                      lds(&ws.uy[s0][ly][lz + 4]));
                step_site<EXT>(p, ph, u, N, M, F, dens);
                v = dvec4{::fma(p.dt2, F[0], v.x), ::fma(p.dt2, F[1], v.y), ::fma(p.dt2, F[2], v.z),
                          ::fma(p.dt2, F[3], v.w)};
                const double t[4] = {::fma(p.dt, v.x, ph[0]), ::fma(p.dt, v.y, ph[1]), ::fma(p.dt, v.z, ph[2]),
                                     ::fma(p.dt, v.w, ph[3])};
                const double rn = rsqrt(dot4(t, t));  // within an ulp of 1/sqrt, without its division
                if (valid) {
                    const size_t site = (size_t)x * sx + col_site;
                    store4<double>(vel_out + site, v);
                    store4<double>(phi_out + site, dvec4{t[0] * rn, t[1] * rn, t[2] * rn, t[3] * rn});
                    const double f2 = dot4(F, F);
#pragma unroll
                    for (int i = 0; i < 4; ++i) acc[i] += dens[i];
                    acc[4] += f2;
                    // (f2 >= 0: ordered as its bits; NaN, above infinity's, is passed over)
                    const long long fb = __double_as_longlong(f2);
                    if (fb <= 0x7ff0000000000000LL) mx = max(mx, fb);
                    if constexpr (EXT) acc[6] += dens[4];
                }
            }
            __syncwarp();  // the run's planes are done with before the next run's first arrives
        }

        // ---- sums: each warp's quantities over its lanes, then the CTA's warps
        {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            // three exchanges leave each lane one of the eight quantities
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) {
                const bool up = lane & o;
#pragma unroll
                for (int q = 0; q < o; ++q) {
                    const double keep = up ? acc[q + o] : acc[q], send = up ? acc[q] : acc[q + o];
                    acc[q] = keep + __shfl_xor_sync(0xffffffffu, send, o);
                }
            }
            double v = acc[0];  // of quantity lane & 7
            v += __shfl_xor_sync(0xffffffffu, v, 8);
            v += __shfl_xor_sync(0xffffffffu, v, 16);
            if (lane < kSums64) sm.red[warp][lane] = lane == 5 ? __longlong_as_double(mx) : v;
        }
        __syncthreads();
        if (tid < kSums64) {
            double v = sm.red[0][tid];
            for (int w = 1; w < warps; ++w) v = tid == 5 ? fmax(v, sm.red[w][tid]) : v + sm.red[w][tid];
            p.parts[(size_t)blockIdx.x * kPartialDoubles + tid] = v;
            __threadfence();
        }
        __syncthreads();
        if (tid == 0) sm.last = atomicAdd(&p.ctrl->done, 1u) == gridDim.x - 1;
        __syncthreads();
        if (sm.last) {
            // ---- the last CTA sums the records, 4 threads per warp and quantity;
            // thread 0 fetches the control fields it needs meanwhile
            __threadfence();
            StepControl ctl;
            if (tid == 0) ctl = load_control(p.ctrl);
            const int q = tid & 7;
            double v = 0.0;
            for (int i0 = tid >> 3; i0 < (int)gridDim.x; i0 += 32 * warps) {
                double t[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int i = i0 + 4 * warps * j;
                    t[j] = i < (int)gridDim.x ? __ldcg(p.parts + (size_t)i * kPartialDoubles + q) : 0.0;
                }
                if (q == 5) {
#pragma unroll
                    for (int j = 0; j < 8; ++j) v = fmax(v, t[j]);
                } else {
                    v += ((t[0] + t[1]) + (t[2] + t[3])) + ((t[4] + t[5]) + (t[6] + t[7]));
                }
            }
#pragma unroll
            for (int o = 8; o <= 16; o <<= 1) {
                const double t = __shfl_xor_sync(0xffffffffu, v, o);
                v = q == 5 ? fmax(v, t) : v + t;
            }
            if (lane < kSums64) sm.red[warp][lane] = v;
            __syncthreads();
            if (tid < kSums64) {
                double t = sm.red[0][tid];
                for (int w = 1; w < warps; ++w) t = tid == 5 ? fmax(t, sm.red[w][tid]) : t + sm.red[w][tid];
                sm.tot[tid] = t * p.scale[tid];
            }
            __syncthreads();
            if (tid == 0 || tid == 32) {
                // thread 0 decides and publishes, thread 32 forms the report
                const double *t = sm.tot;
                const double nsites = (double)(p.n0 - 4) * (double)(p.n1 - 4) * (double)(p.n2 - 4);
                const double tot[kPartialDoubles] = {t[0], t[1], t[2], t[3], t[4], t[5], nsites, t[6]};
                if (p.slab_rec) {
                    // one x-slab of a larger lattice: the arrest decision needs
                    // every slab's sums, so this step only leaves its record
                    if (tid == 0) {
#pragma unroll
                        for (int i = 0; i < kPartialDoubles; ++i) p.slab_rec[i] = tot[i];
                        p.ctrl->done = 0;
                    }
                } else if (tid == 0) {
                    decide_step(p.ctrl, ctl, tot, p.h3, p.mode, pred);
                } else {
                    report_step(p.ctrl, tot, p.h3);
                }
            }
        }
        const bool more = step < p.steps;
        if (!p.fuse_fix && !more) return;
        // ---- every CTA (all resident: a cooperative launch) waits, bounded, for
        // the decision and corrects its own sites when the prediction was wrong
        if (tid == 0) {
            sm.fix = wait_until([&] { return ld_acquire_s64(&p.ctrl->steps) != steps0; }) ? __ldcg(&p.ctrl->fix) : 2;
            ++steps0;
        }
        __syncthreads();
        const int fix = sm.fix;
        if (fix == 2) {
            if (tid == 0) atomicExch(&p.ctrl->status, (int)DEV_TIMEOUT);
            return;
        }
        if (fix != 0) correct_sites<TZ>(p, cur, fix, u0, u1, ly, lz);
        if (!more) return;
        if (fix != 0) {
            // the next step reads its neighbours' corrected sites: the last CTA to
            // arrive clears the correction, which the others wait for
            __syncthreads();
            if (tid == 0) {
                // released before the arrival and acquired after it: the last CTA's
                // release below then covers every CTA's corrected sites
                __threadfence();
                const bool last = atomicAdd(&p.ctrl->done, 1u) == gridDim.x - 1;
                __threadfence();
                if (last) {
                    p.ctrl->done = 0;
                    st_release_s32(&p.ctrl->fix, 0);
                } else if (!wait_until([&] { return ld_acquire_s32(&p.ctrl->fix) == 0; })) {
                    sm.fix = 2;
                    atomicExch(&p.ctrl->status, (int)DEV_TIMEOUT);
                }
            }
            __syncthreads();
            if (sm.fix == 2) return;
        }
    }
}

// Shares of `units` (columns of nix planes) for nw warps: contiguous ranges
// whose largest cost is as small as a greedy cover allows, a run costing its
// planes and half a plane for its ends (four planes of which only u_y and u_z
// are formed).  Returns twice that cost; fills start[0 .. nw].
static int share_units(int units, int nix, int nw, int *start)
{
    auto cover = [&](int cap) {  // warps used, or nw + 1
        int pos = 0, w = 0;
        while (pos < units) {
            if (w == nw) return nw + 1;
            start[w++] = pos;
            for (int budget = cap, first = 1; pos < units; first = 0) {
                const int col_end = (pos / nix + 1) * nix;
                int take = (budget - 1) / 2;
                if (take < 1) {
                    if (!first) break;
                    take = 1;
                }
                take = std::min(take, col_end - pos);
                pos += take;
                budget -= 2 * take + 1;
                if (pos < col_end) break;
            }
        }
        for (int i = w; i <= nw; ++i) start[i] = units;
        return w;
    };
    // (a warp's share and one run per column it may touch)
    int lo = 1, hi = 2 * ((units + nw - 1) / nw) + (units / nix / nw + 2) + 2;
    while (cover(hi) > nw) hi *= 2;
    while (lo < hi) {
        const int mid = lo + (hi - lo) / 2;
        if (cover(mid) <= nw) hi = mid;
        else lo = mid + 1;
    }
    (void)cover(hi);
    return hi;
}

// Warps per CTA (one CTA per SM) and their shares: 8, 6 or 4 warps, whichever
// leaves the busiest SM less to do.  The FP64 pipe is the SM's, so a warp's
// share costs the warps on its SM times its planes.  Odd counts load the SM's
// four schedulers unevenly (5 warps: 9% slower on 128^3); 6 and 4 warps keep
// the pipe 0.7% and 2% less busy than 8 (128^3: 1205, 1219 and 1196 us), but
// 48^3, 4.8 units per warp of 4, took 84.7 us with 4 and 87.2 with 8 (even
// shares; 78.5 with 4 and these).
// Remembered for the last geometry of the thread.
static int plan_warps(long long units, int nix, int sms, int *start)
{
    static thread_local long long key_units = -1;
    static thread_local int key_nix = 0, key_sms = 0, warps = 0, plan[kMaxShare + 1];
    if (units != key_units || nix != key_nix || sms != key_sms) {
        static const struct {
            int warps;
            double busy;
        } kChoices[] = {{8, 1.0}, {6, 0.993}, {4, 0.98}};
        double best = -1.0;
        int trial[kMaxShare + 1];
        for (const auto &c : kChoices) {
            const double cost = share_units((int)units, nix, c.warps * sms, trial) * c.warps / c.busy;
            if (best < 0.0 || cost < best) {
                best = cost;
                warps = c.warps;
                memcpy(plan, trial, (size_t)(c.warps * sms + 1) * sizeof(int));
            }
        }
        key_units = units, key_nix = nix, key_sms = sms;
    }
    memcpy(start, plan, (size_t)(warps * sms + 1) * sizeof(int));
    return warps;
}

template <bool EXT, int TZ> static cudaError_t launch_shape(F64Params &p, int steps, int sms, cudaStream_t s)
{
    using S = ColumnShape<TZ>;
    p.nzt = (p.n2 - 4 + TZ - 1) / TZ;
    p.units = (long long)((p.n1 - 4 + S::TY - 1) / S::TY) * p.nzt * p.nix;
    if (p.units > 0x7fffffffLL) return cudaErrorInvalidValue;
    constexpr int smem_max = (int)(sizeof(StepSmem64) + kMaxWarps * sizeof(WarpSmem<TZ>));
    static_assert(smem_max <= 227 * 1024, "one CTA per SM");
    sms = std::min(sms, kMaxShare / kMaxWarps);
    const int warps = plan_warps(p.units, p.nix, sms, p.start);
    int used = warps * sms;  // warps with units
    while (used > 1 && p.start[used - 1] == p.units) --used;
    cudaError_t e = cudaFuncSetAttribute(k_step_f64<EXT, TZ>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = p.fuse_fix || p.steps > 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((used + warps - 1) / warps));
    cfg.blockDim = dim3(32 * warps);
    cfg.dynamicSmemBytes = sizeof(StepSmem64) + warps * sizeof(WarpSmem<TZ>);
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    for (int left = steps; left > 0; left -= p.steps) {
        p.steps = std::min(p.steps, left);
        e = cudaLaunchKernelEx(&cfg, k_step_f64<EXT, TZ>, p);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// SMs that kernels on stream s run on: a green context's share, else the
// device's.  A cooperative launch of more CTAs than fit on them is refused.
static cudaError_t stream_sms(cudaStream_t s, int *sms)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    static const auto entry = [](const char *name) -> void * {
        void *fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        return cudaGetDriverEntryPointByVersion(name, &fn, 12040, cudaEnableDefault, &q) == cudaSuccess &&
                       q == cudaDriverEntryPointSuccess
                   ? fn
                   : nullptr;
    };
    static const auto green_of = reinterpret_cast<PFN_cuStreamGetGreenCtx_v12040>(entry("cuStreamGetGreenCtx"));
    static const auto resource =
        reinterpret_cast<PFN_cuGreenCtxGetDevResource_v12040>(entry("cuGreenCtxGetDevResource"));
    CUgreenCtx green = nullptr;
    CUdevResource r;
    if (green_of && resource && green_of(s, &green) == CUDA_SUCCESS && green &&
        resource(green, &r, CU_DEV_RESOURCE_TYPE_SM) == CUDA_SUCCESS && r.sm.smCount > 0)
        *sms = std::min(*sms, (int)r.sm.smCount);
    return cudaSuccess;
}

cudaError_t launch_steps_f64(const skyrme_lattice &lat, const FlowArgs &a, int steps, cudaStream_t s)
{
    F64Params p = {};
    for (int i = 0; i < 2; ++i) {
        p.phi[i] = static_cast<dvec4 *>(a.phi[i]);
        p.vel[i] = static_cast<dvec4 *>(a.vel[i]);
    }
    p.ctrl = static_cast<Ctrl *>(a.ctrl);
    p.parts = a.step_parts;
    p.slab_rec = a.slab_rec;
    p.n0 = a.n[0], p.n1 = a.n[1], p.n2 = a.n[2];
    p.nix = p.n0 - 4;
    p.mode = a.mode;
    p.fuse_fix = a.mode == SKYRME_ARRESTED && !a.slab_rec;
    // A launch runs as many steps as update kLaunchSites sites, but kLaunchSteps at
    // most (a step of the smallest lattices is all fixed costs, 20 us): 2 to 5 ms.
    // More save nothing, and other streams' kernels start between launches.
    const double sites = (double)(p.n0 - 4) * (p.n1 - 4) * (p.n2 - 4);
    const double most = std::min((double)kLaunchSteps, kLaunchSites / sites);
    p.steps = a.slab_rec ? 1 : (int)std::max(1.0, std::min((double)steps, most));
    const double k1 = 1.0 / (12.0 * a.h), k2 = k1 * k1, B = 12.0 * k2 * k2;
    p.dt = a.dt;
    p.dt2 = 2.0 * a.dt * B;
    p.K144 = 144.0 * a.h * a.h;
    p.bm2 = a.m * a.m / B;
    p.my2 = a.my * a.my, p.mz2 = a.mz * a.mz, p.mw2 = a.mw * a.mw;
    p.m2x2 = 2.0 * a.m * a.m;
    p.bmy2 = p.my2 / B, p.bmz2 = p.mz2 / B, p.bmw2 = p.mw2 / B;
    p.c6b = a.c6 * k2;
    const bool ext = lattice_extended(lat);
    const double scale[kSums64] = {k2, k2 * k2, ext ? 1.0 : p.m2x2, -0.050660591821168885 * k2 * k1,  // -1/(2 pi^2)
                                   4.0 * B * B, 4.0 * B * B, a.c6 * k2 * k2 * k2, 0.0};
    for (int q = 0; q < kSums64; ++q) p.scale[q] = scale[q];
    p.h3 = a.h * a.h * a.h;
    int sms = 0;
    const cudaError_t e = stream_sms(s, &sms);
    if (e != cudaSuccess) return e;
    // the column that pads the lattice less (4 x 8 forms twice the halo: 1%)
    const long long iy = p.n1 - 4, iz = p.n2 - 4;
    const long long pad16 = (iy + 1) / 2 * 2 * ((iz + 15) / 16 * 16), pad8 = (iy + 3) / 4 * 4 * ((iz + 7) / 8 * 8);
    if (101 * pad8 < 100 * pad16)
        return ext ? launch_shape<true, 8>(p, steps, sms, s) : launch_shape<false, 8>(p, steps, sms, s);
    return ext ? launch_shape<true, 16>(p, steps, sms, s) : launch_shape<false, 16>(p, steps, sms, s);
}

}  // namespace skyrme
