// energy.cu -- the energy, baryon-number and virial reduction of the current
// field (Section 2.1, Eq. "SkyrmeEnergy_phi"; Eq. "B0_components"; the Section
// 7.8 densities), in either precision.
//
// The densities need first derivatives only (13 sites per site), so this is a
// pass of its own rather than the step's arithmetic: no second or mixed
// derivatives and no force.
//
// FP32 (k_energy_tma): a CTA streams chunks of (y, z) tiles of 512 sites along
// x.  A producer warp brings the haloed planes into an 8-slot shared-memory
// ring by TMA; eight consumer warps keep the five field values of their
// x-stencils in registers and read y and z neighbours from the ring, two rows
// per thread, so that a site costs 7 shared loads instead of 9.  Packed pair
// arithmetic with the stencils' 1/h factors left out (they scale the sums in
// FP64), every density added error-free (two-sum) and the block sums in
// double-float, so no FP32 reduction error enters.
//   Bound: shared-memory wavefronts (34 of 128 bytes per 32 sites) and issue
//   (about 110 instructions per 32 sites).  256^3: 103 us, 272 MB
//   from DRAM (625 us in the step's tile kernel, 135 us with the neighbours
//   read through L1, which waits for DRAM every plane).
// FP64 (k_energy): bound by the FP64 pipe (about 105 instructions per site), so
// threads read their neighbours through L1, one site each.
// Persistent CTAs walk the (tile, chunk) items and leave one partial record
// each; the last CTA sums the records in a fixed order.
#include <cuda_runtime.h>

#include <algorithm>

#include "packed_f32.cuh"
#include "skyrme_device.cuh"
#include "skyrme_internal.h"
#include "tma.cuh"

namespace skyrme {

constexpr int kEnergyThreads = 256;
constexpr int kEnergySums = 5;  // e2, e4, potential, det, e6

template <typename T> struct EnergyParams {
    const vec4_t<T> *phi[2];
    Ctrl *ctrl;
    double *parts;
    int n0, n1, n2;
    int nzt, ncol, chunk, items;  // z tiles, (y, z) tiles, planes per item, items in all
    T m2, my2, mz2, mw2;
    double scale[kEnergySums];  // of the sums, 1/h factors and h^3 included
};

// The unscaled densities of one site: tr A and the quartic form of
// A_ij = u_i.u_j (u_i = 12h d_i phi), the potential (1 - phi^0 for the
// standard model, the whole potential with the Section 7.8 terms) and
// D = det[phi, u_x, u_y, u_z].
template <typename T> struct SiteDens {
    T e2, e4, e0, det;
};

// tr A^2 - A_ij A_ij over 2 as the sum of the principal 2x2 minors
template <typename T>
__device__ __forceinline__ T quartic(T xx, T yy, T zz, T xy, T xz, T yz)
{
    return xx * (yy + zz) + yy * zz - (xy * xy + xz * xz + yz * yz);
}

template <typename T, bool EXT>
__device__ __forceinline__ T potential(const T ph[4], const EnergyParams<T> &p)
{
    const T u = one_minus_phi0<T>(ph);
    if constexpr (!EXT) return u;
    const T u2 = u * u;
    return T(2) * p.m2 * u + p.my2 * one_minus_phi0_sq<T>(ph, u) + p.mz2 * u2 +
           T(0.5) * p.mw2 * u2 * u2;
}

template <bool EXT>
__device__ __forceinline__ SiteDens<float> site_densities(const float4 &c, const P4 &ux,
                                                          const P4 &uy, const P4 &uz,
                                                          const EnergyParams<float> &p)
{
    const P4 f = ld4(c);
    const float xx = dot(ux, ux), yy = dot(uy, uy), zz = dot(uz, uz);
    const float xy = dot(ux, uy), xz = dot(ux, uz), yz = dot(uy, uz);
    SiteDens<float> r;
    r.e2 = xx + yy + zz;
    r.e4 = quartic(xx, yy, zz, xy, xz, yz);
    const float ph[4] = {c.x, c.y, c.z, c.w};
    r.e0 = potential<float, EXT>(ph, p);
    // 2x2 minors of the rows (phi, u_x) and (u_y, u_z)
    const float s01 = f.a.x * ux.a.y - ux.a.x * f.a.y;
    const float2 s23 = __ffma2_rn(bc(-ux.a.x), f.b, __fmul2_rn(bc(f.a.x), ux.b));    // s02, s03
    const float2 s45 = __ffma2_rn(bc(-ux.a.y), f.b, __fmul2_rn(bc(f.a.y), ux.b));    // s12, s13
    const float s6 = f.b.x * ux.b.y - ux.b.x * f.b.y;                                // s23
    const float q01 = uy.a.x * uz.a.y - uz.a.x * uy.a.y;
    const float2 q23 = __ffma2_rn(bc(-uz.a.x), uy.b, __fmul2_rn(bc(uy.a.x), uz.b));
    const float2 q45 = __ffma2_rn(bc(-uz.a.y), uy.b, __fmul2_rn(bc(uy.a.y), uz.b));
    const float q6 = uy.b.x * uz.b.y - uz.b.x * uy.b.y;
    r.det = s01 * q6 - s23.x * q45.y + s23.y * q45.x + s45.x * q23.y - s45.y * q23.x + s6 * q01;
    return r;
}

template <bool EXT>
__device__ __forceinline__ SiteDens<double> site_densities(const dvec4 &c, const dvec4 &ux,
                                                           const dvec4 &uy, const dvec4 &uz,
                                                           const EnergyParams<double> &p)
{
    auto dp = [](const dvec4 &a, const dvec4 &b) { return a.x * b.x + a.y * b.y + a.z * b.z + a.w * b.w; };
    const double xx = dp(ux, ux), yy = dp(uy, uy), zz = dp(uz, uz);
    const double xy = dp(ux, uy), xz = dp(ux, uz), yz = dp(uy, uz);
    SiteDens<double> r;
    r.e2 = xx + yy + zz;
    r.e4 = quartic(xx, yy, zz, xy, xz, yz);
    const double ph[4] = {c.x, c.y, c.z, c.w};
    r.e0 = potential<double, EXT>(ph, p);
    r.det = (c.x * ux.y - ux.x * c.y) * (uy.z * uz.w - uz.z * uy.w) -
            (c.x * ux.z - ux.x * c.z) * (uy.y * uz.w - uz.y * uy.w) +
            (c.x * ux.w - ux.x * c.w) * (uy.y * uz.z - uz.y * uy.z) +
            (c.y * ux.z - ux.y * c.z) * (uy.x * uz.w - uz.x * uy.w) -
            (c.y * ux.w - ux.y * c.w) * (uy.x * uz.z - uz.x * uy.z) +
            (c.z * ux.w - ux.z * c.w) * (uy.x * uz.y - uz.x * uy.y);
    return r;
}

// u = 8 (p1 - m1) - (p2 - m2) = 12h d phi
__device__ __forceinline__ P4 first_difference(const float4 &m2, const float4 &m1, const float4 &p1,
                                               const float4 &p2)
{
    return fd1u(ld4(m2), ld4(m1), ld4(p1), ld4(p2), kW8());
}
__device__ __forceinline__ dvec4 first_difference(const dvec4 &m2, const dvec4 &m1, const dvec4 &p1,
                                                  const dvec4 &p2)
{
    return dvec4{::fma(8.0, p1.x - m1.x, m2.x - p2.x), ::fma(8.0, p1.y - m1.y, m2.y - p2.y),
                 ::fma(8.0, p1.z - m1.z, m2.z - p2.z), ::fma(8.0, p1.w - m1.w, m2.w - p2.w)};
}

// A thread's running sums
template <typename T> struct EnergyAcc;
template <> struct EnergyAcc<double> {
    double s[kEnergySums] = {0, 0, 0, 0, 0};
    template <bool EXT> __device__ __forceinline__ void add(const SiteDens<double> &d)
    {
        s[0] += d.e2, s[1] += d.e4, s[2] += d.e0, s[3] += d.det;
        if constexpr (EXT) s[4] = ::fma(d.det, d.det, s[4]);
    }
};
template <> struct EnergyAcc<float> {
    float2 s24 = {0.f, 0.f}, c24 = {0.f, 0.f}, s0b = {0.f, 0.f}, c0b = {0.f, 0.f};
    float s6 = 0.f, c6 = 0.f;
    template <bool EXT> __device__ __forceinline__ void add(const SiteDens<float> &d)
    {
        two_sum_acc(s24, c24, make_float2(d.e2, d.e4));
        two_sum_acc(s0b, c0b, make_float2(d.e0, d.det));
        if constexpr (EXT) two_sum_acc1(s6, c6, d.det * d.det);
    }
};

// Block sums in a fixed order, one warp per quantity: each lane its 8 entries
// as a pairwise tree, then a butterfly; tot[] of warp 0 holds the totals.
// buf: kEnergySums * kEnergyThreads entries.
__device__ __forceinline__ void block_totals(const EnergyAcc<double> &a, double *buf, int tid)
{
#pragma unroll
    for (int q = 0; q < kEnergySums; ++q) buf[q * kEnergyThreads + tid] = a.s[q];
    __syncthreads();
    const int lane = tid & 31, warp = tid >> 5;
    double r = 0.0;
    if (warp < kEnergySums) {
        const double *c = buf + warp * kEnergyThreads + lane;
        r = ((c[0] + c[32]) + (c[64] + c[96])) + ((c[128] + c[160]) + (c[192] + c[224]));
        r = warp_sum(r);
    }
    __syncthreads();
    if (warp < kEnergySums && lane == 0) buf[warp] = r;
    __syncthreads();
}
__device__ __forceinline__ void block_totals(const EnergyAcc<float> &a, double *buf, int tid)
{
    DF *d = reinterpret_cast<DF *>(buf);
    const float s[kEnergySums] = {a.s24.x, a.s24.y, a.s0b.x, a.s0b.y, a.s6};
    const float c[kEnergySums] = {a.c24.x, a.c24.y, a.c0b.x, a.c0b.y, a.c6};
    if (tid < kEnergyThreads) {  // not the producer warp
#pragma unroll
        for (int q = 0; q < kEnergySums; ++q) {
            DF v;
            two_sum(s[q], c[q], v.hi, v.lo);
            d[q * kEnergyThreads + tid] = v;
        }
    }
    __syncthreads();
    const int lane = tid & 31, warp = tid >> 5;
    DF r = {0.f, 0.f};
    if (warp < kEnergySums) {
        DF x[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) x[k] = d[warp * kEnergyThreads + lane + 32 * k];
        df_tree<8>(x);
        r = x[0];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) r = df_add(r, df_shfl_xor(r, o));
    }
    __syncthreads();
    if (warp < kEnergySums && lane == 0) buf[warp] = df_value(r);
    __syncthreads();
}

// The CTA's record, and in the last CTA the totals of all records into the
// control block.  buf: the block totals (block_totals).  All the block's
// threads take part; the first five warps sum.
__device__ __forceinline__ void finish_energy(Ctrl *c, double *parts, const double (&scale)[kEnergySums],
                                              double *buf, int *s_last, int tid)
{
    if (tid == 0) {
        double *rec = parts + (size_t)blockIdx.x * kPartialDoubles;
#pragma unroll
        for (int i = 0; i < kEnergySums; ++i) rec[i] = buf[i];
        __threadfence();
        *s_last = atomicAdd(&c->edone, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!*s_last) return;
    __threadfence();
    // warp q sums quantity q of every record, eight loads in flight per lane
    const int lane = tid & 31, warp = tid >> 5;
    if (warp < kEnergySums) {
        double r = 0.0;
        for (int i0 = 0; i0 < (int)gridDim.x; i0 += 256) {
            double v[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int i = i0 + lane + 32 * j;
                v[j] = i < (int)gridDim.x ? __ldcg(parts + (size_t)i * kPartialDoubles + warp) : 0.0;
            }
            r += ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
        }
        r = warp_sum(r);
        // (no sextic term: 0, also where the sum of the squares overflows)
        if (lane == 0) buf[warp] = warp == 4 && scale[4] == 0.0 ? 0.0 : scale[warp] * r;
    }
    __syncthreads();
    if (tid == 0) {
        const double E2 = buf[0], E4 = buf[1], E0 = buf[2], B = buf[3], E6 = buf[4];
        const double E = E2 + E4 + E0 + E6;
        c->energy[0] = E;
        c->energy[1] = E2;
        c->energy[2] = E4;
        c->energy[3] = E0;
        c->energy[4] = B;
        c->energy[5] = -E2 + E4 - 3.0 * E0 + 3.0 * E6;
        c->e6_energy = E6;
        if (!(isfinite(E) && isfinite(B)) && c->status != DEV_TIMEOUT) c->status = DEV_NONFINITE;
        c->edone = 0;
    }
}

// One site per thread, neighbours through L1: FP64 fields, and FP32 fields
// where the driver has no tensor-map encoder.
template <typename T, bool EXT, int TZ>
__global__ void __launch_bounds__(kEnergyThreads, 2) k_energy(const __grid_constant__ EnergyParams<T> p)
{
    constexpr int TY = kEnergyThreads / TZ;
    __shared__ double buf[kEnergySums * kEnergyThreads];
    __shared__ int s_last;
    const int tid = threadIdx.x;
    const vec4_t<T> *__restrict__ phi = __ldcg(&p.ctrl->cur) ? p.phi[1] : p.phi[0];
    const size_t sx = (size_t)p.n1 * p.n2;
    const int sy = p.n2;
    EnergyAcc<T> acc;
    for (int it = blockIdx.x; it < p.items; it += gridDim.x) {
        // columns fastest: CTAs in flight share halo rows in L2
        const int k = it / p.ncol, col = it - k * p.ncol;
        const int y = 2 + (col / p.nzt) * TY + tid / TZ, z = 2 + (col % p.nzt) * TZ + tid % TZ;
        if (y > p.n1 - 3 || z > p.n2 - 3) continue;
        const int xa = 2 + k * p.chunk, xb = min(xa + p.chunk, p.n0 - 2);
        const vec4_t<T> *q = phi + (size_t)xa * sx + (size_t)y * sy + z;  // the centre
        vec4_t<T> m2 = load4<T>(q - 2 * sx), m1 = load4<T>(q - sx), c = load4<T>(q), p1 = load4<T>(q + sx);
#pragma unroll 5
        for (int x = xa; x < xb; ++x) {
            const vec4_t<T> p2 = load4<T>(q + 2 * sx);
            const vec4_t<T> ym2 = load4<T>(q - 2 * sy), ym1 = load4<T>(q - sy);
            const vec4_t<T> yp1 = load4<T>(q + sy), yp2 = load4<T>(q + 2 * sy);
            const vec4_t<T> zm2 = load4<T>(q - 2), zm1 = load4<T>(q - 1);
            const vec4_t<T> zp1 = load4<T>(q + 1), zp2 = load4<T>(q + 2);
            acc.template add<EXT>(site_densities<EXT>(c, first_difference(m2, m1, p1, p2),
                                                      first_difference(ym2, ym1, yp1, yp2),
                                                      first_difference(zm2, zm1, zp1, zp2), p));
            m2 = m1, m1 = c, c = p1, p1 = p2;
            q += sx;
        }
    }
    block_totals(acc, buf, tid);
    finish_energy(p.ctrl, p.parts, p.scale, buf, &s_last, tid);
}

// Shared memory of the streaming kernel
constexpr int kRingSlots = 8;
template <int TZ> struct __align__(128) EnergySmem {
    static constexpr int TY = 512 / TZ;
    float4 plane[kRingSlots][TY + 4][TZ + 4];
    double buf[kEnergySums * kEnergyThreads];
    unsigned long long full[kRingSlots], empty[kRingSlots];
    int last, flag;
};
struct PlaneMaps {
    CUtensorMap map[2];  // haloed planes of phi[0], phi[1]
};

__device__ __forceinline__ void mbar_arrive(unsigned long long *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

template <bool EXT, int TZ>
__global__ void __launch_bounds__(kEnergyThreads + 32, 2)
    k_energy_tma(const __grid_constant__ PlaneMaps maps, const __grid_constant__ EnergyParams<float> p)
{
    using Smem = EnergySmem<TZ>;
    constexpr int TY = Smem::TY;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    Smem &sm = *reinterpret_cast<Smem *>(smem_raw);
    const int tid = threadIdx.x, warp = tid >> 5;
    if (tid == 0) {
        for (int s = 0; s < kRingSlots; ++s) {
            mbar_init(&sm.full[s], 1);
            mbar_init(&sm.empty[s], kEnergyThreads / 32);
        }
        mbar_fence_init();
        sm.flag = 0;
    }
    __syncthreads();
    EnergyAcc<float> acc;
    if (warp == kEnergyThreads / 32) {
        // ---- producer: every plane of this CTA's items, in order
        if ((tid & 31) == 0) {
            const CUtensorMap *map = &maps.map[__ldcg(&p.ctrl->cur)];
            uint32_t g = 0;
            bool ok = true;
            for (int it = blockIdx.x; it < p.items && ok; it += gridDim.x) {
                const int k = it / p.ncol, col = it - k * p.ncol;
                const int y0 = (col / p.nzt) * TY, z0 = (col % p.nzt) * TZ;  // of the halo
                const int xa = 2 + k * p.chunk, xb = min(xa + p.chunk, p.n0 - 2);
                for (int x = xa - 2; x < xb + 2; ++x, ++g) {
                    const int s = g % kRingSlots;
                    // the slot's previous plane has been read by every warp
                    if (g >= kRingSlots && !mbar_wait_flag(&sm.empty[s], (g / kRingSlots - 1) & 1u, &sm.flag)) {
                        ok = false;
                        break;
                    }
                    // those reads (generic proxy) before the copy's writes (async proxy)
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    mbar_expect_tx(&sm.full[s], (TY + 4) * (TZ + 4) * 16);
                    tma_plane(&sm.plane[s][0][0], map, &sm.full[s], 4 * z0, y0, x);
                }
            }
            if (!ok) *(volatile int *)&sm.flag = 1;
            // copies in flight land before the CTA ends (the consumers have
            // waited for every plane unless a wait failed)
            for (uint32_t q = g > kRingSlots ? g - kRingSlots : 0; q < g; ++q)
                (void)mbar_wait(&sm.full[q % kRingSlots], (q / kRingSlots) & 1u, ok ? kWaitLimitNs : 50000000ull);
        }
    } else {
        const int r0 = 2 * (tid / TZ), tz = tid % TZ;
        uint32_t g = 0;
        for (int it = blockIdx.x; it < p.items; it += gridDim.x) {
            const int k = it / p.ncol, col = it - k * p.ncol;
            const int y = 2 + (col / p.nzt) * TY + r0, z = 2 + (col % p.nzt) * TZ + tz;
            const bool v0 = y <= p.n1 - 3 && z <= p.n2 - 3, v1 = y + 1 <= p.n1 - 3 && z <= p.n2 - 3;
            const int xa = 2 + k * p.chunk, len = min(p.chunk, p.n0 - 2 - xa);
            float4 m2[2], m1[2], c[2], p1[2];
#pragma unroll 5
            for (int i = 0; i < len + 4; ++i, ++g) {
                const int s = g % kRingSlots;
                if (!mbar_wait_flag(&sm.full[s], (g / kRingSlots) & 1u, &sm.flag))
                    *(volatile int *)&sm.flag = 1;
                const float4 p2[2] = {sm.plane[s][r0 + 2][tz + 2], sm.plane[s][r0 + 3][tz + 2]};
                if (i >= 2) {
                    // the plane two back: its neighbours are read now, the
                    // x-stencil's values having arrived (a run's first two
                    // planes are never centres)
                    const int sc = (g - 2) % kRingSlots;
                    if (i >= 4) {
                        const float4(*P)[TZ + 4] = sm.plane[sc];
                        const float4 ym2 = P[r0][tz + 2], ym1 = P[r0 + 1][tz + 2];
                        const float4 yp2 = P[r0 + 4][tz + 2], yp3 = P[r0 + 5][tz + 2];
                        const SiteDens<float> d0 = site_densities<EXT>(
                            c[0], first_difference(m2[0], m1[0], p1[0], p2[0]),
                            first_difference(ym2, ym1, c[1], yp2),
                            first_difference(P[r0 + 2][tz], P[r0 + 2][tz + 1], P[r0 + 2][tz + 3], P[r0 + 2][tz + 4]), p);
                        if (v0) acc.add<EXT>(d0);
                        const SiteDens<float> d1 = site_densities<EXT>(
                            c[1], first_difference(m2[1], m1[1], p1[1], p2[1]),
                            first_difference(ym1, c[0], yp2, yp3),
                            first_difference(P[r0 + 3][tz], P[r0 + 3][tz + 1], P[r0 + 3][tz + 3], P[r0 + 3][tz + 4]), p);
                        if (v1) acc.add<EXT>(d1);
                    }
                    __syncwarp();
                    if ((tid & 31) == 0) mbar_arrive(&sm.empty[sc]);
                }
#pragma unroll
                for (int r = 0; r < 2; ++r) m2[r] = m1[r], m1[r] = c[r], c[r] = p1[r], p1[r] = p2[r];
            }
            // the run's last two planes are not centres either
            __syncwarp();
            if ((tid & 31) == 0) {
                mbar_arrive(&sm.empty[(g - 2) % kRingSlots]);
                mbar_arrive(&sm.empty[(g - 1) % kRingSlots]);
            }
        }
    }
    __syncthreads();
    const bool failed = sm.flag != 0;
    if (failed) {
        // a plane never landed: record it; the totals become NaN
        if (tid == 0) atomicExch(&p.ctrl->status, (int)DEV_TIMEOUT);
        acc.s24 = acc.c24 = acc.s0b = acc.c0b = make_float2(__int_as_float(0x7fc00000), __int_as_float(0x7fc00000));
    }
    block_totals(acc, sm.buf, tid);
    finish_energy(p.ctrl, p.parts, p.scale, sm.buf, &sm.last, tid);
}

static cudaError_t sm_count_of(int *sms)
{
    int dev = 0;
    const cudaError_t e = cudaGetDevice(&dev);
    return e != cudaSuccess ? e : cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev);
}

// Planes per item, of `nix`, for `ctas` CTAs and ncol tiles: the length whose
// rounds of items take the fewest planes, a run counting one plane more than
// its centres (its first and last two planes are only staged).
static int energy_chunk(int nix, int ncol, int ctas)
{
    int best = 1;
    long long best_cost = -1;
    for (int c = 1; c <= std::min(nix, 64); ++c) {
        const long long items = (long long)ncol * ((nix + c - 1) / c);
        const long long cost = (items + ctas - 1) / ctas * (c + 1);
        if (best_cost < 0 || cost <= best_cost) best = c, best_cost = cost;
    }
    return best;
}

template <typename T, bool EXT, int TZ>
static cudaError_t launch_energy_tz(const skyrme_lattice &lat, EnergyParams<T> p, cudaStream_t s)
{
    int sms = 0;
    cudaError_t e = sm_count_of(&sms);
    if (e != cudaSuccess) return e;
    // two CTAs per SM; the partial-record space holds at least 152 * 8 records
    const int resident = std::min(152 * 8, 2 * sms);
    const int nix = p.n0 - 4;
    p.nzt = (p.n2 - 4 + TZ - 1) / TZ;
    if constexpr (sizeof(T) == 4) {
        PlaneMaps maps;
        constexpr int TY = EnergySmem<TZ>::TY;
        if (make_plane_map(&maps.map[0], p.phi[0], lat, 4 * (TZ + 4), TY + 4) &&
            make_plane_map(&maps.map[1], p.phi[1], lat, 4 * (TZ + 4), TY + 4)) {
            p.ncol = p.nzt * ((p.n1 - 4 + TY - 1) / TY);
            p.chunk = energy_chunk(nix, p.ncol, resident);
            p.items = p.ncol * ((nix + p.chunk - 1) / p.chunk);
            constexpr int smem = (int)sizeof(EnergySmem<TZ>);
            e = cudaFuncSetAttribute(k_energy_tma<EXT, TZ>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
            if (e != cudaSuccess) return e;
            k_energy_tma<EXT, TZ><<<std::min(p.items, resident), kEnergyThreads + 32, smem, s>>>(maps, p);
            return cudaGetLastError();
        }
    }
    constexpr int TY = kEnergyThreads / TZ;
    p.ncol = p.nzt * ((p.n1 - 4 + TY - 1) / TY);
    p.chunk = energy_chunk(nix, p.ncol, resident);
    p.items = p.ncol * ((nix + p.chunk - 1) / p.chunk);
    k_energy<T, EXT, TZ><<<std::min(p.items, resident), kEnergyThreads, 0, s>>>(p);
    return cudaGetLastError();
}

template <typename T>
static cudaError_t launch_energy_t(const skyrme_lattice &lat, const FlowArgs &a, cudaStream_t s)
{
    EnergyParams<T> p;
    for (int i = 0; i < 2; ++i) p.phi[i] = static_cast<const vec4_t<T> *>(a.phi[i]);
    p.ctrl = static_cast<Ctrl *>(a.ctrl);
    p.parts = a.energy_parts;
    p.n0 = a.n[0], p.n1 = a.n[1], p.n2 = a.n[2];
    p.m2 = T(a.m * a.m);
    p.my2 = T(a.my * a.my), p.mz2 = T(a.mz * a.mz), p.mw2 = T(a.mw * a.mw);
    const bool ext = lattice_extended(lat);
    // u = 12h d phi: e2, e4, det, e6 carry k1^2, k1^4, k1^3, k1^6
    const double h3 = a.h * a.h * a.h, k1 = 1.0 / (12.0 * a.h), k2 = k1 * k1;
    p.scale[0] = h3 * k2;
    p.scale[1] = h3 * k2 * k2;
    p.scale[2] = ext ? h3 : h3 * (2.0 * a.m * a.m);
    p.scale[3] = h3 * k2 * k1 * -0.050660591821168885;  // b = -det / (2 pi^2)
    p.scale[4] = h3 * k2 * k2 * k2 * a.c6;
    const bool narrow = tile_geometry(lat).tz == 16;  // the z tile that pads the lattice less
    if (ext)
        return narrow ? launch_energy_tz<T, true, 16>(lat, p, s) : launch_energy_tz<T, true, 32>(lat, p, s);
    return narrow ? launch_energy_tz<T, false, 16>(lat, p, s) : launch_energy_tz<T, false, 32>(lat, p, s);
}

cudaError_t launch_energy(const skyrme_lattice &lat, const FlowArgs &a, cudaStream_t s)
{
    return lat.precision == 64 ? launch_energy_t<double>(lat, a, s)
                               : launch_energy_t<float>(lat, a, s);
}

}  // namespace skyrme
