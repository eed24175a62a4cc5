// Vector form of the fused time step for 3D domains with 16-bit deviation
// storage: the arithmetic of step_kernel.cuh, operation by operation (the two
// give the same bits), with the work split into two launches per step and four
// consecutive sites along x per thread.
//
// Launch 1, heat_vec_kernel: the lagged heat update of step n-1,
//   (f^{n-1}, aux^{n-1}, phi^n) -> (f^n, aux^n) and u^n into a work field.
// Launch 2, phi_vec_kernel: the phase-field update of step n,
//   (g^n, phi^n, u^n) -> (g^{n+1}, phi^{n+1}).
// The lagged state between steps is the step kernel's, so either kernel can
// take over at any step.
//
// Why: step_kernel is bound by instruction issue (1210 thread-instructions a
// site with FP16 deviations, 73 % issue-active, 30 % of HBM at 256^3).  Apart,
// the heat update is computed once per site instead of on every halo (111
// instructions a site, bound by HBM: 127 us at 256^3, 66 % of the DRAM rate),
// and both launches read and write four sites per instruction, which leaves
// 408 instructions a site for the phase field.  The work field costs 8 of
// 104 bytes a site.  Measured, us a step (step_kernel / this): D3Q15 FP16
// 512^3 5289 / 3782 (stochastic rounding 7147 / 5936), 256^3 719 / 551, 351^3
// with walls 2307 / 1682, 207 x 174 x 190 397 / 296; 256^3 D3Q19 838 / 690,
// D3Q27 1260 / 980.  Rows that are not whole vectors are padded in memory
// (DomainDev::px); a row's last partial vector is computed whole, what falls into
// the padding is never read.  Full (FP32) storage measured 2-8 % slower this way
// (the vectors in flight need twice the registers) and stays with step_kernel;
// the heat launch apart before a one-site phase-field march was not measured.
#pragma once

#include <algorithm>

#include "step_kernel.cuh"

namespace lbpf {

// Four consecutive stored deviations are loaded in two steps, so that many
// loads can be in flight in few registers: raw bits, then the values.
template <class T>
__device__ __forceinline__ uint2 raw4(const T* p)
{
    static_assert(sizeof(T) == 2, "16-bit deviations");
    return __ldg(reinterpret_cast<const uint2*>(p));
}
template <class T>
__device__ __forceinline__ void unpack2(uint2 a, float2 (&v)[2])
{
    if constexpr (std::is_same<T, __half>::value) {
        v[0] = __half22float2(*reinterpret_cast<const __half2*>(&a.x));
        v[1] = __half22float2(*reinterpret_cast<const __half2*>(&a.y));
    } else {  // BF16: the upper half of an FP32
        v[0] = make_float2(__uint_as_float(a.x << 16), __uint_as_float(a.x & 0xFFFF0000u));
        v[1] = make_float2(__uint_as_float(a.y << 16), __uint_as_float(a.y & 0xFFFF0000u));
    }
}
// Four floats as pairs.
__device__ __forceinline__ void lds_v(const float* p, float2 (&v)[2])
{
    const float4 a = *reinterpret_cast<const float4*>(p);
    v[0] = make_float2(a.x, a.y);
    v[1] = make_float2(a.z, a.w);
}
__device__ __forceinline__ void st_v(float* p, const float2 (&v)[2])
{
    *reinterpret_cast<float4*>(p) = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
}
// element k of a vector of pairs
__device__ __forceinline__ float& el(float2 (&v)[2], int k)
{
    return k & 1 ? v[k >> 1].y : v[k >> 1].x;
}
template <class T>
__device__ __forceinline__ void load4(const T* p, float (&v)[4])
{
    float2 t[2];
    unpack2<T>(raw4(p), t);
    v[0] = t[0].x;
    v[1] = t[0].y;
    v[2] = t[1].x;
    v[3] = t[1].y;
}
__device__ __forceinline__ void load4(const float* p, float (&v)[4])
{
    const float4 a = __ldg(reinterpret_cast<const float4*>(p));
    v[0] = a.x;
    v[1] = a.y;
    v[2] = a.z;
    v[3] = a.w;
}
__device__ __forceinline__ void store4(float* p, const float (&v)[4])
{
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
// Rounded deviations of four sites (h: their hashes for the stochastic form).
template <class S>
__device__ __forceinline__ void store_dev(typename S::T* p, const float (&v)[4], const uint32_t (&h)[4], uint32_t pop)
{
    using T = typename S::T;
    uint32_t b[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        T t;
        if constexpr (UsesSR<S>::value)
            t = from_real_sr<T>(v[k], sr_bits(h[k], pop));
        else
            t = from_real<T, float>(v[k]);
        b[k] = *reinterpret_cast<const uint16_t*>(&t);
    }
    *reinterpret_cast<uint2*>(p) = make_uint2(b[0] | b[1] << 16, b[2] | b[3] << 16);
}

// Index maps of one axis: periodic, or reflected at a wall.
template <bool WALLS>
__device__ __forceinline__ int wrap_axis(int v, int n, bool wall)
{
    if (WALLS && wall) return reflect_index(v, n);
    return v < 0 ? v + n : (v >= n ? v - n : v);
}

// ---- launch 1 ---------------------------------------------------------------
// A thread owns four sites along x and marches over planes [z0, z1), keeping
// h = aux + phi / 2 of its own column at z - 1, z, z + 1 in registers; rows
// y +- 1 and the sites x - 1, x + 4 come from global memory (L1).  With
// collide == 0 (the state is synchronised) only u^n and aux^n are formed.  One
// launch covers a group of domains (HeatGrid): nseg runs of zlen planes each in
// grid z.

// The launch over the first m of n domains: as many in a row, with or without
// walls alike, as keep at least half of the blocks busy when all get the
// largest one's, in the grid's limits (vec_applies holds a domain's own ny and
// nz to them).  A launch a domain costs its latency each time: FP16, us a step,
// a launch each / grouped (the march): 64 domains of 48^3 513 / 343 (474), 64 of
// 64^3 930 / 665 (760), 8 of 128^3 581 / 547 (727).
struct HeatGrid {
    int m, zlen, nseg;
    dim3 grid;
};
inline HeatGrid heat_grid(const DomainDev* h, int n)
{
    HeatGrid g{};
    long long gx = 0, gy = 0, nz = 0, work = 0;
    while (g.m < n && (h[g.m].bc != 0) == (h[0].bc != 0)) {
        const DomainDev& d = h[g.m];
        const long long bx = (d.px / 4 + kHeatX - 1) / kHeatX, by = (d.ny + kHeatY - 1) / kHeatY;
        const long long ax = std::max(gx, bx), ay = std::max(gy, by), az = std::max(nz, (long long)d.nz);
        const long long w = work + bx * by * d.nz;
        if (g.m > 0 && (ax * ay * az * (g.m + 1) > 2 * w || az * (g.m + 1) > 65535)) break;
        gx = ax;
        gy = ay;
        nz = az;
        work = w;
        ++g.m;
    }
    g.zlen = 16;
    while (g.zlen > 1 && gx * gy * ((nz + g.zlen - 1) / g.zlen) * g.m < 152 * 8) g.zlen /= 2;
    g.nseg = (int)((nz + g.zlen - 1) / g.zlen);
    g.grid = dim3((unsigned)gx, (unsigned)gy, (unsigned)(g.nseg * g.m));
    return g;
}

template <class UL, class S, bool WALLS>
__global__ void __launch_bounds__(kHeatX* kHeatY) heat_vec_kernel(const DomainDev* dp, int cur, int fcur, int acur,
                                                                 int collide, int zlen, int nseg,
                                                                 const int* counters)
{
    using T = typename S::T;
    constexpr int QU = UL::Q;
    static_assert(UL::D == 3 && QU == 7 && S::dev, "D3Q7, 16-bit deviations");
    const DomainDev& d = dp[(int)blockIdx.z / nseg];
    const int nx = d.nx, ny = d.ny, nz = d.nz;
    const int x = ((int)blockIdx.x * kHeatX + (int)threadIdx.x) * 4, y = (int)blockIdx.y * kHeatY + (int)threadIdx.y;
    if (x >= nx || y >= ny) return;
    const int z0 = (int)blockIdx.z % nseg * zlen, z1 = min(z0 + zlen, nz);
    if (z0 >= nz) return;
    const long long n = d.n, nxy = (long long)d.px * ny;
    const bool wX = WALLS && (d.bc & LBPF_BC_WALL_X), wY = WALLS && (d.bc & LBPF_BC_WALL_Y),
               wZ = WALLS && (d.bc & LBPF_BC_WALL_Z);
    const T* __restrict__ fc = static_cast<const T*>(d.f[fcur]);
    T* __restrict__ fn = static_cast<T*>(d.f[fcur ^ 1]);
    const float* __restrict__ auxc = static_cast<const float*>(d.aux[acur]);
    float* __restrict__ auxn = static_cast<float*>(d.aux[acur ^ 1]);
    const float* __restrict__ phi = static_cast<const float*>(d.phi[cur]);
    float* __restrict__ uo = static_cast<float*>(d.u_work);
    const float ieu = d.r32.inv_eta_u, om_u = 1.f - ieu;
    const uint32_t seed = UsesSR<S>::value ? (uint32_t)counters[2 + cur] : 0u;
    const long long row = (long long)y * d.px + x;  // in-plane offset of the vector
    const int ke = min(3, nx - 1 - x);              // the vector's last site (the rest is row padding)

    if (!collide) {
        for (int z = z0; z < z1; ++z) {
            const long long s = z * nxy + row;
            float ph[4], u[4], a[4];
            load4(phi + s, ph);
            load4(auxc + s, a);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                u[k] = a[k] + 0.5f * ph[k];
                a[k] = u[k] - 0.5f * ph[k];
            }
            store4(auxn + s, a);
            store4(uo + s, u);
        }
        return;
    }

    const int xm = wrap_axis<WALLS>(x - 1, nx, wX), xp = wrap_axis<WALLS>(x + ke + 1, nx, wX);
    const int ym = wrap_axis<WALLS>(y - 1, ny, wY), yp = wrap_axis<WALLS>(y + 1, ny, wY);
    const long long rym = (long long)ym * d.px + x, ryp = (long long)yp * d.px + x, r0 = (long long)y * d.px;
    auto load_h = [&](long long s, float (&h)[4], float (&ph)[4]) {
        load4(phi + s, ph);
        load4(auxc + s, h);
#pragma unroll
        for (int k = 0; k < 4; ++k) h[k] += 0.5f * ph[k];
    };
    float hm[4], hc[4], hp[4], ph[4], php[4], tmp[4];
    load_h((long long)wrap_axis<WALLS>(z0 - 1, nz, wZ) * nxy + row, hm, tmp);
    load_h(z0 * nxy + row, hc, ph);
    for (int z = z0; z < z1; ++z) {
        const long long zo = z * nxy, zm = (long long)wrap_axis<WALLS>(z - 1, nz, wZ) * nxy,
                        zp = (long long)wrap_axis<WALLS>(z + 1, nz, wZ) * nxy;
        const long long s = zo + row;
        load_h(zp + row, hp, php);
        float hym[4], hyp[4];
        load_h(zo + rym, hym, tmp);
        load_h(zo + ryp, hyp, tmp);
        const float hxm = auxc[zo + r0 + xm] + 0.5f * phi[zo + r0 + xm];
        const float hxp = auxc[zo + r0 + xp] + 0.5f * phi[zo + r0 + xp];
        // the array of direction j >= 1 is j - 1
        const T *f1 = fc, *f2 = fc + n, *f3 = fc + 2 * n, *f4 = fc + 3 * n, *f5 = fc + 4 * n, *f6 = fc + 5 * n;
        float l1[4], l2[4], l3[4], l4[4], l5[4], l6[4], p2[4], p4[4], p5[4], p6[4], d0[4];
        load4(f1 + s, l1);
        load4(f2 + s, l2);
        load4(f3 + s, l3);
        load4(f4 + s, l4);
        load4(f5 + s, l5);
        load4(f6 + s, l6);
        load4(f2 + zo + rym, p2);
        load4(f4 + zo + ryp, p4);
        load4(f5 + zm + row, p5);
        load4(f6 + zp + row, p6);
        const float e1 = to_real(f1[zo + r0 + xm]), e3 = to_real(f3[zo + r0 + xp]);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            d0[k] = 0.f;
            d0[k] -= l1[k];
            d0[k] -= l2[k];
            d0[k] -= l3[k];
            d0[k] -= l4[k];
            d0[k] -= l5[k];
            d0[k] -= l6[k];
        }
        float fv[QU][4], u[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float hs[QU] = {hc[k], k > 0 ? hc[k > 0 ? k - 1 : 0] : hxm, hym[k],
                                  k == ke ? hxp : hc[k < 3 ? k + 1 : 3],
                                  hyp[k], hm[k], hp[k]};
            const float pv[QU] = {d0[k], k > 0 ? l1[k > 0 ? k - 1 : 0] : e1, p2[k],
                                  k == ke ? e3 : l3[k < 3 ? k + 1 : 3],
                                  p4[k], p5[k], p6[k]};
            u[k] = 0.f;
#pragma unroll
            for (int j = 0; j < QU; ++j) {
                const float fj = float(UL::w(j)) * hs[j] + om_u * pv[j];
                fv[j][k] = fj;
                u[k] += fj;
            }
        }
        if constexpr (WALLS) {
            const int loyz = (wY && y == 0 ? 2 : 0) | (wZ && z == 0 ? 4 : 0);
            const int hiyz = (wY && y == ny - 1 ? 2 : 0) | (wZ && z == nz - 1 ? 4 : 0);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int lo = loyz | (wX && x + k == 0 ? 1 : 0), hi = hiyz | (wX && x + k == nx - 1 ? 1 : 0);
                if (lo | hi) {
                    float t[QU];
#pragma unroll
                    for (int j = 0; j < QU; ++j) t[j] = fv[j][k];
                    mirror_refill<UL, float>(t, lo, hi);
                    u[k] = 0.f;
#pragma unroll
                    for (int j = 0; j < QU; ++j) {
                        fv[j][k] = t[j];
                        u[k] += t[j];
                    }
                }
            }
        }
        uint32_t hh[4] = {0u, 0u, 0u, 0u};
        if constexpr (UsesSR<S>::value) {
#pragma unroll
            for (int k = 0; k < 4; ++k) hh[k] = sr_hash((uint32_t)(((long long)z * ny + y) * nx + x + k), seed);
        }
#pragma unroll
        for (int j = 1; j < QU; ++j) {
            float o[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) o[k] = fv[j][k] - float(UL::w(j)) * u[k];
            store_dev<S>(fn + (j - 1) * n + s, o, hh, 32u + j);
        }
        float a[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) a[k] = u[k] - 0.5f * ph[k];
        store4(auxn + s, a);
        store4(uo + s, u);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            hm[k] = hc[k];
            hc[k] = hp[k];
            ph[k] = php[k];
        }
    }
}

// ---- launch 2 ---------------------------------------------------------------
// A block of eight warps owns a 64 x 12 column of sites and marches along z as
// step_kernel does; two block-wide barriers a plane separate the phases.
//   Coefficient phase (plane z + 1): warps 0-6 compute the four-site vectors of
//   the 14 rows (tile and halo rows), warp 7 the two halo columns.
//   Output phase (plane z): warps 0-5 stream and store the 12 rows, warp 6
//   computes the row segments' end sites (below), warp 7 copies the next phi
//   plane.
// Rings in shared memory: four phi planes (tile + 2 sites), three planes of the
// coefficients (c1, c2 negated, s, vx, vy, vz), six arrays of 64 x 14 and one
// record per row for each halo column: 85 KB, two blocks an SM.
// Every global access of a population is one aligned vector of four sites.  A
// direction with e_x = +-1 is computed on the source vector (all of whose
// inputs are aligned): the destination's g_i(y) is shifted against it by one
// lane shuffle, and the result back by another; the one destination site of a
// row segment whose source lies beyond the segment is computed apart (warp 6).
// What bounds it: latency.  16 warps an SM at 128 registers (the populations of
// four sites in flight) keep 45 % of the issue slots and 54 % of the shared
// memory pipe busy at 256^3 (418 us, 35 % of the DRAM rate), the barriers being
// the largest stall.  Tried: two sites
// a thread with 64 registers and 32 warps (15 % slower: as many spills and
// 20 % more instructions), 14 rows with one helper warp (3 % slower at 512^3:
// that warp was the longest path), loads that skip L1 (10 % slower: spilled
// registers and halo rows hit there).
constexpr int kVecV = 4;                // sites a thread
constexpr int kVecLX = kVecTX / kVecV;  // lanes a row segment
constexpr int kVecNT = kVecLX * (kVecTY + 4);

template <class PL>
struct VecSmem {
    static constexpr int CR = kVecTY + 2;                    // coefficient rows
    static constexpr int CA = CR * kVecTX;                   // one coefficient array of a plane
    static constexpr int EDGE = CR * 2 * 6;                  // halo column records of a plane
    static constexpr int CP = 6 * CA;                        // floats of one coefficient plane
    static constexpr int PX = kVecTX + 8, PY = kVecTY + 4;   // phi frame (tile starts at 4, 2)
    static constexpr int PP = PX * PY;
    static constexpr int NPH = 4, NC = 3;
    static constexpr int END = kVecTY * 2 * 9;                // end-site populations of a plane
    static constexpr size_t bytes = sizeof(float) * (size_t)(NPH * PP + NC * (CP + EDGE) + END);
};

// One direction pair (e_x = +1, e_x = -1 with the same e_y, e_z) of lattice PL.
template <class PL>
LBPF_HD constexpr int dir_index(int ex, int ey, int ez)
{
    for (int i = 0; i < PL::Q; ++i)
        if (PL::ex(i) == ex && PL::ey(i) == ey && PL::ez(i) == ez) return i;
    return -1;
}

template <class PL, class S, bool WALLS>
__device__ __forceinline__ void phi_vec_item(const StepArgs& args, const WorkItem it, float* smem)
{
    using T = typename S::T;
    using SM = VecSmem<PL>;
    static_assert(S::dev && sizeof(T) == 2, "16-bit deviations");
    constexpr int QG = PL::Q;
    constexpr int CA = SM::CA, CP = SM::CP, PX = SM::PX, PP = SM::PP;
    constexpr unsigned FULL = 0xffffffffu;
    float* s_phi = smem;
    float* s_co = smem + SM::NPH * PP;
    float* s_edge = s_co + SM::NC * CP;
    float* s_end = s_edge + SM::NC * SM::EDGE;

    const DomainDev& dm = args.doms[it.dom];
    const int nx = dm.nx, ny = dm.ny, nz = dm.nz;
    const int P = dm.px;  // row pitch
    const long long n = dm.n, nxy = (long long)P * ny;
    const int x0 = it.x0, y0 = it.y0, z0 = it.z0, z1 = it.z1;
    const int tw = min(kVecTX, nx - x0), th = min(kVecTY, ny - y0);
    const int tid = threadIdx.x;
    // the last two rows' threads: copies and halo columns (index hl of HN); the
    // two rows before them own no output row and compute the end sites (hp)
    constexpr int HN = 2 * kVecLX;
    const int hl = tid - kVecLX * (kVecTY + 2), hp = tid - kVecLX * kVecTY;
    const bool helper = hl >= 0;
    const T* __restrict__ gc = static_cast<const T*>(dm.g[args.cur]);
    T* __restrict__ gn = static_cast<T*>(dm.g[args.cur ^ 1]);
    const float* __restrict__ phic = static_cast<const float*>(dm.phi[args.cur]);
    float* __restrict__ phin = static_cast<float*>(dm.phi[args.cur ^ 1]);
    const float* __restrict__ uc = static_cast<const float*>(dm.u_work);
    const uint32_t seed = UsesSR<S>::value ? (uint32_t)args.counters[2 + args.cur] : 0u;
    const float De2 = dm.r32.De2, qphi = dm.r32.qphi, lam = dm.r32.lambda;
    const bool wX = WALLS && (dm.bc & LBPF_BC_WALL_X), wY = WALLS && (dm.bc & LBPF_BC_WALL_Y),
               wZ = WALLS && (dm.bc & LBPF_BC_WALL_Z);
    const bool dd = args.grad == LBPF_GRAD_DD;
    auto wy = [&](int v) { return wrap_axis<WALLS>(v, ny, wY); };
    auto wz = [&](int v) { return wrap_axis<WALLS>(v, nz, wZ); };
    auto wx = [&](int v) { return wrap_axis<WALLS>(v, nx, wX); };
    auto phi_plane = [&](int z) { return s_phi + ((z + 8) & 3) * PP; };
    auto edge_plane = [&](int z) { return s_edge + ((z + 3) % 3) * SM::EDGE; };
    auto co_plane = [&](int z) { return s_co + ((z + 3) % 3) * CP; };

    // phi plane z (tile + 2 sites) into its ring slot, by threads t0 of nt (a
    // multiple of 32): 16-byte chunks of the rows, 16 a row, then single columns
    auto copy_phi = [&](int z, int t0, int nt) {
        const float* src = phic + (long long)wz(z) * nxy;
        float* dst = phi_plane(z);
        const int c = t0 & 15;
        if (4 * c + 4 <= tw)
            for (int r = t0 >> 4; r < th + 4; r += nt >> 4) {
                const float* g = src + ((long long)wy(y0 + r - 2) * P + x0 + 4 * c);
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                                 (unsigned)__cvta_generic_to_shared(dst + r * PX + 4 + 4 * c)),
                             "l"(g));
            }
        // single columns: the two left of the tile, the sites of a row's last
        // partial vector and the two right of the tile
        const int sh = tw & 3 ? 3 : 2, q = t0 & ((1 << sh) - 1);
        const int qx = q < 2 ? 2 + q : 4 + (tw & ~3) + (q - 2);
        if (qx >= 4 + tw + 2) {
            asm volatile("cp.async.commit_group;");
            return;
        }
        const int gq = wx(x0 + qx - 4);
        for (int r = t0 >> sh; r < th + 4; r += nt >> sh) {
            const float* g = src + ((long long)wy(y0 + r - 2) * P + gq);
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(
                             (unsigned)__cvta_generic_to_shared(dst + r * PX + qx)),
                         "l"(g));
        }
        asm volatile("cp.async.commit_group;");
    };

    // coefficients of one site from phi, its gradient and u
    auto coefficients = [&](float ph, float Gx, float Gy, float Gz, float u, float& c1, float& c2, float& sc, float& vx,
                            float& vy, float& vz) {
        float a = 1.f, Nx = 0.f, Ny = 0.f, Nz = 0.f;
        anisotropy<float, 3>(dm.cr[0], Gx, Gy, Gz, a, Nx, Ny, Nz);
        const float A2 = a * a;
        const float iA2 = recip<float>(A2);
        const float ieta = recip<float>(A2 * De2 + 0.5f);
        const float omp = (1.f - ph) * (1.f + ph);
        const float Qphi = (ph - lam * u * omp) * omp;
        const float vf = -De2 * ieta * iA2;
        sc = (ph + qphi * Qphi) * iA2;
        c1 = (1.f - ieta) * iA2;
        c2 = 1.f - iA2;  // minus (1 - a^2) / a^2
        vx = vf * Nx;
        vy = vf * Ny;
        vz = vf * Nz;
    };
    constexpr bool EDGES_XY = dir_index<PL>(1, 1, 0) >= 0;  // D3Q19 / D3Q27
    constexpr bool CORNERS = dir_index<PL>(1, 1, 1) >= 0;   // D3Q15 / D3Q27

    constexpr int V = kVecV, H = V / 2;
    // vector task: coefficient row cr, columns V lx .. of plane z; u of these
    // sites is passed in
    auto coef_vec = [&](int z, int cr, int lx, float2(&u)[H]) {
        const float* pm = phi_plane(z - 1) + (cr + 1) * PX + 4 + V * lx;
        const float* pc = phi_plane(z) + (cr + 1) * PX + 4 + V * lx;
        const float* pp = phi_plane(z + 1) + (cr + 1) * PX + 4 + V * lx;
        // r[k]: phi at x - 1 + k of row (dy, dz) (ends only where needed)
        auto row_ends = [&](const float* b, bool ends, float(&r)[V + 2]) {
            float2 a[H];
            lds_v(b, a);
#pragma unroll
            for (int k = 0; k < V; ++k) r[k + 1] = el(a, k);
            r[0] = ends ? b[-1] : 0.f;
            r[V + 1] = ends ? b[V] : 0.f;
        };
        float r00[V + 2];
        row_ends(pc, true, r00);
        float G[3][V];
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int k = 0; k < V; ++k) G[a][k] = 0.f;
        if (dd) {
            float ry[2][V + 2], rz[2][V + 2], rc[4][V + 2];  // rows (dy,0), (0,dz), (dy,dz): + before -
            row_ends(pc + PX, EDGES_XY, ry[0]);
            row_ends(pc - PX, EDGES_XY, ry[1]);
            row_ends(pp, EDGES_XY, rz[0]);
            row_ends(pm, EDGES_XY, rz[1]);
            row_ends(pp + PX, CORNERS, rc[0]);
            row_ends(pm + PX, CORNERS, rc[1]);
            row_ends(pp - PX, CORNERS, rc[2]);
            row_ends(pm - PX, CORNERS, rc[3]);
#pragma unroll
            for (int i = 1; i < QG; ++i) {
                if (i > opposite<PL>(i)) continue;
                const int ex = PL::ex(i), ey = PL::ey(i), ez = PL::ez(i);
                auto at = [&](int sx, int sy, int sz, int k) -> float {
                    const int j = 1 + k + sx;
                    if (sy == 0 && sz == 0) return r00[j];
                    if (sz == 0) return ry[sy > 0 ? 0 : 1][j];
                    if (sy == 0) return rz[sz > 0 ? 0 : 1][j];
                    return rc[(sy > 0 ? 0 : 2) + (sz > 0 ? 0 : 1)][j];
                };
#pragma unroll
                for (int k = 0; k < V; ++k) {
                    const float df = at(ex, ey, ez, k) - at(-ex, -ey, -ez, k);
                    const float wd = float(PL::w(i)) * df;
                    if (ex) G[0][k] += float(ex) * wd;
                    if (ey) G[1][k] += float(ey) * wd;
                    if (ez) G[2][k] += float(ez) * wd;
                }
            }
            const float kk = float(1.0 / PL::E2);
#pragma unroll
            for (int a = 0; a < 3; ++a)
#pragma unroll
                for (int k = 0; k < V; ++k) G[a][k] *= kk;
        } else {
#pragma unroll
            for (int k = 0; k < V; ++k) {
                G[0][k] = 0.5f * (r00[k + 2] - r00[k]);
                G[1][k] = 0.5f * (pc[PX + k] - pc[-PX + k]);
                G[2][k] = 0.5f * (pp[k] - pm[k]);
            }
        }
        float2 o[6][H];
#pragma unroll
        for (int k = 0; k < V; ++k)
            coefficients(r00[k + 1], G[0][k], G[1][k], G[2][k], el(u, k), el(o[0], k), el(o[1], k), el(o[2], k),
                         el(o[3], k), el(o[4], k), el(o[5], k));
        float* co = co_plane(z) + cr * kVecTX + V * lx;
#pragma unroll
        for (int c = 0; c < 6; ++c) st_v(co + c * CA, o[c]);
    };
    // one halo column site: row cr, side 0 (x0 - 1) or 1 (x0 + tw)
    auto coef_edge = [&](int z, int cr, int side, float u) {
        const int px = side ? 4 + tw : 3;
        const float* pm = phi_plane(z - 1) + (cr + 1) * PX + px;
        const float* pc = phi_plane(z) + (cr + 1) * PX + px;
        const float* pp = phi_plane(z + 1) + (cr + 1) * PX + px;
        float Gx = 0.f, Gy = 0.f, Gz = 0.f;
        if (dd) {
#pragma unroll
            for (int i = 1; i < QG; ++i) {
                if (i > opposite<PL>(i)) continue;
                const int ex = PL::ex(i), ey = PL::ey(i), ez = PL::ez(i);
                const float* pa = ez > 0 ? pp : (ez < 0 ? pm : pc);
                const float* pb = ez > 0 ? pm : (ez < 0 ? pp : pc);
                const float df = pa[ey * PX + ex] - pb[-ey * PX - ex];
                const float wd = float(PL::w(i)) * df;
                if (ex) Gx += float(ex) * wd;
                if (ey) Gy += float(ey) * wd;
                if (ez) Gz += float(ez) * wd;
            }
            const float kk = float(1.0 / PL::E2);
            Gx *= kk;
            Gy *= kk;
            Gz *= kk;
        } else {
            Gx = 0.5f * (pc[1] - pc[-1]);
            Gy = 0.5f * (pc[PX] - pc[-PX]);
            Gz = 0.5f * (pp[0] - pm[0]);
        }
        float c1, c2, sc, vx, vy, vz;
        coefficients(pc[0], Gx, Gy, Gz, u, c1, c2, sc, vx, vy, vz);
        float2* co = reinterpret_cast<float2*>(edge_plane(z) + (cr * 2 + side) * 6);
        co[0] = make_float2(c1, c2);
        co[1] = make_float2(sc, vx);
        co[2] = make_float2(vy, vz);
    };

    // this thread's vector task: row cr of the coefficient plane
    const int lx = tid & (kVecLX - 1);
    const int cr = tid / kVecLX;
    const bool vtask = !helper && V * lx < tw && cr <= th + 1;
    const long long urow = (long long)wy(y0 + cr - 1) * P + x0 + V * lx;
    auto load_u = [&](int z, float2(&u)[H]) {
        if (vtask) lds_v(uc + (long long)wz(z) * nxy + urow, u);
    };
    // halo columns: helper thread t the site of row t / 2, side t & 1
    static_assert(HN >= 2 * (kVecTY + 2), "one halo column site a helper thread");
    const bool etask = helper && (hl >> 1) < th + 2;
    const long long erow = (long long)wy(y0 + (hl >> 1) - 1) * P + wx(hl & 1 ? x0 + tw : x0 - 1);
    auto load_ue = [&](int z) { return etask ? __ldg(uc + (long long)wz(z) * nxy + erow) : 0.f; };

    // The populations that output_plane(z) is the first to touch (plane z, or
    // z + 1 for the directions with e_z = -1), requested into L2.
    // Helper thread t takes row t / 2 of the tile with halo rows, its first
    // line or its last (the same where rows are aligned to lines).
    const long long prow = (long long)wy(y0 + (hl >> 1) - 1) * P + x0 + (hl & 1 ? tw - 1 : 0);
    const bool ptask = etask && (!(hl & 1) || P % 64 != 0);
    auto prefetch_g = [&](int z) {
        if (!ptask) return;
        const T* pa = gc + ((long long)wz(z) * nxy + prow);
        const T* pb = gc + ((long long)wz(z + 1) * nxy + prow);
#pragma unroll
        for (int i = 1; i < QG; ++i)
            asm volatile("prefetch.global.L2 [%0];" ::"l"((PL::ez(i) < 0 ? pb : pa) + (long long)(i - 1) * n));
    };
    // phi of plane z into L2, ahead of its copy: thread t half of row t / 2
    const long long frow = (long long)wy(y0 + (hl >> 1) - 1) * P + min(x0 + (hl & 1) * 32, nx - 1);
    auto prefetch_phi = [&](int z) {
        if (etask) asm volatile("prefetch.global.L2 [%0];" ::"l"(phic + ((long long)wz(z) * nxy + frow)));
    };

    // output geometry
    const int r = cr;            // tile row
    const int ll = (tw - 1) / V;   // last lane of the segment
    const bool live = r < th && lx <= ll;
    const bool first = lx == 0, last = lx == ll;
    // threads without a vector (beyond the tile) read the nearest one
    const int gy = y0 + min(r, th - 1), gx = x0 + V * min(lx, ll);
    const uint32_t rowm = (uint32_t)wy(gy - 1) * P + gx, row0 = (uint32_t)gy * P + gx, rowp = (uint32_t)wy(gy + 1) * P + gx;

    // The first (last) site of each row segment: its new populations with e_x =
    // +1 (-1), whose sources are the halo column.  Helper thread t: row t / 2,
    // side t & 1.
    auto end_sites = [&](int z) {
        const int rr = hp >> 1, side = hp & 1, y = y0 + rr;
        if (rr >= th) return;
        const uint32_t xd = side ? x0 + tw - 1 : x0, xs = side ? wx(x0 + tw) : wx(x0 - 1);
        const uint32_t zo = (uint32_t)z * (uint32_t)nxy, zm = (uint32_t)wz(z - 1) * (uint32_t)nxy,
                       zp = (uint32_t)wz(z + 1) * (uint32_t)nxy;
        const uint32_t ym = (uint32_t)wy(y - 1) * P, yc = (uint32_t)y * P, yp = (uint32_t)wy(y + 1) * P;
        const float ph = phi_plane(z)[(rr + 2) * PX + 4 + (side ? tw - 1 : 0)];
        T lo[9], gp[9];
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            const int ey = q % 3 - 1, ez = q / 3 - 1;
            const int ip = dir_index<PL>(1, ey, ez), im = dir_index<PL>(-1, ey, ez);
            if (ip < 0) continue;
            const T* ga = gc + (long long)((side ? im : ip) - 1) * n;
            gp[q] = ga[(ez > 0 ? zm : (ez < 0 ? zp : zo)) + (ey > 0 ? ym : (ey < 0 ? yp : yc)) + xs];
            lo[q] = ga[zo + yc + xd];
        }
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            const int ey = q % 3 - 1, ez = q / 3 - 1;
            const int ip = dir_index<PL>(1, ey, ez);
            if (ip < 0) continue;
            const float w = float(PL::w(ip));
            const float2* co = reinterpret_cast<const float2*>(edge_plane(z - ez) + ((rr + 1 - ey) * 2 + side) * 6);
            const float2 a = co[0], b = co[1], c = co[2];
            s_end[hp * 9 + q] = pull_new<float>(1, ey, ez, w, a.x, -a.y, b.x, side ? -b.y : b.y, c.x, c.y,
                                                to_real(gp[q]), fma_rn(w, ph, to_real(lo[q])));
        }
    };

    auto output_plane = [&](int z) {
        // sites of the destination and of the source row of a direction (y - ey,
        // z - ez); a domain has fewer than 2^31 sites
        const uint32_t zo = (uint32_t)z * (uint32_t)nxy, zm = (uint32_t)wz(z - 1) * (uint32_t)nxy,
                       zp = (uint32_t)wz(z + 1) * (uint32_t)nxy;
        auto src = [&](int ey, int ez) -> uint32_t {
            return (ez > 0 ? zm : (ez < 0 ? zp : zo)) + (ey > 0 ? rowm : (ey < 0 ? rowp : row0));
        };
        const uint32_t s = zo + row0;
        const float* cpm = co_plane(z - 1) + (r + 1) * kVecTX + V * lx;
        const float* cpc = co_plane(z) + (r + 1) * kVecTX + V * lx;
        const float* cpp = co_plane(z + 1) + (r + 1) * kVecTX + V * lx;
        float2 ph[H];
        lds_v(phi_plane(z) + (r + 2) * PX + 4 + V * lx, ph);
        // the thread's population vectors are requested AHEAD directions before
        // their use (4 registers a direction, the space the new populations take
        // over one by one): all at once, but 12 of D3Q27's 26, whose space does
        // not suffice (256^3 FP16, 12 / all: D3Q15 551 / 549 us, D3Q19 723 / 689,
        // D3Q27 980 / 1083)
        constexpr int AHEAD = QG > 19 ? 12 : QG;
        uint2 ra[QG], rb[QG];
        auto request = [&](int i) {
            ra[i] = raw4(gc + (long long)(i - 1) * n + s);
            rb[i] = raw4(gc + (long long)(i - 1) * n + src(PL::ey(i), PL::ez(i)));
        };
#pragma unroll
        for (int i = 1; i < QG; ++i)
            if (i <= AHEAD) request(i);
        // new populations; the rest population comes last (its deviation is
        // minus the sum of the others).  Directions i, i + 1 that differ in the
        // sign of e_x share their coefficient vectors.
        float2 gnew[QG][H], d0[H];
#pragma unroll
        for (int h = 0; h < H; ++h) d0[h] = make_float2(0.f, 0.f);
        struct Coef {
            float2 c1[H], c2[H], cs[H], vx[H], vy[H], vz[H];
        };
        auto load_coef = [&](int ey, int ez, bool wantx, Coef& c) {
            const float* co = (ez > 0 ? cpm : (ez < 0 ? cpp : cpc)) - ey * kVecTX;
            lds_v(co, c.c1);
            lds_v(co + CA, c.c2);
            lds_v(co + 2 * CA, c.cs);
            if (wantx) lds_v(co + 3 * CA, c.vx);
            if (ey) lds_v(co + 4 * CA, c.vy);
            if (ez) lds_v(co + 5 * CA, c.vz);
        };
        auto direction = [&](int i, const Coef& c) {
            const int ex = PL::ex(i), ey = PL::ey(i), ez = PL::ez(i);
            const float2 w = make_float2(float(PL::w(i)), float(PL::w(i))), one = make_float2(-1.f, -1.f);
            float2 gp[H], gl[H], v[H], gs[H];
            if (i > 0 && i + AHEAD < QG) request(i + AHEAD);
            if (i > 0) {
                float2 lo[H];
                unpack2<T>(ra[i], lo);
                unpack2<T>(rb[i], gp);
#pragma unroll
                for (int h = 0; h < H; ++h) {
                    d0[h] = __ffma2_rn(lo[h], one, d0[h]);  // d0 - lo
                    gl[h] = __ffma2_rn(w, ph[h], lo[h]);
                }
            } else {
#pragma unroll
                for (int h = 0; h < H; ++h) {
                    gl[h] = __ffma2_rn(w, ph[h], d0[h]);
                    gp[h] = d0[h];
                }
            }
            // g_i(y) against the source vector: element k belongs to x + k + ex
            float t = 0.f;
            if (ex > 0) t = __shfl_down_sync(FULL, el(gl, 0), 1, kVecLX);
            if (ex < 0) t = __shfl_up_sync(FULL, el(gl, V - 1), 1, kVecLX);
#pragma unroll
            for (int k = 0; k < V; ++k) el(gs, k) = k + ex < 0 || k + ex >= V ? t : el(gl, (k + ex) & (V - 1));
            // pull_new on pairs (c2 is stored negated; a - v as fma(v, -1, a))
#pragma unroll
            for (int h = 0; h < H; ++h) {
                float2 a = c.cs[h];
                if (ex) a = ex > 0 ? __fadd2_rn(a, c.vx[h]) : __ffma2_rn(c.vx[h], one, a);
                if (ey) a = ey > 0 ? __fadd2_rn(a, c.vy[h]) : __ffma2_rn(c.vy[h], one, a);
                if (ez) a = ez > 0 ? __fadd2_rn(a, c.vz[h]) : __ffma2_rn(c.vz[h], one, a);
                v[h] = __ffma2_rn(w, a, __ffma2_rn(c.c1[h], gp[h], __fmul2_rn(c.c2[h], gs[h])));
            }
            if (ex > 0) {
                t = __shfl_up_sync(FULL, el(v, V - 1), 1, kVecLX);
            } else if (ex < 0) {
                t = __shfl_down_sync(FULL, el(v, 0), 1, kVecLX);
            }
#pragma unroll
            for (int k = 0; k < V; ++k) el(gnew[i], k) = k - ex < 0 || k - ex >= V ? t : el(v, (k - ex) & (V - 1));
        };
#pragma unroll
        for (int i = 1; i < QG; ++i) {
            const int m = reflect_dir<PL>(i, 1);
            if (PL::ex(i) != 0 && m == i - 1) continue;  // done with its partner
            Coef c;
            load_coef(PL::ey(i), PL::ez(i), PL::ex(i) != 0, c);
            direction(i, c);
            if (PL::ex(i) != 0 && m == i + 1) direction(i + 1, c);
        }
        {
            Coef c;
            load_coef(0, 0, false, c);
            direction(0, c);
        }
        // the end sites' populations from beyond the segment (end_sites)
        asm volatile("bar.sync 1, %0;" ::"n"(kVecLX * (kVecTY + 2)) : "memory");
        if (first || last) {
            const int ke = (tw - 1) & (V - 1);  // the segment's last site in its vector
#pragma unroll
            for (int i = 1; i < QG; ++i) {
                if (PL::ex(i) == 0) continue;
                const float t = s_end[(r * 2 + (PL::ex(i) > 0 ? 0 : 1)) * 9 + (PL::ez(i) + 1) * 3 + PL::ey(i) + 1];
                if (PL::ex(i) > 0 && first) el(gnew[i], 0) = t;
                if (PL::ex(i) < 0 && last) {
#pragma unroll
                    for (int k = 0; k < V; ++k)
                        if (k == ke) el(gnew[i], k) = t;
                }
            }
        }
        if (!live) return;
        float2 pn[H];
#pragma unroll
        for (int h = 0; h < H; ++h) {
            pn[h] = make_float2(0.f, 0.f);
#pragma unroll
            for (int kk = 0; kk < QG; ++kk) pn[h] = __fadd2_rn(pn[h], gnew[(kk + 1) % QG][h]);
        }
        if constexpr (WALLS) {
            // populations from beyond a wall: mirrored partners, axis by axis
            // (an x wall holds the first or last site of one vector)
            const int kh = nx - 1 - gx;  // element on the high x wall, if 0 .. 3
            const bool xl = wX && gx == 0, xh = wX && kh < V, yl = wY && gy == 0, yh = wY && gy == ny - 1,
                       zl = wZ && z == 0, zh = wZ && z == nz - 1;
            if (xl | xh | yl | yh | zl | zh) {
#pragma unroll
                for (int i = 1; i < QG; ++i) {
                    const int m = reflect_dir<PL>(i, 1);
                    if (PL::ex(i) > 0 && xl) gnew[i][0].x = gnew[m][0].x;
                    if (PL::ex(i) < 0 && xh) {
#pragma unroll
                        for (int k = 0; k < V; ++k)
                            if (k == kh) el(gnew[i], k) = el(gnew[m], k);
                    }
                }
#pragma unroll
                for (int h = 0; h < H; ++h) {
#pragma unroll
                    for (int i = 1; i < QG; ++i)
                        if ((PL::ey(i) > 0 && yl) || (PL::ey(i) < 0 && yh)) gnew[i][h] = gnew[reflect_dir<PL>(i, 2)][h];
#pragma unroll
                    for (int i = 1; i < QG; ++i)
                        if ((PL::ez(i) > 0 && zl) || (PL::ez(i) < 0 && zh)) gnew[i][h] = gnew[reflect_dir<PL>(i, 4)][h];
                }
                const bool yz = yl | yh | zl | zh;
#pragma unroll
                for (int h = 0; h < H; ++h) {
                    float2 t = gnew[0][h];
#pragma unroll
                    for (int i = 1; i < QG; ++i) t = __fadd2_rn(t, gnew[i][h]);
                    if (yz || (xl && h == 0) || (xh && kh == 2 * h)) pn[h].x = t.x;
                    if (yz || (xh && kh == 2 * h + 1)) pn[h].y = t.y;
                }
            }
        }
        st_v(phin + s, pn);
        uint32_t hh[V] = {};
        if constexpr (UsesSR<S>::value) {
#pragma unroll
            for (int k = 0; k < V; ++k) hh[k] = sr_hash(((uint32_t)z * ny + gy) * nx + gx + k, seed);
        }
#pragma unroll
        for (int i = 1; i < QG; ++i) {
            float o[V];
#pragma unroll
            for (int k = 0; k < V; ++k) o[k] = fma_rn(-float(PL::w(i)), el(pn, k), el(gnew[i], k));
            store_dev<S>(gn + (long long)(i - 1) * n + s, o, hh, (uint32_t)i);
        }
    };

    // Iteration z: coefficients of plane z + 1, then the output of plane z (the
    // first two iterations only fill the coefficient ring).  During the output
    // phase the helpers copy phi of plane z + 3 over plane z - 1, which nothing
    // reads any more.
    for (int p = z0 - 2; p <= z0; ++p) copy_phi(p, tid, kVecNT);
    float2 u[H] = {};
    float ue = load_ue(z0 - 1);
    load_u(z0 - 1, u);
    asm volatile("cp.async.wait_group 0;" ::: "memory");
#pragma unroll 1
    for (int z = z0 - 2; z < z1; ++z) {
        __syncthreads();
        if (vtask) {
            coef_vec(z + 1, cr, lx, u);
            if (z + 1 < z1) load_u(z + 2, u);
        } else if (helper) {
            if (z + 1 >= z0 && z + 1 < z1) prefetch_g(z + 1);
            if (etask) coef_edge(z + 1, hl >> 1, hl & 1, ue);
            if (z + 1 < z1) ue = load_ue(z + 2);
        }
        __syncthreads();
        if (helper) {
            if (z + 1 < z1) {
                copy_phi(z + 3, hl, HN);
                if (z + 3 <= z1) prefetch_phi(z + 4);
            }
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        } else if (z >= z0) {
            if (hp < 0) {
                output_plane(z);
            } else {
                end_sites(z);
                // lanes without an end site leave end_sites early; the arrival is
                // one instruction of the whole warp (bar is the aligned form)
                __syncwarp();
                asm volatile("bar.arrive 1, %0;" ::"n"(kVecLX * (kVecTY + 2)) : "memory");
            }
        }
    }
}

template <class PL, class S, bool WALLS>
__global__ void __launch_bounds__(kVecNT, 2) phi_vec_kernel(const StepArgs args)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_next;
    int* counter = args.counters + args.cur;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        args.counters[args.cur ^ 1] = 0;
        if constexpr (UsesSR<S>::value) args.counters[2 + (args.cur ^ 1)] = args.counters[2 + args.cur] + 1;
    }
    for (;;) {
        if (threadIdx.x == 0) s_next = atomicAdd(counter, 1);
        __syncthreads();
        const int k = s_next;
        if (k >= args.n_items) break;
        phi_vec_item<PL, S, WALLS>(args, args.items[k], reinterpret_cast<float*>(smem_raw));
        __syncthreads();
    }
}

}  // namespace lbpf
