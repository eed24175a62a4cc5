// One-tile form of the fused step for small 2D domains: the arithmetic of
// step_kernel.cuh, operation by operation, with a block per tile instead of a
// march (rounded explicitly where an expression leaves a choice, in the way the
// march's compiled form rounds: the results are the same bits).  A thread owns one
// site of a 32 x 8 region: it requests everything its site needs from global
// memory at once (phi and aux of the region plus one site into shared memory, its
// pulled heat populations, its local and pulled phase-field populations), then
// heat update, gradient, anisotropy and coefficients of the site, one barrier, and
// the phase-field update of the inner 30 x (RY - 2) sites.
//
// Why: a step of a small domain costs one chain of dependent memory latencies.
// The march has five of them and a fetched work item per launch, the tile has
// one: 128^2 FP32 3.2 us a step against 8.9 (22 with the march's former
// eight-row items), at 512^2 10.2 against 18.5.  The ring of sites around a
// tile is computed more than once (1.42 coefficients a site), so large domains
// keep the march (8000^2: 2030 against 1859 us).  A region of 16 rows measured
// 4.1 us at 128^2 and 39.4 at 1024^2 (37.0; fewer, longer blocks), in FP64 25.6
// at 128^2 against 13.9 and 400 at 1200^2 against 420.
#pragma once

#include "step_kernel.cuh"

namespace lbpf {

template <class PL, class UL, class S, bool WALLS>
__global__ void __launch_bounds__(kTileRX* kTileRY) tile_step_kernel(const StepArgs args)
{
    static_assert(PL::D == 2 && UL::D == 2, "2D");
    using R = typename S::Real;
    using T = typename S::T;
    constexpr bool DEV = S::dev;
    constexpr int QG = PL::Q, QU = UL::Q, RY = kTileRY, NT = kTileRX * RY;
    constexpr int FX = kTileRX + 2, FY = RY + 2, FN = FX * FY;  // phi frame: region + 1 site
    constexpr bool SR = UsesSR<S>::value;
    __shared__ R s_phi[FN], s_h[FN];
    __shared__ __align__(16) R s_c1[NT], s_c2[NT], s_s[NT], s_vx[NT], s_vy[NT];

    const WorkItem it = args.items[blockIdx.x];
    const DomainDev& dm = args.doms[it.dom];
    const int nx = dm.nx, ny = dm.ny;
    const long long n = dm.n;
    const int x0 = it.x0, y0 = it.y0;
    const int tw = min(kTileRX - 2, nx - x0), th = min(RY - 2, ny - y0);
    const int tid = threadIdx.x, lx = tid % kTileRX, ly = tid / kTileRX;
    const bool collide = args.collide != 0, use_index = dm.use_index != 0;
    const bool need_h = collide || DEV;
    const uint32_t seed = SR ? (uint32_t)args.counters[2 + args.cur] : 0u;
    if (blockIdx.x == 0 && tid == 0) {
        args.counters[args.cur ^ 1] = 0;
        if (SR) args.counters[2 + (args.cur ^ 1)] = args.counters[2 + args.cur] + 1;  // next step's rounding seed
    }
    const T* __restrict__ gc = static_cast<const T*>(dm.g[args.cur]);
    T* __restrict__ gn = static_cast<T*>(dm.g[args.cur ^ 1]);
    const R* __restrict__ phic = static_cast<const R*>(dm.phi[args.cur]);
    R* __restrict__ phin = static_cast<R*>(dm.phi[args.cur ^ 1]);
    const T* __restrict__ fc = static_cast<const T*>(dm.f[args.fcur]);
    T* __restrict__ fn = static_cast<T*>(dm.f[args.fcur ^ 1]);
    const R* __restrict__ auxc = static_cast<const R*>(dm.aux[args.acur]);
    R* __restrict__ auxn = static_cast<R*>(dm.aux[args.acur ^ 1]);
    const int8_t* __restrict__ Ic = dm.I[args.cur];
    int8_t* __restrict__ In = dm.I[args.cur ^ 1];

    const int bcm = WALLS ? dm.bc : 0;
    const bool wX = (bcm & LBPF_BC_WALL_X) != 0, wY = (bcm & LBPF_BC_WALL_Y) != 0;
    auto wrapx = [&](int v) {
        if (WALLS && wX) return reflect_index(v, nx);
        return v < 0 ? v + nx : (v >= nx ? v - nx : v);
    };
    auto wrapy = [&](int v) {
        if (WALLS && wY) return reflect_index(v, ny);
        return v < 0 ? v + ny : (v >= ny ? v - ny : v);
    };

    // the region's active part: tile + 1 site; this thread's site
    const bool active = lx < tw + 2 && ly < th + 2;
    const int ux = x0 + lx - 1, uy = y0 + ly - 1;  // before wrapping
    const bool inner = active && lx >= 1 && lx <= tw && ly >= 1 && ly <= th;
    int gx = 0, gy = 0, gxm = 0, gxp = 0, gym = 0, gyp = 0;
    if (active) {
        gx = wrapx(ux);
        gy = wrapy(uy);
        gxm = wrapx(gx - 1);
        gxp = wrapx(gx + 1);
        gym = wrapy(gy - 1);
        gyp = wrapy(gy + 1);
    }
    auto site = [&](int ex, int ey) -> long long {  // the neighbour at (ex, ey)
        return (long long)(ey < 0 ? gym : (ey > 0 ? gyp : gy)) * nx + (ex < 0 ? gxm : (ex > 0 ? gxp : gx));
    };
    const long long s = (long long)gy * nx + gx;

    // -- every load of the step ---------------------------------------------
    R pv[2], av[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const int k = tid + j * NT, fy = k / FX, fx = k - fy * FX;
        pv[j] = av[j] = R(0);
        if (k < FN && fx < tw + 4 && fy < th + 4) {
            const long long q = (long long)wrapy(y0 + fy - 2) * nx + wrapx(x0 + fx - 2);
            pv[j] = phic[q];
            if (need_h) av[j] = auxc[q];
        }
    }
    static_assert(FN <= 2 * NT, "two frame sites a thread");
    R fl[QU], floc[DEV ? QU : 1];
    if (active) {
#pragma unroll
        for (int j = 0; j < QU; ++j) {
            if (collide) {
                if (!DEV)
                    fl[j] = to_real(fc[(long long)j * n + site(-UL::ex(j), -UL::ey(j))]);
                else if (j > 0) {
                    fl[j] = to_real(fc[(long long)(j - 1) * n + site(-UL::ex(j), -UL::ey(j))]);
                    floc[DEV ? j : 0] = to_real(fc[(long long)(j - 1) * n + s]);
                }
            } else if (!DEV) {
                fl[j] = to_real(fc[(long long)j * n + s]);
            }
        }
    }
    R gl[QG], gp[QG];
    if (inner) {
#pragma unroll
        for (int i = 0; i < QG; ++i) {
            if (DEV && i == 0) continue;
            const T* a = gc + (long long)(DEV ? i - 1 : i) * n;
            gl[i] = to_real(a[s]);
            if (i > 0) gp[i] = to_real(a[site(-PL::ex(i), -PL::ey(i))]);
        }
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const int k = tid + j * NT;
        if (k < FN) {
            s_phi[k] = pv[j];
            if (need_h) s_h[k] = av[j] + R(0.5) * pv[j];
        }
    }
    __syncthreads();

    const int fk = (ly + 1) * FX + lx + 1;  // this site in the frame
    R phy = R(0);
    if (active) {
        const DomainPar<R>& par = par_of<R>(dm);
        const R ieu = par.inv_eta_u, om_u = R(1) - ieu;
        const R ph = s_phi[fk];
        phy = ph;
        R u = 0;
        if (collide) {
            R fv[QU];
            R d0 = 0;
            if (DEV) {
#pragma unroll
                for (int j = 1; j < QU; ++j) d0 -= floc[DEV ? j : 0];
            }
#pragma unroll
            for (int j = 0; j < QU; ++j) {
                const R hs = s_h[fk - UL::ey(j) * FX - UL::ex(j)];
                const R fj = fma_rn(R(UL::w(j)), hs, mul_rn(om_u, DEV && j == 0 ? d0 : fl[j]));
                fv[j] = fj;
                u += fj;
            }
            if constexpr (WALLS) {
                // (sites beyond a wall are ghosts whose values are never used)
                const bool real = (!wX || (ux >= 0 && ux < nx)) && (!wY || (uy >= 0 && uy < ny));
                const int lo = (wX && gx == 0 ? 1 : 0) | (wY && gy == 0 ? 2 : 0);
                const int hi = (wX && gx == nx - 1 ? 1 : 0) | (wY && gy == ny - 1 ? 2 : 0);
                if (real && (lo | hi)) {
                    mirror_refill<UL, R>(fv, lo, hi);
                    u = 0;
#pragma unroll
                    for (int j = 0; j < QU; ++j) u += fv[j];
                }
            }
            if (inner) {
                if (!DEV) {
#pragma unroll
                    for (int j = 0; j < QU; ++j) fn[(long long)j * n + s] = from_real<T, R>(fv[j]);
                } else {
                    const uint32_t h = SR ? sr_hash((uint32_t)s, seed) : 0u;
#pragma unroll
                    for (int j = 1; j < QU; ++j) {
                        const R v = fv[j] - R(UL::w(j)) * u;
                        if constexpr (SR)
                            fn[(long long)(j - 1) * n + s] = from_real_sr<T>(v, sr_bits(h, 32u + j));
                        else
                            fn[(long long)(j - 1) * n + s] = from_real<T, R>(v);
                    }
                }
            }
        } else {
            if (!DEV) {
#pragma unroll
                for (int j = 0; j < QU; ++j) u += fl[j];
            } else {
                u = s_h[fk];  // C^n + phi^n / 2
            }
        }
        if (inner) auxn[s] = DEV ? (u - R(0.5) * ph) : fma_rn(u, ieu, -(R(0.5) * ph));

        // gradient of phi^n (Sec. 4.2)
        R Gx = 0, Gy = 0;
        if (args.grad == LBPF_GRAD_DD) {
#pragma unroll
            for (int i = 1; i < QG; ++i) {
                if (i > opposite<PL>(i)) continue;
                const int ex = PL::ex(i), ey = PL::ey(i);
                const R dd = s_phi[fk + ey * FX + ex] - s_phi[fk - ey * FX - ex];
                if (ex) Gx = fma_rn(R(ex) * R(PL::w(i)), dd, Gx);
                if (ey) Gy = fma_rn(R(ey) * R(PL::w(i)), dd, Gy);
            }
            const R k = R(1.0 / PL::E2);
            Gx *= k;
            Gy *= k;
        } else {
            Gx = R(0.5) * (s_phi[fk + 1] - s_phi[fk - 1]);
            Gy = R(0.5) * (s_phi[fk + FX] - s_phi[fk - FX]);
        }

        // crystal index (Sec. 4.3)
        int cryst = 1;
        if (use_index) {
            int Iv = Ic[s];
            if (Iv == 0 && Gx * Gx + Gy * Gy > par.xi2) {
#pragma unroll
                for (int i = 1; i < QG; ++i) {
                    const int v = Ic[site(PL::ex(i), PL::ey(i))];
                    if (Iv == 0 && v != 0) Iv = v;
                }
            }
            if (inner) In[s] = (int8_t)Iv;
            cryst = Iv;
        }

        R a = 1, Nx = 0, Ny = 0;
        if (cryst > 0 && cryst <= dm.n_crystals) {
            R n2 = 0;
            anisotropy<R, 2>(dm.cr[cryst - 1], Gx, Gy, R(0), a, Nx, Ny, n2);
        }
        const R De2 = par.De2, qphi = par.qphi, lam = par.lambda;
        R iA2 = R(1), ieta = par.ieta1;
        if (sizeof(R) == 4 || a != R(1)) {  // (FP64 divides: not where there is no interface)
            const R A2 = a * a;
            iA2 = recip<R>(A2);
            ieta = recip<R>(A2 * De2 + R(0.5));
        }
        const R omp = (R(1) - ph) * (R(1) + ph);
        const R Qphi = (ph - lam * u * omp) * omp;
        const R vf = -De2 * ieta * iA2;
        s_c1[tid] = (R(1) - ieta) * iA2;
        s_c2[tid] = iA2 - R(1);
        s_s[tid] = DEV ? (ph + qphi * Qphi) * iA2 : fma_rn(qphi, Qphi, mul_rn(ph, ieta)) * iA2;
        s_vx[tid] = vf * Nx;
        s_vy[tid] = vf * Ny;
    }
    __syncthreads();
    if (!inner) return;

    // phase-field collision + streaming (see output_plane of step_kernel)
    R gnew[QG];
    R phinew = 0, d0 = 0;
#pragma unroll
    for (int k = 0; k < QG; ++k) {
        const int i = DEV ? (k + 1) % QG : k;
        const int ex = PL::ex(i), ey = PL::ey(i);
        const int c = tid - ey * kTileRX - ex;
        R l, p;
        if (!DEV) {
            l = gl[i];
            p = i == 0 ? l : gp[i];
        } else if (i > 0) {
            d0 = sub_rn(d0, gl[i]);
            l = fma_rn(R(PL::w(i)), phy, gl[i]);
            p = gp[i];
        } else {
            l = fma_rn(R(PL::w(0)), phy, d0);
            p = d0;
        }
        const R v = pull_new<R>(ex, ey, 0, R(PL::w(i)), s_c1[c], s_c2[c], s_s[c], ex ? s_vx[c] : R(0), ey ? s_vy[c] : R(0),
                                R(0), p, l);
        phinew = add_rn(phinew, v);
        gnew[i] = v;
    }
    if constexpr (WALLS) {
        const int lo = (wX && gx == 0 ? 1 : 0) | (wY && gy == 0 ? 2 : 0);
        const int hi = (wX && gx == nx - 1 ? 1 : 0) | (wY && gy == ny - 1 ? 2 : 0);
        if (lo | hi) {
            mirror_refill<PL, R>(gnew, lo, hi);
            phinew = 0;
#pragma unroll
            for (int i = 0; i < QG; ++i) phinew += gnew[i];
        }
    }
    phin[s] = phinew;
    if (!DEV) {
#pragma unroll
        for (int i = 0; i < QG; ++i) gn[(long long)i * n + s] = from_real<T, R>(gnew[i]);
    } else {
        const uint32_t h = SR ? sr_hash((uint32_t)s, seed) : 0u;
#pragma unroll
        for (int i = 1; i < QG; ++i) {
            const R v = fma_rn(-R(PL::w(i)), phinew, gnew[i]);
            if constexpr (SR)
                gn[(long long)(i - 1) * n + s] = from_real_sr<T>(v, sr_bits(h, (uint32_t)i));
            else
                gn[(long long)(i - 1) * n + s] = from_real<T, R>(v);
        }
    }
}

}  // namespace lbpf
