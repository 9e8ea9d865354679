// Generic RKL2 conduction kernels: one thread per cell, any dtype (float /
// double), 1-3 active axes, periodic or Dirichlet boundaries.  The stage
// kernel serves 1D grids, 2D FP32 grids with a finite limiter floor and what
// the tiled and column-march kernels do not cover; each cell evaluates the
// fluxes on all of its faces straight from global memory (L1/L2 absorb the
// neighbour re-reads).  The face fluxes, the advection step and the statistics
// of every grid are here too.
#include <algorithm>

#include "rkl_launch.h"

namespace rkl {
namespace {

template <typename R>
struct Field {
    const R* T;
    const R* b;
    KGrid<R> g;

    // T at a cell that may lie one cell outside the grid on active axes.
    __device__ __forceinline__ R t(int i, int j, int k) const
    {
        if (g.bc == 1) {
            if (i < 0 || i >= g.n[0] || j < 0 || j >= g.n[1] || k < 0 || k >= g.n[2]) return g.bcv;
        } else {
            i = wrap(i, g.n[0]);
            j = wrap(j, g.n[1]);
            k = wrap(k, g.n[2]);
        }
        return T[((int64_t)k * g.n[1] + j) * g.n[0] + i];
    }
    // Component e of b; ghosts copy the nearest interior cell (Dirichlet).
    __device__ __forceinline__ R bc(int e, int i, int j, int k) const
    {
        if (g.bc == 1) {
            i = clampi(i, g.n[0]);
            j = clampi(j, g.n[1]);
            k = clampi(k, g.n[2]);
        } else {
            i = wrap(i, g.n[0]);
            j = wrap(j, g.n[1]);
            k = wrap(k, g.n[2]);
        }
        return b[(int64_t)e * g.ncell + ((int64_t)k * g.n[1] + j) * g.n[0] + i];
    }
};

// Flux component d on the face between P = (i,j,k) and P + e_d.
template <typename R, int NDIM, bool SPITZER, bool SAT>
__device__ __forceinline__ R face(const Field<R>& f, const KPhys<R>& p, int d, int i, int j, int k)
{
    int P[3] = {i, j, k};
    int Q[3] = {i, j, k};
    Q[d] += 1;
    R TL = f.t(P[0], P[1], P[2]);
    R TR = f.t(Q[0], Q[1], Q[2]);
    R gn = (TR - TL) * f.g.inv_dx[d];
    R gt[2] = {R(0), R(0)};
    R bt[2] = {R(0), R(0)};
    // Appendix C: MC-limited transverse gradients where the face's lower
    // temperature is below the floor (an infinite floor limits everywhere)
    const bool limit = p.limiter && fmin(TL, TR) < p.lfloor;
    int m = 0;
#pragma unroll
    for (int e = 0; e < NDIM; ++e) {
        if (e == d) continue;
        int Pp[3] = {P[0], P[1], P[2]}, Pm[3] = {P[0], P[1], P[2]};
        int Qp[3] = {Q[0], Q[1], Q[2]}, Qm[3] = {Q[0], Q[1], Q[2]};
        Pp[e] += 1; Qp[e] += 1; Pm[e] -= 1; Qm[e] -= 1;
        if (limit) {
            const R upL = f.t(Pp[0], Pp[1], Pp[2]) - TL, downL = TL - f.t(Pm[0], Pm[1], Pm[2]);
            const R upR = f.t(Qp[0], Qp[1], Qp[2]) - TR, downR = TR - f.t(Qm[0], Qm[1], Qm[2]);
            gt[m] = mc_limit(mc_limit(upL, downL), mc_limit(upR, downR)) * f.g.inv_dx[e];
        } else {
            gt[m] = (f.t(Pp[0], Pp[1], Pp[2]) + f.t(Qp[0], Qp[1], Qp[2])
                   - f.t(Pm[0], Pm[1], Pm[2]) - f.t(Qm[0], Qm[1], Qm[2])) * f.g.inv_4dx[e];
        }
        bt[m] = R(0.5) * (f.bc(e, P[0], P[1], P[2]) + f.bc(e, Q[0], Q[1], Q[2]));
        ++m;
    }
    R bn = R(0.5) * (f.bc(d, P[0], P[1], P[2]) + f.bc(d, Q[0], Q[1], Q[2]));
    return face_flux<R, SPITZER, SAT>(TL, TR, gn, gt[0], gt[1], bn, bt[0], bt[1], p);
}

template <typename R>
struct StageArgs {
    const R* Y0;
    R* MY0;
    const R* Yjm1;
    const R* Yjm2;
    R* Yj;
    const R* coef_tab;
    int j;
    int mode;
};

template <typename R, int NDIM, bool SPITZER, bool SAT>
__global__ void __launch_bounds__(256) stage_generic_kernel(KGrid<R> g, KPhys<R> p, StageArgs<R> a,
                                                            const R* __restrict__ b, KCoef<R> cf,
                                                            unsigned* status)
{
    int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= g.ncell) return;
    int i = (int)(c % g.n[0]);
    int64_t r = c / g.n[0];
    int j = (int)(r % g.n[1]);
    int k = (int)(r / g.n[1]);

    // the field whose M is taken: Y0 for stage 1 / Euler, Yjm1 otherwise
    Field<R> f{a.mode == 2 || a.mode == 0 ? a.Yjm1 : a.Y0, b, g};
    R div = R(0);
#pragma unroll
    for (int d = 0; d < NDIM; ++d) {
        int lo[3] = {i, j, k};
        lo[d] -= 1;
        R Fhi = face<R, NDIM, SPITZER, SAT>(f, p, d, i, j, k);
        R Flo = face<R, NDIM, SPITZER, SAT>(f, p, d, lo[0], lo[1], lo[2]);
        div += (Fhi - Flo) * g.inv_dx[d];
    }
    R M = -div;
    if (a.mode == 0) {
        a.Yj[c] = M;
        return;
    }
    if (a.coef_tab) {
        const R* t = a.coef_tab + 4 * a.j;
        cf.mu = t[0]; cf.nu = t[1]; cf.mt = t[2]; cf.gt = t[3];
    }
    R y0 = a.Y0[c];
    R y;
    if (a.mode == 1) {
        if (a.MY0) a.MY0[c] = M;
        y = y0 + cf.mt * M;
    } else {
        R inc = cf.mu * (a.Yjm1[c] - y0) + cf.nu * (a.Yjm2[c] - y0) + cf.mt * M + cf.gt * a.MY0[c];
        y = y0 + inc;
    }
    check_value<R, SPITZER>(y, status);
    a.Yj[c] = y;
}

template <typename R, int NDIM, bool SPITZER, bool SAT>
__global__ void __launch_bounds__(256) flux_generic_kernel(KGrid<R> g, KPhys<R> p, const R* __restrict__ T,
                                                           const R* __restrict__ b, R* Fx, R* Fy, R* Fz)
{
    int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= g.ncell) return;
    int i = (int)(c % g.n[0]);
    int64_t r = c / g.n[0];
    int j = (int)(r % g.n[1]);
    int k = (int)(r / g.n[1]);
    Field<R> f{T, b, g};
    R* F[3] = {Fx, Fy, Fz};
#pragma unroll
    for (int d = 0; d < NDIM; ++d) F[d][c] = face<R, NDIM, SPITZER, SAT>(f, p, d, i, j, k);
}

// The same faces on 3D grids without a limiter: a thread per (x, y) column
// marches `nzc` planes with 32-bit offsets fixed at its start, each plane's
// T and b read once per thread and handed to the next (17 reads a cell; the
// kernel above does 64-bit divisions and about 60).  The flux is face_flux
// on the same operands with its fused multiply-adds spelled out as the kernel
// above has them: the surrogate's features round these fluxes to BF16 and
// the network's output follows every rounding that flips, so the bits have to
// stay (left to the compiler the z-face came out in another order).  96^3 FP32 Spitzer: 54 -> 15 us.
template <typename R, bool SPITZER, bool SAT>
__device__ __forceinline__ R face_flux_fused(R TL, R TR, R gn, R g1, R g2, R bn, R b1, R b2, const KPhys<R>& p)
{
    const R Tf = R(0.5) * (TL + TR);
    const R kpar = kappa_par<R, SPITZER>(Tf, p);
    const R kperp = p.kperp * kpar;
    const R bdg = fma(b2, g2, fma(bn, gn, b1 * g1));
    R Fn = fma(-kpar * bn, bdg, -(kperp * gn));
    if (SAT) {
        const R F1 = fma(-kpar * b1, bdg, -(kperp * g1));
        const R F2 = fma(-kpar * b2, bdg, -(kperp * g2));
        const R Fmag = dsqrt<R>(fma(F2, F2, fma(Fn, Fn, F1 * F1)));
        const R Tq = p.upwind ? (Fn >= R(0) ? TL : TR) : Tf;
        const R q = p.q0 * Tq * dsqrt<R>(Tq);
        Fn = ddiv<R>(q, q + Fmag) * Fn;
    }
    return Fn;
}

template <typename R, bool SPITZER, bool SAT>
__global__ void __launch_bounds__(256) flux3_kernel(KGrid<R> g, KPhys<R> p, const R* __restrict__ T,
                                                    const R* __restrict__ b, R* __restrict__ Fx, R* __restrict__ Fy,
                                                    R* __restrict__ Fz, int nzc)
{
    const int nx = g.n[0], ny = g.n[1], nz = g.n[2];
    const int i = blockIdx.x * 32 + (threadIdx.x & 31), j = blockIdx.y * 8 + (threadIdx.x >> 5);
    if (i >= nx || j >= ny) return;
    const bool dir = g.bc == 1;
    auto at = [&](int v, int n) { return dir ? clampi(v, n) : wrap(v, n); };
    const int im = at(i - 1, nx), ip = at(i + 1, nx), jm = at(j - 1, ny), jp = at(j + 1, ny);
    const bool gxm = dir && i == 0, gxp = dir && i == nx - 1, gym = dir && j == 0, gyp = dir && j == ny - 1;
    const int oc = j * nx + i, oxm = j * nx + im, oxp = j * nx + ip, oym = jm * nx + i, oyp = jp * nx + i;
    const int opp = jp * nx + ip, opm = jm * nx + ip, omp = jp * nx + im;
    const int z0 = blockIdx.z * nzc, z1 = min(z0 + nzc, nz);
    auto t = [&](int64_t pl, int q, bool ghost) { return ghost ? g.bcv : T[pl + q]; };
    struct Q {
        R c, xm, xp, ym, yp;
        R b[3];
    };
    auto read = [&](int z, int64_t& pl) -> Q {
        pl = (int64_t)at(z, nz) * g.plane;
        const bool zg = dir && (z < 0 || z >= nz);
        Q q;
        q.c = t(pl, oc, zg);
        q.xm = t(pl, oxm, zg || gxm);
        q.xp = t(pl, oxp, zg || gxp);
        q.ym = t(pl, oym, zg || gym);
        q.yp = t(pl, oyp, zg || gyp);
#pragma unroll
        for (int e = 0; e < 3; ++e) q.b[e] = b[e * g.ncell + pl + oc];
        return q;
    };
    const R hf = R(0.5);
    int64_t pl, pn;
    const bool zm = dir && z0 == 0;
    const int64_t pm = (int64_t)at(z0 - 1, nz) * g.plane;
    R mc = t(pm, oc, zm), mx = t(pm, oxp, zm || gxp), my = t(pm, oyp, zm || gyp);
    Q c = read(z0, pl);
    for (int z = z0; z < z1; ++z) {
        const Q n = read(z + 1, pn);
        const R pp = t(pl, opp, gxp || gyp), pd = t(pl, opm, gxp || gym), mp = t(pl, omp, gxm || gyp);
        R bx[3], by[3];
#pragma unroll
        for (int e = 0; e < 3; ++e) {
            bx[e] = b[e * g.ncell + pl + oxp];
            by[e] = b[e * g.ncell + pl + oyp];
        }
        Fx[pl + oc] = face_flux_fused<R, SPITZER, SAT>(c.c, c.xp, (c.xp - c.c) * g.inv_dx[0],
                                                 (c.yp + pp - c.ym - pd) * g.inv_4dx[1],
                                                 (n.c + n.xp - mc - mx) * g.inv_4dx[2], hf * (c.b[0] + bx[0]),
                                                 hf * (c.b[1] + bx[1]), hf * (c.b[2] + bx[2]), p);
        Fy[pl + oc] = face_flux_fused<R, SPITZER, SAT>(c.c, c.yp, (c.yp - c.c) * g.inv_dx[1],
                                                 (c.xp + pp - c.xm - mp) * g.inv_4dx[0],
                                                 (n.c + n.yp - mc - my) * g.inv_4dx[2], hf * (c.b[1] + by[1]),
                                                 hf * (c.b[0] + by[0]), hf * (c.b[2] + by[2]), p);
        Fz[pl + oc] = face_flux_fused<R, SPITZER, SAT>(c.c, n.c, (n.c - c.c) * g.inv_dx[2],
                                                 (c.xp + n.xp - c.xm - n.xm) * g.inv_4dx[0],
                                                 (c.yp + n.yp - c.ym - n.ym) * g.inv_4dx[1], hf * (c.b[2] + n.b[2]),
                                                 hf * (c.b[0] + n.b[0]), hf * (c.b[1] + n.b[1]), p);
        mc = c.c;
        mx = c.xp;
        my = c.yp;
        c = n;
        pl = pn;
    }
}

// Threads per block: 256, halved (down to one warp) while the grid would
// leave SMs idle -- small FP64 grids (the 100 x 100 ring) are bound by the
// per-SM FP64 rate, so they need every SM more than full blocks.
int sm_count()
{
    static int nsm = 0;
    if (nsm == 0) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || nsm <= 0)
            nsm = 152;
    }
    return nsm;
}
// Whether the marching kernels of the face fluxes and of the advection (tiles of
// 32 x 8 columns, `nzc` planes a thread, 3D) beat one thread per cell.  FP32:
// idle lanes cost nothing while all warps are resident at once, and from eight
// columns on the march's cheaper addressing outweighs them (rows of 4 cells, 368
// x 41 of them: 0.8 of the speed; of 8, 805 x 20: 1.2).  FP64 runs at the FP64
// rate either way, so idle lanes and uneven SMs are lost time and large grids of
// full tiles gain 0-6% (flux: 256^3 3.59 -> 3.40 ms, but 64^3 62 against 68 us
// and 40 x 208 x 123 0.23 against 0.35 ms).
template <typename R>
bool march_pays(const KGrid<R>& g, int nzc)
{
    if (g.plane >= ((int64_t)1 << 31) || g.n[1] > 8 * 65535) return false;
    const int64_t warps = (int64_t)((g.n[0] + 31) / 32) * g.n[1] * ((g.n[2] + nzc - 1) / nzc);
    if (sizeof(R) == 8) return g.n[0] % 32 == 0 && g.n[1] % 8 == 0 && warps >= 128 * (int64_t)sm_count();
    return g.n[0] >= 8 || warps <= 16 * (int64_t)sm_count();
}
int generic_block(int64_t ncell)
{
    int tpb = 256;
    while (tpb > 32 && (ncell + tpb - 1) / tpb < 2 * (int64_t)sm_count()) tpb /= 2;
    return tpb;
}

template <typename R, int NDIM, bool SPITZER, bool SAT>
cudaError_t stage_impl(const void* grid, const void* phys, const StageIO& io, const void* coef,
                       unsigned* status, cudaStream_t st)
{
    const KGrid<R>& g = *static_cast<const KGrid<R>*>(grid);
    const KPhys<R>& p = *static_cast<const KPhys<R>*>(phys);
    StageArgs<R> a{static_cast<const R*>(io.Y0), static_cast<R*>(io.MY0),
                   static_cast<const R*>(io.Yjm1), static_cast<const R*>(io.Yjm2),
                   static_cast<R*>(io.Yj), static_cast<const R*>(io.coef_tab), io.j, io.mode};
    KCoef<R> cf = coef ? *static_cast<const KCoef<R>*>(coef) : KCoef<R>{R(0), R(0), R(0), R(0)};
    const int tpb = generic_block(g.ncell);
    const int64_t blocks = (g.ncell + tpb - 1) / tpb;
    stage_generic_kernel<R, NDIM, SPITZER, SAT><<<(unsigned)blocks, tpb, 0, st>>>(
        g, p, a, static_cast<const R*>(io.b), cf, status);
    return cudaGetLastError();
}

template <typename R, int NDIM, bool SPITZER, bool SAT>
cudaError_t flux_impl(const void* grid, const void* phys, const void* T, const void* b, void* F[3],
                      cudaStream_t st)
{
    const KGrid<R>& g = *static_cast<const KGrid<R>*>(grid);
    const KPhys<R>& p = *static_cast<const KPhys<R>*>(phys);
    const int nzc = std::max(4, (g.n[2] + 65534) / 65535);
    if (NDIM == 3 && !p.limiter && march_pays(g, nzc)) {
        const dim3 grid((g.n[0] + 31) / 32, (g.n[1] + 7) / 8, (g.n[2] + nzc - 1) / nzc);
        flux3_kernel<R, SPITZER, SAT><<<grid, 256, 0, st>>>(g, p, static_cast<const R*>(T), static_cast<const R*>(b),
                                                            static_cast<R*>(F[0]), static_cast<R*>(F[1]),
                                                            static_cast<R*>(F[2]), nzc);
        return cudaGetLastError();
    }
    const int tpb = generic_block(g.ncell);
    const int64_t blocks = (g.ncell + tpb - 1) / tpb;
    flux_generic_kernel<R, NDIM, SPITZER, SAT><<<(unsigned)blocks, tpb, 0, st>>>(
        g, p, static_cast<const R*>(T), static_cast<const R*>(b), static_cast<R*>(F[0]),
        static_cast<R*>(F[1]), static_cast<R*>(F[2]));
    return cudaGetLastError();
}

// --------------------------------------------------------------------------
// Operator splitting (Section 3): the hyperbolic step as the passive
// advection dT/dt = -div(u T) of the energy density by a cell-centred
// velocity u ([3][ncell], ghosts copy the nearest interior cell as b does),
// conservative donor cell: face velocity = mean of the two cells, face flux
// = u_f T(upwind cell).

template <typename R>
__device__ __forceinline__ R adv_flux(const Field<R>& f, int d, int i, int j, int k)
{
    int Q[3] = {i, j, k};
    Q[d] += 1;
    const R uf = R(0.5) * (f.bc(d, i, j, k) + f.bc(d, Q[0], Q[1], Q[2]));
    return uf * (uf >= R(0) ? f.t(i, j, k) : f.t(Q[0], Q[1], Q[2]));
}

template <typename R, int NDIM>
__global__ void __launch_bounds__(256) advect_kernel(KGrid<R> g, const R* __restrict__ T, const R* __restrict__ u,
                                                     R* __restrict__ Tout, R dt)
{
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= g.ncell) return;
    const int i = (int)(c % g.n[0]);
    const int64_t r = c / g.n[0];
    const int j = (int)(r % g.n[1]);
    const int k = (int)(r / g.n[1]);
    const Field<R> f{T, u, g};
    R div = R(0);
#pragma unroll
    for (int d = 0; d < NDIM; ++d) {
        int lo[3] = {i, j, k};
        lo[d] -= 1;
        div += (adv_flux(f, d, i, j, k) - adv_flux(f, d, lo[0], lo[1], lo[2])) * g.inv_dx[d];
    }
    Tout[c] = T[c] - dt * div;
}

// The same step on 3D grids with 32-bit offsets: a thread per (x, y) column
// marches `nzc` planes and keeps the z-face flux and the next plane's T and
// u_z in registers, so that every z-face is evaluated once; the in-plane
// neighbours come through L1.  Bound by HBM (5 words a cell): the kernel
// above spent its time on 64-bit divisions and both faces of every axis.
// 192 x 128 x 96 Dirichlet FP32, cold caches: 52 -> 19 us.
template <typename R>
__global__ void __launch_bounds__(256) advect3_kernel(KGrid<R> g, const R* __restrict__ T, const R* __restrict__ u,
                                                      R* __restrict__ Tout, R dt, int nzc)
{
    const int nx = g.n[0], ny = g.n[1], nz = g.n[2];
    const int i = blockIdx.x * 32 + (threadIdx.x & 31), j = blockIdx.y * 8 + (threadIdx.x >> 5);
    if (i >= nx || j >= ny) return;
    const bool dir = g.bc == 1;
    auto at = [&](int v, int n) { return dir ? clampi(v, n) : wrap(v, n); };
    const int z0 = blockIdx.z * nzc, z1 = min(z0 + nzc, nz);
    const int im = at(i - 1, nx), ip = at(i + 1, nx), jm = at(j - 1, ny), jp = at(j + 1, ny);
    const int o = j * nx + i, oxm = j * nx + im, oxp = j * nx + ip, oym = jm * nx + i, oyp = jp * nx + i;
    const bool gxm = dir && i == 0, gxp = dir && i == nx - 1, gym = dir && j == 0, gyp = dir && j == ny - 1;
    const R* ux = u;
    const R* uy = u + g.ncell;
    const R* uz = u + 2 * g.ncell;
    auto plane = [&](int z) { return (int64_t)at(z, nz) * g.plane; };
    auto t = [&](int64_t pl, int q, bool ghost) { return ghost ? g.bcv : T[pl + q]; };
    auto flux = [](R ul, R uh, R Tl, R Th) {
        const R uf = R(0.5) * (ul + uh);
        return uf * (uf >= R(0) ? Tl : Th);
    };
    int64_t pl = plane(z0), pn = plane(z0 - 1);
    R Tc = T[pl + o], wc = uz[pl + o];
    R Fl = flux(uz[pn + o], wc, t(pn, o, dir && z0 == 0), Tc);
    for (int z = z0; z < z1; ++z) {
        pn = plane(z + 1);
        const R Tn = t(pn, o, dir && z == nz - 1), wn = uz[pn + o];
        const R uc = ux[pl + o], vc = uy[pl + o];
        const R Fh = flux(wc, wn, Tc, Tn);
        R div = R(0);
        div += (flux(uc, ux[pl + oxp], Tc, t(pl, oxp, gxp)) - flux(ux[pl + oxm], uc, t(pl, oxm, gxm), Tc)) * g.inv_dx[0];
        div += (flux(vc, uy[pl + oyp], Tc, t(pl, oyp, gyp)) - flux(uy[pl + oym], vc, t(pl, oym, gym), Tc)) * g.inv_dx[1];
        div += (Fh - Fl) * g.inv_dx[2];
        Tout[pl + o] = Tc - dt * div;
        Fl = Fh;
        Tc = Tn;
        wc = wn;
        pl = pn;
    }
}

template <typename R>
cudaError_t advect_impl(const LaunchCfg& c, const void* grid, const void* T, const void* u, void* Tout, double dt,
                        cudaStream_t st)
{
    const KGrid<R>& g = *static_cast<const KGrid<R>*>(grid);
    const int tpb = generic_block(g.ncell);
    const unsigned blocks = (unsigned)((g.ncell + tpb - 1) / tpb);
    const R* Tp = static_cast<const R*>(T);
    const R* up = static_cast<const R*>(u);
    R* op = static_cast<R*>(Tout);
    // two planes per thread: more of them serialise the loads of a plane behind
    // the last one's (7 planes: 24 us on 192 x 128 x 96)
    const int nzc = std::max(2, (g.n[2] + 65534) / 65535);
    if (c.ndim == 1) advect_kernel<R, 1><<<blocks, tpb, 0, st>>>(g, Tp, up, op, (R)dt);
    else if (c.ndim == 2) advect_kernel<R, 2><<<blocks, tpb, 0, st>>>(g, Tp, up, op, (R)dt);
    else if (march_pays(g, nzc)) {
        const dim3 xy((g.n[0] + 31) / 32, (g.n[1] + 7) / 8);
        advect3_kernel<R><<<dim3(xy.x, xy.y, (g.n[2] + nzc - 1) / nzc), 256, 0, st>>>(g, Tp, up, op, (R)dt, nzc);
    } else advect_kernel<R, 3><<<blocks, tpb, 0, st>>>(g, Tp, up, op, (R)dt);
    return cudaGetLastError();
}

template <typename R, int NDIM>
cudaError_t stage_dispatch_phys(const LaunchCfg& c, const void* grid, const void* phys,
                                const StageIO& io, const void* coef, unsigned* status, cudaStream_t st)
{
    if (c.spitzer) {
        if (c.saturate) return stage_impl<R, NDIM, true, true>(grid, phys, io, coef, status, st);
        return stage_impl<R, NDIM, true, false>(grid, phys, io, coef, status, st);
    }
    if (c.saturate) return stage_impl<R, NDIM, false, true>(grid, phys, io, coef, status, st);
    return stage_impl<R, NDIM, false, false>(grid, phys, io, coef, status, st);
}

template <typename R>
cudaError_t stage_dispatch_ndim(const LaunchCfg& c, const void* grid, const void* phys,
                                const StageIO& io, const void* coef, unsigned* status, cudaStream_t st)
{
    switch (c.ndim) {
        case 1: return stage_dispatch_phys<R, 1>(c, grid, phys, io, coef, status, st);
        case 2: return stage_dispatch_phys<R, 2>(c, grid, phys, io, coef, status, st);
        case 3: return stage_dispatch_phys<R, 3>(c, grid, phys, io, coef, status, st);
    }
    return cudaErrorInvalidValue;
}

template <typename R, int NDIM>
cudaError_t flux_dispatch_phys(const LaunchCfg& c, const void* grid, const void* phys, const void* T,
                               const void* b, void* F[3], cudaStream_t st)
{
    if (c.spitzer) {
        if (c.saturate) return flux_impl<R, NDIM, true, true>(grid, phys, T, b, F, st);
        return flux_impl<R, NDIM, true, false>(grid, phys, T, b, F, st);
    }
    if (c.saturate) return flux_impl<R, NDIM, false, true>(grid, phys, T, b, F, st);
    return flux_impl<R, NDIM, false, false>(grid, phys, T, b, F, st);
}

template <typename R>
cudaError_t flux_dispatch_ndim(const LaunchCfg& c, const void* grid, const void* phys, const void* T,
                               const void* b, void* F[3], cudaStream_t st)
{
    switch (c.ndim) {
        case 1: return flux_dispatch_phys<R, 1>(c, grid, phys, T, b, F, st);
        case 2: return flux_dispatch_phys<R, 2>(c, grid, phys, T, b, F, st);
        case 3: return flux_dispatch_phys<R, 3>(c, grid, phys, T, b, F, st);
    }
    return cudaErrorInvalidValue;
}

// ---------------------------------------------------------------------------
// Statistics (max, min, sum) of a grid array in a fixed reduction order.
//
// The FP64 units of this GPU retire two lanes per SM and clock, so a 64-bit
// compare per lane and shuffle step costs more than reading the array: with
// FP64 folds the pass over 256^3 FP32 cells took 37 us against 10 us of
// memory time, and 860 thousand FP64 cells took 32 us.  The extrema are
// therefore kept in the data's own type (FP32) or as order-preserving
// integers (FP64), both exact, with a NaN flag beside them; only the sum
// (energy), and only when asked for, is FP64 arithmetic.

template <typename R>
struct Ext;

template <>
struct Ext<float> {
    float mx = -INFINITY, mn = INFINITY;
    int nan = 0;
    __device__ __forceinline__ void add(float v)
    {
        mx = fmaxf(mx, v);
        mn = fminf(mn, v);
        nan |= v != v;
    }
    __device__ __forceinline__ float max_value() const { return nan ? NAN : mx; }
    __device__ __forceinline__ float min_value() const { return nan ? NAN : mn; }
};

template <>
struct Ext<double> {
    // the total order of the doubles as signed integers
    static __device__ __forceinline__ long long key(long long b) { return b ^ ((b >> 63) & 0x7fffffffffffffffll); }
    long long mx = key((long long)0xfff0000000000000ull), mn = 0x7ff0000000000000ll;    // -inf, +inf
    int nan = 0;
    __device__ __forceinline__ void add(double v)
    {
        const long long b = __double_as_longlong(v), k = key(b);
        mx = max(mx, k);
        mn = min(mn, k);
        nan |= (b & 0x7fffffffffffffffll) > 0x7ff0000000000000ll;
    }
    __device__ __forceinline__ double max_value() const { return nan ? NAN : __longlong_as_double(key(mx)); }
    __device__ __forceinline__ double min_value() const { return nan ? NAN : __longlong_as_double(key(mn)); }
};

// Folds the block's extrema and (SUM) sum into thread 0 (256 threads).
template <typename R, bool SUM>
__device__ __forceinline__ void block_fold(Ext<R>& e, double& sm)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        e.mx = max(e.mx, __shfl_xor_sync(0xffffffffu, e.mx, o));
        e.mn = min(e.mn, __shfl_xor_sync(0xffffffffu, e.mn, o));
        if (SUM) sm += __shfl_xor_sync(0xffffffffu, sm, o);
    }
    __shared__ decltype(Ext<R>::mx) smx[8], smn[8];
    __shared__ double ss[8];
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    e.nan = __syncthreads_or(e.nan);
    if (l == 0) { smx[w] = e.mx; smn[w] = e.mn; ss[w] = sm; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int q = 1; q < 8; ++q) {
            e.mx = max(e.mx, smx[q]);
            e.mn = min(e.mn, smn[q]);
            if (SUM) sm += ss[q];
        }
    }
}

// What the statistics run over: an array, or the rate lambda(c) = sum_d
// |u_d| / dx_d of a velocity (the denominator of Eq. dt_h), four cells at a
// time where the arrays allow it.
template <typename R>
struct ArraySrc {
    const R* T;
    __device__ __forceinline__ R at(int64_t c) const { return T[c]; }
    __device__ __forceinline__ float4 at4(int64_t c) const { return reinterpret_cast<const float4*>(T)[c]; }
    __device__ __forceinline__ bool wide(int64_t n) const
    {
        return sizeof(R) == 4 && (n & 3) == 0 && (reinterpret_cast<uintptr_t>(T) & 15) == 0;
    }
};
template <typename R, int NDIM>
struct RateSrc {
    const R* u;
    int64_t n;
    R inv[3];
    __device__ __forceinline__ R at(int64_t c) const
    {
        R v = R(0);
#pragma unroll
        for (int d = 0; d < NDIM; ++d) v += fabs(u[(int64_t)d * n + c]) * inv[d];
        return v;
    }
    __device__ __forceinline__ float4 at4(int64_t c) const
    {
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int d = 0; d < NDIM; ++d) {
            const float4 w = reinterpret_cast<const float4*>(u + (int64_t)d * n)[c];
            const float s = (float)inv[d];
            v.x += fabsf(w.x) * s; v.y += fabsf(w.y) * s; v.z += fabsf(w.z) * s; v.w += fabsf(w.w) * s;
        }
        return v;
    }
    __device__ __forceinline__ bool wide(int64_t n) const
    {
        return sizeof(R) == 4 && (n & 3) == 0 && (reinterpret_cast<uintptr_t>(u) & 15) == 0;
    }
};

// The extrema (and sum) of cells 0 .. n - 1 of a source over one grid of
// blocks or one block: thread t0 of `stride` threads.
template <typename R, bool SUM, class Src>
__device__ __forceinline__ void thread_stats(const Src& src, int64_t n, int64_t t0, int64_t stride, Ext<R>& e,
                                             double& sm)
{
    auto fold = [&](R v) {
        e.add(v);
        if (SUM) sm += (double)v;
    };
    if (src.wide(n)) {
        const int64_t n4 = n / 4;
        int64_t c = t0;
        // four independent 16-byte loads in flight per thread
        for (; c + 3 * stride < n4; c += 4 * stride) {
            float4 v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = src.at4(c + u * stride);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                fold((R)v[u].x); fold((R)v[u].y); fold((R)v[u].z); fold((R)v[u].w);
            }
        }
        for (; c < n4; c += stride) {
            const float4 v = src.at4(c);
            fold((R)v.x); fold((R)v.y); fold((R)v.z); fold((R)v.w);
        }
    } else {
        int64_t c = t0;
        for (; c + 3 * stride < n; c += 4 * stride) {
            R v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = src.at(c + u * stride);
#pragma unroll
            for (int u = 0; u < 4; ++u) fold(v[u]);
        }
        for (; c < n; c += stride) fold(src.at(c));
    }
}

// Each block leaves its partial {max, min, sum}; the block that finishes
// last (ticket counter at partials[3 * kStatsBlocks], reset by that block)
// folds all partials in a fixed order, so the result does not depend on
// which block is last.
template <typename R, bool SUM, class Src>
__global__ void __launch_bounds__(256) stats_kernel(Src src, int64_t n, double* partials, double* out,
                                                    unsigned* status)
{
    Ext<R> e;
    double sm = 0.0;
    thread_stats<R, SUM>(src, n, (int64_t)blockIdx.x * blockDim.x + threadIdx.x, (int64_t)gridDim.x * blockDim.x, e, sm);
    block_fold<R, SUM>(e, sm);
    __shared__ bool last;
    unsigned* ticket = reinterpret_cast<unsigned*>(partials + 3 * kStatsBlocks);
    if (threadIdx.x == 0) {
        // the extrema in the data's own type, at the head of their slots
        *reinterpret_cast<R*>(&partials[3 * blockIdx.x]) = e.max_value();
        *reinterpret_cast<R*>(&partials[3 * blockIdx.x + 1]) = e.min_value();
        if (SUM) partials[3 * blockIdx.x + 2] = sm;
        __threadfence();
        last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    e = Ext<R>();
    sm = 0.0;
    for (int q = threadIdx.x; q < (int)gridDim.x; q += blockDim.x) {
        e.add(__ldcg(reinterpret_cast<const R*>(&partials[3 * q])));
        e.add(__ldcg(reinterpret_cast<const R*>(&partials[3 * q + 1])));
        if (SUM) sm += __ldcg(&partials[3 * q + 2]);
    }
    block_fold<R, SUM>(e, sm);
    if (threadIdx.x == 0) {
        out[0] = (double)e.max_value();
        out[1] = (double)e.min_value();
        out[2] = sm;
        unsigned st = status ? *status : 0u;
        out[3] = (double)st;
        if (status) *status = 0u;
        *ticket = 0u;
    }
}

}  // namespace

cudaError_t launch_stage_generic(const LaunchCfg& c, const void* grid, const void* phys,
                                 const StageIO& io, const void* coef, unsigned* status, cudaStream_t st)
{
    if (c.dtype == 1) return stage_dispatch_ndim<double>(c, grid, phys, io, coef, status, st);
    return stage_dispatch_ndim<float>(c, grid, phys, io, coef, status, st);
}

double generic_cells(int64_t ncell)
{
    const int tpb = generic_block(ncell);
    const int64_t blocks = (ncell + tpb - 1) / tpb;
    const double k = (double)blocks / sm_count();
    return tpb * (k > 8.0 ? k + 0.4 : (double)((blocks + sm_count() - 1) / sm_count()));
}

cudaError_t launch_advect(const LaunchCfg& c, const void* grid, const void* T, const void* u, void* Tout, double dt,
                          cudaStream_t st)
{
    if (c.dtype == 1) return advect_impl<double>(c, grid, T, u, Tout, dt, st);
    return advect_impl<float>(c, grid, T, u, Tout, dt, st);
}

cudaError_t launch_flux_generic(const LaunchCfg& c, const void* grid, const void* phys, const void* T,
                                const void* b, void* F[3], cudaStream_t st)
{
    if (c.dtype == 1) return flux_dispatch_ndim<double>(c, grid, phys, T, b, F, st);
    return flux_dispatch_ndim<float>(c, grid, phys, T, b, F, st);
}

namespace {

// two 16-byte loads a thread at least: more blocks only queue at the ticket
int stats_blocks(int64_t n, size_t esize)
{
    const int per = esize == 8 ? 1024 : 2048;
    return (int)std::min<int64_t>(kStatsBlocks, (n + per - 1) / per);
}

template <typename R>
cudaError_t rate_stats(const LaunchCfg& c, const KGrid<R>& g, const R* u, double* partials, double* out,
                       cudaStream_t st)
{
    const int nb = stats_blocks(g.ncell, sizeof(R));
    auto go = [&](auto src) {
        src.u = u;
        src.n = g.ncell;
        for (int d = 0; d < 3; ++d) src.inv[d] = g.inv_dx[d];
        stats_kernel<R, false><<<nb, 256, 0, st>>>(src, g.ncell, partials, out, (unsigned*)nullptr);
    };
    if (c.ndim == 1) go(RateSrc<R, 1>{});
    else if (c.ndim == 2) go(RateSrc<R, 2>{});
    else go(RateSrc<R, 3>{});
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_stats(int dtype, const void* T, int64_t n, double* partials, double* out,
                         unsigned* status, cudaStream_t st, bool need_sum)
{
    const int nb = stats_blocks(n, dtype == 1 ? 8 : 4);
    if (dtype == 1) {
        const ArraySrc<double> src{static_cast<const double*>(T)};
        if (need_sum) stats_kernel<double, true><<<nb, 256, 0, st>>>(src, n, partials, out, status);
        else stats_kernel<double, false><<<nb, 256, 0, st>>>(src, n, partials, out, status);
    } else {
        const ArraySrc<float> src{static_cast<const float*>(T)};
        if (need_sum) stats_kernel<float, true><<<nb, 256, 0, st>>>(src, n, partials, out, status);
        else stats_kernel<float, false><<<nb, 256, 0, st>>>(src, n, partials, out, status);
    }
    return cudaGetLastError();
}

cudaError_t launch_rate_stats(const LaunchCfg& c, const void* grid, const void* u, double* partials, double* out,
                              cudaStream_t st)
{
    if (c.dtype == 1)
        return rate_stats<double>(c, *static_cast<const KGrid<double>*>(grid), static_cast<const double*>(u), partials,
                                  out, st);
    return rate_stats<float>(c, *static_cast<const KGrid<float>*>(grid), static_cast<const float*>(u), partials, out,
                             st);
}

// ---------------------------------------------------------------------------
// Segmented extrema of the problems of an ensemble: block c folds chunk c
// (cells [cstart[c], cstart[c] + clen[c]) of one problem), then one warp per
// problem folds that problem's chunks pchunk[p] .. pchunk[p+1]-1.  FP32 folds
// (see Ext): 33.5 million cells took 236 us with FP64 ones.

namespace {

__global__ void __launch_bounds__(256) seg_stats_kernel(const float* __restrict__ T, const int64_t* cstart,
                                                        const int* clen, float2* partials)
{
    Ext<float> e;
    double none = 0.0;
    thread_stats<float, false>(ArraySrc<float>{T + cstart[blockIdx.x]}, clen[blockIdx.x], threadIdx.x, blockDim.x, e, none);
    block_fold<float, false>(e, none);
    if (threadIdx.x == 0) partials[blockIdx.x] = make_float2(e.max_value(), e.min_value());
}

__global__ void seg_stats_final_kernel(const float2* partials, const int* pchunk, int nprob, double* out)
{
    const int p = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int l = threadIdx.x & 31;
    if (p >= nprob) return;
    Ext<float> e;
    for (int q = pchunk[p] + l; q < pchunk[p + 1]; q += 32) {
        e.add(partials[q].x);
        e.add(partials[q].y);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        e.mx = fmaxf(e.mx, __shfl_xor_sync(0xffffffffu, e.mx, o));
        e.mn = fminf(e.mn, __shfl_xor_sync(0xffffffffu, e.mn, o));
        e.nan |= __shfl_xor_sync(0xffffffffu, e.nan, o);
    }
    if (l == 0) {
        out[2 * p + 0] = (double)e.max_value();
        out[2 * p + 1] = (double)e.min_value();
    }
}

}  // namespace

cudaError_t launch_stats_segmented(const float* T, const int64_t* cstart, const int* clen, int nchunk,
                                   const int* pchunk, int nprob, float* partials, double* out, cudaStream_t st)
{
    float2* part = reinterpret_cast<float2*>(partials);
    seg_stats_kernel<<<nchunk, 256, 0, st>>>(T, cstart, clen, part);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    seg_stats_final_kernel<<<(nprob + 7) / 8, 256, 0, st>>>(part, pchunk, nprob, out);
    return cudaGetLastError();
}

}  // namespace rkl
