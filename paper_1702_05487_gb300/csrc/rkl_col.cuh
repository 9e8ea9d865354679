// Column-march stage kernels of the RKL2 conduction super-step for FP64 grids,
// 3D and 2D (rkl_plane.cu has the packed FP32 form of the 2D one), periodic or
// Dirichlet, limiter at any floor.  One thread per cell column,
// marching along the slowest axis; every face is evaluated once:
//
//   3D  eight warps of a block cover LPR columns x 256 / LPR rows of a plane
//       (LPR = 32, 16 or 8 lanes per row, whichever leaves the fewest lanes
//       beyond the grid) and march in z.  The x-face below a cell comes from
//       the lane to the left by a shuffle, the y-face from the row below
//       through shared memory (one barrier per plane), the z-face from the
//       previous plane in registers.  Two more warps march the row below the
//       tile (its y-faces) and the column left of it (its x-faces).
//   2D  a warp covers 31 columns (lane 0 repeats the column to the left for
//       its x-face) and marches in y; no shared memory, no barrier.
//
// Fields are read straight from global memory: a block's plane is a few KB
// and its neighbours are the block's own rows, so L1 serves the re-reads.
// What bounds the kernel in FP64 is the FP64 rate (two lanes per SM and
// clock: 16 clocks a warp instruction), hence every face once, the folded
// face constants, one scale for all axes on cubic cells, an own square root
// and integer checks of the result: about 95 FP64 operations per cell and
// stage against about 305 in the generic kernel, which evaluates both faces
// of every axis.  112 x 96 x 80 FP64 stage (Spitzer): generic 419 us, this
// kernel 176 us; 100 x 100 Dirichlet 8.2 -> 3.1 us.  Narrow grids stay with the
// generic kernel (col_stage_pays).
#pragma once

#include <algorithm>
#include <cmath>

#include "rkl_launch.h"

namespace rkl {
namespace col {

constexpr int NW = 8;                    // warps of a 3D block that own cells
constexpr int NT = 32 * (NW + 2);        // and the two for its low faces
constexpr int NW2 = 4;                   // warps of a 2D block (independent of one another)

template <typename R>
struct Args {
    const R* Tin;        // field whose M is taken (Y_{j-1}, or Y_0 at stage 1)
    const R* b;          // [ndim][ncell]
    const R* Y0;
    const R* Yjm2;
    const R* MY0in;
    R* MY0out;           // stage 1 only
    R* out;              // Y_j, or M(T) in mode 0
    const R* coef_tab;   // if non-null: stage coefficients at coef_tab[4 j]
    int j;
    int mode;
};

// Square root of an FP64 number: the reciprocal square root estimate r of the
// PTX ISA refined by one third-order (Householder) step, sqrt(x) = t (1 + e / 2
// + 3 e^2 / 8) with t = x r, e = 1 - t r, five FP64 operations.  The rounding of
// t is part of e; with |e| <= 2^-19 the remainder 5 e^3 / 16 is below 2^-58 of the
// root: within 0.52 ulp.  Of 25 million roots 0.06% were not the rounded one, by
// at most 0.515 ulp; the error of M against 80-bit arithmetic is that with sqrt()
// and below the generic kernel's (rms 2.2e-16 against 2.6e-16 of M's rms).  With
// sqrt() a Spitzer stage takes 5% longer and a saturated one 10%.  Anything but
// positive normal numbers takes sqrt().
__device__ __forceinline__ double root(double x)
{
    if ((unsigned)__double2hiint(x) - 0x00100000u >= 0x7fe00000u) return sqrt(x);
    double r;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    const double t = x * r, e = fma(-t, r, 1.0);
    return fma(t * e, fma(e, 0.375, 0.5), t);
}

// Constants of the folded face flux (the packed form of the FP32 tile
// kernels, in either type): with B = b_L + b_R and Ts = T_L + T_R the halves
// of the face averages and -kappa_par0 become one constant, fscale, that the
// divergence absorbs.  Saturation at the face temperature cancels Ts^1.5
// between q and |F|; the upwind form returns F itself (fscale = 1).
//
// CUBE (equal spacings): gradients are taken in units of 1 / (4 dx), so that
// the transverse ones are plain sums of slopes; 1 / (4 dx) joins the
// constants.
template <typename R>
struct FaceC {
    R nk, kp4, fscale, sat;
    R idn[3], idt[3];       // factors of the normal difference and of the summed slopes
    R idl[3];               // factor of a limited slope
};

template <typename R, bool SP, bool SAT, bool CUBE>
__device__ __forceinline__ FaceC<R> face_consts(const KPhys<R>& p, const KGrid<R>& g)
{
    FaceC<R> k;
    const R unit = CUBE ? g.inv_4dx[0] : R(1);
    k.nk = R(-0.25) * p.kappa0 * (SP ? R(0.17677669529663688110) : R(1)) * unit;    // 2^-2.5
    k.kp4 = R(4) * p.kperp;
    k.fscale = (SAT && p.upwind) ? R(1) : k.nk;
    k.sat = SAT ? -k.nk / (p.q0 * R(0.35355339059327376220)) : R(0);               // 2^-1.5
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        k.idn[d] = CUBE ? R(4) : g.inv_dx[d];
        k.idt[d] = CUBE ? R(1) : g.inv_4dx[d];
        k.idl[d] = CUBE ? R(4) : g.inv_dx[d];
    }
    return k;
}

// Normal flux / fscale on a face.  ND == 2: one transverse direction (g2,
// B2 unused).
template <typename R, int ND, bool SP, bool SAT>
__device__ __forceinline__ R face(R TL, R TR, R gn, R g1, R g2, R Bn, R B1, R B2, const FaceC<R>& k,
                                  const KPhys<R>& p)
{
    const R Ts = TL + TR;
    R bdg = Bn * gn + B1 * g1;
    if (ND == 3) bdg += B2 * g2;
    R X = Bn * bdg;
    const bool perp = k.kp4 != R(0);
    if (perp) X += k.kp4 * gn;
    if (!SAT) return SP ? (Ts * Ts) * root(Ts) * X : X;
    R Y1 = B1 * bdg;
    R Y2 = ND == 3 ? B2 * bdg : R(0);
    if (perp) {
        Y1 += k.kp4 * g1;
        if (ND == 3) Y2 += k.kp4 * g2;
    }
    R V2 = X * X + Y1 * Y1;
    if (ND == 3) V2 += Y2 * Y2;
    if (!p.upwind) {
        const R sTs = root(Ts), Vm = root(V2);
        if (SP) return ddiv<R>((Ts * Ts) * sTs * X, k.sat * (Ts * Vm) + R(1));
        const R T15 = Ts * sTs;
        return ddiv<R>(T15 * X, k.sat * Vm + T15);
    }
    const R nk = SP ? k.nk * (Ts * Ts) * root(Ts) : k.nk;
    const R Fn = nk * X;
    const R Tq = Fn >= R(0) ? TL : TR;
    const R q = p.q0 * Tq * root(Tq);
    return ddiv<R>(q, q + fabs(nk) * root(V2)) * Fn;
}

// A cell's transverse slope along one axis: the centred difference and, with
// LIM, the limited slope MC(T+ - T0, T0 - T-) beside it.
template <typename R, bool LIM>
struct Slope {
    R c;
    R l;
};
template <typename R, bool LIM>
__device__ __forceinline__ Slope<R, LIM> slope(R Tp, R T0, R Tm)
{
    Slope<R, LIM> s;
    s.c = Tp - Tm;
    s.l = LIM ? mc_limit<R>(Tp - T0, T0 - Tm) : R(0);
    return s;
}
// Transverse gradient along axis d at a face from its two cells' slopes.
template <typename R, bool LIM, bool CUBE>
__device__ __forceinline__ R grad(const Slope<R, LIM>& a, const Slope<R, LIM>& b, const FaceC<R>& k, int d, bool limit)
{
    if (LIM && limit) return mc_limit<R>(a.l, b.l) * k.idl[d];
    return CUBE ? a.c + b.c : (a.c + b.c) * k.idt[d];
}
template <typename R, bool LIM>
__device__ __forceinline__ bool limited(R TL, R TR, const KPhys<R>& p)
{
    return LIM && fmin(TL, TR) < p.lfloor;
}

// An index wrapped (periodic) or clamped (Dirichlet, outside: a ghost cell).
struct Idx {
    int i;
    bool ghost;
};
__device__ __forceinline__ Idx index(int i, int n, int bc)
{
    if (bc == 1) return Idx{clampi(i, n), i < 0 || i >= n};
    int r = i % n;
    return Idx{r < 0 ? r + n : r, false};
}

template <typename R>
__device__ __forceinline__ void load_coef(const Args<R>& a, KCoef<R>& cf)
{
    if (a.mode != 0 && a.coef_tab) {
        const R* t = a.coef_tab + 4 * a.j;
        cf.mu = t[0]; cf.nu = t[1]; cf.mt = t[2]; cf.gt = t[3];
    }
}

// Status bits of a stage value (integer arithmetic: the FP64 units are the
// scarce ones): ST_NONFINITE for NaN and infinities, with SP ST_NONPOSITIVE
// for anything not above zero.
template <bool SP>
__device__ __forceinline__ unsigned bad_bits(float y)
{
    const int b = __float_as_int(y);
    return ((b & 0x7f800000) == 0x7f800000 ? ST_NONFINITE : 0u) | (SP && b <= 0 ? ST_NONPOSITIVE : 0u);
}
template <bool SP>
__device__ __forceinline__ unsigned bad_bits(double y)
{
    const int h = __double2hiint(y);
    return ((h & 0x7ff00000) == 0x7ff00000 ? ST_NONFINITE : 0u) |
           (SP && __double_as_longlong(y) <= 0 ? ST_NONPOSITIVE : 0u);
}

// The stage update of one cell from its M; y0, yj2 and my0 are the cell's
// Y0, Y_{j-2} and M(Y0) (stages j >= 2).  Returns the status bits.
template <typename R, bool SP>
__device__ __forceinline__ unsigned emit(const Args<R>& a, const KCoef<R>& cf, R* out, R* MY0out, R M, R T, R y0, R yj2,
                                         R my0)
{
    if (a.mode == 0) {
        *out = M;
        return 0u;
    }
    R y;
    if (a.mode == 1) {
        if (a.MY0out) *MY0out = M;
        y = T + cf.mt * M;
    } else {
        y = y0 + (cf.mu * (T - y0) + cf.nu * (yj2 - y0) + cf.mt * M + cf.gt * my0);
    }
    *out = y;
    return bad_bits<SP>(y);
}

// --------------------------------------------------------------------------
// 3D

// In-plane offsets and ghost flags of a cell and its neighbours.
struct Nbr {
    int c, xm, xp, ym, yp, pp, pm, mp;     // (x, y): p / m one up / down; pm = (x + 1, y - 1), mp = (x - 1, y + 1)
    unsigned g;                            // bit k: the k-th of these is a Dirichlet ghost
};

__device__ __forceinline__ Nbr neighbours(int i, int j, int nx, int ny, int bc)
{
    const Idx x0 = index(i, nx, bc), xm = index(i - 1, nx, bc), xp = index(i + 1, nx, bc);
    const Idx y0 = index(j, ny, bc), ym = index(j - 1, ny, bc), yp = index(j + 1, ny, bc);
    auto at = [&](const Idx& x, const Idx& y) { return y.i * nx + x.i; };
    Nbr n;
    n.c = at(x0, y0);
    n.xm = at(xm, y0);
    n.xp = at(xp, y0);
    n.ym = at(x0, ym);
    n.yp = at(x0, yp);
    n.pp = at(xp, yp);
    n.pm = at(xp, ym);
    n.mp = at(xm, yp);
    const bool gx = x0.ghost, gy = y0.ghost;
    n.g = (gx || gy ? 1u : 0u) | (xm.ghost || gy ? 2u : 0u) | (xp.ghost || gy ? 4u : 0u) |
          (gx || ym.ghost ? 8u : 0u) | (gx || yp.ghost ? 16u : 0u) | (xp.ghost || yp.ghost ? 32u : 0u) |
          (xp.ghost || ym.ghost ? 64u : 0u) | (xm.ghost || yp.ghost ? 128u : 0u);
    return n;
}

template <typename R>
struct Smem3 {
    R Fy[2][32 * (NW + 1)];     // y-faces: row r's lower face at [r LPR + lx] (row 0: the tile's bottom)
    R FxLo[2][32];              // x-faces on the tile's left boundary
};

template <typename R, bool SP, bool SAT, bool LIM, bool CUBE>
__global__ void __launch_bounds__(NT, 2)
col3_kernel(KGrid<R> g, KPhys<R> p, Args<R> a, KCoef<R> cf, unsigned* status, int nzchunk, int lpr)
{
    __shared__ Smem3<R> sm;
    using S = Slope<R, LIM>;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int rows = NW * (32 / lpr);
    // warps 0 .. 7 own the tile's cells, warp 8 the row below it, warp 9 the
    // column left of it
    const bool bottom = w == NW, left = w == NW + 1;
    const int lx = left ? -1 : lane & (lpr - 1);
    const int row = bottom ? -1 : (left ? lane & (rows - 1) : w * (32 / lpr) + lane / lpr);
    const int nx = g.n[0], ny = g.n[1], nz = g.n[2], bc = g.bc;
    const int i0 = blockIdx.x * lpr, j0 = blockIdx.y * rows, z0 = blockIdx.z * nzchunk;
    const int nzc = min(nzchunk, nz - z0);
    const bool active = w < NW && i0 + lx < nx && j0 + row < ny;
    load_coef(a, cf);

    // lanes beyond the grid repeat its last column or row
    const Nbr n = neighbours(min(i0 + lx, nx - 1), min(j0 + row, ny - 1), nx, ny, bc);
    const R bcv = g.bcv;
    auto plane = [&](int k, bool& zghost) -> int64_t {      // -1 <= z0 + k <= nz
        int z = z0 + k;
        zghost = bc == 1 && (z < 0 || z >= nz);
        if (z < 0) z = bc == 1 ? 0 : nz - 1;
        if (z >= nz) z = bc == 1 ? nz - 1 : 0;
        return (int64_t)z * g.plane;
    };
    auto ld = [&](const R* base, int o, bool ghost) -> R { return ghost ? bcv : base[o]; };

    const FaceC<R> fk = face_consts<R, SP, SAT, CUBE>(p, g);
    const R cx = -fk.fscale * g.inv_dx[0], cy = -fk.fscale * g.inv_dx[1], cz = -fk.fscale * g.inv_dx[2];

    // what a plane hands to the next: T of the cell, one column right and one
    // row up, the cell's x / y slopes and b
    struct Q {
        R c, r, u;
        S gx, gy;
        R b[3];
    };
    auto read = [&](int k) -> Q {
        bool zg;
        const int64_t pl = plane(k, zg);
        const R* T = a.Tin + pl;
        Q q;
        q.c = ld(T, n.c, zg || (n.g & 1u));
        const R xm = ld(T, n.xm, zg || (n.g & 2u));
        q.r = ld(T, n.xp, zg || (n.g & 4u));
        const R ym = ld(T, n.ym, zg || (n.g & 8u));
        q.u = ld(T, n.yp, zg || (n.g & 16u));
#pragma unroll
        for (int e = 0; e < 3; ++e) q.b[e] = a.b[e * g.ncell + pl + n.c];
        q.gx = slope<R, LIM>(q.r, q.c, xm);
        q.gy = slope<R, LIM>(q.u, q.c, ym);
        return q;
    };
    auto zface = [&](const Q& L, const Q& H) -> R {
        const bool lim = limited<R, LIM>(L.c, H.c, p);
        return face<R, 3, SP, SAT>(L.c, H.c, (H.c - L.c) * fk.idn[2], grad<R, LIM, CUBE>(L.gx, H.gx, fk, 0, lim),
                                   grad<R, LIM, CUBE>(L.gy, H.gy, fk, 1, lim), L.b[2] + H.b[2], L.b[0] + H.b[0],
                                   L.b[1] + H.b[1], fk, p);
    };

    chain_wait();
    Q A = read(-1), B = read(0);
    R Fzl = w < NW ? zface(A, B) : R(0);
    R Tmc = A.c, Tmr = A.r, Tmu = A.u;
    unsigned bad = 0u;

    for (int q = 0; q < nzc; ++q) {
        bool zg;
        const int64_t pl = plane(q, zg);            // inside the grid: zg false
        const R* T = a.Tin + pl;
        const Q N = read(q + 1);
        const R Tpp = ld(T, n.pp, n.g & 32u), Tpm = ld(T, n.pm, n.g & 64u), Tmp = ld(T, n.mp, n.g & 128u);
        R bR[3], bU[3];
#pragma unroll
        for (int e = 0; e < 3; ++e) {
            bR[e] = a.b[e * g.ncell + pl + n.xp];
            bU[e] = a.b[e * g.ncell + pl + n.yp];
        }
        R y0 = R(0), yj2 = R(0), my0 = R(0);
        if (a.mode == 2 && w < NW) {
            y0 = a.Y0[pl + n.c];
            yj2 = a.Yjm2[pl + n.c];
            my0 = a.MY0in[pl + n.c];
        }
        const int par = q & 1;
        const S gz = slope<R, LIM>(N.c, B.c, Tmc);
        R Fx = R(0), Fy = R(0), Fz = R(0);
        if (!bottom) {
            const S gzR = slope<R, LIM>(N.r, B.r, Tmr), gyR = slope<R, LIM>(Tpp, B.r, Tpm);
            const bool lim = limited<R, LIM>(B.c, B.r, p);
            Fx = face<R, 3, SP, SAT>(B.c, B.r, (B.r - B.c) * fk.idn[0], grad<R, LIM, CUBE>(B.gy, gyR, fk, 1, lim),
                                     grad<R, LIM, CUBE>(gz, gzR, fk, 2, lim), B.b[0] + bR[0], B.b[1] + bR[1],
                                     B.b[2] + bR[2], fk, p);
            if (left) sm.FxLo[par][row] = Fx;
        }
        if (!left) {
            const S gzU = slope<R, LIM>(N.u, B.u, Tmu), gxU = slope<R, LIM>(Tpp, B.u, Tmp);
            const bool lim = limited<R, LIM>(B.c, B.u, p);
            Fy = face<R, 3, SP, SAT>(B.c, B.u, (B.u - B.c) * fk.idn[1], grad<R, LIM, CUBE>(B.gx, gxU, fk, 0, lim),
                                     grad<R, LIM, CUBE>(gz, gzU, fk, 2, lim), B.b[1] + bU[1], B.b[0] + bU[0],
                                     B.b[2] + bU[2], fk, p);
            sm.Fy[par][(row + 1) * lpr + lx] = Fy;
        }
        if (w < NW) Fz = zface(B, N);
        // one barrier per plane: the other half of Fy / FxLo is written only
        // after every thread has passed it, that is, has read this half's
        // previous plane
        __syncthreads();
        if (w < NW) {
            const R Fyl = sm.Fy[par][row * lpr + lx];
            R Fxl = __shfl_up_sync(0xffffffffu, Fx, 1, lpr);
            if (lx == 0) Fxl = sm.FxLo[par][row];
            const R M = cx * (Fx - Fxl) + cy * (Fy - Fyl) + cz * (Fz - Fzl);
            if (active)
                bad |= emit<R, SP>(a, cf, a.out + pl + n.c, a.MY0out + pl + n.c, M, B.c, y0, yj2, my0);
        }
        Fzl = Fz;
        Tmc = B.c;
        Tmr = B.r;
        Tmu = B.u;
        B = N;
    }
    chain_release();
    if (bad) atomicOr(status, bad);
}

// --------------------------------------------------------------------------
// 2D

template <typename R, bool SP, bool SAT, bool LIM, bool CUBE>
__global__ void __launch_bounds__(32 * NW2)
col2_kernel(KGrid<R> g, KPhys<R> p, Args<R> a, KCoef<R> cf, unsigned* status, int nychunk, int ntx, int nitems)
{
    using S = Slope<R, LIM>;
    const int lane = threadIdx.x & 31, item = blockIdx.x * NW2 + (threadIdx.x >> 5);
    if (item >= nitems) return;                     // whole warps
    const int nx = g.n[0], ny = g.n[1], bc = g.bc;
    const int i = (item % ntx) * 31 - 1 + lane, r0 = (item / ntx) * nychunk;
    const int nyc = min(nychunk, ny - r0);
    const bool active = lane > 0 && i < nx;
    load_coef(a, cf);

    const int ic = min(i, nx - 1);                  // lanes beyond the grid repeat its last column
    const Idx x0 = index(ic, nx, bc), xm = index(ic - 1, nx, bc), xp = index(ic + 1, nx, bc);
    const R bcv = g.bcv;
    const R* bx = a.b;
    const R* by = a.b + g.ncell;

    const FaceC<R> fk = face_consts<R, SP, SAT, CUBE>(p, g);
    const R cx = -fk.fscale * g.inv_dx[0], cy = -fk.fscale * g.inv_dx[1];

    struct Q {
        R c, r;             // T of the cell and one column right
        S gx;
        R b[2], bR[2];      // b there
    };
    // 32-bit element offsets: the launcher keeps 2^31 cells and more away
    auto read = [&](int k) -> Q {                   // -1 <= r0 + k <= ny + 1
        int y = r0 + k;
        const bool yg = bc == 1 && (y < 0 || y >= ny);
        if (bc == 1) y = clampi(y, ny);
        else {
            y = y < 0 ? y + ny : y;
            y = y >= ny ? y - ny : y;
            y = y >= ny ? y - ny : y;               // one row, and two past the end
        }
        const unsigned ro = (unsigned)y * (unsigned)nx, oc = ro + x0.i, om = ro + xm.i, op = ro + xp.i;
        Q q;
        q.c = yg || x0.ghost ? bcv : a.Tin[oc];
        const R l = yg || xm.ghost ? bcv : a.Tin[om];
        q.r = yg || xp.ghost ? bcv : a.Tin[op];
        q.b[0] = bx[oc];
        q.b[1] = by[oc];
        q.bR[0] = bx[op];
        q.bR[1] = by[op];
        q.gx = slope<R, LIM>(q.r, q.c, l);
        return q;
    };
    auto yface = [&](const Q& L, const Q& H) -> R {
        const bool lim = limited<R, LIM>(L.c, H.c, p);
        return face<R, 2, SP, SAT>(L.c, H.c, (H.c - L.c) * fk.idn[1], grad<R, LIM, CUBE>(L.gx, H.gx, fk, 0, lim), R(0),
                                   L.b[1] + H.b[1], L.b[0] + H.b[0], R(0), fk, p);
    };

    chain_wait();
    Q A = read(-1), B = read(0), N = read(1);
    R Fyl = yface(A, B);
    R Tmc = A.c, Tmr = A.r;
    unsigned bad = 0u;
    unsigned o = (unsigned)r0 * (unsigned)nx + x0.i;
    for (int q = 0; q < nyc; ++q, o += nx) {
        Q P = N;
        if (q + 1 < nyc) P = read(q + 2);           // in flight while row q is computed
        R y0 = R(0), yj2 = R(0), my0 = R(0);
        if (a.mode == 2) {
            y0 = a.Y0[o];
            yj2 = a.Yjm2[o];
            my0 = a.MY0in[o];
        }
        const S gy = slope<R, LIM>(N.c, B.c, Tmc), gyR = slope<R, LIM>(N.r, B.r, Tmr);
        const bool lim = limited<R, LIM>(B.c, B.r, p);
        const R Fx = face<R, 2, SP, SAT>(B.c, B.r, (B.r - B.c) * fk.idn[0], grad<R, LIM, CUBE>(gy, gyR, fk, 1, lim),
                                         R(0), B.b[0] + B.bR[0], B.b[1] + B.bR[1], R(0), fk, p);
        const R Fy = yface(B, N);
        const R Fxl = __shfl_up_sync(0xffffffffu, Fx, 1);
        const R M = cx * (Fx - Fxl) + cy * (Fy - Fyl);
        if (active) bad |= emit<R, SP>(a, cf, a.out + o, a.MY0out + o, M, B.c, y0, yj2, my0);
        Fyl = Fy;
        Tmc = B.c;
        Tmr = B.r;
        B = N;
        N = P;
    }
    chain_release();
    if (bad) atomicOr(status, bad);
}

int sms();      // rkl_col.cu

// Lanes per row of a 3D block: of 32, 16 and 8 the fewest lanes beyond the
// grid (columns and rows), the widest among equals.
inline int lanes_per_row(int nx, int ny)
{
    int best = 32;
    double waste = 1e300;
    for (int l = 32; l >= 8; l /= 2) {
        const int rows = NW * 32 / l;
        const double c = (double)((nx + l - 1) / l * l) * ((ny + rows - 1) / rows * rows);
        if (c < waste * 0.999) {
            waste = c;
            best = l;
        }
    }
    return best;
}

// Length of a block's march and its cost.
struct Chunk {
    int len;
    double cost;
};

// 3D, cost in planes of a lone block (7.2 us FP64 Spitzer, 4.7 constant, 13
// saturated, 18 limited).  A chunk costs its planes and 0.5 (limited 0.6) for its
// first z-face.  The fullest SM decides: K blocks on it take K times as long, at
// the FP64 rate; one on every SM takes 1.6 times as long as one on every second
// SM (limited 1.15).  CTAs start in z order, so the short last chunks of the
// columns come last.  An SM takes two blocks at a time: near the end of the third
// limited one, some take a fourth.  Fitted to chunks of 1 .. 64 planes on 44 grids
// (8 x 6 x 8 to 100^3, columns of 3 x 500 and 4 x 5000) with each flux: the choice
// is 0.4% (limited 2%) above the best on average.
inline Chunk chunk3(int64_t cols, int nz, bool lim)
{
    const double p = lim ? 0.6 : 0.5, one = lim ? 1.15 : 1.6;
    auto at = [&](int64_t K) { return K == 1 ? one : (double)K; };
    Chunk best{1, 1e300};
    for (int c = 1; c <= 64 && c <= nz; ++c) {
        const int64_t chunks = (nz + c - 1) / c, blocks = cols * chunks;
        const int last = nz - (int)(chunks - 1) * c;
        const double k = (double)blocks / sms();
        double cost;
        if (k <= 0.5) cost = c + p;
        else if (k > 12.0) cost = (c + p) * (k + 0.3);
        else {
            const int64_t K = (blocks + sms() - 1) / sms();
            const bool tail = chunks > 1 && blocks - (K - 1) * sms() <= cols && K > 1;
            const double full = lim && k > 2.6 && k <= 3.0 ? 4.0 : at(K);
            cost = tail ? (c + p) * at(K - 1) + (last + p) * (full - at(K - 1)) : (c + p) * full;
        }
        if (cost < best.cost - 1e-9) best = Chunk{c, cost};
    }
    return best;
}

// 2D, cost in rows of a warp at the FP64 rate (0.56 us a row and SM, FP64
// Spitzer).  With more than 96 rows an SM: 32 warps an SM, at most 32 rows each.
// Below, 1 to 6 rows: a warp alone takes 4.4 a row and 4.8 to start; an SM takes
// its warps' rows one after the other, with 0.8 more per warp for its first
// y-face, and the fullest SM decides.  Limited blocks on more than every second SM: 1.4
// times; one-row warps beyond four blocks an SM wait for a second round.  Fitted
// like the above on 30 grids (8 x 8 to 60000 x 31).
inline Chunk chunk2(int64_t ntx, int ny, bool lim)
{
    const double rows = (double)ntx * ny / sms();
    if (rows > 96.0) {
        const int c = (int)std::min(32.0, std::ceil(rows / 32.0));
        return Chunk{c, rows * (1.0 + 0.8 / c)};
    }
    Chunk best{1, 1e300};
    for (int c = 1; c <= 6 && c <= ny; ++c) {
        const int64_t blocks = (ntx * ((ny + c - 1) / c) + NW2 - 1) / NW2;
        const int64_t full = (blocks + sms() - 1) / sms();
        const double alone = (4.4 * c + 4.8) * (lim && 2 * blocks > sms() ? 1.4 : 1.0);
        const double cost = std::max(alone, NW2 * full * (c + 0.8)) + (full > 4 && c == 1 ? 8.0 : 0.0);
        if (cost < best.cost - 1e-9) best = Chunk{c, cost};
    }
    return best;
}

// Blocks of a plane, and warps of a row.
struct Cols {
    int lpr, bx, by;
};
inline Cols cols3(int nx, int ny)
{
    const int lpr = lanes_per_row(nx, ny), rows = NW * 32 / lpr;
    return Cols{lpr, (nx + lpr - 1) / lpr, (ny + rows - 1) / rows};
}
inline int cols2(int nx) { return (nx + 30) / 31; }

template <typename R, bool SP, bool SAT, bool LIM, bool CUBE>
cudaError_t launch_nd(const LaunchCfg& c, const KGrid<R>& g, const KPhys<R>& p, const Args<R>& a, const KCoef<R>& cf,
                      unsigned* status, int chunk, cudaStream_t st, bool chained)
{
    if (c.ndim == 3) {
        const Cols q = cols3(g.n[0], g.n[1]);
        const int nzc = chunk > 0 ? chunk : chunk3((int64_t)q.bx * q.by, g.n[2], LIM).len;
        const dim3 grid(q.bx, q.by, (g.n[2] + nzc - 1) / nzc);
        return launch_chained(col3_kernel<R, SP, SAT, LIM, CUBE>, grid, NT, 0, st, chained, g, p, a, cf, status, nzc,
                              q.lpr);
    }
    const int ntx = cols2(g.n[0]), ch = chunk > 0 ? chunk : chunk2(ntx, g.n[1], LIM).len;
    const int64_t items = (int64_t)ntx * ((g.n[1] + ch - 1) / ch);
    return launch_chained(col2_kernel<R, SP, SAT, LIM, CUBE>, (unsigned)((items + NW2 - 1) / NW2), 32 * NW2, 0, st,
                          chained, g, p, a, cf, status, ch, ntx, (int)items);
}

template <typename R, bool SP, bool SAT>
cudaError_t launch_form(const LaunchCfg& c, const KGrid<R>& g, const KPhys<R>& p, const Args<R>& a, const KCoef<R>& cf,
                        unsigned* status, int chunk, cudaStream_t st, bool chained)
{
    bool cube = true;
    for (int d = 1; d < c.ndim; ++d) cube = cube && g.inv_dx[d] == g.inv_dx[0];
    if (c.limiter)
        return cube ? launch_nd<R, SP, SAT, true, true>(c, g, p, a, cf, status, chunk, st, chained)
                    : launch_nd<R, SP, SAT, true, false>(c, g, p, a, cf, status, chunk, st, chained);
    return cube ? launch_nd<R, SP, SAT, false, true>(c, g, p, a, cf, status, chunk, st, chained)
                : launch_nd<R, SP, SAT, false, false>(c, g, p, a, cf, status, chunk, st, chained);
}

template <typename R>
Args<R> stage_args(const StageIO& io)
{
    return Args<R>{static_cast<const R*>(io.mode == 1 ? io.Y0 : io.Yjm1), static_cast<const R*>(io.b),
                   static_cast<const R*>(io.Y0), static_cast<const R*>(io.Yjm2), static_cast<const R*>(io.MY0),
                   io.mode == 1 ? static_cast<R*>(io.MY0) : nullptr, static_cast<R*>(io.Yj),
                   static_cast<const R*>(io.coef_tab), io.j, io.mode};
}

template <typename R>
cudaError_t launch(const LaunchCfg& c, const KGrid<R>& g, const KPhys<R>& p, const StageIO& io, const KCoef<R>& cf,
                   unsigned* status, int chunk, cudaStream_t st)
{
    const Args<R> a = stage_args<R>(io);
    if (c.spitzer)
        return c.saturate ? launch_form<R, true, true>(c, g, p, a, cf, status, chunk, st, io.chained)
                          : launch_form<R, true, false>(c, g, p, a, cf, status, chunk, st, io.chained);
    return c.saturate ? launch_form<R, false, true>(c, g, p, a, cf, status, chunk, st, io.chained)
                      : launch_form<R, false, false>(c, g, p, a, cf, status, chunk, st, io.chained);
}

}  // namespace col
}  // namespace rkl
