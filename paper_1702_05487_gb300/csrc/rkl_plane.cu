// Packed 2D FP32 stage kernel: the column march of rkl_col.cuh with two
// neighbouring cells per thread in packed FP32 pair instructions.
//
// A warp covers 60 columns: 30 lanes own a pair each, lane 0 holds the pair
// to the left (its x-face) and lane 31 the pair to the right, so that a row is
// read once, two cells a lane, and every neighbour comes by shuffle.  It
// marches up a run of rows; each row is read one row ahead of its use.  No
// shared memory, no barrier.  Even widths read and write pairs as 64-bit
// words; odd ones cell by cell.
//
// 2D grids live in L2 and a stage is a few microseconds, so the scalar march
// was bound by instruction issue (11.2 M warp instructions on 1530 x 1071,
// saturated, 17 us a stage); this kernel issues 7.8 M and takes 12 us.
#include <algorithm>

#include "rkl_col.cuh"
#include "rkl_x2_tile.cuh"

namespace rkl {
namespace col {
namespace {

using x2::add2;
using x2::bc2;
using x2::fma2;
using x2::mul2;
using x2::sub2;

constexpr int COLS = 60;
constexpr int NWP = 4;                   // warps of a block (independent of one another)

// Normal flux / fscale on a pair of faces (x2::face2s with one transverse
// direction).
template <bool SP, bool SAT>
__device__ __forceinline__ float2 face2d(float2 TL, float2 TR, float2 gn, float2 g1, float2 Bn, float2 B1,
                                         const x2::FaceK& k, const KPhys<float>& p)
{
    const float2 Ts = add2(TL, TR);
    const float2 bdg = fma2(Bn, gn, mul2(B1, g1));
    const float2 X = fma2(Bn, bdg, mul2(bc2(k.kp4), gn));
    if (!SAT) {
        if (SP) return mul2(mul2(mul2(Ts, Ts), x2::sqrt2(Ts)), X);
        return X;
    }
    const float2 sTs = x2::sqrt2(Ts);
    const float2 Y1 = fma2(B1, bdg, mul2(bc2(k.kp4), g1));
    const float2 V2 = fma2(Y1, Y1, mul2(X, X));
    if (!p.upwind) {
        const float2 Vm = x2::sqrt2(V2);
        float2 num, den;
        if (SP) {
            num = mul2(mul2(mul2(Ts, Ts), sTs), X);
            den = fma2(bc2(k.sat), mul2(Ts, Vm), bc2(1.f));
        } else {
            const float2 T15 = mul2(Ts, sTs);
            num = mul2(T15, X);
            den = fma2(bc2(k.sat), Vm, T15);
        }
        return make_float2(ddiv<float>(num.x, den.x), ddiv<float>(num.y, den.y));
    }
    const float2 nk = SP ? mul2(mul2(bc2(k.nk), mul2(Ts, Ts)), sTs) : bc2(k.nk);
    const float2 Fn = mul2(nk, X);
    const float2 Fmag = mul2(make_float2(fabsf(nk.x), fabsf(nk.y)), x2::sqrt2(V2));
    const float2 Tq = make_float2(Fn.x >= 0.f ? TL.x : TR.x, Fn.y >= 0.f ? TL.y : TR.y);
    const float2 q = mul2(mul2(bc2(p.q0), Tq), x2::sqrt2(Tq));
    const float2 den = add2(q, Fmag);
    return make_float2(ddiv<float>(q.x, den.x) * Fn.x, ddiv<float>(q.y, den.y) * Fn.y);
}

template <bool SP, bool SAT, bool LIM, bool VEC>
__global__ void __launch_bounds__(32 * NWP)
plane_kernel(KGrid<float> g, KPhys<float> p, Args<float> a, KCoef<float> cf, unsigned* status, int nychunk, int ntx,
             int nitems)
{
    const int lane = threadIdx.x & 31, item = blockIdx.x * NWP + (threadIdx.x >> 5);
    if (item >= nitems) return;                     // whole warps
    const int nx = g.n[0], ny = g.n[1], bc = g.bc;
    const int c = (item % ntx) * COLS - 2 + 2 * lane, r0 = (item / ntx) * nychunk;
    const int nyc = min(nychunk, ny - r0);
    const bool own = lane > 0 && lane < 31;
    const bool act0 = own && c < nx, act1 = own && c + 1 < nx;
    load_coef(a, cf);

    // VEC: nx is even, so a pair is inside the grid, wrapped or a ghost as a whole
    const Idx x0 = index(c, nx, bc), x1 = index(c + 1, nx, bc);
    const float bcv = g.bcv;
    const float* bx = a.b;
    const float* by = a.b + g.ncell;
    auto pair = [&](const float* A, unsigned ro) -> float2 {
        if (VEC && x1.i == x0.i + 1) return *reinterpret_cast<const float2*>(A + ro + x0.i);
        return make_float2(A[ro + x0.i], A[ro + x1.i]);
    };
    auto left = [](float2 v) { return __shfl_up_sync(0xffffffffu, v.y, 1); };      // column c - 1
    auto right = [](float2 v) { return __shfl_down_sync(0xffffffffu, v.x, 1); };   // column c + 2

    const x2::FaceK fk = x2::face_consts<SP, SAT>(p);
    const float2 idx = bc2(g.inv_dx[0]), idy = bc2(g.inv_dx[1]);
    const float2 i4x = bc2(g.inv_4dx[0]), i4y = bc2(g.inv_4dx[1]);
    const float2 ilx = bc2(4.f * g.inv_dx[0]), ily = bc2(4.f * g.inv_dx[1]);
    const float2 cx = bc2(-fk.fscale * g.inv_dx[0]), cy = bc2(-fk.fscale * g.inv_dx[1]);

    struct Raw {
        float2 T, bx, by;
    };
    struct Row {
        float2 T, bx, by, gx;
        float r;                                    // T at column c + 2
    };
    auto read = [&](int k) -> Raw {                 // -1 <= r0 + k <= ny + 1
        int y = r0 + k;
        const bool yg = bc == 1 && (y < 0 || y >= ny);
        if (bc == 1) y = clampi(y, ny);
        else {
            y = y < 0 ? y + ny : y;
            y = y >= ny ? y - ny : y;
            y = y >= ny ? y - ny : y;
        }
        const unsigned ro = (unsigned)y * (unsigned)nx;
        Raw q;
        q.T = pair(a.Tin, ro);
        q.bx = pair(bx, ro);
        q.by = pair(by, ro);
        if (yg || x0.ghost) q.T.x = bcv;
        if (yg || x1.ghost) q.T.y = bcv;
        return q;
    };
    auto row = [&](const Raw& q) -> Row {
        Row w;
        w.T = q.T;
        w.bx = q.bx;
        w.by = q.by;
        w.r = right(q.T);
        w.gx = x2::cslope<LIM>(make_float2(q.T.y, w.r), q.T, make_float2(left(q.T), q.T.x));
        return w;
    };
    auto yface = [&](const Row& L, const Row& H) -> float2 {
        return face2d<SP, SAT>(L.T, H.T, mul2(sub2(H.T, L.T), idy), x2::fgrad<LIM>(L.gx, H.gx, i4x, ilx),
                               add2(L.by, H.by), add2(L.bx, H.bx), fk, p);
    };

    chain_wait();
    const Raw ra = read(-1), rb = read(0);
    Raw rn = read(1);
    const Row A = row(ra);
    Row B = row(rb);
    float2 Fyl = yface(A, B);
    float2 Tm = A.T;
    float Tmr = A.r;
    unsigned bad = 0u;
    unsigned o = (unsigned)r0 * (unsigned)nx + x0.i;
    for (int q = 0; q < nyc; ++q, o += nx) {
        Raw rp = rn;
        if (q + 1 < nyc) rp = read(q + 2);          // in flight while row q is computed
        float2 y0 = bc2(0.f), yj2 = bc2(0.f), my0 = bc2(0.f);
        if (a.mode == 2 && act0) {
            auto get = [&](const float* A_) {
                if (VEC) return *reinterpret_cast<const float2*>(A_ + o);
                return make_float2(A_[o], act1 ? A_[o + 1] : 0.f);
            };
            y0 = get(a.Y0);
            yj2 = get(a.Yjm2);
            my0 = get(a.MY0in);
        }
        const Row N = row(rn);
        const float2 gy = x2::cslope<LIM>(N.T, B.T, Tm);
        const float2 gyR = make_float2(gy.y, x2::cslope1<LIM>(N.r, B.r, Tmr));
        const float2 TR = make_float2(B.T.y, B.r);
        const float2 Fx = face2d<SP, SAT>(B.T, TR, mul2(sub2(TR, B.T), idx), x2::fgrad<LIM>(gy, gyR, i4y, ily),
                                          add2(B.bx, make_float2(B.bx.y, right(B.bx))),
                                          add2(B.by, make_float2(B.by.y, right(B.by))), fk, p);
        const float2 Fy = yface(B, N);
        const float2 Fxl = make_float2(left(Fx), Fx.x);
        const float2 M = fma2(sub2(Fx, Fxl), cx, mul2(sub2(Fy, Fyl), cy));
        if (act0) {
            auto put = [&](float* A_, float2 v) {
                if (VEC) *reinterpret_cast<float2*>(A_ + o) = v;
                else {
                    A_[o] = v.x;
                    if (act1) A_[o + 1] = v.y;
                }
            };
            float2 y = M;
            if (a.mode == 1) {
                if (a.MY0out) put(a.MY0out, M);
                y = fma2(bc2(cf.mt), M, B.T);
            } else if (a.mode == 2) {
                y = add2(y0, fma2(bc2(cf.mu), sub2(B.T, y0),
                                  fma2(bc2(cf.nu), sub2(yj2, y0), fma2(bc2(cf.mt), M, mul2(bc2(cf.gt), my0)))));
            }
            if (a.mode != 0) bad |= bad_bits<SP>(y.x) | (act1 ? bad_bits<SP>(y.y) : 0u);
            put(a.out, y);
        }
        Fyl = Fy;
        Tm = B.T;
        Tmr = B.r;
        B = N;
        rn = rp;
    }
    chain_release();
    if (bad) atomicOr(status, bad);
}

template <bool SP, bool SAT, bool LIM>
cudaError_t launch_plane(const KGrid<float>& g, const KPhys<float>& p, const Args<float>& a, const KCoef<float>& cf,
                         unsigned* status, int chunk, cudaStream_t st, bool chained)
{
    const int ntx = (g.n[0] + COLS - 1) / COLS;
    // rows per warp: about 24 warps per SM, at most 32 rows
    const int64_t warps = (int64_t)24 * sms();
    const int ch = chunk > 0 ? chunk : (int)std::min<int64_t>(32, std::max<int64_t>(1, ((int64_t)ntx * g.n[1] + warps - 1) / warps));
    const int64_t items = (int64_t)ntx * ((g.n[1] + ch - 1) / ch);
    const unsigned blocks = (unsigned)((items + NWP - 1) / NWP);
    auto al8 = [](const void* q) { return (reinterpret_cast<uintptr_t>(q) & 7u) == 0; };
    const bool vec = (g.n[0] & 1) == 0 && al8(a.Tin) && al8(a.b) && al8(a.Y0) && al8(a.Yjm2) && al8(a.MY0in) &&
                     al8(a.MY0out) && al8(a.out);
    if (vec)
        return launch_chained(plane_kernel<SP, SAT, LIM, true>, blocks, 32 * NWP, 0, st, chained, g, p, a, cf, status,
                              ch, ntx, (int)items);
    return launch_chained(plane_kernel<SP, SAT, LIM, false>, blocks, 32 * NWP, 0, st, chained, g, p, a, cf, status, ch,
                          ntx, (int)items);
}

}  // namespace
}  // namespace col

cudaError_t launch_stage_plane(const LaunchCfg& c, const KGrid<float>& g, const KPhys<float>& p, const StageIO& io,
                               const KCoef<float>& cf, unsigned* status, int chunk, cudaStream_t st)
{
    if (c.ndim != 2 || !col_stage_supported(c.dtype, c.ndim, g.n, g.plane) || (c.limiter && !c.lim_all))
        return cudaErrorNotSupported;
    const col::Args<float> a = col::stage_args<float>(io);
    auto go = [&](auto sp, auto sat) {
        constexpr bool SP = decltype(sp)::value, SAT = decltype(sat)::value;
        return c.limiter ? col::launch_plane<SP, SAT, true>(g, p, a, cf, status, chunk, st, io.chained)
                         : col::launch_plane<SP, SAT, false>(g, p, a, cf, status, chunk, st, io.chained);
    };
    using T = std::true_type;
    using F = std::false_type;
    if (c.spitzer) return c.saturate ? go(T{}, T{}) : go(T{}, F{});
    return c.saturate ? go(F{}, T{}) : go(F{}, F{});
}

}  // namespace rkl
