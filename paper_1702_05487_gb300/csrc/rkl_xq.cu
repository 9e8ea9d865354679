// Row-pair FP32 3D stage kernel (the tile body and kernel template are in
// rkl_xq.cuh): launches with the classical flux, the choice of build, the
// z-chunk of a launch, and the persistent ensemble kernel on the row-pair
// tile body.
#include <cmath>

#include "rkl_xq.cuh"

namespace rkl {
namespace xq {

// Persistent ensemble kernel on the row-pair tile body: the work list,
// dependency waits and completion counters of the paired-cell ensemble
// kernel (x2::ens_claim), each item a 64 x 8 tile (or 32 x 16 where the
// problem's txw is 32) of one stage of one problem.
template <bool SP, bool SAT>
__global__ void __launch_bounds__(NTHREADS, kCtasPerSm)
ensemble_q_kernel(const x2::EnsProb* __restrict__ probs, const x2::EnsSeg* __restrict__ segs, int nseg, int total,
                  int* work, unsigned* done, unsigned* status, int* abort_flag, long long spin_limit)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    SmemQ<64>& sm = *reinterpret_cast<SmemQ<64>*>(smem_raw);
    SmemQ<32>& sm32 = *reinterpret_cast<SmemQ<32>*>(smem_raw);
    __shared__ int s_go, s_p, s_j, s_tile;
    for (;;) {
        if (threadIdx.x == 0) {
            int p = 0, j = 0, tile = 0;
            s_go = x2::ens_claim(probs, segs, nseg, total, work, done, status, abort_flag, spin_limit, p, j, tile);
            s_p = p;
            s_j = j;
            s_tile = tile;
        }
        __syncthreads();
        if (!s_go) break;
        const x2::EnsProb& d = probs[s_p];
        const int j = s_j, tile = s_tile;
        const int bx = tile % d.tx, by = (tile / d.tx) % d.ty, bz = tile / (d.tx * d.ty);
        const bool narrow = d.txw == 32;
        const int i0 = bx * d.txw, j0 = by * (narrow ? SmemQ<32>::TY : SmemQ<64>::TY);
        const int z0 = bz * d.nzchunk;
        const int nzc = min(d.nzchunk, d.g.n[2] - z0);
        x2::FastArgs a;
        a.b = d.b;
        a.Y0 = d.T;
        a.coef_tab = d.coef;
        a.j = j;
        KCoef<float> cf{0.f, 0.f, 0.f, 0.f};
        if (j == 1) {
            a.Tin = d.T;
            a.Yjm2 = nullptr;
            a.MY0in = nullptr;
            a.MY0out = d.my0;
            a.out = d.buf[0];
            if (narrow) tile_q<SP, SAT, 1, 32>(sm32, d.g, d.p, a, cf, status, i0, j0, z0, nzc);
            else tile_q<SP, SAT, 1, 64>(sm, d.g, d.p, a, cf, status, i0, j0, z0, nzc);
        } else {
            a.Tin = d.buf[(j - 2) % 3];
            a.Yjm2 = j == 2 ? d.T : d.buf[(j - 3) % 3];
            a.MY0in = d.my0;
            a.MY0out = nullptr;
            a.out = j == d.s ? d.T : d.buf[(j - 1) % 3];
            if (narrow) tile_q<SP, SAT, 2, 32>(sm32, d.g, d.p, a, cf, status, i0, j0, z0, nzc);
            else tile_q<SP, SAT, 2, 64>(sm, d.g, d.p, a, cf, status, i0, j0, z0, nzc);
        }
        if (threadIdx.x == 0) {
            __threadfence();
            atomicAdd(&done[s_p], 1u);
        }
    }
}

template <bool SP, bool SAT>
cudaError_t ensemble_launch_q(const x2::EnsProb* probs, const x2::EnsSeg* segs, int nseg, int total, int* work,
                              unsigned* done, unsigned* status, int* abort_flag, long long spin_limit, int grid,
                              cudaStream_t st)
{
    const int smem = (int)std::max(sizeof(SmemQ<64>), sizeof(SmemQ<32>));
    static bool attr_set = false;
    if (!attr_set) {
        cudaError_t e = cudaFuncSetAttribute(ensemble_q_kernel<SP, SAT>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        attr_set = true;
    }
    if (grid <= 0) {
        int per = 0;
        cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, ensemble_q_kernel<SP, SAT>, NTHREADS, smem);
        if (e != cudaSuccess) return e;
        grid = sm_count() * (per > 0 ? per : 1);
    }
    if (grid > total) grid = total > 0 ? total : 1;
    ensemble_q_kernel<SP, SAT><<<grid, NTHREADS, smem, st>>>(probs, segs, nseg, total, work, done, status, abort_flag,
                                                             spin_limit);
    return cudaGetLastError();
}

// Planes per CTA.  Grids with at least 3.5 waves of CTAs at 16 planes: among
// 16 .. 64, the length that minimises (rounds of resident CTAs) x (planes +
// halo cost), keeping the 3.5 waves (the paired-cell kernel's rule with this
// kernel's tile and occupancy); down to one wave at 16 planes the same cost
// without that floor.  Grids below one wave fill the chip with shorter chunks, a
// chunk costing its planes and 1 for its prologue.  The fullest SM decides: of the
// time of three CTAs (all that an SM holds) two take 0.84 and one alone 0.65 (the
// classical flux on rows in 16-byte chunks: 0.75 and 0.5), a fourth starts the next round, and CTAs start in z order, so the short last
// chunks come last.  Past six CTAs an SM the rounds blur: a third of the CTAs,
// and a tenth more.  Fitted to 1 .. 64 planes on 34 boxes of 0.03 to 5 million
// cells, classical, saturated and limited, in the periodic, DIR and PAD builds:
// the choice is 1% above the best on average, 14%
// at worst.  100 x 150 x 157 saturated, a stage: 34.9 us with the 10 planes of a rule
// without rounds, now 28.8; 16 planes 31.9.  Stage time at 16 planes and now: 32^3 14.2 -> 2.9
// us, 64^3 11.6 -> 4.2, 96^3 14.5 -> 8.9, 128^3 15.7 -> 14.4, 128^3 saturated 23.7
// -> 19.1.
double rounds_cost(int64_t cols, int nz, int nzc, int64_t sms, bool light)
{
    const double F[4] = {0.0, light ? 0.5 : 0.65, light ? 0.75 : 0.84, 1.0};
    const int64_t chunks = (nz + nzc - 1) / nzc, ctas = cols * chunks;
    const int last = nz - (int)(chunks - 1) * nzc;
    const double k = (double)ctas / (double)sms;
    if (k > 6.0) return (nzc + 1.0) * k / 3.0 * 1.1;
    const int64_t K = (ctas + sms - 1) / sms, full = (K - 1) / kCtasPerSm;
    const int r = (int)((K - 1) % kCtasPerSm) + 1;
    if (chunks > 1 && ctas - sms * (K - 1) <= cols)       // the last to start are short ones
        return (nzc + 1.0) * full + (last + 1.0) * F[r] + (r > 1 ? (nzc - last) * F[r - 1] : 0.0);
    return (nzc + 1.0) * (full + F[r]);
}

int auto_nzchunk_q(const KGrid<float>& g, int tx, int ty, bool light)
{
    const int64_t cols = (int64_t)((g.n[0] + tx - 1) / tx) * ((g.n[1] + ty - 1) / ty);
    const int64_t sms = sm_count(), slots = kCtasPerSm * sms;
    const int64_t at16 = cols * ((g.n[2] + 15) / 16);
    const bool many = at16 * 2 >= 7 * slots, wave = at16 >= slots;
    int best = 32;
    double cost = 1e300;
    for (int nzc = wave ? 16 : 1; nzc <= 64; ++nzc) {
        double cst;
        if (wave) {
            const int64_t chunks = (g.n[2] + nzc - 1) / nzc;
            if (many && cols * chunks * 2 < 7 * slots) continue;
            const int64_t rounds = (cols * chunks + slots - 1) / slots;
            cst = (double)rounds * (std::min(nzc, g.n[2]) + 2.5);
        } else {
            cst = rounds_cost(cols, g.n[2], std::min(nzc, g.n[2]), sms, light);
        }
        if (cst < cost - 1e-9) {
            cost = cst;
            best = nzc;
        }
    }
    return best;
}

}  // namespace xq

x2::FastArgs x2_args(const StageIO& io);      // rkl_x2.cu

bool xq_stage_supported(const LaunchCfg& c, const KGrid<float>& g)
{
    return c.dtype == 0 && c.ndim == 3 && (!c.limiter || c.lim_all) && g.bc == 0 && (g.n[0] % 4) == 0 &&
           g.ncell < ((int64_t)1 << 31);
}

cudaError_t launch_stage_xq(const LaunchCfg& c, const KGrid<float>& g, const KPhys<float>& p, const StageIO& io,
                            const KCoef<float>& coef, unsigned* status, int nzchunk, cudaStream_t st, int txw)
{
    if (!xq_stage_supported(c, g) || (txw != 64 && txw != 32)) return cudaErrorNotSupported;
    const x2::FastArgs a = x2_args(io);
    // the limited build comes with 64-column tiles only
    if (c.limiter) txw = 64;
    if (nzchunk <= 0) nzchunk = xq::auto_nzchunk_q(g, txw, txw == 64 ? xq::SmemQ<64>::TY : xq::SmemQ<32>::TY,
                                                  !c.limiter && !c.saturate);
    if (c.limiter) return xq::launch_q_lim(c.spitzer != 0, c.saturate != 0, io.mode, g, p, a, coef, status, nzchunk, st, io.chained);
    if (c.saturate)
        return xq::launch_q_sat(c.spitzer != 0, p.kperp == 0.f, txw, io.mode, g, p, a, coef, status, nzchunk, st, io.chained);
    if (c.spitzer) {
        if (txw == 32) return xq::launch_q_mode<true, false, 32, false>(io.mode, g, p, a, coef, status, nzchunk, st, io.chained);
        return xq::launch_q_mode<true, false, 64, false>(io.mode, g, p, a, coef, status, nzchunk, st, io.chained);
    }
    if (txw == 32) return xq::launch_q_mode<false, false, 32, false>(io.mode, g, p, a, coef, status, nzchunk, st, io.chained);
    return xq::launch_q_mode<false, false, 64, false>(io.mode, g, p, a, coef, status, nzchunk, st, io.chained);
}

bool xg_stage_supported(const LaunchCfg& c, const KGrid<float>& g)
{
    // 65535 tiles of 8 rows
    return c.dtype == 0 && c.ndim == 3 && (!c.limiter || c.lim_all) && g.ncell < ((int64_t)1 << 31) &&
           g.n[1] <= 8 * 65535;
}

// GEN against the one-cell tiled kernel (32 x 8 tiles, an L1-served march that
// skips what lies outside) on rows of a few cells, from one wave of CTAs on
// (smaller grids need GEN's short chunks).  M of 500 x 500 rows with walls: 3
// cells 304 against 226 us, 17 cells 0.88 and 31 cells 1.06 of its speed; periodic rows
// of 1 cell 0.75, of 2 cells 1.26.
bool xg_stage_pays(const LaunchCfg& c, const KGrid<float>& g)
{
    if (g.n[0] % 4 == 0) return true;                   // DIR
    const int64_t at16 = (int64_t)((g.n[1] + 7) / 8) * ((g.n[2] + 15) / 16);
    const int narrow = g.bc == 0 ? 1 : (c.limiter ? 12 : 20);
    return g.n[0] > narrow || at16 < xq::kCtasPerSm * (int64_t)sm_count();
}

cudaError_t launch_stage_xg(const LaunchCfg& c, const KGrid<float>& g, const KPhys<float>& p, const StageIO& io,
                            const KCoef<float>& coef, unsigned* status, int nzchunk, cudaStream_t st)
{
    if (!xg_stage_supported(c, g)) return cudaErrorNotSupported;
    const x2::FastArgs a = x2_args(io);
    const bool dir = g.bc == 1 && g.n[0] % 4 == 0;
    int nzc = nzchunk > 0 ? nzchunk
                          : xq::auto_nzchunk_q(g, 64, xq::SmemQ<64>::TY, dir && !c.limiter && !c.saturate);
    nzc = std::max(nzc, (g.n[2] + 65534) / 65535);      // the grid's z limit
    if (dir)
        return (c.limiter ? xq::launch_q_dir_lim : xq::launch_q_dir)(c.spitzer != 0, c.saturate != 0, io.mode, g, p, a,
                                                                     coef, status, nzc, st, io.chained);
    if (c.limiter) return xq::launch_q_gen_lim(c.spitzer != 0, c.saturate != 0, io.mode, g, p, a, coef, status, nzc, st, io.chained);
    return xq::launch_q_gen(c.spitzer != 0, c.saturate != 0, io.mode, g, p, a, coef, status, nzc, st, io.chained);
}

namespace xq {

// Rows of nx cells (T, and the three components of b) into rows of `pitch`
// cells, four at a time; blockIdx.y: array.  The padding is not read.
__global__ void __launch_bounds__(256) pack_rows_kernel(const float* __restrict__ T, const float* __restrict__ b,
                                                        float* __restrict__ pT, float* __restrict__ pb, unsigned chunks,
                                                        int nx, int pitch, int64_t ncell, int64_t npad)
{
    const unsigned q = blockIdx.x * 256u + threadIdx.x, cpr = (unsigned)pitch / 4u;
    if (q >= chunks) return;
    const unsigned row = q / cpr, c = 4u * (q - row * cpr);
    const float* s = (blockIdx.y == 0 ? T : b + (int64_t)(blockIdx.y - 1) * ncell) + (int64_t)row * nx + c;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    const int n = nx - (int)c;
    v.x = s[0];
    if (n > 1) v.y = s[1];
    if (n > 2) v.z = s[2];
    if (n > 3) v.w = s[3];
    reinterpret_cast<float4*>(blockIdx.y == 0 ? pT : pb + (int64_t)(blockIdx.y - 1) * npad)[q] = v;
}
__global__ void __launch_bounds__(256) unpack_rows_kernel(const float* __restrict__ pT, float* __restrict__ T,
                                                          unsigned chunks, int nx, int pitch)
{
    const unsigned q = blockIdx.x * 256u + threadIdx.x, cpr = (unsigned)pitch / 4u;
    if (q >= chunks) return;
    const unsigned row = q / cpr, c = 4u * (q - row * cpr);
    const float4 v = reinterpret_cast<const float4*>(pT)[q];
    float* d = T + (int64_t)row * nx + c;
    const int n = nx - (int)c;
    d[0] = v.x;
    if (n > 1) d[1] = v.y;
    if (n > 2) d[2] = v.z;
    if (n > 3) d[3] = v.w;
}

}  // namespace xq

cudaError_t launch_pack_rows(const KGrid<float>& g, const void* T, const void* b, void* pT, void* pb, cudaStream_t st)
{
    const int64_t chunks = g.ncell / 4, ncell = (int64_t)g.n[0] * g.n[1] * g.n[2];
    xq::pack_rows_kernel<<<dim3((unsigned)((chunks + 255) / 256), 4), 256, 0, st>>>(
        static_cast<const float*>(T), static_cast<const float*>(b), static_cast<float*>(pT), static_cast<float*>(pb),
        (unsigned)chunks, g.n[0], g.pitch, ncell, g.ncell);
    return cudaGetLastError();
}
cudaError_t launch_unpack_rows(const KGrid<float>& g, const void* pT, void* T, cudaStream_t st)
{
    const int64_t chunks = g.ncell / 4;
    xq::unpack_rows_kernel<<<(unsigned)((chunks + 255) / 256), 256, 0, st>>>(
        static_cast<const float*>(pT), static_cast<float*>(T), (unsigned)chunks, g.n[0], g.pitch);
    return cudaGetLastError();
}
cudaError_t launch_stage_xp(const LaunchCfg& c, const KGrid<float>& g, const KPhys<float>& p, const StageIO& io,
                            const KCoef<float>& coef, unsigned* status, int nzchunk, cudaStream_t st)
{
    if (!xg_stage_supported(c, g) || g.pitch % 4 != 0) return cudaErrorNotSupported;
    int nzc = nzchunk > 0 ? nzchunk : xq::auto_nzchunk_q(g, 64, xq::SmemQ<64>::TY, false);
    nzc = std::max(nzc, (g.n[2] + 65534) / 65535);      // the grid's z limit
    return (c.limiter ? xq::launch_q_pad_lim : xq::launch_q_pad)(c.spitzer != 0, c.saturate != 0, io.mode, g, p,
                                                                 x2_args(io), coef, status, nzc, st, io.chained);
}

cudaError_t launch_ensemble_xq(bool spitzer, bool saturate, const x2::EnsProb* probs, const x2::EnsSeg* segs,
                               int nseg, int total, int* work, unsigned* done, unsigned* status, int* abort_flag,
                               long long spin_limit, int grid, cudaStream_t st)
{
    if (spitzer) {
        if (saturate)
            return xq::ensemble_launch_q<true, true>(probs, segs, nseg, total, work, done, status, abort_flag,
                                                     spin_limit, grid, st);
        return xq::ensemble_launch_q<true, false>(probs, segs, nseg, total, work, done, status, abort_flag,
                                                  spin_limit, grid, st);
    }
    if (saturate)
        return xq::ensemble_launch_q<false, true>(probs, segs, nseg, total, work, done, status, abort_flag,
                                                  spin_limit, grid, st);
    return xq::ensemble_launch_q<false, false>(probs, segs, nseg, total, work, done, status, abort_flag, spin_limit,
                                               grid, st);
}

}  // namespace rkl
