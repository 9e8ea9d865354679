// Column-march stage kernels (rkl_col.cuh) and the rule for the grids they
// take.
#include "rkl_col.cuh"

namespace rkl {
namespace col {

int sms()
{
    static int n = 0;
    if (n == 0) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0)
            n = 152;
    }
    return n;
}

}  // namespace col

// 2D grids with 32-bit element offsets, FP64 3D grids with 32-bit offsets in
// a plane and block counts that fit a launch; the rest stays with the
// generic kernel.
bool col_stage_supported(int dtype, int ndim, const int n[3], int64_t plane)
{
    if (ndim == 2) return plane < ((int64_t)1 << 31) - ((int64_t)1 << 21);
    return ndim == 3 && dtype == 1 && plane < ((int64_t)1 << 31) && n[1] <= 8 * 65535 && n[2] <= 65535;
}

// Idle lanes of a march are lost time, so narrow grids stay with one thread per
// cell.  FP64: the march's cost against the generic kernel's, which the cells on
// its fullest SM decide beyond the time of a single one (96 cells take as long as
// a lone block's plane, 13 as long as a warp's row, small numbers longer).  A
// Spitzer stage: 12 x 18 x 508 march 80, generic 58 us; 4 x 3 x 5000 330 and 39;
// 112 x 96 x 80 176 and 419; 2D 2 x 10^5 315 and 65.  Over 225 grids with five
// fluxes the choice is at most 3% slower than the generic kernel.  FP32 rows of up to five cells
// cost what a warp's row costs once there are more of them than warps (10^5 rows
// of one cell, saturated: 32 against 7.6 us a stage).
bool col_stage_pays(const LaunchCfg& c, const int n[3])
{
    const bool lim = c.limiter != 0;
    if (c.dtype == 0) return n[0] > 5 || n[1] <= 128 * col::sms();
    const double cells = generic_cells((int64_t)n[0] * n[1] * n[2]);
    if (c.ndim == 2) {
        const double few = lim ? 90.0 : (c.saturate ? 160.0 : (c.spitzer ? 230.0 : 280.0));
        const double generic = std::max({15.0, cells / 13.0, (cells + few) / 17.5});
        return col::chunk2(col::cols2(n[0]), n[1], lim).cost <= generic;
    }
    const col::Cols q = col::cols3(n[0], n[1]);
    const double least = lim || c.saturate || c.spitzer ? 2.5 : 3.5;
    const double generic = std::max({least, cells / 96.0, (cells + 170.0) / 124.0});
    return col::chunk3((int64_t)q.bx * q.by, n[2], lim).cost <= generic;
}

cudaError_t launch_stage_col(const LaunchCfg& c, const KGrid<double>& g, const KPhys<double>& p, const StageIO& io,
                             const KCoef<double>& coef, unsigned* status, int chunk, cudaStream_t st)
{
    if (!col_stage_supported(c.dtype, c.ndim, g.n, g.plane)) return cudaErrorNotSupported;
    return col::launch<double>(c, g, p, io, coef, status, chunk, st);
}

}  // namespace rkl
