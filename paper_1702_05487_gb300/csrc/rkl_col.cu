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

cudaError_t launch_stage_col(const LaunchCfg& c, const KGrid<double>& g, const KPhys<double>& p, const StageIO& io,
                             const KCoef<double>& coef, unsigned* status, cudaStream_t st)
{
    if (!col_stage_supported(c.dtype, c.ndim, g.n, g.plane)) return cudaErrorNotSupported;
    return col::launch<double>(c, g, p, io, coef, status, st);
}

}  // namespace rkl
