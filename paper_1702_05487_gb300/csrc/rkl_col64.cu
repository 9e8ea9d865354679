// Column-march stage kernels (rkl_col.cuh), FP64 instances, in a translation
// unit of their own so that they compile beside the FP32 ones.
#include "rkl_col.cuh"

namespace rkl {

cudaError_t launch_stage_col(const LaunchCfg& c, const KGrid<double>& g, const KPhys<double>& p, const StageIO& io,
                             const KCoef<double>& coef, unsigned* status, cudaStream_t st)
{
    if (!col_stage_supported(c.dtype, c.ndim, g.n, g.plane)) return cudaErrorNotSupported;
    return col::launch<double>(c, g, p, io, coef, status, st);
}

}  // namespace rkl
