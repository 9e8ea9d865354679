// Row-pair stage kernel for row-padded arrays (rkl_xq.cuh, PAD
// builds), MC limiter at every face; a translation unit of its own so that it compiles
// beside the others.
#include "rkl_xq.cuh"

namespace rkl {
namespace xq {

cudaError_t launch_q_pad_lim(bool sp, bool sat, int mode, const KGrid<float>& g, const KPhys<float>& p,
                             const x2::FastArgs& a, const KCoef<float>& cf, unsigned* status, int nzchunk,
                             cudaStream_t st, bool chained)
{
    if (sp) {
        if (sat) return launch_q_mode<true, true, 64, false, true, Q_PAD>(mode, g, p, a, cf, status, nzchunk, st, chained);
        return launch_q_mode<true, false, 64, false, true, Q_PAD>(mode, g, p, a, cf, status, nzchunk, st, chained);
    }
    if (sat) return launch_q_mode<false, true, 64, false, true, Q_PAD>(mode, g, p, a, cf, status, nzchunk, st, chained);
    return launch_q_mode<false, false, 64, false, true, Q_PAD>(mode, g, p, a, cf, status, nzchunk, st, chained);
}

}  // namespace xq
}  // namespace rkl
