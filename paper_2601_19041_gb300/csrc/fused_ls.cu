// The one-ant-per-quad form of the fused cluster kernel (fused.cuh) for groups
// with local search.
#include "fused.cuh"

namespace hac {

cudaError_t launch_fused_quad_ls(const FusedArgs &A, const FusedLaunch &L)
{
    if (A.kp_cap <= 16) return launch_fused_form<8, 4, true>(A, L);
    if (A.kp_cap <= 20) return launch_fused_form<8, 5, true>(A, L);
    return launch_fused_form<8, 8, true>(A, L);
}

}  // namespace hac
