// The fused cluster kernel (fused.cuh) with one ant per lane pair or lane, for groups
// without local search.
#include "fused.cuh"

namespace hac {

cudaError_t launch_fused_lane(const FusedArgs &A, const FusedLaunch &L)
{
    const int G = A.kp_cap / 4;   // slot groups; lane h of a pair holds groups 2j + h
    if (A.apw == 32) {
        if (G <= 3) return launch_fused_form<32, 3, false>(A, L);
        if (G <= 5) return launch_fused_form<32, 5, false>(A, L);
        return launch_fused_form<32, 8, false>(A, L);
    }
    if (G <= 4) return launch_fused_form<16, 2, false>(A, L);
    if (G <= 6) return launch_fused_form<16, 3, false>(A, L);
    return launch_fused_form<16, 4, false>(A, L);
}

}  // namespace hac
