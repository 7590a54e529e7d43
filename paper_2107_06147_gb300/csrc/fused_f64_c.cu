// fused_f64_c.cu -- double instantiations of the fused trajectory kernel for N in {8192}.
#include "fused.cuh"
#include "fused_launch.cuh"

namespace qt {

cudaError_t fused_launch_f64_c(int N, const Tables<double> &tb, const LaunchArgs &a, int sm_count, int max_ctas,
                             cudaStream_t s, FusedInfo *info, bool query_only, int variant)
{
    switch (N) {
    case 8192: return tb.potential == 1 ? fused_go<double, 8192, 5>(tb, a, sm_count, max_ctas, s, info, query_only)
                                  : a.trace_every > 0 ? fused_go<double, 8192, 4>(tb, a, sm_count, max_ctas, s, info, query_only)
                                  : fused_go<double, 8192, 0>(tb, a, sm_count, max_ctas, s, info, query_only);
    default: return cudaErrorInvalidValue;
    }
}

} // namespace qt
