// fused_f64_b.cu -- double instantiations of the fused trajectory kernel for N in {2048, 4096}.
#include "fused.cuh"
#include "fused_launch.cuh"

namespace qt {
cudaError_t fused_launch_f64_c(int N, const Tables<double> &tb, const LaunchArgs &a, int sm_count, int max_ctas,
                             cudaStream_t s, FusedInfo *info, bool query_only, int variant);

cudaError_t fused_launch_f64_b(int N, const Tables<double> &tb, const LaunchArgs &a, int sm_count, int max_ctas,
                             cudaStream_t s, FusedInfo *info, bool query_only, int variant)
{
    switch (N) {
    case 2048: return tb.potential == 1 ? fused_go<double, 2048, 5>(tb, a, sm_count, max_ctas, s, info, query_only)
                                  : a.trace_every > 0 ? fused_go<double, 2048, 4>(tb, a, sm_count, max_ctas, s, info, query_only)
                                  : fused_go<double, 2048, 0>(tb, a, sm_count, max_ctas, s, info, query_only);
    case 4096: return tb.potential == 1 ? fused_go<double, 4096, 5>(tb, a, sm_count, max_ctas, s, info, query_only)
                                  : a.trace_every > 0 ? fused_go<double, 4096, 4>(tb, a, sm_count, max_ctas, s, info, query_only)
                                  : fused_go<double, 4096, 0>(tb, a, sm_count, max_ctas, s, info, query_only);
    default: return fused_launch_f64_c(N, tb, a, sm_count, max_ctas, s, info, query_only, variant);
    }
}

} // namespace qt
