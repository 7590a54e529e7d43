// fused_f32_b.cu -- float instantiations of the fused trajectory kernel for N in {2048, 4096}.
#include "fused.cuh"
#include "fused_ksu32.cuh"
#include "fused_launch.cuh"

namespace qt {
cudaError_t fused_launch_f32_c(int N, const Tables<float> &tb, const LaunchArgs &a, int sm_count, int max_ctas,
                             cudaStream_t s, FusedInfo *info, bool query_only, int variant);

cudaError_t fused_launch_f32_b(int N, const Tables<float> &tb, const LaunchArgs &a, int sm_count, int max_ctas,
                             cudaStream_t s, FusedInfo *info, bool query_only, int variant)
{
    // the per-step summary runs the traced twin of the context's plan, the KSU potential its own kernel
    if (tb.potential == 1) variant = 0;
    else if (a.trace_every > 0) variant = variant >= 2 ? 6 : 0;
    switch (N) {
    case 2048:
        switch (variant) {
        case 1: return fused_go<float, 2048, 1>(tb, a, sm_count, max_ctas, s, info, query_only);
        case 2: return fused_go<float, 2048, 2>(tb, a, sm_count, max_ctas, s, info, query_only);
        case 3: return fused_go<float, 2048, 3>(tb, a, sm_count, max_ctas, s, info, query_only);
        case 6: return fused_go<float, 2048, 6>(tb, a, sm_count, max_ctas, s, info, query_only);
        default: return tb.potential == 1 ? ksu32_go<2048>(tb, a, sm_count, max_ctas, s, info, query_only)
                                  : a.trace_every > 0 ? fused_go<float, 2048, 4>(tb, a, sm_count, max_ctas, s, info, query_only)
                                  : fused_go<float, 2048, 0>(tb, a, sm_count, max_ctas, s, info, query_only);
        }
    case 4096:   // (variant 1 is variant 0: FusedBounds)
        switch (variant) {
        case 2: return fused_go<float, 4096, 2>(tb, a, sm_count, max_ctas, s, info, query_only);
        case 3: return fused_go<float, 4096, 3>(tb, a, sm_count, max_ctas, s, info, query_only);
        case 6: return fused_go<float, 4096, 6>(tb, a, sm_count, max_ctas, s, info, query_only);
        default: return tb.potential == 1 ? ksu32_go<4096>(tb, a, sm_count, max_ctas, s, info, query_only)
                                  : a.trace_every > 0 ? fused_go<float, 4096, 4>(tb, a, sm_count, max_ctas, s, info, query_only)
                                  : fused_go<float, 4096, 0>(tb, a, sm_count, max_ctas, s, info, query_only);
        }
    default: return fused_launch_f32_c(N, tb, a, sm_count, max_ctas, s, info, query_only, variant);
    }
}

} // namespace qt
