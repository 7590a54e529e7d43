// fused_f32_a.cu -- float instantiations of the fused trajectory kernel for N in {16, 32, 64, 128, 256, 512, 1024}.
#include "fused.cuh"
#include "fused_ksu32.cuh"
#include "fused_launch.cuh"

namespace qt {
cudaError_t fused_launch_f32_b(int N, const Tables<float> &tb, const LaunchArgs &a, int sm_count, int max_ctas,
                             cudaStream_t s, FusedInfo *info, bool query_only, int variant);

cudaError_t fused_launch_f32(int N, const Tables<float> &tb, const LaunchArgs &a, int sm_count, int max_ctas,
                             cudaStream_t s, FusedInfo *info, bool query_only, int variant)
{
    switch (N) {
    case 16: return tb.potential == 1 ? ksu32_go<16>(tb, a, sm_count, max_ctas, s, info, query_only)
                                  : a.trace_every > 0 ? fused_go<float, 16, 4>(tb, a, sm_count, max_ctas, s, info, query_only)
                                  : fused_go<float, 16, 0>(tb, a, sm_count, max_ctas, s, info, query_only);
    case 32: return tb.potential == 1 ? ksu32_go<32>(tb, a, sm_count, max_ctas, s, info, query_only)
                                  : a.trace_every > 0 ? fused_go<float, 32, 4>(tb, a, sm_count, max_ctas, s, info, query_only)
                                  : fused_go<float, 32, 0>(tb, a, sm_count, max_ctas, s, info, query_only);
    case 64: return tb.potential == 1 ? ksu32_go<64>(tb, a, sm_count, max_ctas, s, info, query_only)
                                  : a.trace_every > 0 ? fused_go<float, 64, 4>(tb, a, sm_count, max_ctas, s, info, query_only)
                                  : fused_go<float, 64, 0>(tb, a, sm_count, max_ctas, s, info, query_only);
    case 128: return tb.potential == 1 ? ksu32_go<128>(tb, a, sm_count, max_ctas, s, info, query_only)
                                  : a.trace_every > 0 ? fused_go<float, 128, 4>(tb, a, sm_count, max_ctas, s, info, query_only)
                                  : fused_go<float, 128, 0>(tb, a, sm_count, max_ctas, s, info, query_only);
    case 256: return tb.potential == 1 ? ksu32_go<256>(tb, a, sm_count, max_ctas, s, info, query_only)
                                  : a.trace_every > 0 ? fused_go<float, 256, 4>(tb, a, sm_count, max_ctas, s, info, query_only)
                                  : fused_go<float, 256, 0>(tb, a, sm_count, max_ctas, s, info, query_only);
    case 512: return tb.potential == 1 ? ksu32_go<512>(tb, a, sm_count, max_ctas, s, info, query_only)
                                  : a.trace_every > 0 ? fused_go<float, 512, 4>(tb, a, sm_count, max_ctas, s, info, query_only)
                                  : fused_go<float, 512, 0>(tb, a, sm_count, max_ctas, s, info, query_only);
    case 1024: return tb.potential == 1 ? ksu32_go<1024>(tb, a, sm_count, max_ctas, s, info, query_only)
                                  : a.trace_every > 0 ? fused_go<float, 1024, 4>(tb, a, sm_count, max_ctas, s, info, query_only)
                                  : fused_go<float, 1024, 0>(tb, a, sm_count, max_ctas, s, info, query_only);
    default: return fused_launch_f32_b(N, tb, a, sm_count, max_ctas, s, info, query_only, variant);
    }
}

} // namespace qt
