// level_fp32_ns2.cu -- FP32-path Euler--Maruyama level kernels with two samples per thread (a
// translation unit of their own, compiled in parallel with the one-sample kernels; the Milstein and
// antithetic ones in level_fp32_ns2_mil.cu).
#include "level_kernel.cuh"

namespace mlmcgb {
const void *level_ns2_kernel_fp32(int payoff, int mt, int scheme, bool anti, bool long_lanes)
{
    if (scheme != 0 || anti) return level_ns2_kernel_fp32_other(payoff, mt, scheme, anti, long_lanes);
    if (mt == 4) return select_ns2_by_payoff<float, 4, false, false>(payoff, long_lanes);
    if (mt == 0) return select_ns2_by_payoff<float, 0, false, false>(payoff, long_lanes);
    return nullptr;
}
}  // namespace mlmcgb
