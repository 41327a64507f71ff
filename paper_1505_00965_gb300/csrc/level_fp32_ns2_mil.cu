// level_fp32_ns2_mil.cu -- two samples per thread: FP32 Milstein and antithetic kernels (M = 4).
#include "level_kernel.cuh"

namespace mlmcgb {
const void *level_ns2_kernel_fp32_other(int payoff, int mt, int scheme, bool anti, bool long_lanes)
{
    if (mt != 4) return nullptr;
    if (anti)
        return scheme == 1 ? select_ns2_by_payoff<float, 4, true, true>(payoff, long_lanes)
                           : select_ns2_by_payoff<float, 4, false, true>(payoff, long_lanes);
    return select_ns2_by_payoff<float, 4, true, false>(payoff, long_lanes);
}
}  // namespace mlmcgb
