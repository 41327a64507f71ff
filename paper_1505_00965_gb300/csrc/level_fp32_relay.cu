// level_fp32_relay.cu -- FP32-path level kernels for launches of few, long paths (level_relay_kernel).
#include "level_kernel.cuh"
#include "mlmc.h"

namespace mlmcgb {
const void *level_relay_kernel_fp32(int payoff, int mt, bool split, int scheme, bool long_lanes, bool positive)
{
    if (mt < 0) return nullptr;
    if (scheme == MLMC_MILSTEIN)
        return mt == 4 ? select_relay<4, true>(payoff, split, long_lanes, positive)
                       : select_relay<0, true>(payoff, split, long_lanes, positive);
    return mt == 4 ? select_relay<4, false>(payoff, split, long_lanes, positive)
                   : select_relay<0, false>(payoff, split, long_lanes, positive);
}
}  // namespace mlmcgb
