// level_fp64_library.cu -- Milstein level kernels of FP64 paths on the CUDA library's normals (a translation
// unit of their own, compiled in parallel).
#include "level_kernel.cuh"

namespace mlmcgb {
const void *level_kernel_fp64_library(int payoff, int mt, bool split, bool long_lanes, bool positive)
{
    if (mt == 4)
        return split ? select_by_payoff<double, 4, true, kLibrary>(payoff, long_lanes, positive)
                     : select_by_payoff<double, 4, false, kLibrary>(payoff, long_lanes);
    if (mt == 0)
        return split ? select_by_payoff<double, 0, true, kLibrary>(payoff, long_lanes, positive)
                     : select_by_payoff<double, 0, false, kLibrary>(payoff, long_lanes);
    return nullptr;
}
const void *level_anti_kernel_fp64_library(int payoff, int mt, bool long_lanes)
{
    if (mt == 4) return select_anti_by_payoff<double, 4, kLibrary>(payoff, long_lanes);
    if (mt == 0) return select_anti_by_payoff<double, 0, kLibrary>(payoff, long_lanes);
    return nullptr;
}
}  // namespace mlmcgb
