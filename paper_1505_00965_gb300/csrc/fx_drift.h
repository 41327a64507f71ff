// fx_drift.h -- the drift of fixed-point steps (host constants and their use in a path's loop).
#pragma once
#include <cmath>
#include <cstdint>

#ifdef __CUDACC__
#define MLMC_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define MLMC_HOST_DEVICE inline
#endif

namespace mlmcgb {

// The drift of a step in units of 2^-u: rh whole units and the fraction rest 2^-32.  A path's steps go in
// groups of equal drift, rh or rh + 1 as the running sum of the fractions carries, so the drift of any
// run of groups is within one group's steps (in units) of the exact one.  (One rounded drift for all
// steps was up to half a unit off in each: 7e-13 of S after 2^24 steps, twice the walk of FP64 roundings.)
struct FxDrift {
    int64_t rh;
    uint32_t rest;
};
// more: units that each step's other products drop on average (Milstein).
inline FxDrift fx_drift(double drift, int u, double more = 0.0)
{
    const double x = std::ldexp(drift, u), r = std::floor(x), rest = x - r + more;
    return {(int64_t)r + (int64_t)std::floor(rest), (uint32_t)std::ldexp(rest - std::floor(rest), 32)};
}
// The mean of what fx_mul64(a, b) lacks of a b 2^-64 over a: half a unit for each cross product and a
// quarter of the low words' product, with b's own words.
inline double fx_dropped_mean(uint64_t b)
{
    const uint32_t lo = (uint32_t)b;
    return (b >> 32 ? 0.5 : 0.0) + (lo ? 0.5 : 0.0) + std::ldexp((double)lo, -33);
}
// The sum ahead of group g (half a unit to begin with: a single group takes the nearest unit), and the
// drift of the next group.
MLMC_HOST_DEVICE uint32_t fx_drift_sum(uint32_t rest, int g) { return 0x80000000u + rest * (uint32_t)g; }
MLMC_HOST_DEVICE int64_t fx_drift_next(int64_t rh, uint32_t rest, uint32_t &sum)
{
    const uint32_t next = sum + rest;
    rh += next < sum ? 1 : 0;
    sum = next;
    return rh;
}
// Philox calls of a group.  Euler--Maruyama: 256 steps, whose 2^-55 S does not see; what the fine steps
// take, the coarse ones do too.  Milstein: single calls, since its coarse path has the FP64 drift.
template <bool MILSTEIN> constexpr int kDriftCalls = MILSTEIN ? 1 : 64;

}  // namespace mlmcgb
