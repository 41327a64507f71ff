// engine.h -- internal interface between the C ABI and the level kernels.
#pragma once
#include <cmath>
#include <cstddef>
#include <cstdint>

namespace mlmcgb {

// Payoff codes, equal to the public mlmc_payoff_kind values.
enum : int { kEuropean = 0, kAsian = 1, kLookback = 2, kDigital = 3, kLinear = 100, kGeoAsian = 101 };

// Time-stepping schemes of the level kernels: the public mlmc_scheme values of the GBM model, and Milstein
// FP64 paths on the library's normals (path_scheme).
enum : int { kEuler = 0, kMilstein = 1, kLibrary = 16 };

// Everything one level launch needs, passed by value as the kernel argument.
struct LevelParams {
    double S0;        // initial value
    double disc;      // exp(-r T)
    double K, Q;      // strike, digital cash
    double a;         // sigma * sqrt(h), h = T / M^l
    double rh;        // r * fine step
    double inv_nf;    // 1 / M^l
    double inv_nc;    // 1 / M^(l-1)
    double sqrt_h;    // sqrt(h): Brownian increment scale of one fine step
    double sqrt_tg;   // sqrt(T / 16): scale of the control variate's grid increments
    double h;         // fine step T / M^l
    // FP32 payoff constants of the call options on paths relative to S0 (rel_payoff): disc S0,
    // -disc K, and for the fine (f) and coarse (c) path disc S0 / n, disc S0 / (2 n) - disc K
    float pay_dS0, pay_mdK, pay_af, pay_bf, pay_ac, pay_bc;
    // FP64 constants of the payoffs formed in fixed point (fx_fixed): disc S0 and K / S0
    double pay_dS0_64, pay_k64;
    // FP64 steps in fixed point (fx_steps): their unit is 2^-fx, 0 where they run in FP64; sigma sqrt(h)
    // and sigma^2 h / 2 in units of 2^-(fx + 6), the whole units of r h
    // (Milstein: r h - sigma^2 h / 2) in 2^-fx
    uint64_t fx_a, fx_c2;
    int64_t fx_rh;
    uint32_t fx_rest;  // the fraction of a unit that fx_rh lacks (fx_drift.h)
    int fx;
    // samples of one Philox block at most (level 0; M^l = 4 with M = 4) whose payoff is formed in the
    // same units: 1 - K / S0, and whether it fits
    int64_t fx_base;
    int fx_fixed;
    uint64_t first;   // first sample index
    uint64_t N;       // number of samples
    uint32_t key0, key1;  // Philox key (seed low, seed high)
    uint32_t ctr3;        // Philox counter word 3: (tag << 16) | level
    uint32_t rkey[20];    // Philox round keys: key0 + i W_A, key1 + i W_B for rounds i = 0..9
    int level, M;
    int nf;           // fine steps M^l
    int lanes;        // lanes per sample (1 = one thread per sample)
    int small;        // 1 when M^l < 4: 4 / M^l samples share one Philox block
    int payoff;       // payoff code (the batched kernel selects its code path from it)
    double c2;        // sigma^2 h / 2: the Milstein term's scale on the fine grid
    int scheme;       // 0 Euler--Maruyama, 1 Milstein
    int fine_only;    // 1: Y = P_l alone (single-level estimator)
    int u23;          // FP64 arithmetic on the FP32 stream's 23-bit uniforms
    int antithetic;   // antithetic estimator (read by the kernel of levels with M^l < 4)
    double *partials; // [gridDim.x][4] block partial sums (workspace)
    double *out;      // [4] level sums (device)
    unsigned *ticket; // completion counter (workspace), zero between launches
    double *y_out;    // optional per-sample Y, NULL = off
};

// Workspace layout: the completion ticket in the first 256 bytes, then the FP64 partial sums
// of `blocks` blocks.  The ticket sits at a fixed offset so that launches of any grid size can
// share one workspace: it is zero between launches, while the partials need no initial value.
constexpr size_t kTicketBytes = 256;
inline size_t workspace_bytes_for_blocks(int blocks)
{
    return kTicketBytes + (size_t)blocks * 4 * sizeof(double);
}

// Kernel selection.  `mt` is 4 for the M = 4 specialisation, 0 for the generic-M kernel and
// -1 for the kernel of levels with M^l < 4.  `long_lanes`: a lane runs more than kLongLaneSteps
// fine steps of its path (M^l / lanes), for which the FP32 arithmetic-Asian kernels add the
// running sum in two levels (partials of 256 steps).  `positive`: every fine and coarse step
// factor 1 + d is positive for any normal the stream can produce, so the split lookback kernels
// keep no running minimum (no chunk of a path starts below zero).
constexpr long kLongLaneSteps = 4096;
const void *level_kernel_fp32(int payoff, int mt, bool split, int scheme, bool long_lanes, bool positive = false);
// Milstein kernels (level_fp32_mil.cu, level_fp64_mil.cu), selected by the two above.
const void *level_kernel_fp32_milstein(int payoff, int mt, bool split, bool long_lanes, bool positive);
const void *level_kernel_fp64_milstein(int payoff, int mt, bool split, bool long_lanes, bool positive);
// The same kernels with FP64 steps on the CUDA library's normals (level_fp64_library.cu).
const void *level_kernel_fp64_library(int payoff, int mt, bool split, bool long_lanes, bool positive);
const void *level_anti_kernel_fp64_library(int payoff, int mt, bool long_lanes);
// Level sums of FP64 Milstein paths of more than 1024 fine steps over fewer than 4096 samples (of more
// than 512 over fewer than 64) take the library's logarithm, root and sine, and FP64 steps, operation for
// operation.  P_l - P_{l-1} of strong order 1 shrinks like 1 / n while the rounding of its two paths grows
// like sqrt(n), so few samples' sums agree to 1e-9 only between forms that round alike; over N samples the
// difference falls like 1 / sqrt(N).  Largest
// difference of fixed-point sums to the library's (norm of the four sums, 2640 launches of 1e4 to 3e8 steps, coupled
// and antithetic, S0 = K = 100, r = 0.05, sigma = 0.2) by fine steps, M and samples below 64 / 512 / 4096 / above:
//    1024 (2)  1.1e-9  1.4e-10  8.8e-11  1.5e-11     4096 (4)   2.0e-9  3.3e-10  1.5e-10  4.4e-11
//    2048 (2)  4.4e-9  5.1e-10  8.9e-11  3.6e-11    16384 (4)   7.0e-8  1.7e-8   5.3e-10  1.8e-10
//    8192 (2)  4.6e-8  5.3e-9   5.7e-10  2.6e-10    65536 (4)   3.9e-7  3.7e-8   1.7e-8   4.5e-10 (3 launches)
// Beyond 16384 steps the least number of samples grows with n^3, which keeps n^1.5 / sqrt(N).  The library's
// form takes 24.9 ms for 3e8 steps, fixed point 1.7.  The adaptive drivers (many) keep fixed point: their sums
// build up over rounds, and no result of theirs divides by a deep level's sum alone.  Euler--Maruyama, of
// strong order 1/2, keeps fixed point too: over 3000 drawn launches of every kind three differed by more than
// 1e-9, of 9, 10 and 39 samples at 65536 steps whose Y nearly cancel; against extended precision the
// fixed-point sums were the nearer ones there (4.8e-10, 8.2e-10, 1.1e-10 against 2.0e-9, 1.2e-9, 1.8e-9).  The
// single-level estimator has no such difference.
constexpr long kMilsteinFixedSteps = 512, kMilsteinFewSteps = 1024, kMilsteinCubeSteps = 16384;
constexpr double kMilsteinFewSamples = 64.0, kMilsteinFixedSamples = 4096.0;
constexpr uint64_t kManySamples = UINT64_MAX;
inline int path_scheme(bool fp64, int scheme, bool single_level, long nf, uint64_t N)
{
    if (!fp64 || scheme != kMilstein || single_level || nf <= kMilsteinFixedSteps) return scheme;
    if (nf <= kMilsteinFewSteps) return (double)N < kMilsteinFewSamples ? kLibrary : scheme;
    const double over = nf > kMilsteinCubeSteps ? (double)nf / kMilsteinCubeSteps : 1.0;
    return (double)N < kMilsteinFixedSamples * over * over * over ? kLibrary : scheme;
}
// Antithetic level kernels (level_anti_fp32.cu, level_anti_fp64.cu): mt = 4 (M = 4) or 0 (M = 2).
const void *level_anti_kernel_fp32(int payoff, int mt, int scheme, bool long_lanes);
const void *level_anti_kernel_fp64(int payoff, int mt, int scheme, bool long_lanes);
// Two samples per thread (level_fp32_ns2.cu, level_fp32_ns2_mil.cu): FP32 paths, one thread per
// sample, at most 512 threads per block; Euler--Maruyama for mt = 4 or 0, Milstein and the antithetic
// estimator for mt = 4 (NULL where there is none).
const void *level_ns2_kernel_fp32(int payoff, int mt, int scheme, bool anti, bool long_lanes);
const void *level_ns2_kernel_fp32_other(int payoff, int mt, int scheme, bool anti, bool long_lanes);
constexpr int kNs2MaxThreads = 512;
// The planners' default of two samples per thread: FP32 whole paths with M = 4 and at least one Philox
// block.  The two-sample kernel takes the same samples per thread in the same order on the same grid
// (a thread's unpaired last sample runs alone).  One block (level 1), 4e7 samples, one against two:
// European 155.9 / 149.7 us, Asian 164.0 / 159.8, lookback 160.3 / 155.5, digital 179.8 / 172.3,
// Milstein 171.5-194.8 / 162.3-182.3, antithetic 166.0-194.2 / 159.6-188.6; even at 2e6 and below.
constexpr long kNs2MinSteps = 4;
inline const void *default_ns2_kernel(int precision_is_fp32, int payoff, int M, long nf, int scheme, bool anti, int threads)
{
    if (!precision_is_fp32 || M != 4 || nf < kNs2MinSteps || threads > kNs2MaxThreads) return nullptr;
    return level_ns2_kernel_fp32(payoff, 4, scheme, anti, nf > kLongLaneSteps);
}
// Launches of few, long FP32 paths (level_fp32_relay.cu): mt = 4 or 0, call and digital options; a block
// of 128 or 256 threads per 32 lanes, NULL where there is none.
const void *level_relay_kernel_fp32(int payoff, int mt, bool split, int scheme, bool long_lanes, bool positive);
// Threads of their blocks for `lane_warps` warps of lanes of `calls` Philox calls on `sms` SMs; 0 where
// the plain kernels are faster.  Timed against them on levels 4..8 at 4 to 1216 lane warps (152 SMs):
// level 8 on 32 lanes 41 against 90 us up to 152 lane warps, 62 against 92 at 500, 86 against 105 at
// 900, 104 against 106 at 1216; 64 calls per lane 19 against 25 us at 152, even at 900; whole paths of
// 64 calls even at 400.  256 threads win up to about 400 lane warps (level 6 whole paths: 57 against 70
// us at 152, 68 against 79 at 304, 111 against 108 at 500).
inline int relay_threads(double lane_warps, long calls, int sms)
{
    const double per_sm = lane_warps / sms;
    if (calls < 64 || per_sm > (calls < 128 ? 2.0 : 6.0)) return 0;
    return per_sm <= 2.6 ? 256 : 128;
}
// The lanes-per-path model of both planners (plan_level and the device rounds): the time of w waves
// of lane-items in whole waves (a partial last wave after whole ones costs min(1, kLanesTailSlope f
// + kLanesTailBase) at fill f), a split step's cost relative to a whole-path one, and the least steps
// of a lane.  Below one wave FP32 paths wait on latency: min(1, 3 w), and a quarter of a wave at
// least.  FP64 paths, integer arithmetic of four times the instructions per step, fill a scheduler
// with a few warps: launches of levels 3..7 at 0.02..0.96 waves took 0.26 of a wave up to w = 0.06,
// then 0.34, 0.56 and 0.82 at w = 0.16, 0.32 and 0.64 (3112 samples: level 4 76 -> 31 us, level 6
// 0.96 -> 0.12 ms against one lane each).
constexpr double kLanesTailSlope = 1.25, kLanesTailBase = 0.1, kLanesSplitStep = 1.08;
__host__ __device__ inline double lane_waves(double w, bool fp64)
{
    const double full = floor(w), tail = kLanesTailSlope * (w - full) + kLanesTailBase;
    if (w >= 1.0) return full + (tail < 1.0 ? tail : 1.0);
    const double part = fp64 ? 0.2 + 0.95 * w : 3.0 * w, least = fp64 ? 0.26 : 0.25;
    return part < least ? least : part < 1.0 ? part : 1.0;
}
// FP64, 1000 samples: level 3 takes 19.4 us on lanes of 32 steps, 15.3 of 16 and 14.4 of 8; level 4 20.5, 16.5
// and 18.5 (128 threads per block).
__host__ __device__ constexpr long min_lane_steps(bool fp64) { return fp64 ? 8 : 256; }
// The control variate's level-estimator kernel (cv_level.cu) for a payoff on level `level` with
// refinement M: compiled for M^l = 1, 4, 16 at M = 4, else for a run-time M^l; NULL for an unknown
// payoff.
const void *cv_level_kernel_fp32(int payoff, int level, int M);
// Level kernel of the QUINTIC_ODE model (ode.cu): precision, scheme (EM or tamed EM).
const void *ode_level_kernel(int precision, int scheme);
const void *level_kernel_fp64(int payoff, int mt, bool split, int scheme, bool long_lanes, bool positive = false);

// Batched rounds: one chunk of samples of one task (a level of one problem).
struct BatchChunk {
    uint64_t first;   // first sample of the chunk
    uint32_t task;    // index into the task array
    uint32_t count;   // samples in the chunk
};
// Chunks [begin, end) belong to one task; the header counts tasks and chunks of the round.
struct BatchRange {
    uint32_t begin, end;
};
struct BatchHeader {
    uint32_t n_tasks, n_chunks;
};
// Persistent batch kernel and its fixed-order reduction, per precision and M specialisation
// (mt = 4 or 0).
const void *batch_kernel_fp32(int mt);
const void *batch_kernel_fp64(int mt);
const void *batch_reduce_kernel();

}  // namespace mlmcgb
