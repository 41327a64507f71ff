// normal64.cuh -- Box--Muller normals for FP64 paths in 64-bit fixed point.
//
// The normals of one Philox block's word pair (xa, xb) are rho cos(2 pi u2), rho sin(2 pi u2) with
// rho = sqrt(-2 ln u1) and 32-bit (or, on the FP32 path's stream, 23-bit) uniforms.  GB300 runs 2
// FP64 operations per SM per clock (1.65 measured) against 24 widening 32-bit integer multiplies, 64
// integer adds and 16 MUFU operations, so one FP64 instruction costs as much as 12 or more widening
// multiplies.  CUDA's double-precision log, sqrt and sincospi took 32 of the 36.5 FP64
// instructions of a coupled step.  Here the whole pair is 34 widening integer multiplies and no FP64:
//
//   ln u1    u = w 2^-32 with an integer w: w normalised to mu in [1/2, 1), c = k / 512 the
//            multiple of 1/512 nearest 1 / mu (a hardware reciprocal), s = mu c - 1 exactly as a
//            32-bit integer in units of 2^-41 (|s| < 2^-10), and
//            -ln u = n ln 2 + ln c - (s - s^2/2 + s^3/3 - s^4/4 + s^5/5 - ...), table + series
//            (the argument reduction of Tang, "Table-driven implementation of the logarithm
//            function in IEEE floating-point arithmetic", ACM TOMS 16, 1990);
//   sqrt     a 24-bit hardware reciprocal root, then one third-order correction
//            p (1 + r/2 + 3 r^2/8), p = x y, r = 1 - p y (the binomial series of (1 - r)^(-1/2));
//   cos, sin quadrant, 4096 angles per quadrant by table, the rotation by the remaining angle
//            delta < pi/8192 as three shears with tan(delta / 2) and sin(delta) from their Taylor
//            series (nine 32-bit products; the four of the addition theorems take twelve).  With this
//            many angles the series' one further term is small enough for FP32, whose pipe idles:
//            512 angles took seven more products of the multiplier, which bounds the paths (digital
//            level 2, 1e7 samples: 0.902 -> 0.850 ms; Asian level 5, 3.0e5 samples: 1.759 -> 1.663 ms).
//
// Error (against quadruple precision, 3e6 random words and the edges of every reduction): cos and sin
// 2^-61.2 rms and 2^-58.2 at most, rho 2^-58.8 rms, 2^-56.8 at most from rho = 1/2 on and 2^-53.7 at
// most (rho about 2^-4).  The library's log and sqrt give rho with 2^-53.6 rms; the fixed-point error is
// absolute where theirs shrinks with rho: below rho = 0.2 (one word in 64) it is 2^-55.6 to 2^-57.1 rms by
// octave of 1 - u against 2^-56.7 to 2^-58.6, next to u = 1 (1 - u < 2^-10) 2^-56.2 against 2^-59.0
// (2^-59.2 with the cubic term in 64 bits there: 1.1 % more time, no digit of a sum).  An
// FP64 normal of size 1 to 2 rounds by up to 2^-53.
#pragma once
#include <cstdint>
#ifndef __CUDACC__
#include <cmath>
#include <cstring>
#endif

#include "normal64_tables.h"

namespace mlmcgb {

// The hardware operations, and stand-ins for them where a host compiler includes this file (the
// accuracy test): the reductions tolerate any reciprocal (root) within 2^-22.5.
#ifdef __CUDACC__
#define MLMC_FX __device__ __forceinline__
MLMC_FX uint32_t fx_mulhi(uint32_t a, uint32_t b) { return __umulhi(a, b); }
MLMC_FX int32_t fx_mulhi_s(int32_t a, int32_t b) { return __mulhi(a, b); }
// Left shift that brings the top bit to bit 31 (one instruction); -1 for 0.
MLMC_FX int fx_norm(uint32_t a)
{
    int n;
    asm("bfind.shiftamt.u32 %0, %1;" : "=r"(n) : "r"(a));
    return n;
}
// a << n, 0 for n beyond 31 (n taken unsigned).
MLMC_FX uint32_t fx_shl(uint32_t a, int n)
{
    uint32_t y;
    asm("shl.b32 %0, %1, %2;" : "=r"(y) : "r"(a), "r"(n));
    return y;
}
MLMC_FX float fx_rcp(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
MLMC_FX float fx_rsqrt(float x)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
MLMC_FX uint32_t fx_bits(float x) { return __float_as_uint(x); }
MLMC_FX uint32_t fx_round(float x) { return __float2uint_rn(x); }
MLMC_FX float fx_float(uint32_t x) { return __uint2float_rn(x); }
// The high word of (hi, lo) << k and the low word of (hi, lo) >> k, k < 32.
MLMC_FX uint32_t fx_shl_hi(uint32_t lo, uint32_t hi, int k) { return __funnelshift_l(lo, hi, k); }
MLMC_FX uint32_t fx_shr_lo(uint32_t lo, uint32_t hi, int k) { return __funnelshift_r(lo, hi, k); }
#else
#define MLMC_FX inline
MLMC_FX uint32_t fx_mulhi(uint32_t a, uint32_t b) { return (uint32_t)(((uint64_t)a * b) >> 32); }
MLMC_FX int32_t fx_mulhi_s(int32_t a, int32_t b) { return (int32_t)(((int64_t)a * b) >> 32); }
MLMC_FX int fx_norm(uint32_t a) { return a ? __builtin_clz(a) : -1; }
MLMC_FX uint32_t fx_shl(uint32_t a, int n) { return (uint32_t)n > 31u ? 0u : a << n; }
MLMC_FX float fx_rcp(float x) { return 1.0f / x; }
MLMC_FX float fx_rsqrt(float x) { return (float)(1.0 / std::sqrt((double)x)); }
MLMC_FX uint32_t fx_bits(float x)
{
    uint32_t u;
    std::memcpy(&u, &x, sizeof(u));
    return u;
}
MLMC_FX uint32_t fx_round(float x) { return (uint32_t)std::llrint(x); }
MLMC_FX float fx_float(uint32_t x) { return (float)x; }
MLMC_FX uint32_t fx_shl_hi(uint32_t lo, uint32_t hi, int k) { return k ? (hi << k) | (lo >> (32 - k)) : hi; }
MLMC_FX uint32_t fx_shr_lo(uint32_t lo, uint32_t hi, int k) { return k ? (lo >> k) | (hi << (32 - k)) : lo; }
using std::fmaf;
using std::fminf;
#endif

MLMC_FX uint64_t fx_wide(uint32_t a, uint32_t b) { return (uint64_t)a * b; }
MLMC_FX uint64_t fx_join(uint32_t lo, uint32_t hi) { return ((uint64_t)hi << 32) | lo; }

// The high 64 bits of a b, at most 2 below the exact value (the product of the low words and the
// carries of the cross products' low words are left out).
MLMC_FX uint64_t fx_mul64(uint64_t a, uint64_t b)
{
    const uint32_t al = (uint32_t)a, ah = (uint32_t)(a >> 32), bl = (uint32_t)b, bh = (uint32_t)(b >> 32);
    return fx_wide(ah, bh) + fx_mulhi(al, bh) + fx_mulhi(ah, bl);
}
// The high 64 bits of the 96-bit product a b, at most 1 below.
MLMC_FX uint64_t fx_mul64x32(uint64_t a, uint32_t b)
{
    return fx_wide((uint32_t)(a >> 32), b) + fx_mulhi((uint32_t)a, b);
}

// The uniform of a Philox word x as (w mod 2^32) 2^-32 in (0, 1], w = 0 standing for 2^32: the FP64
// stream's w = x + 1, or the FP32 path's u = 1 - (x mod 2^23) 2^-23, w = -(x << 9).  One multiply-add
// with uniform factors.
MLMC_FX uint32_t fx_word(uint32_t x, bool u23) { return x * (u23 ? 0u - 512u : 1u) + (u23 ? 0u : 1u); }

// sqrt(-2 ln(w 2^-32)) in units of 2^-60 (w = 0 stands for 2^32: the result is 0).
MLMC_FX uint64_t fx_radius(uint32_t w, const uint64_t *tab)
{
    const int n = fx_norm(w);
    const uint32_t m = fx_shl(w, n) | 0x80000000u;
    // k = 512 c, by a magic-number rounding of 2^41 / m
    const uint32_t k = fx_bits(fmaf(fx_rcp(fx_float(m)), 0x1p41f, 12582912.0f)) & 0x7FFu;
    const int32_t s = (int32_t)(m * k);  // m k - 2^41: the multiple of 2^32 drops out
    // n ln 2 + ln c in units of 2^-59; the entry before n = 0 takes w = 0 (n = -1, k = 1024) to 0
    const uint64_t A = tab[kFxLn2 + n] + tab[kFxLnC + k];
    // F = -ln u = A - (s - s^2/2 + s^3/3 - s^4/4 + s^5/5)
    const uint64_t q = (uint64_t)((int64_t)s * s);              // s^2: 2^-82, below 2^62
    const uint32_t s2 = (uint32_t)(q >> 32);                    // 2^-50
    const uint32_t br = 0x55555555u - (uint32_t)(s >> 11) + fx_mulhi(s2, 3277u);  // (1/3 - s/4 + s^2/5) 2^32
    const int64_t tail = (int64_t)s * (int32_t)fx_mulhi(s2, br);  // 2^-91
    uint64_t F = (uint64_t)((int64_t)s * -(1 << 18) + (int64_t)A) + (q >> 24) - (uint64_t)(int64_t)(int32_t)(tail >> 32);
    int extra = 0;
    // next to u = 1 (n = 0, c = 1; one word in 1024) the table part is 0 and the series alone, in units
    // of 2^-71, keeps the digits that F loses
    if (A == 0) {
        F = (q >> 12) - ((uint64_t)(int64_t)s << 30) - (uint64_t)(tail >> 20);
        extra = 6;
    }
    // sqrt(2 F): F normalised to x 2^64 by an even shift, x in [1/4, 1)
    const int e = fx_norm((uint32_t)(F >> 32)) & 30;
    const uint32_t xh = fx_shl_hi((uint32_t)F, (uint32_t)(F >> 32), e), xl = (uint32_t)F << e;
    // 1 / sqrt(x) in units of 2^-31: the hardware's, lowered by 2^-22 (above its error of 2^-22.9) ...
    const uint32_t y0 = (fx_bits(fminf(fx_rsqrt(fx_float(xh)), 0x1.fffffep-16f)) << 8) - 0x200u;
    // ... and corrected by (1 - x y0^2) / 2: x y0^2 in units of 2^-32, less its whole 2^32, is at most
    // 1.5 2^-30 too low; six units less keep p = x y below 1
    const uint64_t xyy = fx_wide(xh, fx_mulhi(y0, y0));
    const uint32_t y = y0 + (uint32_t)fx_mulhi_s((int32_t)(y0 >> 1),
                                                 (int32_t)(0u - 6u - fx_shr_lo((uint32_t)xyy, (uint32_t)(xyy >> 32), 30)));
    const uint64_t p = fx_mul64x32(fx_join(xl, xh), y);         // x y: 2^-63
    // 1 - p y in units of 2^-62, below 2^-28.4; four units more than the products' roundings keep it
    // above 0 and stand for the halves that the shifts below drop
    const uint64_t r = (uint64_t(1) << 62) + 4u - fx_mul64x32(p, y);
    // sqrt(x) = p (1 + r / 2); the next term, 3 r^2 / 8, is below 2^-58 and 2^-61 on average
    const uint64_t corr = fx_wide((uint32_t)(p >> 32), fx_shr_lo((uint32_t)r, (uint32_t)(r >> 32), 2));  // 2^-92
    const uint64_t root = p + (corr >> 29);                     // 2^-63
    const int sh = (e >> 1) + extra;
    return fx_join(fx_shr_lo((uint32_t)root, (uint32_t)(root >> 32), sh), (uint32_t)(root >> 32) >> sh);
}

// |cos| and |sin| of 2 pi t 2^-32 reduced to the first quadrant, in units of 2^-62; in quadrant
// q = t >> 30, (cos, sin) = (c, s), (-s, c), (-c, -s), (s, -c) for q = 0..3.
MLMC_FX void fx_circle(uint32_t t, const uint64_t *tab, uint64_t &c, uint64_t &s)
{
    const uint32_t i = (t >> 18) & 4095u;
    const uint64_t C = tab[kFxCos + i], S = tab[kFxCos + 4096 - i];
    const uint32_t dt = t << 14;                                // delta = 2 pi dt 2^-46 < pi / 8192
    const uint64_t D = fx_mul64x32(kFxTwoPi60, dt);             // delta: 2^-74
    // sin delta = delta - e and tan(delta / 2) = (delta + e / 2) / 2 with e = delta^3 / 6 (the next terms
    // are below 2^-61), itself below 2^-36.6 and so in FP32, in units of 2^-68
    const float df = (float)(int32_t)(uint32_t)(D >> 32);       // 2^-42
    const uint32_t e = fx_round(df * df * (df * (0x1p-58f / 6)));
    const uint64_t v = D - ((uint64_t)e << 6);
    const uint64_t w = D + ((uint64_t)e << 5);                  // tan(delta / 2): 2^-75
    // the rotation by delta as three shears: c1 = C - w S, s = S + v c1, c = c1 - w s
    const uint64_t c1 = C - (fx_mul64(w, S) >> 11);             // products in units of 2^-73, 2^-72
    s = S + (fx_mul64(v, c1) >> 10);
    c = c1 - (fx_mul64(w, s) >> 11);
}
// Signs of the cosine and sine of angle t as all-ones masks, and whether they trade places.
MLMC_FX uint64_t fx_cos_sign(uint32_t t) { return (uint64_t)(int64_t)((int32_t)(t + 0x40000000u) >> 31); }
MLMC_FX uint64_t fx_sin_sign(uint32_t t) { return (uint64_t)(int64_t)((int32_t)t >> 31); }
MLMC_FX bool fx_swapped(uint32_t t) { return (t & 0x40000000u) != 0; }

// The two normals of a word pair, in units of 2^-58.
constexpr double kFxZ = 0x1p-58;
MLMC_FX void fx_pair(uint32_t xa, uint32_t xb, bool u23, const uint64_t *tab, int64_t &z0, int64_t &z1)
{
    const uint64_t rho = fx_radius(fx_word(xa, u23), tab);
    const uint32_t t = fx_word(xb, u23);
    uint64_t c, s;
    fx_circle(t, tab, c, s);
    const uint64_t m0 = fx_cos_sign(t), m1 = fx_sin_sign(t);
    z0 = (int64_t)((fx_mul64(rho, fx_swapped(t) ? s : c) ^ m0) - m0);
    z1 = (int64_t)((fx_mul64(rho, fx_swapped(t) ? c : s) ^ m1) - m1);
}

// x 2^-unit rounded to FP64 (half up), x at least 2^32; `any` also takes smaller x and 0.
template <bool any = false> MLMC_FX uint64_t fx_double_bits(uint64_t x, int unit)
{
    uint32_t hi = (uint32_t)(x >> 32), lo = (uint32_t)x;
    int top = 1023 + 62 - unit;
    if (any && hi == 0) {
        hi = lo;
        lo = 0;
        top -= 32;
    }
    const int n = fx_norm(hi);
    const uint32_t vh = fx_shl_hi(lo, hi, n & 31), vl = lo << (n & 31);
    const uint64_t r = fx_join(fx_shr_lo(vl, vh, 11), (vh >> 11) + (uint32_t)(top - n) * 0x100000u) + ((vl >> 10) & 1u);
    return any && hi == 0 ? 0 : r;
}

// The high 64 bits of the signed product a b, within 2 and without a bias: the addend stands for the
// half that the shift drops and the mean quarter of the low words' product, which is left out (a
// bias would add up over a path's steps).  |a| and |b| must not both be near 2^63.
MLMC_FX int64_t fx_mul64s(int64_t a, int64_t b)
{
    const int32_t ah = (int32_t)(a >> 32), bh = (int32_t)(b >> 32);
    const int32_t al = (int32_t)((uint32_t)a >> 1), bl = (int32_t)((uint32_t)b >> 1);
    const int64_t cross = (int64_t)ah * bl + 0x60000000 + (int64_t)bh * al;
    return (int64_t)ah * bh + (cross >> 31);
}

// Running products G_k = (1 + d_0) .. (1 + d_{k-1}) of four increments as D_k = G_k - 1, all in units of
// 2^-(64 - up) (fx_mul64s returns units of 2^-(64 - 2 up)).
MLMC_FX void fx_products(int64_t d0, int64_t d1, int64_t d2, int64_t d3, int up, int64_t &D2, int64_t &D3, int64_t &D4)
{
    D2 = d0 + d1 + (int64_t)((uint64_t)fx_mul64s(d0, d1) << up);
    D3 = D2 + d2 + (int64_t)((uint64_t)fx_mul64s(D2, d2) << up);
    D4 = D3 + d3 + (int64_t)((uint64_t)fx_mul64s(D3, d3) << up);
}

// Relative increments d = r h + sigma dW of one word pair's two fine steps in units of 2^-u:
// A is sigma sqrt(h) in units of 2^-(u + 6), rh is r h in units of 2^-u.
MLMC_FX void fx_increment_pair(uint32_t xa, uint32_t xb, bool u23, const uint64_t *tab, uint64_t A, int64_t rh,
                               int64_t &d0, int64_t &d1)
{
    const uint64_t ra = fx_mul64(fx_radius(fx_word(xa, u23), tab), A);
    const uint32_t t = fx_word(xb, u23);
    uint64_t c, s;
    fx_circle(t, tab, c, s);
    const uint64_t m0 = fx_cos_sign(t), m1 = fx_sin_sign(t);
    d0 = rh + (int64_t)((fx_mul64(ra, fx_swapped(t) ? s : c) ^ m0) - m0);
    d1 = rh + (int64_t)((fx_mul64(ra, fx_swapped(t) ? c : s) ^ m1) - m1);
}
// The Milstein increment r h - c2 + sigma sqrt(h) z + c2 z^2 from z in units of 2^-58; A and C2 in
// units of 2^-(u + 6), rhm in units of 2^-u.  |z| < 2^61 leaves room to square 8 z, so that z^2 keeps units of
// 2^-58 (2^-52 from z itself: rms error 2^-51.4 where an FP64 product has 2^-52.3).  The product with A drops
// as much for z as for -z; what the one with C2 drops is never negative, and the drift carries its mean
// (fx_dropped_mean).
MLMC_FX int64_t fx_increment_milstein(int64_t z, uint64_t A, uint64_t C2, int64_t rhm)
{
    const uint64_t m = (uint64_t)(z >> 63), y = ((uint64_t)z ^ m) - m, y8 = y << 3;
    return rhm + (int64_t)(((fx_mul64(y, A) ^ m) - m) + fx_mul64(fx_mul64(y8, y8), C2));
}

#ifdef __CUDACC__
__device__ __forceinline__ double fx_to_double(uint64_t x, int unit)
{
    return __longlong_as_double((long long)fx_double_bits(x, unit));
}
// The FP64 pipe converts a signed 64-bit integer in one operation, 64 cycles per warp and scheduler
// against 60 of the integer pipes; the steps keep those busy.
__device__ __forceinline__ double fx_to_double_signed(int64_t x, int unit)
{
    const double d = (double)x;
    const int hi = __double2hiint(d);
    return __hiloint2double(hi ? hi - (unit << 20) : 0, __double2loint(d));
}
// The block's copy of the tables (37 KB of shared memory, one instance per kernel), filled by
// fx_load_tables (16 bytes a copy, all of a thread's in flight together), which ends with a block barrier.
__device__ __forceinline__ uint64_t *fx_tables()
{
    __shared__ alignas(16) uint64_t tables[kFxWords];
    return tables;
}
__device__ __forceinline__ void fx_load_tables()
{
    uint64_t *t = fx_tables();
    for (int i = 2 * threadIdx.x; i < kFxWords; i += 2 * blockDim.x)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;"
                     :: "r"((uint32_t)__cvta_generic_to_shared(t + i)), "l"(kFxTables + i) : "memory");
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
}
#endif

}  // namespace mlmcgb
