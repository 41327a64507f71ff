// normal64.cuh -- Box--Muller normals for FP64 paths in 64-bit fixed point.
//
// The normals of one Philox block's word pair (xa, xb) are rho cos(2 pi u2), rho sin(2 pi u2) with
// rho = sqrt(-2 ln u1) and 32-bit (or, on the FP32 path's stream, 23-bit) uniforms.  GB300 runs 2
// FP64 operations per SM per clock against 32 widening 32-bit integer multiplies, 64 integer adds
// and 16 MUFU operations (all measured), so one FP64 instruction costs as much as 16 widening
// multiplies.  CUDA's double-precision log, sqrt and sincospi took 32 of the 36.5 FP64
// instructions of a coupled step.  Here the whole pair is about 60 integer multiplies and no FP64:
//
//   ln u1    u = w 2^-32 with an integer w: w normalised to mu in [1/2, 1), c = k / 512 the
//            multiple of 1/512 nearest 1 / mu (a hardware reciprocal), s = mu c - 1 exactly as a
//            32-bit integer in units of 2^-41 (|s| < 2^-10), and
//            -ln u = n ln 2 + ln c - (s - s^2/2 + s^3/3 - s^4/4 + s^5/5 - ...), table + series
//            (the argument reduction of Tang, "Table-driven implementation of the logarithm
//            function in IEEE floating-point arithmetic", ACM TOMS 16, 1990);
//   sqrt     a 24-bit hardware reciprocal root, then one third-order correction
//            p (1 + r/2 + 3 r^2/8), p = x y, r = 1 - p y (the binomial series of (1 - r)^(-1/2));
//   cos, sin quadrant, 512 angles per quadrant by table, the remaining angle delta < pi/1024 by
//            its Taylor series and the addition theorems.
//
// Absolute error of a normal: below 2^-56 (checked against quadruple precision over the edges of
// every reduction and 10^8 random words), a quarter of the rounding of an FP64 normal of size 1.
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
MLMC_FX int fx_clz(uint32_t a) { return __clz((int)a); }
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
MLMC_FX float fx_float(uint32_t x) { return __uint2float_rn(x); }
// The high word of (hi, lo) << k and the low word of (hi, lo) >> k, k < 32.
MLMC_FX uint32_t fx_shl_hi(uint32_t lo, uint32_t hi, int k) { return __funnelshift_l(lo, hi, k); }
MLMC_FX uint32_t fx_shr_lo(uint32_t lo, uint32_t hi, int k) { return __funnelshift_r(lo, hi, k); }
#else
#define MLMC_FX inline
MLMC_FX uint32_t fx_mulhi(uint32_t a, uint32_t b) { return (uint32_t)(((uint64_t)a * b) >> 32); }
MLMC_FX int fx_clz(uint32_t a) { return a ? __builtin_clz(a) : 32; }
MLMC_FX float fx_rcp(float x) { return 1.0f / x; }
MLMC_FX float fx_rsqrt(float x) { return (float)(1.0 / std::sqrt((double)x)); }
MLMC_FX uint32_t fx_bits(float x)
{
    uint32_t u;
    std::memcpy(&u, &x, sizeof(u));
    return u;
}
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

// sqrt(-2 ln(w 2^-32)) in units of 2^-60, w = y + 1 (w = 0 stands for 2^32: the result is 0).
MLMC_FX uint64_t fx_radius(uint32_t y, const uint64_t *tab)
{
    const uint32_t w = y + 1u;
    const int n = fx_clz(w);
    const uint32_t m = w << (n & 31);
    // k = 512 c, by a magic-number rounding of 2^41 / m
    const uint32_t k = fx_bits(fmaf(fx_rcp(fx_float(m)), 0x1p41f, 12582912.0f)) - 0x4B400000u;
    const int32_t s = (int32_t)(m * k);  // m k - 2^41: the multiple of 2^32 drops out
    const uint64_t A = tab[kFxLn2 + (n & 31)] + tab[kFxLnC + ((k - 512u) & 1023u)];  // units of 2^-59
    // B = -(s - s^2/2 + s^3/3 - s^4/4 + s^5/5) in units of 2^-71
    const uint64_t q = (uint64_t)((int64_t)s * s);              // 2^-82, below 2^62
    const uint32_t s2 = (uint32_t)(q >> 30);                    // 2^-52
    const uint32_t br = 0x55555555u - (uint32_t)(s >> 11) + fx_mulhi(s2, 819u);  // (1/3 - s/4 + s^2/5) 2^32
    const int64_t tail = (int64_t)s * (int32_t)fx_mulhi(s2, br);  // 2^-93
    const int64_t B = (int64_t)(q >> 12) - ((int64_t)s << 30) - (tail >> 22);
    // close to u = 1 (n = 0, c = 1) the table part is 0 and B alone keeps its extra bits
    const bool near1 = A == 0;
    const uint64_t F = near1 ? (uint64_t)B : A + (uint64_t)(B >> 12);
    // sqrt(2 F): F normalised to x 2^64 by an even shift, x in [1/4, 1)
    const int e = fx_clz((uint32_t)(F >> 32)) & 30;
    const uint32_t xh = fx_shl_hi((uint32_t)F, (uint32_t)(F >> 32), e), xl = (uint32_t)F << e;
    const uint32_t yr = fx_bits(fminf(fx_rsqrt(fx_float(xh)), 0x1.fffffep-16f));
    // 1 / sqrt(x) in units of 2^-31, lowered by two units of its last place (2^-22, above the
    // reciprocal root's error of 2^-22.9) so that p = x y stays below 1
    const uint32_t yi = (yr << 8) - 0x200u;
    const uint64_t p = fx_mul64x32(fx_join(xl, xh), yi);        // x y: 2^-63
    const int64_t r = (int64_t)((uint64_t(1) << 62) - fx_mul64x32(p, yi));  // 1 - p y: 2^-62, |r| < 2^42
    const int32_t rh = (int32_t)(r >> 11);
    const uint32_t rr = (uint32_t)(((int64_t)rh * rh) >> 32);   // r^2: 2^-70
    const uint64_t E = (uint64_t)(r + (int64_t)((3u * (rr >> 2)) >> 8)) << 21;  // r + 3 r^2 / 4: 2^-83
    const int32_t Eh = (int32_t)(E >> 32), ph = (int32_t)(p >> 32), pl = (int32_t)((uint32_t)p >> 1);
    const int64_t corr = (int64_t)ph * Eh + (((int64_t)pl * Eh) >> 31) + (int64_t)fx_mulhi((uint32_t)ph, (uint32_t)E);
    const uint64_t root = p + (uint64_t)(corr >> 20);           // 2^-63
    const int sh = (e >> 1) + (near1 ? 6 : 0);
    const uint64_t rho = fx_join(fx_shr_lo((uint32_t)root, (uint32_t)(root >> 32), sh), (uint32_t)(root >> 32) >> sh);
    return w ? rho : 0;
}

// |cos| and |sin| of 2 pi (y + 1) 2^-32 reduced to the first quadrant, in units of 2^-62, and the
// quadrant q: (cos, sin) = (c, s), (-s, c), (-c, -s), (s, -c) for q = 0..3.
MLMC_FX uint32_t fx_circle(uint32_t y, const uint64_t *tab, uint64_t &c, uint64_t &s)
{
    const uint32_t t = y + 1u;
    const uint32_t i = (t >> 21) & 511u;
    const uint64_t C = tab[kFxCos + i], S = tab[kFxCos + 512 - i];
    const uint32_t dt = t << 11;                                // delta = 2 pi dt 2^-43 < pi / 1024
    const uint64_t D = fx_mul64x32(kFxTwoPi60, dt);             // delta: 2^-71
    const uint64_t U = fx_mul64(fx_wide(dt, dt), kFxTwoPiSq59); // delta^2 / 2: 2^-81
    const uint32_t Uh = (uint32_t)(U >> 32);                    // 2^-49
    const uint32_t U2 = fx_mulhi(Uh, Uh);                       // delta^4 / 4: 2^-66
    // u = 1 - cos delta = U - U^2 / 6, v = sin delta = delta - delta (U / 3 - U^2 / 30): 2^-71
    const uint64_t u = (U >> 10) - ((uint64_t)fx_mulhi(U2, 0x2AAAAAABu) << 5);
    const uint32_t g = fx_mulhi(Uh, 0xAAAAAAABu) - fx_mulhi(U2, 2185u);  // 2^-50
    const uint64_t v = D - (fx_wide((uint32_t)(D >> 32), g) >> 18);
    const uint32_t Ch = (uint32_t)(C >> 32), Cl = (uint32_t)C, Sh = (uint32_t)(S >> 32), Sl = (uint32_t)S;
    const uint32_t uh = (uint32_t)(u >> 32), ul = (uint32_t)u, vh = (uint32_t)(v >> 32), vl = (uint32_t)v;
    // cos = C - (C u + S v), sin = S + (C v - S u); products in units of 2^-69.  The sum of the cross
    // products stays below 2^64: 2^30 2^32 twice, 2^32 2^30.7 and 2^32 2^21.4
    const uint64_t xc = fx_wide(Ch, ul) + fx_wide(Sh, vl) + fx_wide(Sl, vh) + fx_wide(Cl, uh);
    const uint64_t pc = fx_wide(Ch, uh) + fx_wide(Sh, vh) + (xc >> 32);
    c = C - (pc >> 7);
    const uint64_t xp = fx_wide(Ch, vl) + fx_wide(Cl, vh);
    const uint64_t xm = fx_wide(Sh, ul) + fx_wide(Sl, uh);
    const int64_t ps = (int64_t)((fx_wide(Ch, vh) + (xp >> 32)) - (fx_wide(Sh, uh) + (xm >> 32)));
    s = S + (uint64_t)(ps >> 7);
    return t >> 30;
}

// The FP64 stream takes the 32 bits of a word; the FP32 path's stream u = 1 - (x mod 2^23) 2^-23,
// the same fixed-point uniform (y + 1) 2^-32 with y = ~(x << 9).
MLMC_FX uint32_t fx_word(uint32_t x, bool u23) { return u23 ? ~(x << 9) : x; }

// The two normals of a word pair, in units of 2^-58.
constexpr double kFxZ = 0x1p-58;
MLMC_FX void fx_pair(uint32_t xa, uint32_t xb, bool u23, const uint64_t *tab, int64_t &z0, int64_t &z1)
{
    const uint64_t rho = fx_radius(fx_word(xa, u23), tab);
    uint64_t c, s;
    const uint32_t q = fx_circle(fx_word(xb, u23), tab, c, s);
    const bool swap = q & 1;
    const uint64_t m0 = (q == 1 || q == 2) ? ~uint64_t(0) : 0, m1 = q >= 2 ? ~uint64_t(0) : 0;
    z0 = (int64_t)((fx_mul64(rho, swap ? s : c) ^ m0) - m0);
    z1 = (int64_t)((fx_mul64(rho, swap ? c : s) ^ m1) - m1);
}

// x 2^-unit rounded to FP64 (half up), x at least 2^32; `any` also takes smaller x and 0.
template <bool any = false> MLMC_FX uint64_t fx_double_bits(uint64_t x, int unit)
{
    uint32_t hi = (uint32_t)(x >> 32), lo = (uint32_t)x;
    int n = fx_clz(hi);
    if (any && hi == 0) {
        hi = lo;
        lo = 0;
        n = 32 + fx_clz(hi);
    }
    const uint32_t vh = fx_shl_hi(lo, hi, n & 31), vl = lo << (n & 31);
    const uint64_t r = fx_join(fx_shr_lo(vl, vh, 11), (vh >> 11) + (uint32_t)(1023 + 62 - unit - n) * 0x100000u) +
                       ((vl >> 10) & 1u);
    return any && x == 0 ? 0 : r;
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

// Relative increments d = r h + sigma dW of one word pair's two fine steps in units of 2^-u:
// A is sigma sqrt(h) in units of 2^-(u + 6), rh is r h in units of 2^-u.
MLMC_FX void fx_increment_pair(uint32_t xa, uint32_t xb, bool u23, const uint64_t *tab, uint64_t A, int64_t rh,
                               int64_t &d0, int64_t &d1)
{
    const uint64_t ra = fx_mul64(fx_radius(fx_word(xa, u23), tab), A);
    uint64_t c, s;
    const uint32_t q = fx_circle(fx_word(xb, u23), tab, c, s);
    const bool swap = q & 1;
    const uint64_t m0 = (q == 1 || q == 2) ? ~uint64_t(0) : 0, m1 = q >= 2 ? ~uint64_t(0) : 0;
    d0 = rh + (int64_t)((fx_mul64(ra, swap ? s : c) ^ m0) - m0);
    d1 = rh + (int64_t)((fx_mul64(ra, swap ? c : s) ^ m1) - m1);
}
// The Milstein increment r h - c2 + sigma sqrt(h) z + c2 z^2 from z in units of 2^-58; A and C2 in
// units of 2^-(u + 6), rhm in units of 2^-u.
MLMC_FX int64_t fx_increment_milstein(int64_t z, uint64_t A, uint64_t C2, int64_t rhm)
{
    const uint64_t m = (uint64_t)(z >> 63), y = ((uint64_t)z ^ m) - m;
    return rhm + (int64_t)(((fx_mul64(y, A) ^ m) - m) + fx_mul64(fx_mul64(y, y) << 6, C2));
}

#ifdef __CUDACC__
__device__ __forceinline__ double fx_to_double(uint64_t x, int unit)
{
    return __longlong_as_double((long long)fx_double_bits(x, unit));
}
__device__ __forceinline__ double fx_to_double_signed(int64_t x, int unit)
{
    const uint64_t m = (uint64_t)(x >> 63);
    return __longlong_as_double((long long)(fx_double_bits<true>(((uint64_t)x ^ m) - m, unit) | (m << 63)));
}
// The block's copy of the tables (8.5 KB of shared memory, one instance per kernel), filled by
// fx_load_tables, which ends with a block barrier.
__device__ __forceinline__ uint64_t *fx_tables()
{
    __shared__ uint64_t tables[kFxWords];
    return tables;
}
__device__ __forceinline__ void fx_load_tables()
{
    uint64_t *t = fx_tables();
    for (int i = threadIdx.x; i < kFxWords; i += blockDim.x) t[i] = kFxTables[i];
    __syncthreads();
}
#endif

}  // namespace mlmcgb
