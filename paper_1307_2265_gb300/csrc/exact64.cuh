// Correctly rounded FP64 division, square root and comparisons on the integer
// pipe.
//
// What bounds the FP64 path is the FP64 pipe: it retires 2 thread operations
// per clock and SM, the integer pipe 64, and issue slots stood 92% empty while
// it was full.  A division or square root costs the FP64 pipe eight to ten
// operations, and a cell-sweep has about 60 of them, so they are done
// here by digit recurrence on the 53-bit significands: an FP32 reciprocal (or
// reciprocal square root) gives about 20 quotient bits per step, each step's
// remainder is kept exactly in 64 bits, and the last remainder decides the
// rounding.  The results are those of IEEE division and square root, round to
// nearest even, bit for bit; operands outside the normal range (zeros aside)
// take the hardware operation.
//
// The functions compile for the host too (a CPU test compares them with the
// host's division and square root, edge cases and deliberately poor seeds
// included).
//
// Measured with the branches of the tracing and of the Riemann sampling merged
// at the same time (ppm_device.cuh): FP64 pipe slots per cell-sweep 1785 ->
// 695, 2^20 Riemann problems 2044 -> 638 us, a step of a walled 100x75x50 grid
// 25.1 -> 10.0 ms, of a 400-patch level (2e7 cells) 200 -> 142 ms, every result
// the same.
#pragma once
#include <cstdint>
#include <cmath>
#include <cstring>

#ifdef __CUDACC__
#define ENZO_HD __host__ __device__ __forceinline__
#else
#define ENZO_HD inline
#endif

namespace enzo {
namespace x64 {

ENZO_HD uint64_t bits(double x)
{
#ifdef __CUDA_ARCH__
    return (uint64_t)__double_as_longlong(x);
#else
    uint64_t u;
    memcpy(&u, &x, 8);
    return u;
#endif
}
ENZO_HD double from_bits(uint64_t u)
{
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)u);
#else
    double x;
    memcpy(&x, &u, 8);
    return x;
#endif
}
ENZO_HD uint32_t hi32(double x) { return (uint32_t)(bits(x) >> 32); }
ENZO_HD uint32_t mulhi(uint32_t a, uint32_t b)
{
#ifdef __CUDA_ARCH__
    return __umulhi(a, b);
#else
    return (uint32_t)(((uint64_t)a * b) >> 32);
#endif
}

// FP32 seeds.  x in [1, 4) as float bits; the relative error of the hardware
// approximations is below 2^-22.5.  The host's are perturbed by seed_noise()
// in the test.
#ifndef __CUDA_ARCH__
inline float &seed_noise()
{
    static thread_local float e = 0.0f;
    return e;
}
#endif
ENZO_HD float rcp_seed(uint32_t b)
{
#ifdef __CUDA_ARCH__
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(__uint_as_float(b)));
    return y;
#else
    float x;
    memcpy(&x, &b, 4);
    return (1.0f / x) * (1.0f + seed_noise());
#endif
}
ENZO_HD float rsqrt_seed(uint32_t b)
{
#ifdef __CUDA_ARCH__
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(__uint_as_float(b)));
    return y;
#else
    float x;
    memcpy(&x, &b, 4);
    return (float)(1.0 / std::sqrt((double)x)) * (1.0f + seed_noise());
#endif
}
// 2^32 y (1 - 2^-21) of a seed y in [1/2, 1]: the sum 1 + y (1 - 2^-21), in
// [1, 2), keeps 23 fraction bits, which the shift leaves.
ENZO_HD uint32_t fix32(float y)
{
#ifdef __CUDA_ARCH__
    return __float_as_uint(__fmaf_rn(y, 1.0f - 4.76837158e-7f, 1.0f)) << 9;
#else
    const float w = std::fmaf(y, 1.0f - 4.76837158e-7f, 1.0f);
    uint32_t b;
    memcpy(&b, &w, 4);
    return b << 9;
#endif
}

// Reciprocal of a normal divisor's significand b = B / 2^52 in [1, 2): Y =
// 2^32 / b from below, 1 - 2^-20.4 < Y b / 2^32 < 1 (the factor 1 - 2^-21
// outweighs the seed's error, the truncation of b to 24 bits and the rounding
// of the sum).  A divisor used several times keeps it.
struct Recip {
    uint64_t B;        // significand with the hidden bit
    uint32_t Y;
    uint32_t hi;       // sign and exponent of the divisor
};

ENZO_HD Recip recip(double b)
{
    Recip r;
    const uint64_t u = bits(b);
    r.hi = (uint32_t)(u >> 32);
    r.B = (u & 0xfffffffffffffull) | 0x10000000000000ull;
    const uint32_t f = 0x3f800000u | ((uint32_t)(u >> 29) & 0x7fffffu);
    r.Y = fix32(rcp_seed(f));
    return r;
}

#ifdef __CUDACC__
__device__ __noinline__ static double div_hw(double a, double b) { return a / b; }
__device__ __noinline__ static double sqrt_hw(double a) { return sqrt(a); }
#endif
ENZO_HD double div_any(double a, double b)
{
#ifdef __CUDA_ARCH__
    return div_hw(a, b);
#else
    return a / b;
#endif
}
ENZO_HD double sqrt_any(double a)
{
#ifdef __CUDA_ARCH__
    return sqrt_hw(a);
#else
    return std::sqrt(a);
#endif
}

// (a 2^k) / b, with r = recip(b); k = -1, 0 or 1, a 2^k exact.
//   a/b in [1, 2) after the shift; q1 = its first 31 bits from below, off by
//   less than 2^10.7, so r1 = A 2^30 - q1 B < 2^63.7 is exact modulo 2^64;
//   q2 adds 20 bits (r2 = r1 2^20 - q2 B < 2^63); t the last three, exact or
//   one short, which r3 >= B tells.  Q = floor(2^53 a/b) has one bit more than
//   the result and a quotient is never a tie, so (Q + 1) >> 1 rounds it.
template <int k = 0>
ENZO_HD double div(double a, double b, const Recip &r)
{
    const uint64_t u = bits(a);
    const uint32_t ah = (uint32_t)(u >> 32);
    uint64_t A = (u & 0xfffffffffffffull) | 0x10000000000000ull;
    const int ea = (int)((ah >> 20) & 0x7ffu), eb = (int)((r.hi >> 20) & 0x7ffu);
    const bool zero = (u << 1) == 0;
    int e = ea - eb + 1022 + k;                 // biased exponent less one (the hidden bit adds it)
    const bool less = A < r.B;
    A = less ? A << 1 : A;
    e -= less ? 1 : 0;
    const bool ok = (unsigned)(eb - 1) < 2046u && (zero || ((unsigned)(ea - 1) < 2046u && (unsigned)(e - 1) < 2044u));
    if (!ok) return div_any(k == 0 ? a : (k > 0 ? a + a : 0.5 * a), b);
    const uint32_t q1 = mulhi((uint32_t)(A >> 22), r.Y);
    const uint64_t r1 = (A << 30) - q1 * r.B;
    const uint32_t q2 = mulhi((uint32_t)(r1 >> 32), r.Y);
    const uint64_t r2 = (r1 << 20) - q2 * r.B;
    const uint32_t t = mulhi((uint32_t)(r2 >> 32), r.Y) >> 17;
    const uint64_t r3 = (r2 << 3) - t * r.B;
    const uint64_t Q = ((uint64_t)q1 << 23) + ((uint64_t)q2 << 3) + t + (r3 >= r.B ? 1u : 0u);
    uint64_t v = ((uint64_t)(uint32_t)e << 52) + ((Q + 1) >> 1);
    v = zero ? 0 : v;
    return from_bits(v | ((uint64_t)((ah ^ r.hi) & 0x80000000u) << 32));
}

ENZO_HD double div(double a, double b) { return div<0>(a, b, recip(b)); }

// sqrt(x).  m = x with an even exponent taken out, in [1, 4); R = 2^32/sqrt(m)
// from below.  g1 = sqrt(m) 2^30 from below, off by less than 2^10.7; rem1 =
// m 2^60 - g1^2.  d2 = rem1 R (g1 + d2/2^20 stays below: the linear step
// overshoots by half of R's own shortfall); rem2 = m 2^100 - g2^2 < 2^64; t
// the last three bits, exact or one short.  No square root is a tie.
ENZO_HD double sqrt_rn(double x)
{
    const uint64_t u = bits(x);
    const uint32_t h = (uint32_t)(u >> 32);
    const unsigned ex = h >> 20;                        // sign included: negative falls out
    if (ex - 1u >= 2046u) return (u << 1) == 0 ? x : sqrt_any(x);
    const unsigned odd = (ex + 1u) & 1u;                // exponent ex - 1023 odd
    const uint64_t M = (u & 0xfffffffffffffull) | 0x10000000000000ull;
    const uint64_t X = M << (10 + odd);                 // m 2^62
    const uint32_t f = (0x3f800000u + (odd << 23)) | ((uint32_t)(u >> 29) & 0x7fffffu);
    const uint32_t R = fix32(rsqrt_seed(f));
    const uint32_t g1 = mulhi((uint32_t)(X >> 32), R);
    const uint64_t rem1 = (X >> 2) - (uint64_t)g1 * g1;
    const uint32_t d2 = mulhi((uint32_t)(rem1 >> 11), R);
    const uint64_t g2 = ((uint64_t)g1 << 20) + d2;
    const uint64_t rem2 = (rem1 << 40) - (((uint64_t)g1 * d2) << 21) - (uint64_t)d2 * d2;
    const uint32_t t = mulhi((uint32_t)(rem2 >> 32), R) >> 16;
    const uint64_t S0 = (g2 << 3) + t;
    // rem3 = m 2^106 - S0^2 < 2^57, so 32-bit slices of it suffice modulo 2^64
    const uint64_t rem3 = (rem2 << 6) - ((g2 * t) << 4) - (uint64_t)t * t;
    const uint64_t S = S0 + (rem3 > 2 * S0 ? 1u : 0u);
    const uint64_t e = (uint64_t)((ex + 1023u - odd) >> 1) - 1u;
    return from_bits((e << 52) + ((S + 1) >> 1));
}

// x / 6: the significand's exact third.  M 2^3 / 3 (M 2^2 / 3 from 1.5 up)
// has 54 bits, one more than the result, and is never a tie (an odd third
// would make M 2^2 odd).
ENZO_HD double div6(double x)
{
    const uint64_t u = bits(x);
    const uint32_t h = (uint32_t)(u >> 32);
    const unsigned ex = (h >> 20) & 0x7ffu;
    if (ex - 8u >= 2038u) return (u << 1) == 0 ? x : x / 6.0;
    const bool big = (h & 0xfffffu) >= 0x80000u;        // significand of 1.5 or more
    const uint64_t N = ((u & 0xfffffffffffffull) | 0x10000000000000ull) << (big ? 2 : 3);
    const uint32_t nh = (uint32_t)(N >> 32), nl = (uint32_t)N;
    const uint32_t qh = mulhi(nh, 0xAAAAAAABu) >> 1, rh = nh - 3u * qh;
    const uint32_t ql = mulhi(nl, 0xAAAAAAABu) >> 1, rl = nl - 3u * ql;
    const uint64_t Q = ((uint64_t)qh << 32) + (uint64_t)(rh * 0x55555555u) + ql + (rh + rl >= 3u ? 1u : 0u);
    const uint64_t e = (uint64_t)(ex - (big ? 2u : 3u)) - 1u;
    return from_bits(((e << 52) + ((Q + 1) >> 1)) | ((uint64_t)(h & 0x80000000u) << 32));
}

// ---- comparisons (a DSETP costs the FP64 pipe one operation) ---------------

// x >= f, x > f for f > 0 (false for NaN).
ENZO_HD bool ge_pos(double x, double f) { return bits(x) - bits(f) <= 0x7ff0000000000000ull - bits(f); }
ENZO_HD bool gt_pos(double x, double f) { return bits(x) - bits(f) - 1u < 0x7ff0000000000000ull - bits(f); }
// x < f for f > 0 (false for NaN).
ENZO_HD bool lt_pos(double x, double f)
{
    const uint64_t u = bits(x);
    return u < bits(f) || (u >= 0x8000000000000000ull && u <= 0xfff0000000000000ull);
}
// x > 0, x >= 0, x <= 0 (false for NaN).
ENZO_HD bool gt0(double x) { return bits(x) - 1u < 0x7ff0000000000000ull; }
ENZO_HD bool ge0(double x) { return bits(x) <= 0x7ff0000000000000ull || bits(x) == 0x8000000000000000ull; }
ENZO_HD bool lt0(double x) { return bits(x) - 0x8000000000000001ull < 0x7ff0000000000000ull; }
ENZO_HD bool le0(double x) { return bits(x) - 0x8000000000000000ull <= 0x7ff0000000000000ull || bits(x) == 0; }
ENZO_HD bool is_nan(double x) { return (bits(x) << 1) > 0xffe0000000000000ull; }
// a < b.  Magnitudes order as integers, negative ones the other way round.
ENZO_HD bool less(double a, double b)
{
    const int64_t u = (int64_t)bits(a), v = (int64_t)bits(b);
    const int64_t ku = u ^ (int64_t)((uint64_t)(u >> 63) >> 1), kv = v ^ (int64_t)((uint64_t)(v >> 63) >> 1);
    return ku < kv && !is_nan(a) && !is_nan(b) && ((uint64_t)(u | v) << 1) != 0;
}
ENZO_HD bool finite(double x) { return (hi32(x) & 0x7ff00000u) != 0x7ff00000u; }
ENZO_HD double neg_if(bool c, double x) { return from_bits(bits(x) ^ (c ? 0x8000000000000000ull : 0ull)); }
ENZO_HD uint64_t mag(double x) { return bits(x) & 0x7fffffffffffffffull; }
// Magnitude in [2^-511, 2^512): products and quotients of two such numbers are
// normal, and scaling by 4 is an exponent step.
ENZO_HD bool middle(double x) { return ((hi32(x) >> 20) & 0x7ffu) - 512u < 1023u; }

}  // namespace x64
}  // namespace enzo
