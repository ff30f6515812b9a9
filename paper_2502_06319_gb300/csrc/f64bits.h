// f64bits.h -- conversions between FP32 and FP64 and comparisons of FP64 values done on
// their bits, in 32-bit integer instructions.
//
// Why: GB300's FP64 pipe takes 64 clocks per warp instruction and scheduler, and not only
// for arithmetic: every conversion to or from FP64, every FP64 comparison and every FP64
// minimum goes through it.  An FP64-accumulated step (model32.cuh with FP64 sums) had about
// 28 such slots, five of which are the sums themselves; as integer instructions (1-2 clocks
// each) the other 23 cost about 90 issue slots and leave the FP64 pipe to the sums
// (measured beside Acc<COSMICA_PREC_MIXED_F64ACC> in mixed_state.cuh).
//
// Each function gives the bits that the conversion instruction gives (round to nearest
// even, FP32 subnormals flushed to zero) on the values it names; none of them branches, so
// that the step they are part of stays one block.
#pragma once
#include <cstdint>

#if defined(__CUDACC__)
#define COSMICA_HD __host__ __device__ __forceinline__
#else
#define COSMICA_HD inline
#endif

namespace cosmica {
namespace f64bits {

constexpr uint64_t kPiBits = 0x400921FB54442D18ull;      // the double nearest pi
constexpr uint64_t kHalfPiBits = 0x3FF921FB54442D18ull;
constexpr uint64_t kTwoPiBits = 0x401921FB54442D18ull;

// FP32 -> FP64, exact, for every value (a subnormal one gives zero).
COSMICA_HD uint64_t widen(uint32_t u)
{
    // exponent bias 127 -> 1023: add 896 to the exponent field (bit 20 of the high word), or what
    // turns 255 into 2047; a zero stays one
    const uint32_t t = u & 0x7FFFFFFFu;
    const uint32_t bias = t >= 0x7F800000u ? 0x70000000u : 0x38000000u;
    const bool none = t < 0x00800000u;
    const uint32_t hi = (u & 0x80000000u) | (none ? 0u : (t >> 3) + bias);
    return ((uint64_t)hi << 32) | (none ? 0u : u << 29);
}

// FP64 -> FP32, round to nearest even, for |x| < 2^128 (below 2^-126: zero); infinite or a NaN from there to
// 2^129.  Above, and for an infinity or a NaN, a finite number: the caller sees to it that none comes here.
COSMICA_HD uint32_t narrow(uint64_t x)
{
    const uint32_t hi = (uint32_t)(x >> 32), lo = (uint32_t)x;
    const uint32_t m = hi & 0x7FFFFFFFu;
    const uint32_t t = ((m - 0x38000000u) << 3) | (lo >> 29);            // truncated result without its sign
    // the 29 bits below it as a fraction of 2^32: adding 2^31 - 1 + lsb carries exactly when
    // the fraction is above one half, or equal to it with an odd t
    const uint64_t r = (((uint64_t)t << 32) | (uint32_t)(lo << 3)) + (0x7FFFFFFFu + (t & 1u));
    return (m < 0x38100000u ? 0u : (uint32_t)(r >> 32)) | (hi & 0x80000000u);
}

// pi - th as FP32 (the FP64 difference rounded to nearest even), th in [pi/2, pi]: both lie
// within a factor of two, so the FP64 difference is exact (Sterbenz) and is formed as an
// integer multiple of 2^-52.
COSMICA_HD uint64_t pi_minus_units(uint64_t th)
{
    const uint64_t m = (th & 0x000FFFFFFFFFFFFFull) | 0x0010000000000000ull;
    return 0x003243F6A8885A30ull - (m << ((uint32_t)(th >> 52) & 1u ? 0 : 1));
}
COSMICA_HD float pi_minus(uint64_t diff)
{
#if defined(__CUDA_ARCH__)
    const int sh = __clzll((long long)(diff | 1u));
#else
    const int sh = __builtin_clzll(diff | 1u);
#endif
    const uint64_t n = diff << sh;
    // 32 leading bits, the rest folded into a sticky bit below the rounding position
    const uint32_t w = (uint32_t)(n >> 32) | ((uint32_t)n != 0u ? 1u : 0u);
#if defined(__CUDA_ARCH__)
    return __fmul_rn(__uint2float_rn(w), __uint_as_float((uint32_t)(107 - sh) << 23));
#else
    const uint32_t sb = (uint32_t)(107 - sh) << 23;      // 2^(-20 - sh)
    float scale;
    __builtin_memcpy(&scale, &sb, 4);
    return (float)w * scale;
#endif
}

// the double of a 32-bit count, exact
COSMICA_HD uint64_t from_u32(uint32_t n)
{
    if (n == 0u) return 0ull;
#if defined(__CUDA_ARCH__)
    const int sh = __clz(n);
#else
    const int sh = __builtin_clz(n);
#endif
    return ((uint64_t)(1053 - sh) << 52) + ((uint64_t)(n << sh) << 21);   // the leading one carries into the exponent
}

// Bounds for an FP32 sum n = fr + dr, r an FP64 number with the FP32 value fr, 0 <= r <= reach: above the floor
// and below the ceiling, r + dr is at least r_in and below R.  n is off by up to 2^-24 r and 2^-24 of itself; the
// first counts where a step from far out ends beside r_in, hence the share of reach.
COSMICA_HD float vote_floor(float r_in, float reach) { return r_in * 1.000001f + reach * 2.4e-7f; }
COSMICA_HD float vote_ceiling(float R) { return R * 0.999999f; }
constexpr float kMostRise = 1e30f;       // of r in a step where another test bounds r: keeps an infinity out

// FP64 comparisons on the bits, with b > 0 finite: right for every a but NaN.
COSMICA_HD bool less(uint64_t a, uint64_t b) { return (int64_t)a < (int64_t)b; }
// a < 0 or a > b (a = -0 counts as below 0: the caller decides with FP64 comparisons then)
COSMICA_HD bool outside_closed(uint64_t a, uint64_t b) { return a > b; }
// a < 0 or a >= b (likewise)
COSMICA_HD bool outside_half_open(uint64_t a, uint64_t b) { return a >= b; }
COSMICA_HD bool is_finite(uint64_t a) { return ((uint32_t)(a >> 32) & 0x7FFFFFFFu) < 0x7FF00000u; }

}  // namespace f64bits
}  // namespace cosmica
