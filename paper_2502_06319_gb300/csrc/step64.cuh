// step64.cuh -- the FP64 step arranged for GB300's FP64 pipe: bit for bit the values of
// m64::em_step (model64.cuh), in about half of its FP64 instructions.
//
// What bounds it: the FP64 pipe takes 64 clocks per warp instruction and scheduler, whether
// one lane is active or 32 and whether the instruction depends on the last one or not, so a
// step costs its number of FP64 instructions ("slots") times 64 clocks and everything else
// hides behind it.  m64::em_step takes about 1560 slots (full model).  Here:
//   * a division is a reciprocal (an approximate one, then y0 + y0 (e + e^2) with
//     e = 1 - b y0: 3 slots) and 3 slots a quotient, q = RN(a y), q + y (a - b q) -- the
//     correction step of P. Markstein, "Computation of elementary functions on the IBM RISC
//     System/6000 processor", IBM J. Res. Dev. 34 (1990): the correctly rounded quotient
//     when y is the rounded reciprocal.  (y misses that for about one b in 60, by under 2^-7
//     ulp.  The quotient is then one unit off only if it is the nearest to a midpoint that a
//     quotient by this b can be, and b within 2^-8 of the power of two above it: 5 of 480000 such
//     pairs are, none of the others that were tried, about one division in 10^20.)  Quotients with
//     one denominator share the reciprocal; those of the parameter set are stored with it.  A
//     division instruction sequence is 8.7 slots.
//   * terms that are zero by construction (K_rth, K_thph, the shock's without a shock) and
//     values of the parameter set alone are not evaluated;
//   * scalings by powers of two, comparisons, floor, integer conversions, absolute values and
//     the uniforms of the normals are integer operations;
//   * sqrt and the elementary functions keep their operations (detmath64.cuh).
// Whatever leaves the normal range (a pole hit exactly, an overflow) shows as a non-finite
// state, and the step is then taken again by m64::em_step from the old state; so is a step whose
// ln P or angles are outside the range of what is below (odd_range).  The constants' range is the
// caller's to test (fast_step_set): comparisons and switches on the bits would let a NaN that a
// division leaves there pass for a number.
//
// G lanes step one path together (G = 1: a lane a path).  The slot cost does not depend on
// the active lanes, so a launch with fewer paths than lanes spreads each path's independent
// operations over G lanes -- polynomials, groups of up to four quotients, reciprocals or
// square roots, and the normals of G consecutive steps -- and exchanges results by shuffles
// (a few clocks): about 480 slots a step for G = 4.  Every lane of a team
// holds the whole state, and all 32 lanes of the warp execute every shuffle.
//
// Include only from translation units built with -fmad=false.
#pragma once
#include "common.cuh"
#include "detmath64.cuh"
#include "f64bits.h"
#include "model64.cuh"

namespace cosmica {
namespace s64 {

// ---- bits ------------------------------------------------------------------------
__device__ __forceinline__ uint64_t bits(double x) { return (uint64_t)__double_as_longlong(x); }
__device__ __forceinline__ double from_bits(uint64_t b) { return __longlong_as_double((long long)b); }
__device__ __forceinline__ bool lt(double a, double b) { return (int64_t)bits(a) < (int64_t)bits(b); }   // b >= 0, no NaN
// |x| >= b, or a NaN, for a b whose low word is zero
__device__ __forceinline__ bool beyond(double x, double b) { return ((uint32_t)__double2hiint(x) & 0x7FFFFFFFu) >= (uint32_t)__double2hiint(b); }
// x > 0 for any x but a NaN, whose answer is no; a switch held as 0.0 or 1.0
__device__ __forceinline__ bool positive(double x) { return (int64_t)bits(x) > 0 && (int64_t)bits(x) <= 0x7FF0000000000000ll; }
__device__ __forceinline__ bool on(double x) { return __double2hiint(x) != 0; }
// x 2^E for normal results; zeros stay zeros
template <int E>
__device__ __forceinline__ double scale2(double x)
{
    const int hi = __double2hiint(x);
    return __hiloint2double((hi & 0x7FF00000) ? hi + E * 0x100000 : hi, __double2loint(x));
}
__device__ __forceinline__ double neg_if(double x, bool n) { return __hiloint2double(__double2hiint(x) ^ (n ? (int)0x80000000u : 0), __double2loint(x)); }
// floor of |s| < 2^20
__device__ __forceinline__ int ifloor(double s)
{
    const int hi = __double2hiint(s);
    const int e = ((hi >> 20) & 0x7FF) - 1023;
    const uint32_t m = ((uint32_t)hi & 0xFFFFFu) | 0x100000u;
    const int k = e < 0 ? 0 : (int)(m >> ((20 - e) & 31));
    const bool frac = e < 0 ? (((uint32_t)hi & 0x7FFFFFFFu) | (uint32_t)__double2loint(s)) != 0u
                            : ((m & ~(0xFFFFFFFFu << ((20 - e) & 31))) | (uint32_t)__double2loint(s)) != 0u;
    return hi < 0 ? -k - (int)frac : k;
}
__device__ __forceinline__ double from_int(int k)
{
    const uint32_t a = (uint32_t)(k < 0 ? -k : k);
    return from_bits(f64bits::from_u32(a) | ((uint64_t)(k < 0) << 63));
}
// (w + 1/2) 2^-32: the odd integer 2w + 1 times 2^-33
__device__ __forceinline__ double uniform(uint32_t w)
{
    const int lz = __clz((int)w);
    return from_bits(((uint64_t)(1021 - lz) << 52) + (((uint64_t)w * 2u + 1u) << (20 + lz)));
}

// ---- divisions ---------------------------------------------------------------------
// b between 2^-1000 and 2^1000, a zero or above 2^-960 in magnitude and the quotient a normal number (or a zero):
// then nothing underflows.  b = 0 gives a NaN or an infinity.  Every denominator of the step is positive.
__device__ __forceinline__ double recip(double b)
{
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(b));
    const double e = __fma_rn(-b, y, 1.0);
    return __fma_rn(y, __fma_rn(e, e, e), y);
}
__device__ __forceinline__ double quot(double a, double b, double y)
{
    const double q = a * y;
    return __fma_rn(-__fma_rn(b, q, -a), y, q);      // (this sign keeps that of a zero a)
}

// ---- elementary functions (the operations of detmath64.cuh) --------------------------
// One Horner form for exp, sin and cos, so that different lanes can run different ones:
// k = floor(x m + 1/2), r = ((x - k c1) - k c2) - k c3, p = Horner(v) with v = r or r^2 over
// 14 coefficients (leading zeros leave p unchanged: 0 v + c = c).
enum Fn { kExp = 0, kSin = 1, kCos = 2 };
struct FnRow {
    double m, c1, c2, c3, c[14];
};
__device__ const FnRow kFnTable[3] = {
    {dm::kLog2e, dm::kLn2Hi, dm::kLn2Lo, 0.0,
     {1.0 / 6227020800.0, 1.0 / 479001600.0, 1.0 / 39916800.0, 1.0 / 3628800.0, 1.0 / 362880.0, 1.0 / 40320.0,
      1.0 / 5040.0, 1.0 / 720.0, 1.0 / 120.0, 1.0 / 24.0, 1.0 / 6.0, 0.5, 1.0, 1.0}},
    {dm::k2OverPi, dm::kPio2_1, dm::kPio2_2, dm::kPio2_3,
     {0.0, 0.0, 0.0, 0.0, -1.0 / 121645100408832000.0, 1.0 / 355687428096000.0, -1.0 / 1307674368000.0,
      1.0 / 6227020800.0, -1.0 / 39916800.0, 1.0 / 362880.0, -1.0 / 5040.0, 1.0 / 120.0, -1.0 / 6.0, 1.0}},
    {dm::k2OverPi, dm::kPio2_1, dm::kPio2_2, dm::kPio2_3,
     {0.0, 0.0, 0.0, 1.0 / 2432902008176640000.0, -1.0 / 6402373705728000.0, 1.0 / 20922789888000.0,
      -1.0 / 87178291200.0, 1.0 / 479001600.0, -1.0 / 3628800.0, 1.0 / 40320.0, -1.0 / 720.0, 1.0 / 24.0, -0.5, 1.0}},
};
constexpr int kFnStride = 19;      // doubles between rows in shared memory (odd: lanes on different rows, different banks)
constexpr int kFnWords = 3 * kFnStride;

__device__ __forceinline__ void load_table(double *tab)      // whole block; the caller synchronises
{
    for (int i = threadIdx.x; i < 3 * 18; i += blockDim.x)
        tab[(i / 18) * kFnStride + i % 18] = reinterpret_cast<const double *>(kFnTable)[i];
}

// exp(x) for 2^-1 <= result exponents well inside the range, |x| < 700
__device__ __forceinline__ double exp_in(double x)
{
    const int k = ifloor(x * dm::kLog2e + 0.5);
    const double kd = from_int(k);
    const double r = (x - kd * dm::kLn2Hi) - kd * dm::kLn2Lo;
    double p = 1.0 / 6227020800.0;
    p = p * r + 1.0 / 479001600.0;
    p = p * r + 1.0 / 39916800.0;
    p = p * r + 1.0 / 3628800.0;
    p = p * r + 1.0 / 362880.0;
    p = p * r + 1.0 / 40320.0;
    p = p * r + 1.0 / 5040.0;
    p = p * r + 1.0 / 720.0;
    p = p * r + 1.0 / 120.0;
    p = p * r + 1.0 / 24.0;
    p = p * r + 1.0 / 6.0;
    p = p * r + 0.5;
    p = p * r + 1.0;
    p = p * r + 1.0;
    return __hiloint2double(__double2hiint(p) + k * 0x100000, __double2loint(p));
}

__device__ __forceinline__ void quadrant(int k, double sr, double cr, double &sn, double &cs)
{
    const bool odd = k & 1;
    sn = neg_if(odd ? cr : sr, k & 2);
    cs = neg_if(odd ? sr : cr, (k + 1) & 2);
}

// A sheet phase beyond this takes the plain step: ifloor wants |x 2/pi + 1/2| < 2^20, and a start longitude
// is any finite number.
constexpr double kFarAngle = 1e6;
// So do P outside e^-40 .. e^40 GV and theta not in [2^-100, pi] (a step from beside a pole can throw theta so
// far that its fold leaves nothing of it): with them, and with the constants in fast_step_set's range, the
// step's intermediate values stay between about 1e-290 and 1e290 or are zero.
constexpr double kFarLnP = 40.0, kNearPole = 7.888609052210118e-31;
__device__ __forceinline__ bool odd_theta(double th)      // by the high words: up to 5e-10 above pi passes
{
    return (uint32_t)(__double2hiint(th) - __double2hiint(kNearPole)) > (uint32_t)(__double2hiint(kPi) - __double2hiint(kNearPole));
}
__device__ __forceinline__ double reduce(double x, int &k)
{
    k = ifloor(x * dm::k2OverPi + 0.5);
    const double kd = from_int(k);
    return ((x - kd * dm::kPio2_1) - kd * dm::kPio2_2) - kd * dm::kPio2_3;
}
__device__ __forceinline__ void sincos_in(double x, double &sn, double &cs)
{
    int k;
    const double r = reduce(x, k), r2 = r * r;
    double ps = -1.0 / 121645100408832000.0;
    ps = ps * r2 + 1.0 / 355687428096000.0;
    ps = ps * r2 - 1.0 / 1307674368000.0;
    ps = ps * r2 + 1.0 / 6227020800.0;
    ps = ps * r2 - 1.0 / 39916800.0;
    ps = ps * r2 + 1.0 / 362880.0;
    ps = ps * r2 - 1.0 / 5040.0;
    ps = ps * r2 + 1.0 / 120.0;
    ps = ps * r2 - 1.0 / 6.0;
    ps = ps * r2 + 1.0;
    double pc = 1.0 / 2432902008176640000.0;
    pc = pc * r2 - 1.0 / 6402373705728000.0;
    pc = pc * r2 + 1.0 / 20922789888000.0;
    pc = pc * r2 - 1.0 / 87178291200.0;
    pc = pc * r2 + 1.0 / 479001600.0;
    pc = pc * r2 - 1.0 / 3628800.0;
    pc = pc * r2 + 1.0 / 40320.0;
    pc = pc * r2 - 1.0 / 720.0;
    pc = pc * r2 + 1.0 / 24.0;
    pc = pc * r2 - 0.5;
    pc = pc * r2 + 1.0;
    quadrant(k, r * ps, pc, sn, cs);
}
// cos alone: the lane's quadrant needs one of the two polynomials
__device__ __forceinline__ double cos_in(double x)
{
    int k;
    const double r = reduce(x, k), v = r * r;
    const bool odd = k & 1;
    double p = odd ? 0.0 : 1.0 / 2432902008176640000.0;
    p = p * v + (odd ? -1.0 / 121645100408832000.0 : -1.0 / 6402373705728000.0);
    p = p * v + (odd ? 1.0 / 355687428096000.0 : 1.0 / 20922789888000.0);
    p = p * v + (odd ? -1.0 / 1307674368000.0 : -1.0 / 87178291200.0);
    p = p * v + (odd ? 1.0 / 6227020800.0 : 1.0 / 479001600.0);
    p = p * v + (odd ? -1.0 / 39916800.0 : -1.0 / 3628800.0);
    p = p * v + (odd ? 1.0 / 362880.0 : 1.0 / 40320.0);
    p = p * v + (odd ? -1.0 / 5040.0 : -1.0 / 720.0);
    p = p * v + (odd ? 1.0 / 120.0 : 1.0 / 24.0);
    p = p * v + (odd ? -1.0 / 6.0 : -0.5);
    p = p * v + 1.0;
    return neg_if(p * (odd ? r : 1.0), (k + 1) & 2);
}
// log of a positive normal x
__device__ __forceinline__ double log_in(double x)
{
    const uint64_t b = bits(x);
    int e = (int)(b >> 52) - 1023;
    uint64_t mb = (b & 0x000FFFFFFFFFFFFFull) | 0x3FF0000000000000ull;
    if (mb > 0x3FF6A09E667F3BCDull) {      // above the double nearest sqrt 2
        mb -= 0x0010000000000000ull;
        e += 1;
    }
    const double m = from_bits(mb), b1 = m + 1.0;
    const double s = quot(m - 1.0, b1, recip(b1)), s2 = s * s;
    double q = 1.0 / 23.0;
    q = q * s2 + 1.0 / 21.0;
    q = q * s2 + 1.0 / 19.0;
    q = q * s2 + 1.0 / 17.0;
    q = q * s2 + 1.0 / 15.0;
    q = q * s2 + 1.0 / 13.0;
    q = q * s2 + 1.0 / 11.0;
    q = q * s2 + 1.0 / 9.0;
    q = q * s2 + 1.0 / 7.0;
    q = q * s2 + 1.0 / 5.0;
    q = q * s2 + 1.0 / 3.0;
    q = q * s2 + 1.0;
    const double de = from_int(e);
    return de * dm::kLn2Hi + (de * dm::kLn2Lo + scale2<1>(s * q));
}
__device__ __forceinline__ double atan_in(double x)
{
    double a = from_bits(bits(x) & 0x7FFFFFFFFFFFFFFFull);
    const bool inv = lt(1.0, a);
    if (inv) a = quot(1.0, a, recip(a));
    double base = 0.0, y = a;
    if (lt(0.19891236737965800, a)) {
        // (a - c) / (1 + a c) with c = 1 or tan(pi/8)
        const bool far = lt(0.66817863791929891, a);
        const double c = far ? 1.0 : dm::kTanPi_8;
        const double d = 1.0 + a * c;
        y = quot(a - c, d, recip(d));
        base = far ? dm::kPi_4 : dm::kPi_8;
    }
    const double y2 = y * y;
    double q = -1.0 / 23.0;
    q = q * y2 + 1.0 / 21.0;
    q = q * y2 - 1.0 / 19.0;
    q = q * y2 + 1.0 / 17.0;
    q = q * y2 - 1.0 / 15.0;
    q = q * y2 + 1.0 / 13.0;
    q = q * y2 - 1.0 / 11.0;
    q = q * y2 + 1.0 / 9.0;
    q = q * y2 - 1.0 / 7.0;
    q = q * y2 + 1.0 / 5.0;
    q = q * y2 - 1.0 / 3.0;
    q = q * y2 + 1.0;
    double res = base + y * q;
    if (inv) res = dm::kPi_2 - res;
    return neg_if(res, __double2hiint(x) < 0);
}

// Three N(0,1) of step k (m64::normals)
__device__ __forceinline__ void normals(uint64_t seed, uint64_t pid, uint32_t k, double z[3])
{
    const uint4 w = philox_step_block(seed, pid, k);
    const double rho0 = sqrt(neg_if(scale2<1>(log_in(uniform(w.x))), true));
    const double rho2 = sqrt(neg_if(scale2<1>(log_in(uniform(w.z))), true));
    double s1, c1;
    sincos_in(kTwoPi * uniform(w.y), s1, c1);
    z[0] = rho0 * c1;
    z[1] = rho0 * s1;
    z[2] = rho2 * cos_in(kTwoPi * uniform(w.w));
}

// ---- teams of G lanes ------------------------------------------------------------------
template <int G>
struct Team {
    int l;             // lane in the team
    // whether to enter a block that shuffles: the teams of a warp may hold sets with different
    // switches, so it is entered by all of them or by none
    __device__ __forceinline__ bool any(bool mine) const
    {
        if constexpr (G == 1) return mine;
        else return __any_sync(0xffffffffu, mine);
    }
    __device__ __forceinline__ double get(double v, int j) const { return __shfl_sync(0xffffffffu, v, j, G); }
    __device__ __forceinline__ double pick(double a, double b, double c, double d) const
    {
        const double x = (l & 1) ? b : a, y = (l & 1) ? d : c;
        return (l & 2) ? y : x;
    }
    __device__ __forceinline__ void recip4(double a, double b, double c, double d, double (&y)[4]) const
    {
        if constexpr (G == 1) {
            y[0] = recip(a); y[1] = recip(b); y[2] = recip(c); y[3] = recip(d);
        } else {
            const double v = recip(pick(a, b, c, d));
#pragma unroll
            for (int j = 0; j < 4; ++j) y[j] = get(v, j);
        }
    }
    __device__ __forceinline__ void quot4(const double (&n)[4], const double (&b)[4], const double (&y)[4], double (&q)[4]) const
    {
        if constexpr (G == 1) {
#pragma unroll
            for (int j = 0; j < 4; ++j) q[j] = quot(n[j], b[j], y[j]);
        } else {
            const double v = quot(pick(n[0], n[1], n[2], n[3]), pick(b[0], b[1], b[2], b[3]), pick(y[0], y[1], y[2], y[3]));
#pragma unroll
            for (int j = 0; j < 4; ++j) q[j] = get(v, j);
        }
    }
    __device__ __forceinline__ void sqrt4(double a, double b, double c, double d, double (&s)[4]) const
    {
        if constexpr (G == 1) {
            s[0] = sqrt(a); s[1] = sqrt(b); s[2] = sqrt(c); s[3] = sqrt(d);
        } else {
            const double v = sqrt(pick(a, b, c, d));
#pragma unroll
            for (int j = 0; j < 4; ++j) s[j] = get(v, j);
        }
    }
    // exp(x0), exp(x1), sin(th), cos(th): one lane each, one Horner form
    __device__ __forceinline__ void functions(const double *tab, double x0, double x1, double th, double &e0, double &e1,
                                              double &sn, double &cs) const
    {
        const bool trig = l & 2;
        const double *t = tab + (trig ? kSin + (l & 1) : kExp) * kFnStride;
        const double x = pick(x0, x1, th, th);
        const int k = ifloor(x * t[0] + 0.5);
        const double kd = from_int(k);
        const double r = ((x - kd * t[1]) - kd * t[2]) - kd * t[3];
        const double r2 = r * r, v = trig ? r2 : r;
        double p = t[4];
#pragma unroll
        for (int i = 5; i < 18; ++i) p = p * v + t[i];
        // exp: times 2^k; sin: times r; cos: as it is
        p = trig ? p * ((l & 1) ? 1.0 : r) : __hiloint2double(__double2hiint(p) + k * 0x100000, __double2loint(p));
        e0 = get(p, 0);
        e1 = get(p, 1);
        quadrant(__shfl_sync(0xffffffffu, k, 2, G), get(p, 2), get(p, 3), sn, cs);
    }
    __device__ __forceinline__ void sincos(const double *tab, double x, double &sn, double &cs) const
    {
        const double *t = tab + (kSin + (l & 1)) * kFnStride;
        int k;
        const double r = reduce(x, k), v = r * r;
        double p = t[7];                     // the first three coefficients are zero in both rows
#pragma unroll
        for (int i = 8; i < 18; ++i) p = p * v + t[i];
        p = p * ((l & 1) ? 1.0 : r);
        quadrant(k, get(p, 0), get(p, 1), sn, cs);
    }
};

struct Spc {
    double A, aZ, m0, m0sq, aoz, raoz;     // raoz = 1 / aoz
    bool negative;                          // charge
};
__device__ __forceinline__ Spc make_spc(const DevSpecies &s)
{
    const double aoz = s.A / fabs(s.Z);
    return Spc{s.A, fabs(s.Z), s.m0, s.m0 * s.m0, aoz, recip(aoz), s.Z < 0.0};
}

// The step as it is defined, for states outside the fast form's range (by value: only its
// own frame keeps the state in memory).
__device__ __noinline__ m64::State plain_step(const DevParams &p, const DevSpecies &sp, uint64_t seed, uint64_t pid, m64::State x)
{
    m64::em_step(p, sp, seed, pid, x);
    return x;
}

// reflection at r_in and the angles' ranges, by definition
__device__ __forceinline__ void into_range(const DevParams &p, m64::State &o)
{
    if (o.r < p.r_in) o.r = 2.0 * p.r_in - o.r;
    const double t = o.th - kTwoPi * floor(o.th / kTwoPi);
    if (t > kPi) {
        o.th = kTwoPi - t;
        o.ph = o.ph + kPi;
    } else {
        o.th = t;
    }
    // floor(ph / 2 pi) is -1 and 1 on [-2 pi, 0) and [2 pi, 4 pi)
    if (o.ph < 0.0 && o.ph >= -kTwoPi) o.ph = o.ph + kTwoPi;
    else if (o.ph >= kTwoPi && o.ph < 2.0 * kTwoPi) o.ph = o.ph - kTwoPi;
    else o.ph = o.ph - kTwoPi * floor(o.ph / kTwoPi);
}

template <bool EN>
__device__ __forceinline__ bool finite_state(const m64::State &o)
{
    return (!EN | f64bits::is_finite(bits(o.T))) & f64bits::is_finite(bits(o.r)) & f64bits::is_finite(bits(o.th)) &
           f64bits::is_finite(bits(o.ph)) & f64bits::is_finite(bits(o.lnP)) & f64bits::is_finite(bits(o.s));
}

// |dV/dth| with the sign of d|lat|/dth, zero on the equator
__device__ __forceinline__ double toward_equator(double dV, double lat)
{
    return (bits(lat) << 1) == 0 ? 0.0 : neg_if(dV, __double2hiint(lat) >= 0);
}

// One step of x, m64::em_step's values.  ISO: the spherically symmetric model; EN: the energy
// form; no shells, not squashed.  z: the step's normals.  Team lanes hold equal states and
// must all call (shuffles); live = false leaves the state as it was.
template <int G, bool ISO, bool EN>
__device__ __forceinline__ void step(const DevParams &p, const DevSpecies &dsp, const Spc &sp, uint64_t seed, uint64_t pid,
                                     uint32_t max_steps, const double *tab, const Team<G> team, const double z[3], bool live,
                                     m64::State &x)
{
    const F64Params &d = p.d;
    const double r = x.r, th = x.th;
    const bool shock = positive(p.R_ts);
    double y4[4], q4[4], q5[4], q6[4];

    // shock and wind arguments
    double lat = 0.0, wa = 0.0, sa = 0.0, ts = 0.0;
    if constexpr (!ISO) {
        lat = 0.5 * kPi - th;
        const double al = from_bits(bits(lat) & 0x7FFFFFFFFFFFFFFFull);
        wa = quot(al - d.lat_f, d.dlat, d.r_dlat);
    }
    // P, sin, cos, and the wind's exp(2 |wa|)
    double P, ew = 0.0, sn, cs;
    const double wabs = from_bits(bits(wa) & 0x7FFFFFFFFFFFFFFFull);
    const bool wnear = !lt(20.0, wabs);
    if constexpr (G == 1) {
        P = exp_in(x.lnP);
        if (!ISO && wnear) ew = exp_in(scale2<1>(wabs));
        sincos_in(th, sn, cs);
    } else {
        team.functions(tab, x.lnP, wnear ? scale2<1>(wabs) : 0.0, th, P, ew, sn, cs);
    }
    bool odd_range = beyond(x.lnP, kFarLnP) | odd_theta(th);
    double es = 0.0;
    bool snear = false;
    if (shock) {
        sa = quot(r - p.R_ts, p.dts, d.r_dts);
        const double sabs = from_bits(bits(sa) & 0x7FFFFFFFFFFFFFFFull);
        snear = !lt(20.0, sabs);
        if (snear) es = exp_in(scale2<1>(sabs));
    }

    const double pn = quot(P, sp.aoz, sp.raoz);
    const double root = sqrt(pn * pn + sp.m0sq);
    const double ew1 = ew + 1.0, rs = r * sn;
    team.recip4(root, sn, r, ew1, y4);
    const double y_r = y4[2], y_sn = y4[1];
    {
        const double n[4] = {pn, cs, 2.0, 0.0}, b[4] = {root, sn, ew1, 1.0}, y[4] = {y4[0], y4[1], y4[3], 1.0};
        if constexpr (G == 1) {
            q4[0] = quot(n[0], b[0], y[0]);
            q4[1] = quot(n[1], b[1], y[1]);
            q4[2] = ISO ? 0.0 : quot(n[2], b[2], y[2]);
        } else {
            team.quot4(n, b, y, q4);
        }
    }
    const double beta = q4[0], cot = q4[1];

    // wind V(th), dV/dth
    double V, dV = 0.0;
    if constexpr (ISO) {
        V = d.Vs;
    } else {
        const double t = neg_if(wnear ? 1.0 - q4[2] : 1.0, __double2hiint(wa) < 0);
        V = d.Vs + d.hdV * (1.0 + t);
        dV = quot(d.hdV * (1.0 - t * t), d.dlat, d.r_dlat);
        dV = toward_equator(dV, lat);
    }
    // termination shock
    double g = 1.0, dg = 0.0;
    if (shock) {
        double q = 0.0;
        if (snear) {
            const double b = es + 1.0;
            q = quot(2.0, b, recip(b));
        }
        ts = neg_if(snear ? 1.0 - q : 1.0, __double2hiint(sa) < 0);
        g = 1.0 - d.hts * (1.0 + ts);
        dg = neg_if(quot(d.hts * (1.0 - ts * ts), p.dts, d.r_dts), true);
    }
    const double Kbase = p.K0 * beta * P;
    const double Kpar = shock ? Kbase * g : Kbase;
    const double dKpar = shock ? Kbase * dg : 0.0;
    const double rr = r * r, r3 = 3.0 * r;

    double K00, K11, K22, K02 = 0.0, Ar, Ath, Aph = 0.0, l00, l11, l22, l20 = 0.0, dlnP;
    double vd0 = 0.0, vd1 = 0.0, vd2 = 0.0, delta = 0.0, y_rs;
    bool sheet = false;          // its width limits the step
    if constexpr (ISO) {
        K00 = K11 = K22 = Kpar;
        team.recip4(rr, r3, rs, 1.0, y4);
        y_rs = y4[2];
        const double n[4] = {scale2<1>(K00), K11 * cot, scale2<1>(V), 0.0}, b[4] = {r, rr, r3, 1.0},
                     y[4] = {y_r, y4[0], y4[1], 1.0};
        if constexpr (G == 1) {
            for (int j = 0; j < 3; ++j) q4[j] = quot(n[j], b[j], y[j]);
        } else {
            team.quot4(n, b, y, q4);
        }
        Ar = dKpar + q4[0];
        Ath = q4[1];
        dlnP = q4[2];
        l00 = l11 = l22 = sqrt(scale2<1>(Kpar));
    } else {
        const double VV = V * V, Or = d.Omega * r;
        team.recip4(V, VV, rs, r3, y4);
        const double y_V = y4[0], y_VV = y4[1];
        y_rs = y4[2];
        const double y_r3 = y4[3];
        {
            const double n[4] = {Or * sn, Or, d.Omega, dV}, b[4] = {V, V, V, V}, y[4] = {y_V, y_V, y_V, y_V};
            team.quot4(n, b, y, q4);
        }
        const double Gam = q4[0], dphs_dr = q4[2];
        const double G2 = Gam * Gam, og = 1.0 + G2, gg = og * og;
        const double dGam_dth = Gam * (cot - q4[3]);
        const double phs = x.ph + q4[1];
        odd_range |= beyond(phs, kFarAngle);
        double sphs = 0.0, cphs = 0.0;
        const bool hcs = on(p.hcs_on), any_hcs = team.any(hcs);
        if (any_hcs) {
            if constexpr (G == 1) sincos_in(phs, sphs, cphs);
            else team.sincos(tab, phs, sphs, cphs);
        }
        team.recip4(og, gg, rr, 1.0, y4);
        const double y_og = y4[0], y_gg = y4[1], y_rr = y4[2];
        {
            const double n[4] = {1.0, G2, Gam, Gam}, b[4] = {og, og, og, r}, y[4] = {y_og, y_og, y_og, y_r};
            team.quot4(n, b, y, q4);
        }
        const double c2 = q4[0], s2 = q4[1], sc = q4[2], dGam_dr = q4[3];
        const double m1 = 1.0 - G2, r2G = rr * Gam;
        const bool drift = on(p.drift_on);
        sheet = hcs && drift;
        {
            const double n[4] = {neg_if(scale2<1>(Gam) * dGam_dr, true), dGam_dr * m1, neg_if(scale2<1>(r2G * dGam_dth), true),
                                 r * Gam * (3.0 + G2)},
                         b[4] = {gg, gg, gg, gg}, y[4] = {y_gg, y_gg, y_gg, y_gg};
            team.quot4(n, b, y, q4);
        }
        const double dc2 = q4[0], dsc = q4[1], dF_dth = q4[2], dGf_dr = q4[3];

        // tensor
        const double Kpr = p.er * Kpar, Kpt = p.et * Kpar, dK = Kpr - Kpar;
        K00 = Kpar * c2 + Kpr * s2;
        K22 = Kpar * s2 + Kpr * c2;
        K02 = dK * sc;
        K11 = Kpt;
        double Kr00, Kr02;
        if (shock) {
            const double dKpr = p.er * dKpar;
            Kr00 = dKpar * c2 + Kpar * dc2 + dKpr * s2 + Kpr * neg_if(dc2, true);
            Kr02 = (dKpr - dKpar) * sc + dK * dsc;
        } else {
            Kr00 = Kpar * dc2 + Kpr * neg_if(dc2, true);
            Kr02 = dK * dsc;
        }
        double sog = 1.0;
        if constexpr (G == 1) {
            l00 = sqrt(scale2<1>(K00));
            l11 = sqrt(scale2<1>(K11));
            if (hcs) sog = sqrt(og);
        } else {
            double s4[4];
            team.sqrt4(scale2<1>(K00), scale2<1>(K11), og, 1.0, s4);
            l00 = s4[0];
            l11 = s4[1];
            sog = s4[2];
        }
        const double D = quot(P * 1e9, d.dDen, d.r_dDen);
        const double D2r = scale2<1>(D) * r, ogs = og * sog;
        team.recip4(l00, sog, ogs, 1.0, y4);
        {
            // dGf_dth, F, Gf of the drift; d(2K_rr)/r
            const double n[4] = {rr * dGam_dth * m1, rr, r2G, scale2<1>(K00)}, b[4] = {gg, og, og, r}, y[4] = {y_gg, y_og, y_og, y_r};
            team.quot4(n, b, y, q5);
        }
        {
            const double n[4] = {scale2<1>(K02), D2r, scale2<1>(D), neg_if(D2r * Gam * dGam_dth, true)}, b[4] = {l00, sog, ogs, ogs},
                         y[4] = {y4[0], y4[1], y4[2], y4[2]};
            team.quot4(n, b, y, q4);
        }
        {
            const double n[4] = {K11 * cot, K02, neg_if(Or * dV, true), scale2<1>(V)}, b[4] = {rr, r, VV, r3}, y[4] = {y_rr, y_r, y_VV, y_r3};
            team.quot4(n, b, y, q6);
        }
        l20 = q4[0];
        l22 = sqrt(scale2<1>(K22) - l20 * l20);
        Ar = Kr00 + q5[3];
        Ath = q6[0];
        Aph = quot(Kr02 + q6[1], rs, y_rs);
        const double dphs_dth = q6[2];
        dlnP = q6[3];
        const double dGf_dth = q5[0], F = q5[1], Gf = q5[2];

        // current sheet
        double h = 1.0, dh_dr = 0.0, dh_dth = 0.0, dh_dph = 0.0;
        if (any_hcs) {
            const double th_cs = 0.5 * kPi + atan_in(d.ta * sphs);
            const double den = 1.0 + d.ta2 * sphs * sphs;
            const bool rl = lt(d.dmin, q4[1]);
            delta = rl ? q4[1] : d.dmin;
            const double dd_dr = rl ? q4[2] : 0.0, dd_dth = rl ? q4[3] : 0.0;
            team.recip4(den, delta, 1.0, 1.0, y4);
            {
                const double n[4] = {d.ta * cphs, th_cs - th, 0.0, 0.0}, b[4] = {den, delta, 1.0, 1.0}, y[4] = {y4[0], y4[1], 1.0, 1.0};
                if constexpr (G == 1) {
                    q4[0] = quot(n[0], b[0], y[0]);
                    q4[1] = quot(n[1], b[1], y[1]);
                } else {
                    team.quot4(n, b, y, q4);
                }
            }
            const double dthcs = q4[0], u = q4[1];
            const double uabs = from_bits(bits(u) & 0x7FFFFFFFFFFFFFFFull);
            // beyond |u| = 20 the sheet's h is +-1 and its gradient zero
            const bool near = !lt(20.0, uabs);
            double t = 1.0;
            if (near) {
                const double b = exp_in(scale2<1>(uabs)) + 1.0;
                t = 1.0 - quot(2.0, b, recip(b));
            }
            h = neg_if(t, __double2hiint(u) < 0);
            {
                const double n[4] = {dthcs * dphs_dr - u * dd_dr, dthcs * dphs_dth - 1.0 - u * dd_dth, dthcs, 0.0},
                             b[4] = {delta, delta, delta, 1.0}, y[4] = {y4[1], y4[1], y4[1], 1.0};
                if constexpr (G == 1) {
                    if (near)
                        for (int j = 0; j < 3; ++j) q4[j] = quot(n[j], b[j], y[j]);
                } else {
                    team.quot4(n, b, y, q4);
                }
            }
            if (near) {
                const double w = 1.0 - h * h;
                dh_dr = w * q4[0];
                dh_dth = w * q4[1];
                dh_dph = w * q4[2];
            }
            if (!hcs) {
                h = 1.0;
                delta = dh_dr = dh_dth = dh_dph = 0.0;
            }
        }
        if (team.any(drift)) {
            const double CA = quot(beta * P * 1e9 * kDay_s, d.caDen, d.r_caDen);
            const double nCA = neg_if(CA, true);
            const double Wph = nCA * h * Gf;
            const double dWph_dth = nCA * (dh_dth * Gf + h * dGf_dth);
            const double dWph_dr = nCA * (dh_dr * Gf + h * dGf_dr);
            const double dWr_dph = CA * dh_dph * F;
            const double dWr_dth = CA * (dh_dth * F + h * dF_dth);
            const double n[4] = {cot * Wph + dWph_dth, quot(dWr_dph, sn, y_sn) - Wph - r * dWph_dr, neg_if(dWr_dth, true), 0.0},
                         b[4] = {r, r, r, 1.0}, y[4] = {y_r, y_r, y_r, 1.0};
            if constexpr (G == 1) {
                for (int j = 0; j < 3; ++j) q4[j] = quot(n[j], b[j], y[j]);
            } else {
                team.quot4(n, b, y, q4);
            }
            if (drift) {
                const bool s = sp.negative != (__double2hiint(p.polarity) < 0);
                vd0 = neg_if(q4[0], s);
                vd1 = neg_if(q4[1], s);
                vd2 = neg_if(q4[2], s);
            }
        }
    }

    // step length
    const double Ar_tot = Ar - V - vd0;
    const bool fixed = positive(p.dt_fixed);
    double dt = p.dt_fixed, sdt = d.sdt_fixed;
    if (team.any(!fixed)) {
        dt = p.dt_max;
        const double num = d.eps_adv2 * K00, den = Ar_tot * Ar_tot, n2 = p.eps_diff * r * r;
        const double rd = r * delta, n3 = sheet ? p.eps_diff * rd * rd : 0.0;
        if constexpr (G == 1) {
            if (lt(num, dt * den)) dt = quot(num, den, recip(den));
            // a quotient can be below dt only if its numerator is not above dt times the denominator
            // (by the high words, with one unit of slack)
            if (__double2hiint(n2) <= __double2hiint(dt * K00) + 1) {
                const double t2 = quot(n2, K00, recip(K00));
                if (lt(t2, dt)) dt = t2;
            }
            if (sheet && __double2hiint(n3) <= __double2hiint(dt * K11) + 1) {
                const double t3 = quot(n3, K11, recip(K11));
                if (lt(t3, dt)) dt = t3;
            }
        } else {
            team.recip4(den, K00, K11, 1.0, y4);
            const double n[4] = {num, n2, n3, 0.0}, b[4] = {den, K00, K11, 1.0}, y[4] = {y4[0], y4[1], y4[2], 1.0};
            team.quot4(n, b, y, q4);
            if (lt(num, dt * den)) dt = q4[0];
            if (lt(q4[1], dt)) dt = q4[1];
            if (sheet && lt(q4[2], dt)) dt = q4[2];
        }
        if (lt(dt, p.dt_min)) dt = p.dt_min;
        if (fixed) dt = p.dt_fixed;
        else sdt = sqrt(dt);
    }

    // Euler-Maruyama update
    const double Lz_r = l00 * z[0];
    const double Lz_th = l11 * z[1];
    const double Lz_ph = ISO ? l22 * z[2] : l20 * z[0] + l22 * z[2];
    {
        const double n[4] = {vd1, vd2, Lz_th * sdt, Lz_ph * sdt}, b[4] = {r, rs, r, rs}, y[4] = {y_r, y_rs, y_r, y_rs};
        if constexpr (G == 1) {
            q4[0] = ISO ? 0.0 : quot(n[0], b[0], y[0]);
            q4[1] = ISO ? 0.0 : quot(n[1], b[1], y[1]);
            q4[2] = quot(n[2], b[2], y[2]);
            q4[3] = quot(n[3], b[3], y[3]);
        } else {
            team.quot4(n, b, y, q4);
        }
    }
    m64::State o;
    o.r = r + (Ar_tot * dt + Lz_r * sdt);
    if constexpr (ISO) {
        o.th = th + (Ath * dt + q4[2]);
        o.ph = x.ph + q4[3];
    } else {
        o.th = th + ((Ath - q4[0]) * dt + q4[2]);
        o.ph = x.ph + ((Aph - q4[1]) * dt + q4[3]);
    }
    o.T = x.T;
    o.Lam = x.Lam;
    if constexpr (EN) {
        // Eq. 1 backward: A_T = (2/3)(V/r) alpha T, loss L = (2V/(3r)) (1 + beta^2); dlnP = 2V/(3r)
        const double b = x.T + sp.m0;
        const double alpha = quot(x.T + 2.0 * sp.m0, b, recip(b));
        o.T = x.T + dlnP * alpha * x.T * dt;
        o.Lam = x.Lam + dlnP * (1.0 + beta * beta) * dt;
        o.lnP = log_in(sp.aoz * sqrt(o.T * (o.T + 2.0 * sp.m0)));
    } else {
        o.lnP = x.lnP + dlnP * dt;
    }
    // one rarely taken branch for the reflection and the angles' ranges
    if (f64bits::less(bits(o.r), bits(p.r_in)) | f64bits::outside_closed(bits(o.th), f64bits::kPiBits) |
        f64bits::outside_half_open(bits(o.ph), f64bits::kTwoPiBits)) {
        into_range(p, o);
    }
    o.s = x.s + dt;
    o.k = x.k + 1u;
    o.r_old = r;
    o.status = !lt(o.r, p.R_out) ? COSMICA_PATH_EXIT : (o.k >= max_steps ? COSMICA_PATH_STEP_LIMIT : COSMICA_PATH_RUNNING);
    if (live) {
        if (finite_state<EN>(o) & !odd_range) x = o;
        else x = plain_step(p, dsp, seed, pid, x);
    }
}

}  // namespace s64
}  // namespace cosmica
