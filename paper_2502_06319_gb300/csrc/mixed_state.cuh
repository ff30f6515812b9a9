// mixed_state.cuh -- per-lane state of the mixed-precision persistent kernels
// (batched propagation and serving quanta): the particle's identity and the
// accumulated (r, theta, phi, lnP, s), either as compensated float-float
// pairs or in FP64, with the boundary handling of the step.
#pragma once
#include "common.cuh"
#include "f64bits.h"
#include "model32.cuh"

namespace cosmica {

// FP64 <-> FP32 on the bits (f64bits.h)
__device__ __forceinline__ uint64_t bits64(double x) { return (uint64_t)__double_as_longlong(x); }
__device__ __forceinline__ double widen64(float d)
{
    return __longlong_as_double((long long)f64bits::widen(__float_as_uint(d)));
}
__device__ __forceinline__ float narrow64(double x) { return __uint_as_float(f64bits::narrow(bits64(x))); }

struct Lane {
    const float *q;            // field 0 of the particle's FP32 parameter block (see P32)
    float M2, sq;
    uint64_t pid, seed, g;
    uint32_t item, k, max_steps;
};

template <int ACC>
struct Acc;

// compensated FP32 state
template <>
struct Acc<COSMICA_PREC_MIXED> {
    m32::FF r, th, ph;
    m32::FF2 Ps;   // lnP and s, the two that no boundary touches, as packed pairs
    m32::FF Rout;
    float r_in2;   // 2 r_in
    __device__ void init(double r0, double th0, double ph0, double lnP0, double R_out, float r_in, float)
    {
        r = m32::ff_from_double(r0);
        th = m32::ff_from_double(th0);
        ph = m32::ff_from_double(ph0);
        Ps.set(m32::ff_from_double(lnP0), m32::FF{0.0f, 0.0f});
        Rout = m32::ff_from_double(R_out);
        r_in2 = 2.0f * r_in;
    }
    __device__ float fr() const { return r.hi; }
    __device__ float fth() const { return th.hi; }
    __device__ float fph() const { return ph.hi; }
    // distance of theta (hi + lo, in [0, pi]) to the nearer pole, to FP32 accuracy:
    // near pi it is formed from the float-float splits of pi and theta (the high
    // parts subtract exactly), so it keeps its sign and relative accuracy even
    // where the FP32 theta rounds to pi or beyond
    __device__ float pole_distance() const
    {
        if (th.hi < m32::kHalfPiF) return th.hi;
        return __fadd_rn(__fsub_rn(m32::kPiF, th.hi), __fsub_rn(m32::kPiLoF, th.lo));
    }
    // r, theta, phi, lnP and sin(theta) as the step reads them
    __device__ void view(float &fr, float &fth, float &fph, float &flnP, float &sin_th) const
    {
        fr = r.hi; fth = th.hi; fph = ph.hi; flnP = Ps.first().hi;
        sin_th = m32::sin_from_pole_distance(pole_distance());
    }
    // Adds a step's increments (to the state whose view was fr, fth, fph); true when nothing has to
    // be looked at: no boundary, end or non-finite value is near.
    // P: the form accumulates lnP (the energy form integrates T instead and leaves lnP alone);
    // sphere: the outer boundary is r = R_out (a squashed one is tested by its own function)
    template <bool P>
    __device__ bool add(float, float, float, float dr, float dth, float dph, float dlnP, float dt, float r_in, bool sphere)
    {
        m32::ff_add(r, dr);
        m32::ff_add(th, dth);
        m32::ff_add(ph, dph);
        m32::ff_add2(Ps, P ? dlnP : 0.0f, dt);
        return calm(r_in, sphere) & !phi_out();
    }
    // reflect at r_in, fold theta at the poles, wrap phi; all rare branches
    __device__ void boundaries(float r_in)
    {
        const bool fold = th.hi < 0.0f || pole_distance() < 0.0f;   // theta < 0 or theta > pi
        // one rarely taken branch for the three boundaries
        if ((r.hi < r_in) | fold | (ph.hi < 0.0f) | (ph.hi >= m32::kTwoPiF)) {
            if (r.hi < r_in) {           // r <- 2 r_in - r
                r.hi = -r.hi; r.lo = -r.lo;
                m32::ff_add(r, r_in2);
            }
            if (fold) fold_theta();
            if (ph.hi < 0.0f || ph.hi >= m32::kTwoPiF) wrap_phi();
        }
    }
    __device__ void fold_theta()
    {
        // t = th mod 2 pi in [0, 2pi); if t > pi: th = 2pi - t, ph += pi
        const double t0 = m32::ff_to_double(th);
        double t = t0 - kTwoPi * floor(t0 / kTwoPi);
        if (t > kPi) {
            t = kTwoPi - t;
            const double p = m32::ff_to_double(ph) + kPi;
            ph = m32::ff_from_double(p);
        }
        th = m32::ff_from_double(t);
    }
    __device__ void wrap_phi()
    {
        const double p0 = m32::ff_to_double(ph);
        ph = m32::ff_from_double(p0 - kTwoPi * floor(p0 / kTwoPi));
    }
    // no boundary but the longitude's, no end and no non-finite value is anywhere near: false
    // for every state that the rest of boundaries(), exited() or finite() would act on, and for
    // a few others
    __device__ bool calm(float r_in, bool sphere) const
    {
        return (r.hi >= r_in) & (!sphere | (r.hi < Rout.hi)) & (__float_as_uint(th.hi) < __float_as_uint(m32::kPiF)) &
               (ph.hi > -6.28f) & (ph.hi < 12.56f) & isfinite(Ps.first().hi + Ps.second().hi);
    }
    __device__ bool phi_out() const { return !(__float_as_uint(ph.hi) < __float_as_uint(m32::kTwoPiF)); }
    // wrap_phi() for -6.28 < ph < 12.56, where floor(ph / 2 pi) is -1, 0 or 1.  Paths start at one
    // longitude, often 0, and cross it again and again at first (one step in ten of a warp over
    // the paths' lives), so only the three FP64 sums of the definition are left.
    __device__ void wrap_near()
    {
        const double p0 = widen64(ph.hi) + widen64(ph.lo);
        const double turn = ph.hi < 0.0f ? kTwoPi : (f64bits::less(bits64(p0), f64bits::kTwoPiBits) ? 0.0 : -kTwoPi);
        const double p = p0 + turn;
        ph.hi = narrow64(p);
        ph.lo = narrow64(p - widen64(ph.hi));
    }
    __device__ bool exited() const { return m32::ff_ge(r, Rout); }
    __device__ bool finite() const { return isfinite(r.hi + th.hi + ph.hi + Ps.first().hi + Ps.second().hi); }
    __device__ void write(const ExitPtrs &out, uint64_t g) const
    {
        out.r[g] = m32::ff_to_double(r);
        out.th[g] = m32::ff_to_double(th);
        out.ph[g] = m32::ff_to_double(ph);
        out.lnP[g] = m32::ff_to_double(Ps.first());
        out.s[g] = m32::ff_to_double(Ps.second());
    }
};

// FP64 accumulation of FP32 increments.
// The FP64 pipe takes 64 clocks per warp instruction and scheduler, so only the sums stay on it;
// conversions, comparisons and the finiteness test run on the bits (f64bits.h).  The results
// are the same bits.  Measured, conversion instructions and a step in branches against these and a
// step in one block whose vote does not wait for the sums: a lone path's step 2.16 -> 0.51 us, 1.2e5
// paths of 4 heliospheres 854 -> 160 ms.
template <>
struct Acc<COSMICA_PREC_MIXED_F64ACC> {
    double r, th, ph, lnP, s, Rout, r_in;
    float r_lo, r_hi;      // a little inside (r_in, R_out), see add()
    __device__ void init(double r0, double th0, double ph0, double lnP0, double R_out, float r_in_f, float vote_lo)
    {
        r = r0; th = th0; ph = ph0; lnP = lnP0; s = 0.0; Rout = R_out; r_in = (double)r_in_f;
        r_lo = vote_lo;
        r_hi = f64bits::vote_ceiling((float)R_out);
    }
    __device__ float fr() const { return narrow64(r); }
    __device__ float fth() const { return narrow64(th); }
    __device__ float fph() const { return narrow64(ph); }
    // r, theta, phi, lnP and sin(theta) as the step reads them
    __device__ void view(float &fr, float &fth, float &fph, float &flnP, float &sin_th) const
    {
        const uint64_t bt = bits64(th);
        const bool north = f64bits::less(bt, f64bits::kHalfPiBits);
        const uint64_t units = f64bits::pi_minus_units(bt);
        fr = narrow64(r);
        fth = narrow64(th);
        fph = narrow64(ph);
        flnP = narrow64(lnP);
        sin_th = m32::sin_from_pole_distance(north ? fth : f64bits::pi_minus(units));   // of the nearer pole's distance
    }
    // As in the compensated state.  The FP64 sums take 64 clocks each, one after the other, so the
    // step's vote does not wait for them: it looks at the FP32 sums, whose error (two roundings,
    // under 2.4e-7 of the largest r and of 2 pi) is inside the margins, and the sums' finiteness follows
    // from that of the increments (an infinite r has to be seen here: narrow() makes it 1).
    // theta first: the next step's longest chain starts from it.
    template <bool P>
    __device__ bool add(float fr, float fth, float fph, float dr, float dth, float dph, float dlnP, float dt, float, bool sphere)
    {
        const float nr = fr + dr, nth = fth + dth, nph = fph + dph;
        const bool still = (sphere | (dr < f64bits::kMostRise)) & (nr > r_lo) & (!sphere | (nr < r_hi)) & (nth > 1e-5f) &
                           (nth < 3.14158f) & (nph > 1e-5f) & (nph < 6.28317f) & isfinite(dlnP + dt);
        th += widen64(dth); r += widen64(dr);
        if (P) lnP += widen64(dlnP);
        ph += widen64(dph); s += widen64(dt);
        return still;
    }
    __device__ void boundaries(float)
    {
        // one rarely taken branch for the three boundaries; inside it the FP64 comparisons decide
        if (f64bits::less(bits64(r), bits64(r_in)) | f64bits::outside_closed(bits64(th), f64bits::kPiBits) |
            f64bits::outside_half_open(bits64(ph), f64bits::kTwoPiBits)) {
            if (r < r_in) r = 2.0 * r_in - r;
            if (th < 0.0 || th > kPi) {
                double t = th - kTwoPi * floor(th / kTwoPi);
                if (t > kPi) { t = kTwoPi - t; ph += kPi; }
                th = t;
            }
            if (ph < 0.0 || ph >= kTwoPi) ph = ph - kTwoPi * floor(ph / kTwoPi);
        }
    }
    // as in the compensated state, on the high words
    __device__ bool calm(float, bool sphere) const
    {
        return (__double2hiint(r) > __double2hiint(r_in)) & (__double2hiint(r) < (sphere ? __double2hiint(Rout) : 0x7FF00000)) &
               ((uint32_t)__double2hiint(th) < (uint32_t)(f64bits::kPiBits >> 32)) &
               (__double2hiint(ph) < 0x40291EB8) & ((uint32_t)__double2hiint(ph) < 0xC0191EB8u) &
               f64bits::is_finite(bits64(lnP)) & f64bits::is_finite(bits64(s));
    }
    __device__ bool phi_out() const { return f64bits::outside_half_open(bits64(ph), f64bits::kTwoPiBits); }
    __device__ void wrap_near()
    {
        ph += __double2hiint(ph) < 0 ? kTwoPi : (f64bits::less(bits64(ph), f64bits::kTwoPiBits) ? 0.0 : -kTwoPi);
    }
    // (a non-NaN comparison; finite() is asked first)
    __device__ bool exited() const { return !f64bits::less(bits64(r), bits64(Rout)); }
    __device__ bool finite() const
    {
        return f64bits::is_finite(bits64(r)) & f64bits::is_finite(bits64(th)) & f64bits::is_finite(bits64(ph)) &
               f64bits::is_finite(bits64(lnP)) & f64bits::is_finite(bits64(s));
    }
    __device__ void write(const ExitPtrs &out, uint64_t g) const
    {
        out.r[g] = r; out.th[g] = th; out.ph[g] = ph; out.lnP[g] = lnP; out.s[g] = s;
    }
};


// Energy form (Eq. 1): kinetic energy per nucleon T and the loss integral
// Lam = sum L ds of Eq. 4, accumulated with the same precision as the state.
// The momentum form carries nothing.
template <int ACC, bool EN>
struct EnergyAcc {
    __device__ void init(double, float, float) {}
};

template <>
struct EnergyAcc<COSMICA_PREC_MIXED, true> {
    m32::FF T, Lam;
    float m0, aoz;
    __device__ void init(double T0, float m0_, float aoz_)
    {
        T = m32::ff_from_double(T0);
        Lam.hi = 0.0f; Lam.lo = 0.0f;
        m0 = m0_; aoz = aoz_;
    }
    __device__ float fT() const { return T.hi; }
    __device__ void add(float dT, float dLam) { m32::ff_add(T, dT); m32::ff_add(Lam, dLam); }
    __device__ double T64() const { return m32::ff_to_double(T); }
    __device__ double lw() const { return -m32::ff_to_double(Lam); }
};

template <>
struct EnergyAcc<COSMICA_PREC_MIXED_F64ACC, true> {
    double T, Lam;
    float m0, aoz;
    __device__ void init(double T0, float m0_, float aoz_) { T = T0; Lam = 0.0; m0 = m0_; aoz = aoz_; }
    __device__ float fT() const { return narrow64(T); }
    __device__ void add(float dT, float dLam)
    {
        T += widen64(fminf(dT, 3.402823466e38f));   // an infinite T would be 1 to narrow(), 2^128 and more is infinite
        Lam += widen64(dLam);
    }
    __device__ double T64() const { return T; }
    __device__ double lw() const { return -Lam; }
};

// A path between two kernels of one launch: its exact state in its own exit record (float-float
// pairs and doubles both fill the record's 8-byte fields; the energy form keeps T in ln P's
// place and the loss integral in the weight's).
__device__ __forceinline__ double pair_bits(const m32::FF &a) { return __hiloint2double(__float_as_int(a.hi), __float_as_int(a.lo)); }
__device__ __forceinline__ m32::FF from_pair_bits(double v)
{
    m32::FF a;
    a.hi = __int_as_float(__double2hiint(v));
    a.lo = __int_as_float(__double2loint(v));
    return a;
}
template <bool EN>
__device__ __forceinline__ void park(const ExitPtrs &o, uint64_t g, const Acc<COSMICA_PREC_MIXED> &x,
                                     const EnergyAcc<COSMICA_PREC_MIXED, EN> &en)
{
    o.r[g] = pair_bits(x.r); o.th[g] = pair_bits(x.th); o.ph[g] = pair_bits(x.ph);
    o.s[g] = pair_bits(x.Ps.second());
    if constexpr (EN) {
        o.lnP[g] = pair_bits(en.T);
        o.lw[g] = pair_bits(en.Lam);
    } else {
        o.lnP[g] = pair_bits(x.Ps.first());
    }
}
template <bool EN>
__device__ __forceinline__ void unpark(const ExitPtrs &o, uint64_t g, Acc<COSMICA_PREC_MIXED> &x,
                                       EnergyAcc<COSMICA_PREC_MIXED, EN> &en)
{
    x.r = from_pair_bits(o.r[g]); x.th = from_pair_bits(o.th[g]); x.ph = from_pair_bits(o.ph[g]);
    x.Ps.set(EN ? x.Ps.first() : from_pair_bits(o.lnP[g]), from_pair_bits(o.s[g]));
    if constexpr (EN) {
        en.T = from_pair_bits(o.lnP[g]);
        en.Lam = from_pair_bits(o.lw[g]);
    }
}
template <bool EN>
__device__ __forceinline__ void park(const ExitPtrs &o, uint64_t g, const Acc<COSMICA_PREC_MIXED_F64ACC> &x,
                                     const EnergyAcc<COSMICA_PREC_MIXED_F64ACC, EN> &en)
{
    o.r[g] = x.r; o.th[g] = x.th; o.ph[g] = x.ph; o.s[g] = x.s;
    if constexpr (EN) {
        o.lnP[g] = en.T;
        o.lw[g] = en.Lam;
    } else {
        o.lnP[g] = x.lnP;
    }
}
template <bool EN>
__device__ __forceinline__ void unpark(const ExitPtrs &o, uint64_t g, Acc<COSMICA_PREC_MIXED_F64ACC> &x,
                                       EnergyAcc<COSMICA_PREC_MIXED_F64ACC, EN> &en)
{
    x.r = o.r[g]; x.th = o.th[g]; x.ph = o.ph[g]; x.s = o.s[g];
    if constexpr (EN) {
        en.T = o.lnP[g];
        en.Lam = o.lw[g];
    } else {
        x.lnP = o.lnP[g];
    }
}

}  // namespace cosmica
