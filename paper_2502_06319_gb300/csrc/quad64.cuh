// quad64.cuh -- one FP64 step by the four warps of a block, for the last paths of a launch.
//
// What bounds it: a launch ends with a handful of paths many times longer than the rest, and
// their step costs its FP64 instructions ("slots") times 64 clocks on one scheduler while the
// others idle (step64.cuh).  Here each block steps up to eight paths at once, one per team of
// four lanes, and its four warps -- one per scheduler -- take different parts of the same
// step; an exchange through shared memory costs about one slot.
//
//   warp 0  wind, sheet phase, sin/cos, atan, tanh of the sheet, drift, step length, update:
//           the step's serial chain, 242 slots
//   warp 1  sheet width and its gradient, drift geometry, derivatives of the sheet's argument
//   warp 2  tensor, Ito drift, Cholesky factor, noise
//   warp 3  normals of the next four steps (one step per lane), termination shock
//
// Everything up to the wind speed is evaluated by the first three warps alike, which costs
// nothing and saves an exchange.  Meetings: warps 0 and 1 after the atan (barrier 1), 2 and 3
// for the shock (barrier 2), all four before the drift and after the update.  The values are
// those of s64::step, operation by operation; a team whose new state is not finite, or outside
// that form's range, takes the plain step.  The isotropic model has no serial chain to speak
// of: warp 0 takes the step, warp 3 the normals and the shock.
//
// Include only from translation units built with -fmad=false.
#pragma once
#include "step64.cuh"

namespace cosmica {
namespace s64 {

constexpr int kQuadTeams = 8;

struct QuadShared {
    double tab[kFnWords];
    double st[kQuadTeams][5];          // r, th, ph, lnP, T
    double wide[kQuadTeams][2];        // 1 -> 0: sheet half-width, its reciprocal
    double wave[kQuadTeams][3];        // 0 -> 1: th_cs - th, sin and cos of the sheet's phase
    double geo[kQuadTeams][11];        // 1 -> 0
    double ten[kQuadTeams][16];        // 2 -> 0
    double shock[kQuadTeams][2];       // 3 -> 2 (isotropic: -> 0): g, dg/dr
    double z[2][kQuadTeams][4][3];     // 3 -> 2 (isotropic: -> 0)
    int live[2][kQuadTeams];           // by parity of the step: a warp may look while warp 0 is at its end
};

// barrier `id` of whole warps, `threads` in all
__device__ __forceinline__ void meet(int id, int threads)
{
    __syncwarp();
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// what the first three warps evaluate alike: P, theta's functions, the wind
struct Head {
    double P, beta, sn, cot, y_sn, y_r, V, dV;
};
template <bool BETA, bool DV>
__device__ __forceinline__ Head quad_head(const DevParams &p, const Spc &sp, const double *tab, const Team<4> team, double r,
                                          double th, double lnP)
{
    const F64Params &d = p.d;
    Head o;
    const double lat = 0.5 * kPi - th;
    const double wa = quot(from_bits(bits(lat) & 0x7FFFFFFFFFFFFFFFull) - d.lat_f, d.dlat, d.r_dlat);
    const double wabs = from_bits(bits(wa) & 0x7FFFFFFFFFFFFFFFull);
    const bool near = !lt(20.0, wabs);
    double ew, cs, y[4], q[4];
    team.functions(tab, lnP, near ? scale2<1>(wabs) : 0.0, th, o.P, ew, o.sn, cs);
    double pn = 0.0, root = 1.0;
    if constexpr (BETA) {
        pn = quot(o.P, sp.aoz, sp.raoz);
        root = sqrt(pn * pn + sp.m0sq);
    }
    const double ew1 = ew + 1.0;
    team.recip4(root, o.sn, r, ew1, y);
    o.y_sn = y[1];
    o.y_r = y[2];
    const double n[4] = {pn, cs, 2.0, 0.0}, b[4] = {root, o.sn, ew1, 1.0}, yy[4] = {y[0], y[1], y[3], 1.0};
    team.quot4(n, b, yy, q);
    o.beta = q[0];
    o.cot = q[1];
    const double t = neg_if(near ? 1.0 - q[2] : 1.0, __double2hiint(wa) < 0);
    o.V = d.Vs + d.hdV * (1.0 + t);
    o.dV = 0.0;
    if constexpr (DV) {
        o.dV = quot(d.hdV * (1.0 - t * t), d.dlat, d.r_dlat);
        o.dV = toward_equator(o.dV, lat);
    }
    return o;
}

// termination shock factor and its radial derivative
__device__ __forceinline__ void quad_shock(const DevParams &p, double r, double &g, double &dg)
{
    const F64Params &d = p.d;
    const double sa = quot(r - p.R_ts, p.dts, d.r_dts);
    const double sabs = from_bits(bits(sa) & 0x7FFFFFFFFFFFFFFFull);
    double t = 1.0;
    if (!lt(20.0, sabs)) {
        const double b = exp_in(scale2<1>(sabs)) + 1.0;
        t = 1.0 - quot(2.0, b, recip(b));
    }
    const double ts = neg_if(t, __double2hiint(sa) < 0);
    g = 1.0 - d.hts * (1.0 + ts);
    dg = neg_if(quot(d.hts * (1.0 - ts * ts), p.dts, d.r_dts), true);
}

// warp 1: everything of the drift but the sheet's own value
__device__ __forceinline__ void quad_drift(const DevParams &p, const Spc &sp, QuadShared &S, const Team<4> team, int tm,
                                           double r, double th, double lnP)
{
    const F64Params &d = p.d;
    const Head H = quad_head<true, true>(p, sp, S.tab, team, r, th, lnP);
    double y[4], q[4], gq[4];
    const double VV = H.V * H.V, Or = d.Omega * r, rr = r * r;
    team.recip4(H.V, VV, 1.0, 1.0, y);
    const double y_VV = y[1];
    {
        const double n[4] = {Or * H.sn, neg_if(Or * H.dV, true), d.Omega, H.dV}, b[4] = {H.V, VV, H.V, H.V}, yy[4] = {y[0], y_VV, y[0], y[0]};
        team.quot4(n, b, yy, q);
    }
    const double Gam = q[0], dphs_dth = q[1], dphs_dr = q[2];
    const double G2 = Gam * Gam, og = 1.0 + G2, gg = og * og;
    const double dGam_dth = Gam * (H.cot - q[3]);
    const double sog = sqrt(og);
    {
        const double n[4] = {H.P * 1e9, H.beta * H.P * 1e9 * kDay_s, 0.0, 0.0}, b[4] = {d.dDen, d.caDen, 1.0, 1.0},
                     yy[4] = {d.r_dDen, d.r_caDen, 1.0, 1.0};
        team.quot4(n, b, yy, q);
    }
    const double D = q[0], CA = q[1];
    const double D2r = scale2<1>(D) * r, ogs = og * sog;
    team.recip4(sog, ogs, og, gg, y);
    const double y_og = y[2], y_gg = y[3];
    {
        const double n[4] = {D2r, scale2<1>(D), neg_if(D2r * Gam * dGam_dth, true), 0.0}, b[4] = {sog, ogs, ogs, 1.0},
                     yy[4] = {y[0], y[1], y[1], 1.0};
        team.quot4(n, b, yy, q);
    }
    const bool rl = lt(d.dmin, q[0]);
    const double delta = rl ? q[0] : d.dmin;
    const double dd_dr = rl ? q[1] : 0.0, dd_dth = rl ? q[2] : 0.0;
    const double y_delta = recip(delta);
    if (team.l == 0) {
        S.wide[tm][0] = delta;
        S.wide[tm][1] = y_delta;
    }
    meet(1, 64);
    const double diff = S.wave[tm][0], sphs = S.wave[tm][1], cphs = S.wave[tm][2];
    const double den = 1.0 + d.ta2 * sphs * sphs;
    {
        const double n[4] = {d.ta * cphs, diff, 0.0, 0.0}, b[4] = {den, delta, 1.0, 1.0}, yy[4] = {recip(den), y_delta, 1.0, 1.0};
        team.quot4(n, b, yy, q);
    }
    const double dthcs = q[0], u = q[1];
    {
        const double n[4] = {dthcs * dphs_dr - u * dd_dr, dthcs * dphs_dth - 1.0 - u * dd_dth, dthcs, rr}, b[4] = {delta, delta, delta, og},
                     yy[4] = {y_delta, y_delta, y_delta, y_og};
        team.quot4(n, b, yy, q);
    }
    const double m1 = 1.0 - G2, r2G = rr * Gam;
    {
        const double n[4] = {neg_if(scale2<1>(r2G * dGam_dth), true), r * Gam * (3.0 + G2), rr * dGam_dth * m1, r2G}, b[4] = {gg, gg, gg, og},
                     yy[4] = {y_gg, y_gg, y_gg, y_og};
        team.quot4(n, b, yy, gq);
    }
    const double rd = r * delta;
    const double n3 = p.eps_diff * rd * rd;
    if (team.l == 0) {
        double *o = S.geo[tm];
        o[0] = q[0]; o[1] = q[1]; o[2] = q[2];               // d u / d(r, th, ph)
        o[3] = q[3]; o[4] = gq[3];                           // F, Gf
        o[5] = gq[0]; o[6] = gq[1]; o[7] = gq[2];            // dF_dth, dGf_dr, dGf_dth
        o[8] = CA;
        o[9] = n3;
    }
}

// warp 2: tensor, Ito drift, Cholesky factor times the normals
template <bool EN>
__device__ __forceinline__ void quad_tensor(const DevParams &p, const Spc &sp, QuadShared &S, const Team<4> team, int tm,
                                            double r, double th, double lnP, double T, const double *z)
{
    const F64Params &d = p.d;
    const Head H = quad_head<true, false>(p, sp, S.tab, team, r, th, lnP);
    double y[4], q[4];
    const double Or = d.Omega * r, rs = r * H.sn, rr = r * r, r3 = 3.0 * r;
    team.recip4(H.V, r3, rr, rs, y);
    const double y_rr = y[2], y_rs = y[3];
    {
        const double n[4] = {Or * H.sn, scale2<1>(H.V), 0.0, 0.0}, b[4] = {H.V, r3, 1.0, 1.0}, yy[4] = {y[0], y[1], 1.0, 1.0};
        team.quot4(n, b, yy, q);
    }
    const double Gam = q[0], dlnP = q[1];
    const double G2 = Gam * Gam, og = 1.0 + G2, gg = og * og;
    team.recip4(og, gg, 1.0, 1.0, y);
    {
        const double n[4] = {1.0, G2, Gam, Gam}, b[4] = {og, og, og, r}, yy[4] = {y[0], y[0], y[0], H.y_r};
        team.quot4(n, b, yy, q);
    }
    const double c2 = q[0], s2 = q[1], sc = q[2], dGam_dr = q[3];
    {
        const double n[4] = {neg_if(scale2<1>(Gam) * dGam_dr, true), dGam_dr * (1.0 - G2), 0.0, 0.0}, b[4] = {gg, gg, 1.0, 1.0},
                     yy[4] = {y[1], y[1], 1.0, 1.0};
        team.quot4(n, b, yy, q);
    }
    const double dc2 = q[0], dsc = q[1];
    const double Kbase = p.K0 * H.beta * H.P;
    const bool shock = positive(p.R_ts);
    meet(2, 64);
    const double g = S.shock[tm][0], dg = S.shock[tm][1];
    const double Kpar = shock ? Kbase * g : Kbase;
    const double dKpar = shock ? Kbase * dg : 0.0;
    const double Kpr = p.er * Kpar, Kpt = p.et * Kpar, dK = Kpr - Kpar;
    const double K00 = Kpar * c2 + Kpr * s2, K22 = Kpar * s2 + Kpr * c2, K02 = dK * sc, K11 = Kpt;
    double Kr00, Kr02;
    if (shock) {
        const double dKpr = p.er * dKpar;
        Kr00 = dKpar * c2 + Kpar * dc2 + dKpr * s2 + Kpr * neg_if(dc2, true);
        Kr02 = (dKpr - dKpar) * sc + dK * dsc;
    } else {
        Kr00 = Kpar * dc2 + Kpr * neg_if(dc2, true);
        Kr02 = dK * dsc;
    }
    double s4[4];
    team.sqrt4(scale2<1>(K00), scale2<1>(K11), 1.0, 1.0, s4);
    const double l00 = s4[0], l11 = s4[1];
    team.recip4(l00, K00, K11, 1.0, y);
    const double y_K00 = y[1], y_K11 = y[2];
    {
        const double n[4] = {scale2<1>(K02), scale2<1>(K00), K11 * H.cot, K02}, b[4] = {l00, r, rr, r}, yy[4] = {y[0], H.y_r, y_rr, H.y_r};
        team.quot4(n, b, yy, q);
    }
    const double l20 = q[0], Ar = Kr00 + q[1], Ath = q[2];
    const double Aph = quot(Kr02 + q[3], rs, y_rs);
    const double l22 = sqrt(scale2<1>(K22) - l20 * l20);
    double dTa = 0.0, dLa = 0.0;
    if constexpr (EN) {
        const double b = T + sp.m0;
        const double alpha = quot(T + 2.0 * sp.m0, b, recip(b));
        dTa = dlnP * alpha * T;
        dLa = dlnP * (1.0 + H.beta * H.beta);
    }
    const double num = d.eps_adv2 * K00, n2 = p.eps_diff * r * r;
    const double Lz_r = l00 * z[0], Lz_th = l11 * z[1], Lz_ph = l20 * z[0] + l22 * z[2];
    if (team.l == 0) {
        double *o = S.ten[tm];
        o[0] = Ar - H.V; o[1] = Ath; o[2] = Aph; o[3] = dlnP;
        o[4] = Lz_r; o[5] = Lz_th; o[6] = Lz_ph;
        o[7] = num; o[8] = n2; o[9] = K00; o[10] = y_K00; o[11] = K11; o[12] = y_K11;
        o[13] = dTa; o[14] = dLa;
    }
}

// the end of a step, common to both models: new angles into their ranges, status
__device__ __forceinline__ void quad_close(const DevParams &p, m64::State &o, uint32_t max_steps)
{
    if (f64bits::less(bits(o.r), bits(p.r_in)) | f64bits::outside_closed(bits(o.th), f64bits::kPiBits) |
        f64bits::outside_half_open(bits(o.ph), f64bits::kTwoPiBits))
        into_range(p, o);
    o.k += 1u;
    o.status = !lt(o.r, p.R_out) ? COSMICA_PATH_EXIT : (o.k >= max_steps ? COSMICA_PATH_STEP_LIMIT : COSMICA_PATH_RUNNING);
}

// warp 0 of the anisotropic model
template <bool EN>
__device__ __forceinline__ void quad_chain(const DevParams &p, const DevSpecies &dsp, const Spc &sp, uint64_t seed, uint64_t pid,
                                           uint32_t max_steps, QuadShared &S, const Team<4> team, int tm, bool live,
                                           m64::State &x)
{
    const F64Params &d = p.d;
    const double r = x.r, th = x.th;
    const Head H = quad_head<false, false>(p, sp, S.tab, team, r, th, x.lnP);
    bool odd_range = beyond(x.lnP, kFarLnP) | odd_theta(th);
    double y[4], q[4];
    const double Or = d.Omega * r, rs = r * H.sn;
    team.recip4(H.V, rs, 1.0, 1.0, y);
    const double y_rs = y[1];
    const double phs = x.ph + quot(Or, H.V, y[0]);
    odd_range |= beyond(phs, kFarAngle);
    double sphs, cphs;
    team.sincos(S.tab, phs, sphs, cphs);
    const double diff = (0.5 * kPi + atan_in(d.ta * sphs)) - th;
    if (team.l == 0) {
        S.wave[tm][0] = diff;
        S.wave[tm][1] = sphs;
        S.wave[tm][2] = cphs;
    }
    meet(1, 64);
    const double u = quot(diff, S.wide[tm][0], S.wide[tm][1]);
    const double uabs = from_bits(bits(u) & 0x7FFFFFFFFFFFFFFFull);
    double t = 1.0;
    if (!lt(20.0, uabs)) {
        const double b = exp_in(scale2<1>(uabs)) + 1.0;
        t = 1.0 - quot(2.0, b, recip(b));
    }
    const bool hcs = on(p.hcs_on), drift = on(p.drift_on);
    const double h = hcs ? neg_if(t, __double2hiint(u) < 0) : 1.0;
    const double w = hcs ? 1.0 - h * h : 0.0;
    meet(3, 128);
    const double *go = S.geo[tm], *te = S.ten[tm];
    const double F = go[3], Gf = go[4], CA = go[8], nCA = neg_if(CA, true);
    // gradient of h, then the three derivatives of the potential and its longitude term
    const double dh = hcs ? w * team.pick(go[0], go[1], go[2], 0.0) : 0.0;
    const double dh_dr = team.get(dh, 0), dh_dth = team.get(dh, 1), dh_dph = team.get(dh, 2);
    const double a = team.pick(dh_dth, dh_dr, dh_dth, CA) * team.pick(Gf, Gf, F, dh_dph);
    const double c = h * team.pick(go[7], go[6], go[5], 0.0);
    const double v = team.pick(nCA, nCA, CA, F) * (a + c);
    const double dWph_dth = team.get(v, 0), dWph_dr = team.get(v, 1), dWr_dth = team.get(v, 2), dWr_dph = team.get(v, 3);
    const double Wph = nCA * h * Gf;
    const double m = team.pick(H.cot, r, 0.0, 0.0) * team.pick(Wph, dWph_dr, 0.0, 0.0);
    {
        const double n[4] = {team.get(m, 0) + dWph_dth, quot(dWr_dph, H.sn, H.y_sn) - Wph - team.get(m, 1), neg_if(dWr_dth, true), 0.0},
                     b[4] = {r, r, r, 1.0}, yy[4] = {H.y_r, H.y_r, H.y_r, 1.0};
        team.quot4(n, b, yy, q);
    }
    const bool s = sp.negative != (__double2hiint(p.polarity) < 0);
    const double vd0 = drift ? neg_if(q[0], s) : 0.0, vd1 = drift ? neg_if(q[1], s) : 0.0, vd2 = drift ? neg_if(q[2], s) : 0.0;

    // step length
    const double Ar_tot = te[0] - vd0;
    const double den = Ar_tot * Ar_tot;
    double dt = p.dt_max;
    {
        const double n[4] = {te[7], te[8], go[9], 0.0}, b[4] = {den, te[9], te[11], 1.0}, yy[4] = {recip(den), te[10], te[12], 1.0};
        team.quot4(n, b, yy, q);
    }
    if (lt(te[7], dt * den)) dt = q[0];
    if (lt(q[1], dt)) dt = q[1];
    if (hcs && drift && lt(q[2], dt)) dt = q[2];
    if (lt(dt, p.dt_min)) dt = p.dt_min;
    if (positive(p.dt_fixed)) dt = p.dt_fixed;
    const double sdt = sqrt(dt);

    // update: lanes 0 to 3 take r, theta, phi, ln P
    const double e = team.pick(te[4], te[4], te[5], te[6]) * sdt;
    {
        const double n[4] = {vd1, vd2, e, e}, b[4] = {r, rs, r, rs}, yy[4] = {H.y_r, y_rs, H.y_r, y_rs};
        team.quot4(n, b, yy, q);
    }
    const double A = team.pick(Ar_tot, te[1], te[2], te[3]) - team.pick(0.0, q[0], q[1], 0.0);
    const double next = team.pick(r, th, x.ph, x.lnP) + (A * dt + team.pick(team.get(e, 0), q[2], q[3], 0.0));
    m64::State o = x;
    o.r = team.get(next, 0);
    o.th = team.get(next, 1);
    o.ph = team.get(next, 2);
    o.lnP = team.get(next, 3);
    if constexpr (EN) {
        o.T = x.T + te[13] * dt;
        o.Lam = x.Lam + te[14] * dt;
        o.lnP = log_in(sp.aoz * sqrt(o.T * (o.T + 2.0 * sp.m0)));
    }
    o.s = x.s + dt;
    o.r_old = r;
    quad_close(p, o, max_steps);
    if (live) {
        if (finite_state<EN>(o) & !odd_range) x = o;
        else x = plain_step(p, dsp, seed, pid, x);
    }
}

// warp 0 of the isotropic model
template <bool EN>
__device__ __forceinline__ void quad_isotropic(const DevParams &p, const DevSpecies &dsp, const Spc &sp, uint64_t seed,
                                               uint64_t pid, uint32_t max_steps, QuadShared &S, const Team<4> team, int tm,
                                               const double *z, bool live, m64::State &x)
{
    const F64Params &d = p.d;
    const double r = x.r, th = x.th, V = d.Vs;
    const bool odd_range = beyond(x.lnP, kFarLnP) | odd_theta(th);
    double P, unused, sn, cs, y[4], y2[4], q[4];
    team.functions(S.tab, x.lnP, 0.0, th, P, unused, sn, cs);
    const double pn = quot(P, sp.aoz, sp.raoz);
    const double root = sqrt(pn * pn + sp.m0sq);
    const double rs = r * sn, rr = r * r, r3 = 3.0 * r;
    team.recip4(root, sn, r, rs, y);
    team.recip4(rr, r3, 1.0, 1.0, y2);
    {
        const double n[4] = {pn, cs, scale2<1>(V), 0.0}, b[4] = {root, sn, r3, 1.0}, yy[4] = {y[0], y[1], y2[1], 1.0};
        team.quot4(n, b, yy, q);
    }
    const double beta = q[0], cot = q[1], dlnP = q[2];
    const double Kbase = p.K0 * beta * P;
    meet(2, 64);
    const bool shock = positive(p.R_ts);
    const double K = shock ? Kbase * S.shock[tm][0] : Kbase;
    const double dK = shock ? Kbase * S.shock[tm][1] : 0.0;
    {
        const double n[4] = {scale2<1>(K), K * cot, 0.0, 0.0}, b[4] = {r, rr, 1.0, 1.0}, yy[4] = {y[2], y2[0], 1.0, 1.0};
        team.quot4(n, b, yy, q);
    }
    const double Ar_tot = (dK + q[0]) - V, Ath = q[1];
    const double l = sqrt(scale2<1>(K));
    double dt = p.dt_fixed, sdt = d.sdt_fixed;
    const bool fixed = positive(p.dt_fixed);
    if (team.any(!fixed)) {
        double a = p.dt_max;
        const double num = d.eps_adv2 * K, den = Ar_tot * Ar_tot, n2 = p.eps_diff * r * r;
        team.recip4(den, K, 1.0, 1.0, y2);
        const double n[4] = {num, n2, 0.0, 0.0}, b[4] = {den, K, 1.0, 1.0}, yy[4] = {y2[0], y2[1], 1.0, 1.0};
        team.quot4(n, b, yy, q);
        if (lt(num, a * den)) a = q[0];
        if (lt(q[1], a)) a = q[1];
        if (lt(a, p.dt_min)) a = p.dt_min;
        if (!fixed) {
            dt = a;
            sdt = sqrt(a);
        }
    }
    const double e = l * team.pick(z[0], z[1], z[2], 0.0) * sdt;
    const double ends = quot(e, team.pick(1.0, r, rs, 1.0), team.pick(1.0, y[2], y[3], 1.0));
    // lanes 0 to 3 take r, theta, phi, ln P; nothing drives phi but its noise
    const double A = team.pick(Ar_tot, Ath, 0.0, dlnP);
    const double next = team.pick(r, th, x.ph, x.lnP) + (A * dt + team.pick(e, ends, ends, 0.0));
    m64::State o = x;
    o.r = team.get(next, 0);
    o.th = team.get(next, 1);
    o.ph = team.get(next, 2);
    o.lnP = team.get(next, 3);
    if constexpr (EN) {
        const double b = x.T + sp.m0;
        const double alpha = quot(x.T + 2.0 * sp.m0, b, recip(b));
        o.T = x.T + dlnP * alpha * x.T * dt;
        o.Lam = x.Lam + dlnP * (1.0 + beta * beta) * dt;
        o.lnP = log_in(sp.aoz * sqrt(o.T * (o.T + 2.0 * sp.m0)));
    }
    o.s = x.s + dt;
    o.r_old = r;
    quad_close(p, o, max_steps);
    if (live) {
        if (finite_state<EN>(o) & !odd_range) x = o;
        else x = plain_step(p, dsp, seed, pid, x);
    }
}

}  // namespace s64
}  // namespace cosmica
