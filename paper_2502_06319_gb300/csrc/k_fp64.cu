// k_fp64.cu -- FP64 kernels.  Built with -fmad=false: every FP64 expression
// is evaluated exactly as written (no fused multiply-add contraction).
//
//   k_derive          per-parameter-set constants (FP64 and the FP32 block)
//   k_propagate64     the FP64 path: one lane per quasi-particle (Sec. IV.A), refilled from
//                     the work queue, Euler-Maruyama until the path exits (step64.cuh)
//   k_finish64, k_quad64
//                     the last paths of a launch, or all of a small one: teams of lanes,
//                     then the four warps of a block
//   k_propagate_fp64  sets with radial shells or a squashed heliosphere, or with constants
//                     outside the fast step's range: one thread per quasi-particle, the step
//                     as it is defined (model64.cuh)
//   k_debug_*         coefficient / RNG / elementary-function probes used by
//                     the tests through cosmica_debug.h
#include <algorithm>
#include <cstdint>

#include "common.cuh"
#include "internal.h"
#include "model64.cuh"
#include "quad64.cuh"
#include "step64.cuh"

namespace cosmica {

__global__ void k_derive(DevParams *prm, uint32_t n)
{
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    DevParams &p = prm[i];
    const bool iso = p.isotropic != 0.0;
    p.B0 = iso ? 0.0 : m64::field_B0(p);
    // (a spheroid's points are within its tail distance and its flank semi-axis of the Sun, together)
    p.vote_lo = f64bits::vote_floor((float)p.r_in, (float)(p.squashed != 0.0 ? p.R_out * (1.0 + p.hp_tail + p.hp_flank) : p.R_out));
    {
        // in the operations of model64.cuh
        F64Params &d = p.d;
        const double Vs64 = iso ? p.V_const_kms * kDay_s / kAU_km : p.Vs_kms * kDay_s / kAU_km;
        const double Vf64 = p.Vf_kms * kDay_s / kAU_km;
        d.Vs = Vs64;
        d.hdV = iso ? 0.0 : (Vf64 - Vs64) * 0.5;
        d.lat_f = p.lat_fast_deg * kDeg;
        d.dlat = p.dlat_deg * kDeg;
        d.r_dlat = 1.0 / d.dlat;
        d.Omega = iso ? 0.0 : kTwoPi / p.rot_period;
        d.hts = (1.0 - p.ts_f) * 0.5;
        d.r_dts = 1.0 / p.dts;
        double s64, c64;
        dm::sincos(p.tilt_deg * kDeg, &s64, &c64);
        d.ta = s64 / c64;
        d.ta2 = d.ta * d.ta;
        d.dmin = p.dcs_min_deg * kDeg;
        d.dDen = kC_ms * p.B0 * 1e-9 * kAU_m;
        d.r_dDen = 1.0 / d.dDen;
        d.caDen = 3.0 * p.B0 * 1e-9 * kAU_m * kAU_m;
        d.r_caDen = 1.0 / d.caDen;
        d.eps_adv2 = p.eps_adv * 2.0;
        d.sdt_fixed = p.dt_fixed > 0.0 ? sqrt(p.dt_fixed) : 0.0;
    }
    F32Params &f = p.f;
    const double Vs = iso ? p.V_const_kms * kDay_s / kAU_km : p.Vs_kms * kDay_s / kAU_km;
    const double Vf = iso ? Vs : p.Vf_kms * kDay_s / kAU_km;
    f.Vs = (float)Vs;
    f.dV = (float)(Vf - Vs);
    f.lat_f = (float)(p.lat_fast_deg * kDeg);
    f.inv_dlat = (float)(1.0 / (p.dlat_deg * kDeg));
    f.Omega = iso ? 0.0f : (float)(kTwoPi / p.rot_period);
    f.K0 = (float)p.K0;
    f.er = iso ? 1.0f : (float)p.er;
    f.et = iso ? 1.0f : (float)p.et;
    f.ts_drop = (p.R_ts > 0.0) ? (float)(1.0 - p.ts_f) : 0.0f;
    f.R_ts = (float)p.R_ts;
    f.inv_dts = (float)(1.0 / p.dts);
    f.r_in = (float)p.r_in;
    f.dt_max = (float)p.dt_max;
    f.dt_fixed = (float)p.dt_fixed;
    f.dt_min = (float)p.dt_min;
    f.eps_adv2 = (float)(2.0 * p.eps_adv);
    f.eps_diff = (float)p.eps_diff;
    const bool drift = !iso && p.drift_on != 0.0;
    const bool hcs = drift && p.hcs_on != 0.0;
    f.CA0 = drift ? (float)(1e9 * kDay_s / (3.0 * p.B0 * 1e-9 * kAU_m * kAU_m)) : 0.0f;
    f.D2 = iso ? 0.0f : (float)(2.0 * 1e9 / (kC_ms * p.B0 * 1e-9 * kAU_m));
    f.dcs_min = (float)(p.dcs_min_deg * kDeg);
    double sa, ca;
    dm::sincos(p.tilt_deg * kDeg, &sa, &ca);
    const double ta = sa / ca;
    f.ta = (float)ta;
    f.ta2 = (float)(ta * ta);
    f.polarity = (float)p.polarity;
    f.drift = drift ? 1.0f : 0.0f;
    f.hcs = hcs ? 1.0f : 0.0f;
    f.sqrt2er = (float)sqrt(2.0 * (double)f.er);
    f.pad0 = f.pad1 = 0.0f;
    const int ns = (int)p.n_shells;
    const double dR = ns > 0 ? ((p.R_ts > 0.0) ? p.R_ts : p.R_out) / ns : 1.0;
    f.n_sh = (float)ns;
    f.sh_dr = (float)dR;
    f.sh_inv_dr = (float)(1.0 / dR);
    f.sh_w = (float)p.shell_w;
    f.sh_inv_2w = ns > 1 ? (float)(1.0 / (2.0 * p.shell_w)) : 0.0f;
    f.pad2 = f.pad3 = f.pad4 = 0.0f;
    for (int k = 0; k < COSMICA_MAX_SHELLS; ++k) {
        f.sh_K0[k] = (float)p.shell_K0[k];
        f.sh_alpha[k] = (float)(p.shell_tilt_deg[k] * kDeg);
    }
    const bool sq = p.squashed != 0.0;
    f.sq = sq ? 1.0f : 0.0f;
    f.nose_ph = (float)(p.nose_ph - kTwoPi * floor(p.nose_ph / kTwoPi));
    f.sin_nth = (float)sin(p.nose_th);
    f.cos_nth = (float)cos(p.nose_th);
    {
        // shock spheroid with unit nose distance (scaled by ts_R), outer spheroid in AU
        const double a = (1.0 + p.ts_tail) / 2.0, b = p.ts_flank, c = (p.ts_tail - 1.0) / 2.0;
        f.ts_R = (float)p.R_ts;
        f.ts_c = (float)c;
        f.ts_ia2 = (float)(1.0 / (a * a));
        f.ts_ib2 = (float)(1.0 / (b * b));
        f.ts_C = (float)(c * c / (a * a) - 1.0);
        const double A = p.R_out * (1.0 + p.hp_tail) / 2.0, B = p.R_out * p.hp_flank;
        f.hp_c = (float)(p.R_out * (p.hp_tail - 1.0) / 2.0);
        f.hp_ia2 = (float)(1.0 / (A * A));
        f.hp_ib2 = (float)(1.0 / (B * B));
    }
}

__global__ void __launch_bounds__(128) k_propagate_fp64(const DevParams *__restrict__ prm,
                                                        const DevSpecies *__restrict__ spc,
                                                        const DevItem *__restrict__ items,
                                                        const uint64_t *__restrict__ prefix,
                                                        uint32_t n_items, uint64_t n_total,
                                                        ExitPtrs out,
                                                        unsigned long long *__restrict__ steps_total)
{
    const uint64_t g = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    unsigned long long my_steps = 0;
    if (g < n_total) {
        const uint32_t it = find_item(prefix, n_items, g);
        const DevItem item = items[it];
        const DevParams &p = prm[item.param_idx];
        const DevSpecies sp = spc[item.species_idx];
        const uint64_t pid = item.first_pid + (g - prefix[it]);
        m64::State x;
        m64::init_state(sp, item.T, item.r0, item.th0, item.ph0, x);
        while (x.status == COSMICA_PATH_RUNNING) m64::em_step(p, sp, item.seed, pid, x);
        out.r[g] = x.r;
        out.th[g] = x.th;
        out.ph[g] = x.ph;
        out.lnP[g] = x.lnP;
        out.s[g] = x.s;
        out.steps[g] = x.k;
        out.status[g] = (uint8_t)x.status;
        out.item[g] = item.out_item;
        if (out.lw) out.lw[g] = -x.Lam;
        my_steps = x.k;
    }
    if (steps_total) {
        for (int o = 16; o > 0; o >>= 1) my_steps += __shfl_down_sync(0xffffffffu, my_steps, o);
        if ((threadIdx.x & 31) == 0 && my_steps) atomicAdd(steps_total, my_steps);
    }
}

// ---- FP64 paths of the models without shells or squashing -----------------------------
// Bound by the FP64 pipe: a step costs its slots times 64 clocks on the warp's scheduler
// whatever lanes are active (step64.cuh), so
//   * one warp per scheduler (one block of 128 per SM) already fills the pipe; lanes whose
//     path ended take the next one from the queue, most expensive items first;
//   * once no more than 32 paths per SM are left, every lane stores its path in its own exit
//     record and k_finish64 takes them over with four lanes a path, which halves the slots of
//     the step that the launch's slowest paths wait for;
//   * once no more than 8 per SM are left, k_quad64 takes them over with the four warps of a
//     block for up to eight paths (quad64.cuh), which halves the slots on the longest warp again.
// A launch that starts with so few paths starts there.  (A mixture of isotropic and other sets
// stays with k_finish64.)
// Measured against one thread per path with the plain step: a step of the full model 52 us, 29 in
// k_propagate64 (a lane a path), 17.4 in k_finish64 (477 slots, the FP64 pipe 84 % busy), 10.0 in
// k_quad64 (242 slots on its longest warp); 1e4 isotropic paths 91.5 -> 24.0 ms, 2.5e4 paths of the
// full model 1371 -> 318 ms.  The paths are the same bits.
struct Path64 {
    uint64_t g, pid, seed;
    const DevParams *p;
    const DevSpecies *dsp;
    uint32_t out_item, max_steps;
    s64::Spc sp;
};

__device__ __forceinline__ void locate64(const LaunchArgs &a, uint32_t it, uint64_t local, Path64 &P, DevItem &item)
{
    item = a.items[it];
    P.g = a.prefix[it] + local;
    P.pid = item.first_pid + local;
    P.seed = item.seed;
    P.p = a.prm + item.param_idx;
    P.dsp = a.spc + item.species_idx;
    P.out_item = item.out_item;
    P.max_steps = (uint32_t)P.p->max_steps;
    P.sp = s64::make_spc(*P.dsp);
}

// the path in queue slot q, at its start
__device__ __forceinline__ void fresh64(const LaunchArgs &a, uint64_t q, Path64 &P, m64::State &x)
{
    const uint32_t iq = find_item(a.qprefix, a.n_items, q);
    DevItem item;
    locate64(a, a.qitem ? a.qitem[iq] : iq, q - a.qprefix[iq], P, item);
    m64::init_state(*P.dsp, item.T, item.r0, item.th0, item.ph0, x);
}

// the path whose state waits in exit record g (EN: lnP's place holds T, which gives lnP)
template <bool EN>
__device__ __forceinline__ void stored64(const LaunchArgs &a, uint64_t g, Path64 &P, m64::State &x)
{
    const uint32_t it = find_item(a.prefix, a.n_items, g);
    DevItem item;
    locate64(a, it, g - a.prefix[it], P, item);
    m64::init_state(*P.dsp, item.T, item.r0, item.th0, item.ph0, x);
    x.r = a.out.r[g];
    x.th = a.out.th[g];
    x.ph = a.out.ph[g];
    x.s = a.out.s[g];
    x.k = a.out.steps[g];
    x.lnP = a.out.lnP[g];
    if constexpr (EN) {
        x.T = x.lnP;
        x.Lam = -a.out.lw[g];
        x.lnP = dm::log(P.dsp->A / fabs(P.dsp->Z) * sqrt(x.T * (x.T + 2.0 * P.dsp->m0)));
    }
}

template <bool EN>
__device__ __forceinline__ void store64(const ExitPtrs &out, const Path64 &P, const m64::State &x)
{
    const uint64_t g = P.g;
    out.r[g] = x.r;
    out.th[g] = x.th;
    out.ph[g] = x.ph;
    out.lnP[g] = EN && x.status == COSMICA_PATH_RUNNING ? x.T : x.lnP;
    out.s[g] = x.s;
    out.steps[g] = x.k;
    out.status[g] = (uint8_t)x.status;
    out.item[g] = P.out_item;
    if (out.lw) out.lw[g] = -x.Lam;
}

// ISO: 1 every set is isotropic, 0 none, 2 both occur
template <int G, int ISO, bool EN>
__device__ __forceinline__ void step64(const Path64 &P, const double *tab, s64::Team<G> team, const double (&z)[3], bool live,
                                       m64::State &x)
{
    if constexpr (ISO == 2) {
        // teams of a warp may hold different models: all of them run each form that one of them needs
        // (its shuffles take the whole warp), and each keeps its own
        const bool iso = s64::on(P.p->isotropic);
        if (G == 1 ? iso : __any_sync(0xffffffffu, iso))
            s64::step<G, true, EN>(*P.p, *P.dsp, P.sp, P.seed, P.pid, P.max_steps, tab, team, z, live && iso, x);
        if (G == 1 ? !iso : __any_sync(0xffffffffu, !iso))
            s64::step<G, false, EN>(*P.p, *P.dsp, P.sp, P.seed, P.pid, P.max_steps, tab, team, z, live && !iso, x);
    } else {
        s64::step<G, ISO == 1, EN>(*P.p, *P.dsp, P.sp, P.seed, P.pid, P.max_steps, tab, team, z, live, x);
    }
}

template <int ISO, bool EN>
__global__ void __launch_bounds__(128) k_propagate64(LaunchArgs a, uint32_t limit)
{
    const unsigned lane = threadIdx.x & 31u;
    Path64 P;
    m64::State x;
    bool active = false, drained = false;
    uint32_t tick = 0;
    unsigned long long my_steps = 0;
    while (true) {
        const unsigned need = __ballot_sync(0xffffffffu, !active && !drained);
        if (need) {
            unsigned long long base = 0;
            const unsigned leader = __ffs(need) - 1;
            if (lane == leader) base = atomicAdd(a.cursor, (unsigned long long)__popc(need));
            base = __shfl_sync(0xffffffffu, base, leader);
            if (need & (1u << lane)) {
                const uint64_t q = base + __popc(need & ((1u << lane) - 1u));
                if (q < a.n_total) {
                    fresh64(a, q, P, x);
                    active = true;
                }
            }
            if (base + __popc(need) > a.n_total) drained = true;   // a refused lane never asks again
        }
        if (!__any_sync(0xffffffffu, active)) {
            if (drained) break;
            continue;
        }
        // few enough paths left, all of them taken from the queue: hand them over (asked every 8 steps)
        if (limit && (++tick & 7u) == 0u) {
            unsigned few = 0;
            if (lane == 0)
                few = a.n_total - *(volatile unsigned long long *)a.ended <= limit &&
                      *(volatile unsigned long long *)a.cursor >= a.n_total;
            if (__shfl_sync(0xffffffffu, few, 0)) {
                if (active) {
                    store64<EN>(a.out, P, x);
                    a.list[atomicAdd(a.ended + 1, 1ull)] = (uint32_t)P.g;   // at most `limit` paths are left
                }
                break;
            }
        }
        bool end = false;
        if (active) {
            double z[3];
            s64::normals(P.seed, P.pid, x.k, z);
            step64<1, ISO, EN>(P, nullptr, s64::Team<1>{0}, z, true, x);
            end = x.status != COSMICA_PATH_RUNNING;
            if (end) {
                store64<EN>(a.out, P, x);
                my_steps += x.k;
                active = false;
            }
        }
        const unsigned ends = __ballot_sync(0xffffffffu, end);
        if (limit && ends && lane == 0) atomicAdd(a.ended, (unsigned long long)__popc(ends));
    }
    if (a.steps_total) {
        for (int o = 16; o > 0; o >>= 1) my_steps += __shfl_down_sync(0xffffffffu, my_steps, o);
        if (lane == 0 && my_steps) atomicAdd(a.steps_total, my_steps);
    }
}

// Teams of G lanes; team j of warp w takes entry j * warps + w, so that the schedulers share the
// paths evenly.  from: null for the queue's paths from their start, else *n_from indices of
// stored paths.  The last `limit` paths are left to the next kernel (if every path has a team of
// its own: a path that waits for one cannot be left).
template <int G, int ISO, bool EN>
__global__ void __launch_bounds__(128) k_finish64(LaunchArgs a, const uint32_t *from, const unsigned long long *n_from,
                                                  uint32_t *to, unsigned long long *n_to, uint32_t limit)
{
    __shared__ double tab[s64::kFnWords];
    s64::load_table(tab);
    __syncthreads();
    const uint64_t n = from ? *n_from : a.n_total;
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t warps = gridDim.x * (blockDim.x / 32), warp = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
    const s64::Team<G> team{(int)(lane & (G - 1))};
    const bool hand_over = limit != 0 && n <= (uint64_t)warps * (32 / G);
    unsigned long long my_steps = 0;
    for (uint64_t first = warp; first < n; first += (uint64_t)warps * (32 / G)) {
        // a team without a path of its own follows the warp's first one and writes nothing
        uint64_t i = first + (uint64_t)(lane / G) * warps;
        bool live = i < n;
        if (!live) i = first;
        Path64 P;
        m64::State x;
        if (!from) fresh64(a, i, P, x);
        else stored64<EN>(a, from[i], P, x);
        double zs[3];          // normals of step (first of the round) + team lane
        for (uint32_t it = 0; __any_sync(0xffffffffu, live); ++it) {
            if (hand_over && it % 16 == 15) {
                unsigned few = 0;
                if (lane == 0) few = a.n_total - *(volatile unsigned long long *)a.ended <= limit;
                if (__shfl_sync(0xffffffffu, few, 0)) {
                    if (live && team.l == 0) {
                        store64<EN>(a.out, P, x);
                        to[atomicAdd(n_to, 1ull)] = (uint32_t)P.g;   // no more than `limit` paths are left
                    }
                    break;
                }
            }
            if (it % G == 0) s64::normals(P.seed, P.pid, x.k + (uint32_t)team.l, zs);
            const int j = (int)(it % G);
            const double z[3] = {team.get(zs[0], j), team.get(zs[1], j), team.get(zs[2], j)};
            step64<G, ISO, EN>(P, tab, team, z, live, x);
            const bool end = live && x.status != COSMICA_PATH_RUNNING;
            if (end) {
                if (team.l == 0) {
                    store64<EN>(a.out, P, x);
                    my_steps += x.k;
                }
                live = false;
            }
            const unsigned ends = __ballot_sync(0xffffffffu, end && team.l == 0);
            if (hand_over && ends && lane == 0) atomicAdd(a.ended, (unsigned long long)__popc(ends));
        }
    }
    if (a.steps_total && my_steps) atomicAdd(a.steps_total, my_steps);
}

// One block of four warps for up to eight paths: team j of every warp holds path
// j * gridDim.x + blockIdx.x (quad64.cuh).  Shared memory carries the state from warp 0, which
// owns the paths, to the others.
template <bool ISO, bool EN>
__global__ void __launch_bounds__(128, 1) k_quad64(LaunchArgs a, const uint32_t *from, const unsigned long long *n_from)
{
    __shared__ s64::QuadShared S;
    s64::load_table(S.tab);
    const uint64_t n = from ? *n_from : a.n_total;
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const int tm = (int)(lane >> 2);
    const s64::Team<4> team{(int)(lane & 3u)};
    unsigned long long my_steps = 0;
    for (uint64_t first = blockIdx.x; first < n; first += (uint64_t)gridDim.x * s64::kQuadTeams) {
        // a team without a path of its own follows the block's first one and writes nothing
        uint64_t i = first + (uint64_t)tm * gridDim.x;
        bool live = i < n;
        if (!live) i = first;
        Path64 P;
        m64::State x;
        if (!from) fresh64(a, i, P, x);
        else stored64<EN>(a, from[i], P, x);
        const uint32_t k0 = x.k;
        auto draw = [&](uint32_t batch) {      // normals of steps k0 + 4 batch + (0 .. 3)
            double z[3];
            s64::normals(P.seed, P.pid, k0 + 4u * batch + (uint32_t)team.l, z);
            for (int c = 0; c < 3; ++c) S.z[batch & 1u][tm][team.l][c] = z[c];
        };
        auto publish = [&](uint32_t it) {       // the state at the beginning of step `it`
            if (team.l == 0) {
                double *st = S.st[tm];
                st[0] = x.r; st[1] = x.th; st[2] = x.ph; st[3] = x.lnP; st[4] = x.T;
                S.live[it & 1u][tm] = live;
            }
        };
        if (warp == 0) publish(0);
        if (warp == 3) draw(0);
        s64::meet(3, 128);
        for (uint32_t it = 0;; ++it) {
            int any = 0;
            for (int j = 0; j < s64::kQuadTeams; ++j) any |= S.live[it & 1u][j];
            if (!any) break;       // the same answer in all four warps
            const double *st = S.st[tm];
            const double *z = S.z[(it >> 2) & 1u][tm][it & 3u];
            if (warp == 0) {
                if constexpr (ISO) s64::quad_isotropic<EN>(*P.p, *P.dsp, P.sp, P.seed, P.pid, P.max_steps, S, team, tm, z, live, x);
                else s64::quad_chain<EN>(*P.p, *P.dsp, P.sp, P.seed, P.pid, P.max_steps, S, team, tm, live, x);
                if (live && x.status != COSMICA_PATH_RUNNING) {
                    if (team.l == 0) {
                        store64<EN>(a.out, P, x);
                        my_steps += x.k;
                    }
                    live = false;
                }
                publish(it + 1u);
            } else if (warp == 3) {
                double g = 1.0, dg = 0.0;
                if (s64::positive(P.p->R_ts)) s64::quad_shock(*P.p, st[0], g, dg);
                if (team.l == 0) {
                    S.shock[tm][0] = g;
                    S.shock[tm][1] = dg;
                }
                s64::meet(2, 64);
                if ((it & 3u) == 0u) draw((it >> 2) + 1u);
                if constexpr (!ISO) s64::meet(3, 128);
            } else if constexpr (!ISO) {
                if (warp == 1) s64::quad_drift(*P.p, P.sp, S, team, tm, st[0], st[1], st[3]);
                else s64::quad_tensor<EN>(*P.p, P.sp, S, team, tm, st[0], st[1], st[3], st[4], z);
                s64::meet(3, 128);
            }
            s64::meet(3, 128);
        }
        s64::meet(3, 128);     // before the next round's paths are published
    }
    if (a.steps_total && my_steps) atomicAdd(a.steps_total, my_steps);
}

// ---------------------------------------------------------------- debug --
__global__ void k_debug_eval64(const DevParams *__restrict__ prm, const DevSpecies *__restrict__ spc,
                               uint32_t n, const double *__restrict__ st, double *__restrict__ out)
{
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    m64::Coef c;
    m64::eval(prm[0], spc[0], st[4 * i + 0], st[4 * i + 1], st[4 * i + 2], st[4 * i + 3], c);
    double *o = out + (size_t)i * kDebugEvalN;
    o[0] = c.V;   o[1] = c.Gam;  o[2] = c.Kpar; o[3] = c.K00;  o[4] = c.K11;  o[5] = c.K22;
    o[6] = c.K02; o[7] = c.Ar;   o[8] = c.Ath;  o[9] = c.Aph;  o[10] = c.l00; o[11] = c.l11;
    o[12] = c.l20; o[13] = c.l22; o[14] = c.h;  o[15] = c.delta_cs;
    o[16] = c.vd0; o[17] = c.vd1; o[18] = c.vd2; o[19] = c.dlnP; o[20] = c.dt;
}

__global__ void k_debug_fn64(int which, uint32_t n, const double *__restrict__ x, double *__restrict__ y)
{
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double s, c;
    switch (which) {
    case 0: y[i] = dm::exp(x[i]); break;
    case 1: y[i] = dm::log(x[i]); break;
    case 2: dm::sincos(x[i], &s, &c); y[i] = s; break;
    case 3: dm::sincos(x[i], &s, &c); y[i] = c; break;
    case 4: y[i] = dm::tanh(x[i]); break;
    default: y[i] = dm::atan(x[i]); break;
    }
}

// pieces of the fast step (step64.cuh)
__global__ void k_debug_step64(int which, uint32_t n, const double *__restrict__ x, const double *__restrict__ b,
                               double *__restrict__ y)
{
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double v = x[i];
    double s, c;
    switch (which) {
    case 0: y[i] = s64::quot(v, b[i], s64::recip(b[i])); break;
    case 1: y[i] = s64::from_int(s64::ifloor(v)); break;
    case 2: y[i] = s64::uniform((uint32_t)v); break;
    case 3: y[i] = s64::scale2<1>(v); break;
    case 4: y[i] = s64::exp_in(v); break;
    case 5: y[i] = s64::log_in(v); break;
    case 6: s64::sincos_in(v, s, c); y[i] = s; break;
    case 7: s64::sincos_in(v, s, c); y[i] = c; break;
    case 8: y[i] = s64::cos_in(v); break;
    default: y[i] = s64::atan_in(v); break;
    }
}

__global__ void k_debug_normals64(uint64_t seed, uint64_t pid0, uint32_t n, uint32_t step, double *z)
{
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    m64::normals(seed, pid0 + i, step, z + 3 * (size_t)i);
}

__global__ void k_debug_philox(uint32_t n, const uint32_t *__restrict__ ctr, uint32_t k0, uint32_t k1,
                               uint32_t *__restrict__ out)
{
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint4 c = make_uint4(ctr[4 * i], ctr[4 * i + 1], ctr[4 * i + 2], ctr[4 * i + 3]);
    const uint4 w = philox4x32_10(c, k0, k1);
    out[4 * i] = w.x; out[4 * i + 1] = w.y; out[4 * i + 2] = w.z; out[4 * i + 3] = w.w;
}

// ---------------------------------------------------------------- launchers --
static inline unsigned grid_for(uint64_t n, unsigned block) { return (unsigned)((n + block - 1) / block); }

// Paged copy of the FP32 blocks of n parameter sets in quads (see P32): one
// thread per (set, field); the unused slots of the last page stay as they are.
__global__ void k_f32_table(const DevParams *__restrict__ prm, uint32_t n, float *__restrict__ table)
{
    const uint32_t j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n * kF32Fields) return;
    const uint32_t i = j / kF32Fields, f = j - i * kF32Fields;
    table[f32_table_offset(i) + (size_t)(f >> 2) * kSetsPerPage * 4 + (f & 3)] =
        reinterpret_cast<const float *>(&prm[i].f)[f];
}

cudaError_t launch_f32_table(const DevParams *prm, uint32_t n, float *table, cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    cudaGetLastError();
    k_f32_table<<<grid_for(n * kF32Fields, 128), 128, 0, s>>>(prm, n, table);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_derive(DevParams *prm, uint32_t n, cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    cudaGetLastError();
    k_derive<<<grid_for(n, 64), 64, 0, s>>>(prm, n);
    note_launch();
    return cudaGetLastError();
}

template <int ISO, bool EN>
static cudaError_t launch64(const LaunchArgs &a, int sms, cudaStream_t s)
{
    const unsigned n_sms = (unsigned)sms;
    const uint64_t n = a.n_total, teams = 32ull * n_sms, quads = ISO == 2 ? 0 : 8ull * n_sms;
    // the lists hold 32-bit indices
    const uint32_t cap = n <= 0xFFFFFFFFull ? a.list_cap : 0u;
    const uint32_t *from = nullptr;
    const unsigned long long *n_from = nullptr;
    if (n > teams) {
        // a second warp per scheduler fills the gaps between FP64 instructions, but halves the speed
        // of a path: taken when the queue keeps both busy for long
        const unsigned per_sm = n >= 1024ull * n_sms ? 2 : 1;
        const uint32_t limit = (uint32_t)std::min<uint64_t>(teams, cap);
        k_propagate64<ISO, EN><<<n_sms * per_sm, 128, 0, s>>>(a, limit);
        note_launch();
        if (!limit) return cudaGetLastError();
        from = a.list;
        n_from = a.ended + 1;
    }
    if (n > quads) {
        const uint32_t limit = (uint32_t)std::min<uint64_t>(quads, cap);
        uint32_t *to = a.list + (from ? cap : 0u);
        unsigned long long *n_to = a.ended + (from ? 3 : 1);
        k_finish64<4, ISO, EN><<<n_sms, 128, 0, s>>>(a, from, n_from, to, n_to, limit);
        note_launch();
        if (!limit) return cudaGetLastError();
        from = to;
        n_from = n_to;
    }
    if constexpr (ISO != 2) {
        k_quad64<ISO == 1, EN><<<(unsigned)std::min<uint64_t>(n_sms, n), 128, 0, s>>>(a, from, n_from);
        note_launch();
    }
    return cudaGetLastError();
}

cudaError_t launch_propagate_fp64(const LaunchArgs &a, Fp64Variant v, int sms, cudaStream_t s)
{
    if (a.n_total == 0) return cudaSuccess;
    cudaGetLastError();
    if (v.plain) {
        k_propagate_fp64<<<grid_for(a.n_total, 128), 128, 0, s>>>(a.prm, a.spc, a.items, a.prefix, a.n_items,
                                                                 a.n_total, a.out, a.steps_total);
        note_launch();
        return cudaGetLastError();
    }
    if (v.iso && v.aniso) return v.energy ? launch64<2, true>(a, sms, s) : launch64<2, false>(a, sms, s);
    if (v.iso) return v.energy ? launch64<1, true>(a, sms, s) : launch64<1, false>(a, sms, s);
    return v.energy ? launch64<0, true>(a, sms, s) : launch64<0, false>(a, sms, s);
}

cudaError_t launch_debug_eval64(const DevParams *prm, const DevSpecies *spc, uint32_t n, const double *st,
                                double *out, cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    cudaGetLastError();
    k_debug_eval64<<<grid_for(n, 128), 128, 0, s>>>(prm, spc, n, st, out);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_debug_fn64(int which, uint32_t n, const double *x, double *y, cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    cudaGetLastError();
    k_debug_fn64<<<grid_for(n, 256), 256, 0, s>>>(which, n, x, y);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_debug_step64(int which, uint32_t n, const double *x, const double *b, double *y, cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    cudaGetLastError();
    k_debug_step64<<<grid_for(n, 256), 256, 0, s>>>(which, n, x, b, y);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_debug_normals64(uint64_t seed, uint64_t pid0, uint32_t n, uint32_t step, double *z,
                                   cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    cudaGetLastError();
    k_debug_normals64<<<grid_for(n, 256), 256, 0, s>>>(seed, pid0, n, step, z);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_debug_philox(uint32_t n, const uint32_t *ctr, uint32_t k0, uint32_t k1, uint32_t *out,
                                cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    cudaGetLastError();
    k_debug_philox<<<grid_for(n, 256), 256, 0, s>>>(n, ctr, k0, k1, out);
    note_launch();
    return cudaGetLastError();
}

}  // namespace cosmica
