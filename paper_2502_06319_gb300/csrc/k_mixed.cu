// k_mixed.cu -- the batched persistent kernel of the mixed-precision path.
//
// One launch of (SMs x resident blocks) threads drains a device work queue:
// an atomic cursor over the prefix-summed particle counts of all work items
// (parameter set x species x energy).  Each lane owns one quasi-particle at a
// time and steps it until it leaves the heliosphere; a lane whose particle
// exits writes the exit state and immediately takes the next particle from
// the queue (refill), so that warps stay full while the queue lasts despite
// the long tail of exit times.  Lanes needing work in the same step take
// consecutive particles with one atomic per warp.  When the queue is empty and
// the paths left fit a smaller grid, they are handed to another launch of the
// kernel with one warp per scheduler fewer.  The paper's thread-per-
// quasi-particle mapping (Sec. IV.A) is kept; its one-launch-per-energy-bin
// loop (Sec. IV.A, last paragraph) becomes this.
#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "common.cuh"
#include "internal.h"
#include "mixed_state.cuh"
#include "model32.cuh"

namespace cosmica {

namespace {

// ln P0 of every item in place of its T (momentum form; the energy form starts from T): a
// lane taking a path would otherwise spend some 60 slots of the FP64 pipe on it, 64 clocks each
// for its whole warp.
__global__ void k_start_lnP(DevItem *items, const DevSpecies *__restrict__ spc, uint32_t n)
{
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const DevSpecies &sp = spc[items[i].species_idx];
    const double T = items[i].T;
    const double P0 = sp.A / fabs(sp.Z) * sqrt(T * (T + 2.0 * sp.m0));
    items[i].T = log(P0);
}

// the particle `local` of item `it`, at its start
template <int ACC, bool EN>
__device__ __forceinline__ void begin(const LaunchArgs &a, uint32_t it, uint64_t local, Lane &L, Acc<ACC> &x,
                                      EnergyAcc<ACC, EN> &en)
{
    const DevItem item = a.items[it];
    const DevParams &p = a.prm[item.param_idx];
    const DevSpecies &sp = a.spc[item.species_idx];
    L.q = a.f32 + f32_table_offset(item.param_idx);
    L.M2 = sp.aoz_m0_sq;
    L.sq = sp.sgnq;
    L.pid = item.first_pid + local;
    L.seed = item.seed;
    L.g = a.prefix[it] + local;
    L.item = item.out_item;
    L.k = 0;
    L.max_steps = (uint32_t)p.max_steps;
    // item.T: T of the energy form (whose ln P follows from T), ln P0 of the momentum form
    x.init(item.r0, item.th0, item.ph0, EN ? 1.0 : item.T, p.R_out, p.f.r_in, p.vote_lo);
    if constexpr (EN) en.init(item.T, (float)sp.m0, sp.aoz);
}

// Entry q of the launch's source: a queue slot (fresh), or a path parked by the launch before.
template <int ACC, bool EN>
__device__ __forceinline__ void take(const LaunchArgs &a, const MixedStage &st, uint64_t q, Lane &L, Acc<ACC> &x,
                                     EnergyAcc<ACC, EN> &en)
{
    if (!st.from) {
        // queue slot -> (item, index within the item); the exit record keeps item order
        const uint32_t iq = find_item(a.qprefix, a.n_items, q);
        begin<ACC, EN>(a, a.qitem ? a.qitem[iq] : iq, q - a.qprefix[iq], L, x, en);
    } else {
        const uint64_t g = st.from[q];
        const uint32_t it = find_item(a.prefix, a.n_items, g);
        begin<ACC, EN>(a, it, g - a.prefix[it], L, x, en);
        unpark<EN>(a.out, g, x, en);
        L.k = a.out.steps[g];
    }
}

// One Euler-Maruyama step (Eq. 3, Eq. 6) with the normals z0, z1, z2 of step L.k, which become
// those of the next step: the increments are added and nothing else is done.  True when the new
// state has to be looked at (a boundary, an end of the path, or nearly so).  One block without
// branches (in the full-model variant), so that the compiler interleaves the generator with the
// coefficients.
template <int ACC, bool EN, int EXT, bool FULL>
__device__ __forceinline__ bool advance(const float *params, Lane &L, Acc<ACC> &x, EnergyAcc<ACC, EN> &en, float &z0,
                                        float &z1, float &z2)
{
    m32::Drift c;
    const P32<kSetsPerPage> q{params};
    float fr, fth, fph, lnP, sin_th;
    x.view(fr, fth, fph, lnP, sin_th);
    if constexpr (EN) {
        // rigidity from the integrated kinetic energy: P = (A/|Z|) sqrt(T (T + 2 m0))
        const float T = en.fT();
        lnP = __logf(en.aoz * sqrtf(T * (T + 2.0f * en.m0)));
    }
    m32::eval<EXT, FULL, kSetsPerPage>(q, L.M2, L.sq, fr, fth, sin_th, fph, lnP, c);
    const float sdt = sqrtf(c.dt);
    const float dr = fmaf(c.Ar_tot, c.dt, c.l00 * z0 * sdt);
    const float dth = fmaf(c.dth_drift, c.dt, c.l11 * z1 * sdt * c.inv_r);
    const float dph = fmaf(c.dph_drift, c.dt, fmaf(c.l20, z0, c.l22 * z2) * sdt * c.inv_rs);
    if constexpr (EN) {
        // Eq. 1 backward: A_T = (2/3)(V/r) alpha T, loss L = (2V/(3r)) (1 + beta^2)
        const float T = en.fT();
        const float alpha = __fdividef(T + 2.0f * en.m0, T + en.m0);
        en.add(c.dlnP * alpha * T * c.dt, c.dlnP * fmaf(c.beta, c.beta, 1.0f) * c.dt);
    }
    const bool squashed = m32::is_squashed<EXT>(q);
    bool calm = x.template add<!EN>(fr, fth, fph, dr, dth, dph, EN ? 0.0f : c.dlnP * c.dt, c.dt, P32F(q, r_in), !squashed);
    L.k += 1u;
    calm &= L.k < L.max_steps;
    if (squashed) calm &= !m32::outside_squashed(q, x.fr(), x.fth(), x.fph());
    m32::normals(L.seed, L.pid, L.k, z0, z1, z2);
    return !calm;
}

// whether the state after a step needs settle(): a boundary other than the longitude's, an end of
// the path, or nearly so
template <int ACC, int EXT>
__device__ __forceinline__ bool needs_settling(const float *params, const Lane &L, const Acc<ACC> &x)
{
    const P32<kSetsPerPage> q{params};
    const bool squashed = m32::is_squashed<EXT>(q);
    bool calm = x.calm(P32F(q, r_in), !squashed) & (L.k < L.max_steps);
    if (squashed) calm &= !m32::outside_squashed(q, x.fr(), x.fth(), x.fph());
    return !calm;
}

// Boundaries and the three ends of a path; true when the path ended (exit record written).
template <int ACC, bool EN, int EXT>
__device__ __forceinline__ bool settle(const LaunchArgs &a, Lane &L, Acc<ACC> &x, EnergyAcc<ACC, EN> &en,
                                       unsigned long long &my_steps)
{
    const P32<kSetsPerPage> q{L.q};
    x.boundaries(P32F(q, r_in));
    const bool fin = x.finite();
    const bool out = m32::is_squashed<EXT>(q) ? m32::outside_squashed(q, x.fr(), x.fth(), x.fph()) : x.exited();
    const bool lim = L.k >= L.max_steps;
    if (fin & !out & !lim) return false;
    const int status = !fin ? COSMICA_PATH_NONFINITE : (out ? COSMICA_PATH_EXIT : COSMICA_PATH_STEP_LIMIT);
    x.write(a.out, L.g);
    if constexpr (EN) {
        const double T = en.T64();
        a.out.lnP[L.g] = log((double)en.aoz * sqrt(T * (T + 2.0 * (double)en.m0)));
        if (a.out.lw) a.out.lw[L.g] = en.lw();
    } else {
        if (a.out.lw) a.out.lw[L.g] = 0.0;
    }
    a.out.steps[L.g] = L.k;
    a.out.status[L.g] = (uint8_t)status;
    a.out.item[L.g] = L.item;
    my_steps += L.k;
    return true;
}

// Persistent propagation.  Lanes take paths from the source (one atomic per warp for all lanes
// needing work), step them, write the exit record and refill, until the source is drained.
// Then, if the launch has a limit, every warp asks every `period` steps how many paths are
// left, and once they are no more than the limit parks its own for the next launch.
//
// The steps run in an inner loop that ends when some lane of the warp has a boundary or an end
// to see to: one vote and one branch a step.  All lanes of the warp run it, those without a
// path on whatever they hold (nobody looks at the results).  What bounds it: a warp alone on its
// scheduler is bound by its ~400 instructions a step and their dependences, four warps by the
// issue rate.  The loop being one block, the compiler interleaves the generator with the
// coefficients and keeps the parameter set in registers (122-160 instead of 64, so 12 or 16 warps
// per SM instead of 32).  Measured, against a loop that tested everything every step and drew the
// normals after the tests: a lone path's step 0.68 -> 0.30 us (375 instructions), a warp's step
// with four warps per scheduler 1.05 -> 0.87 us, one spectrum of 6e5 paths 144 -> 93 ms, 1.8e6
// paths of 16 heliospheres 893 -> 669 ms.
template <int ACC, bool EN, int EXT, bool FULL>
__global__ void __launch_bounds__(256, 1) k_propagate_mixed(LaunchArgs a, MixedStage st)
{
    const unsigned lane = threadIdx.x & 31u;
    Lane L{};
    Acc<ACC> x{};
    EnergyAcc<ACC, EN> en{};
    // lanes that never get a path step an unremarkable state of the first set
    L.q = a.f32;
    x.init(1.0, 1.0, 1.0, 1.0, 2.0, 0.1f, 0.11f);
    en.init(1.0, 1.0f, 1.0f);
    // a source smaller than the grid is spread evenly over the warps
    const uint64_t n = st.from ? *st.n_from : a.n_total;
    const uint64_t warps = (uint64_t)gridDim.x * (blockDim.x >> 5);
    const bool seat = lane < (n + warps - 1) / warps;
    bool active = false, drained = n == 0;
    float z0 = 0.0f, z1 = 0.0f, z2 = 0.0f;   // normals of the lane's next step
    unsigned long long my_steps = 0;
    uint32_t room = st.limit ? st.period : 0xFFFFFFFFu;   // steps until the next look at the paths left

    while (true) {
        const unsigned need = __ballot_sync(0xffffffffu, seat && !active && !drained);
        if (need) {
            unsigned long long base = 0;
            const unsigned leader = __ffs(need) - 1;
            if (lane == leader) base = atomicAdd(st.cursor, (unsigned long long)__popc(need));
            base = __shfl_sync(0xffffffffu, base, leader);
            if (need & (1u << lane)) {
                const uint64_t q = base + __popc(need & ((1u << lane) - 1u));
                if (q < n) {
                    take<ACC, EN>(a, st, q, L, x, en);
                    m32::normals(L.seed, L.pid, L.k, z0, z1, z2);
                    active = true;
                }
            }
            // a lane that was refused never asks again, so once any lane of the warp is refused the
            // whole warp can stop asking
            if (base + __popc(need) > n) drained = true;
        }
        if (!__any_sync(0xffffffffu, active)) {
            if (drained) break;
            continue;
        }
        if (room == 0) {
            room = st.period;
            // few enough paths left, all of them taken from the source (drained: a lane was refused)
            unsigned few = 0;
            if (drained && lane == 0) few = a.n_total - *(volatile unsigned long long *)a.ended <= st.limit;
            if (__shfl_sync(0xffffffffu, few, 0)) {
                if (active) {
                    park<EN>(a.out, L.g, x, en);
                    a.out.steps[L.g] = L.k;
                    a.out.status[L.g] = COSMICA_PATH_RUNNING;
                    st.to[atomicAdd(st.n_to, 1ull)] = (uint32_t)L.g;   // no more than `limit` paths are left
                }
                break;
            }
        }
        bool see;
        while (true) {
            const bool look = advance<ACC, EN, EXT, FULL>(L.q, L, x, en, z0, z1, z2);
            --room;
            if (!__any_sync(0xffffffffu, (active && look) || room == 0)) continue;
            see = active && look && needs_settling<ACC, EXT>(L.q, L, x);
            if (active && look && !see && x.phi_out()) x.wrap_near();
            if (__any_sync(0xffffffffu, see || room == 0)) break;
        }
        const bool end = see && settle<ACC, EN, EXT>(a, L, x, en, my_steps);
        if (end) active = false;
        const unsigned ends = __ballot_sync(0xffffffffu, end);
        if (ends && lane == 0) atomicAdd(a.ended, (unsigned long long)__popc(ends));
    }
    if (a.steps_total) {
        for (int o = 16; o > 0; o >>= 1) my_steps += __shfl_down_sync(0xffffffffu, my_steps, o);
        if (lane == 0 && my_steps) atomicAdd(a.steps_total, my_steps);
    }
}

// debug: mixed coefficients at given states (FP64 in, FP64 out)
__global__ void k_debug_eval32(const DevParams *__restrict__ prm, const DevSpecies *__restrict__ spc,
                               uint32_t n, const double *__restrict__ st, double *__restrict__ out)
{
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float dbg[kDebugEvalN];
    m32::Drift c;
    m32::eval<m32::kExtAny, false, 1>(P32<1>{reinterpret_cast<const float *>(&prm[0].f)}, spc[0].aoz_m0_sq, spc[0].sgnq,
                              (float)st[4 * i], (float)st[4 * i + 1], m32::sin_theta_f64(st[4 * i + 1]),
                              (float)st[4 * i + 2], (float)st[4 * i + 3], c, dbg);
    for (int j = 0; j < kDebugEvalN; ++j) out[(size_t)i * kDebugEvalN + j] = dbg[j];
}

}  // namespace

// Call fn(acc, energy, extended, full) with each flag as a compile-time constant.
template <class Fn>
static void visit_variant(MixedVariant v, Fn &&fn)
{
    auto on_acc = [&](auto A) {
        auto on_energy = [&](auto E) {
            auto on_ext = [&](auto X) {
                if (v.full) fn(A, E, X, std::true_type{});
                else fn(A, E, X, std::false_type{});
            };
            if (v.extended == m32::kExtNone) on_ext(std::integral_constant<int, m32::kExtNone>{});
            else if (v.extended == m32::kExtShells) on_ext(std::integral_constant<int, m32::kExtShells>{});
            else if (v.extended == m32::kExtSquashed) on_ext(std::integral_constant<int, m32::kExtSquashed>{});
            else on_ext(std::integral_constant<int, m32::kExtAny>{});
        };
        if (v.energy) on_energy(std::true_type{});
        else on_energy(std::false_type{});
    };
    if (v.acc == COSMICA_PREC_MIXED_F64ACC) on_acc(std::integral_constant<int, COSMICA_PREC_MIXED_F64ACC>{});
    else on_acc(std::integral_constant<int, COSMICA_PREC_MIXED>{});
}

int mixed_max_blocks_per_sm(MixedVariant v, unsigned block)
{
    int nb = 0;
    visit_variant(v, [&](auto A, auto E, auto S, auto F) {
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &nb, k_propagate_mixed<decltype(A)::value, decltype(E)::value, decltype(S)::value, decltype(F)::value>,
            (int)block, 0);
    });
    return nb;
}

// A launch of w warps per scheduler whose queue is empty runs on with ever emptier warps, each
// step as slow as the w warps make it; handing the last paths to w - 1 full warps per scheduler,
// and so on down to one, steps them at the speed of those (one warp: 0.3 us a step, four: 0.9).
cudaError_t launch_propagate_mixed(const LaunchArgs &a, MixedVariant v, PersistentShape shape, int sms, cudaStream_t s)
{
    if (a.n_total == 0) return cudaSuccess;
    cudaGetLastError();
    if (!v.energy) {
        k_start_lnP<<<(a.n_items + 63) / 64, 64, 0, s>>>(a.items, a.spc, a.n_items);
        note_launch();
    }
    const unsigned block = 128;                          // of the later launches
    const uint64_t layer = (uint64_t)sms * block;        // one warp per scheduler
    // layers of the next launch: fewer than this one has, and no more than the list holds paths for
    uint64_t layers = 0;
    if (shape.compact_period && a.n_total <= 0xFFFFFFFFull && a.list_cap > 0 && a.n_total > layer) {
        layers = std::min<uint64_t>(((uint64_t)shape.grid * shape.block + layer - 1) / layer, kMixedStages) - 1;
        layers = std::min<uint64_t>(layers, std::max<uint64_t>(1, a.list_cap / layer));
    }
    MixedStage st{};
    st.cursor = a.cursor;
    st.period = shape.compact_period ? shape.compact_period : 64u;
    for (unsigned stage = 0;; ++stage) {
        st.limit = (uint32_t)std::min<uint64_t>(layers * layer, a.list_cap);
        st.to = a.list + (stage & 1u) * (size_t)a.list_cap;
        st.n_to = a.ended + 1 + 2 * stage;
        visit_variant(v, [&](auto A, auto E, auto S, auto F) {
            k_propagate_mixed<decltype(A)::value, decltype(E)::value, decltype(S)::value, decltype(F)::value>
                <<<shape.grid, stage ? block : shape.block, 0, s>>>(a, st);
        });
        note_launch();
        if (layers == 0) break;
        shape.grid = (unsigned)(layers * sms);
        st.from = st.to;
        st.n_from = st.n_to;
        st.cursor = st.n_to + 1;
        --layers;
    }
    return cudaGetLastError();
}

cudaError_t launch_debug_eval32(const DevParams *prm, const DevSpecies *spc, uint32_t n, const double *st,
                                double *out, cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    cudaGetLastError();
    k_debug_eval32<<<(n + 127) / 128, 128, 0, s>>>(prm, spc, n, st, out);
    note_launch();
    return cudaGetLastError();
}

}  // namespace cosmica
