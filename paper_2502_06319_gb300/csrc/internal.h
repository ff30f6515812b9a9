// internal.h -- declarations shared by the translation units of libcosmica
// (launchers implemented in the kernel files, called by the C-ABI layer).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "common.cuh"

namespace cosmica {

constexpr int kDebugEvalN = 21;   // quantities written per state by the debug evaluators

struct LaunchArgs {
    const DevParams *prm;
    const DevSpecies *spc;
    DevItem *items;
    const uint64_t *prefix;
    uint32_t n_items;
    uint64_t n_total;
    ExitPtrs out;
    unsigned long long *steps_total;   // may be null
    unsigned long long *cursor;        // work-queue cursor (persistent kernels)
    const uint32_t *qitem;             // item of each queue slot (null: item order)
    const uint64_t *qprefix;           // prefix sums of particle counts in queue order
    const float *f32;                  // FP32 blocks of the parameter sets, paged field-major (P32)
    // indices of the paths one kernel of the launch leaves to the next: two lists of list_cap
    // (mixed paths use both in turn, the FP64 path the first), and counters cleared like the cursor
    uint32_t *list;
    uint32_t list_cap;
    unsigned long long *ended;         // [0] paths ended; then, per kernel, paths left and their cursor
};

struct PersistentShape {
    unsigned block;
    unsigned grid;
    unsigned compact_period;   // steps between looks at the paths left; 0: never handed over
};

// one kernel of a mixed launch: where its paths come from and where it leaves the last ones
struct MixedStage {
    const uint32_t *from;              // null: the launch's queue, else parked paths, *n_from of them
    const unsigned long long *n_from;
    unsigned long long *cursor;        // of the source
    uint32_t *to;
    unsigned long long *n_to;
    uint32_t limit;                    // leave the last `limit` paths (0: none)
    uint32_t period;
};
constexpr uint32_t kMixedStages = 4;   // most warps per scheduler that hand over step by step

// ---- continuous-batching server -------------------------------------------
// fresh particles of one (request, energy) slice, offered to one quantum
struct ServeItem {
    double T;                  // GeV/n
    uint64_t first_pid;        // pid of the slice's first particle
    uint64_t seed;
    uint64_t exit_idx;         // exit-arena index of the slice's first particle
    uint32_t slot;             // request slot: parameter set and species index
    uint32_t energy;           // energy index within the request
};

// an in-flight particle between two quanta (exact state)
struct Suspended {
    union {
        float f[10];           // compensated pairs (r, th, ph, lnP, s)
        double d[5];           // FP64 accumulation
    };
    uint32_t k, slot, energy, pad;
    uint64_t pid, seed, exit_idx;
};

struct ServeArgs {
    const DevParams *prm;      // per slot
    const DevSpecies *spc;     // per slot
    const ServeItem *items;
    const uint64_t *prefix;
    uint32_t n_items;
    uint64_t n_fresh;
    const Suspended *resume;
    uint64_t n_resume;
    Suspended *suspend;
    unsigned int *n_suspend;
    unsigned long long *cursors;   // [0] fresh, [1] resume
    ExitPtrs arena;
    unsigned int *req_done;        // per slot
    unsigned long long *req_steps; // per slot
    uint32_t budget;               // steps per lane per quantum
    uint32_t idle_slot;            // a resident request's: its parameters are stepped by lanes without a particle
};

// ext: Extensions::kind() of the resident requests; full: every one is the full model (the variant
// without uniform branches)
cudaError_t launch_serve(const ServeArgs &a, int acc, int ext, bool full, PersistentShape shape, cudaStream_t s);
int serve_max_blocks_per_sm(int acc, int ext, bool full, unsigned block);

// extensions of a launch's parameter sets
struct Extensions {
    bool shells = false, no_shells = false, squashed = false, round = false;   // some set has (has not) ...
    void add(const cosmica_params &p)
    {
        (p.n_shells > 0 ? shells : no_shells) = true;
        (p.squashed != 0 ? squashed : round) = true;
    }
    // 0 none, 1 shells in every set, 2 every set squashed, 3 anything else (m32::kExt...)
    int kind() const
    {
        if (!shells && !squashed) return 0;
        if (!no_shells && !squashed) return 1;
        if (!shells && !round) return 2;
        return 3;
    }
};

void note_launch();

cudaError_t launch_derive(DevParams *prm, uint32_t n, cudaStream_t s);
cudaError_t launch_f32_table(const DevParams *prm, uint32_t n, float *table, cudaStream_t s);
// variant of the FP64 kernels
struct Fp64Variant {
    bool energy;
    bool plain;         // some set or species is not one of the fast step's (see fast_step_set): the plain step for all
    bool iso, aniso;    // some set is (not) isotropic
};
// counters of a launch: queue cursor, steps, paths ended, and per kernel paths left and their cursor
constexpr uint32_t kLaunchCounters = 3 + 2 * kMixedStages;
// entries of each of a launch's two lists: at most kMixedStages - 1 warps per scheduler
inline uint32_t list_entries(uint64_t n_total, int sms)
{
    const uint64_t most = (uint64_t)(kMixedStages - 1) * 128u * (uint64_t)sms;
    return n_total > 8ull * (uint64_t)sms ? (uint32_t)(n_total < most ? n_total : most) : 0u;
}
cudaError_t launch_propagate_fp64(const LaunchArgs &a, Fp64Variant v, int sms, cudaStream_t s);

// mixed precision persistent kernel; acc = COSMICA_PREC_MIXED or COSMICA_PREC_MIXED_F64ACC
// compile-time variant of the mixed kernel a launch needs
struct MixedVariant {
    int acc;        // COSMICA_PREC_MIXED or COSMICA_PREC_MIXED_F64ACC
    bool energy;    // energy formulation (Eq. 1) instead of the momentum form
    int extended;   // Extensions::kind() of the launch's parameter sets
    bool full;      // every set is the full model: drift and current sheet on, adaptive step
};
// Sets and species of the FP64 fast step (step64.cuh): no shells, not squashed, and constants between
// 1e-9 and 1e9 (times and step-rule factors: 1e-12 and 1e12).  With ln P and the angles in the range that
// the step itself tests, no operand of its divisions then leaves the range for which they are the correctly
// rounded ones (a shock width of 1e-310 AU, say, has no finite reciprocal).
inline bool fast_step_set(const cosmica_params &p)
{
    auto in = [](double x) { return x >= 1e-9 && x <= 1e9; };
    auto in12 = [](double x) { return x >= 1e-12 && x <= 1e12; };
    if (p.n_shells > 0 || p.squashed != 0 || !in(p.K0) || !in(p.r_in_AU) || !in(p.R_out_AU)) return false;
    if (p.R_ts_AU > 0.0 && !(in(p.R_ts_AU) && in(p.dts_AU) && in(p.ts_K_factor))) return false;
    if (p.dt_fixed_day > 0.0) {
        if (!in12(p.dt_fixed_day)) return false;
    } else if (!in12(p.dt_min_day) || !in12(p.dt_max_day) || !(p.eps_adv == 0.0 || in12(p.eps_adv)) ||
               !(p.eps_diff == 0.0 || in12(p.eps_diff))) {
        return false;
    }
    if (p.isotropic) return p.V_const_kms == 0.0 || in(p.V_const_kms);
    return in(p.kperp_r_frac) && in(p.kperp_th_frac) && in(p.B1AU_nT) && in(p.V_slow_kms) && in(p.V_fast_kms) &&
           in(p.rot_period_day) && in(p.dlat_deg) && p.lat_fast_deg >= -1e9 && p.lat_fast_deg <= 1e9 &&
           (!p.hcs_on || in(p.dcs_min_deg));
}
inline bool fast_step_species(const cosmica_species &s) { return s.m0_GeV >= 1e-9 && s.m0_GeV <= 1e9; }
inline Fp64Variant fp64_variant(const cosmica_params *ps, size_t n, const cosmica_species *sp, size_t n_sp)
{
    Fp64Variant v{ps[0].formulation == 1, false, false, false};
    for (size_t i = 0; i < n; ++i) {
        v.plain = v.plain || !fast_step_set(ps[i]);
        (ps[i].isotropic ? v.iso : v.aniso) = true;
    }
    for (size_t i = 0; i < n_sp; ++i) v.plain = v.plain || !fast_step_species(sp[i]);
    return v;
}
// a set is the full model of the mixed kernels' FULL variant
inline bool full_model(const cosmica_params &p)
{
    return !p.isotropic && p.drift_on && p.hcs_on && !(p.dt_fixed_day > 0.0);
}
cudaError_t launch_propagate_mixed(const LaunchArgs &a, MixedVariant v, PersistentShape shape, int sms, cudaStream_t s);
int mixed_max_blocks_per_sm(MixedVariant v, unsigned block);

struct SpecItem {
    double T;                  // GeV/n
    double A, Z, m0;           // species
    uint32_t sp, pad;          // row of the species in the table of bin weights
};
// table of bin weights [n_sp x nbins] to fill (none if weights is null), species s being that of
// items[sp_item[s]]
struct WeightTable {
    const SpecItem *items;
    const uint32_t *sp_item;
    uint32_t n_sp;
    int lis_kind;
    const double *lnT, *lnJ;
    uint32_t lis_n;
    double *weights;
};
cudaError_t launch_spec_clear(unsigned long long *hist, uint64_t n_hist, cudaStream_t s);
// adds n exit states to the cleared histogram and fills the table of bin weights
cudaError_t launch_histogram(const ExitPtrs &ex, uint64_t n, uint32_t n_items, uint32_t nbins, double x_lo,
                             double dx, unsigned long long *hist, const WeightTable &wt, int sms, cudaStream_t s);
// weights: from launch_histogram, or null (every item evaluates its own); sums: scratch of
// n_items x spectrum_sums_bytes()
constexpr size_t spectrum_sums_bytes() { return 24; }
cudaError_t launch_spectrum(const unsigned long long *hist, uint32_t n_items, uint32_t nbins,
                            double x_lo, double dx, const SpecItem *items, const double *weights, int lis_kind,
                            const double *lis_lnT, const double *lis_lnJ, uint32_t lis_n, void *sums,
                            double *J, double *sigma, cudaStream_t s);

// unbinned estimator: chunks of `per` x 128 exit states of one item, chunk_prefix their prefix sums over items
uint32_t unbinned_per_thread(const uint32_t *n_per_item, uint32_t n_items, int sms);
uint64_t unbinned_chunks(uint64_t n, uint32_t per);
size_t unbinned_partial_bytes();
cudaError_t launch_spectrum_unbinned(const ExitPtrs &ex, const uint64_t *prefix, const uint64_t *chunk_prefix,
                                     uint64_t n_chunks, uint32_t per, void *partials, uint32_t n_items,
                                     const SpecItem *items, int form, int lis_kind, const double *lis_lnT,
                                     const double *lis_lnJ, uint32_t lis_n, double *J, double *sigma, cudaStream_t s);

cudaError_t launch_debug_eval64(const DevParams *prm, const DevSpecies *spc, uint32_t n, const double *st,
                                double *out, cudaStream_t s);
cudaError_t launch_debug_eval32(const DevParams *prm, const DevSpecies *spc, uint32_t n, const double *st,
                                double *out, cudaStream_t s);
cudaError_t launch_debug_fn64(int which, uint32_t n, const double *x, double *y, cudaStream_t s);
cudaError_t launch_debug_step64(int which, uint32_t n, const double *x, const double *b, double *y, cudaStream_t s);
cudaError_t launch_debug_normals64(uint64_t seed, uint64_t pid0, uint32_t n, uint32_t step, double *z,
                                   cudaStream_t s);
cudaError_t launch_debug_normals32(uint64_t seed, uint64_t pid0, uint32_t n, uint32_t step, float *z,
                                   uint32_t *words, cudaStream_t s);
cudaError_t launch_debug_philox(uint32_t n, const uint32_t *ctr, uint32_t k0, uint32_t k1, uint32_t *out,
                                cudaStream_t s);
cudaError_t launch_debug_curand_philox(uint32_t n, uint64_t seed, const unsigned long long *subseq,
                                       const unsigned long long *offset, uint32_t *out, cudaStream_t s);

}  // namespace cosmica
