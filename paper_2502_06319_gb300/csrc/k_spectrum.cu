// k_spectrum.cu -- exit-rigidity histogram and modulated spectrum (Eq. 4).
// Built with -fmad=false so that the bin of every exit is decided by the
// same FP64 operations as its definition: b = floor((lnP / ln 10 - x_lo) / dx).
//
//   k_spec_clear clears the histogram
//   k_histogram  blocks of consecutive exit states count into shared memory and add
//                their nonzero counters to the histogram (integers: deterministic);
//                a few more evaluate the bin weights w_b = J_LIS(T_b) / P_b^2 once per
//                species and bin
//   k_spectrum_warp, k_spectrum
//                one warp or one block per item: J = P0^2 (1/N) sum_b c_b w_b (J = f P^2 is
//                the intensity per unit kinetic energy and f is conserved along
//                a path), and sigma = std of the summand / sqrt(N); fixed-order
//                reductions
//   k_unbinned_chunks, k_unbinned_items
//                unbinned Eq. 4: chunks of an item's exit states, then the item
#include <algorithm>
#include <cmath>
#include <cstdint>

#include "common.cuh"
#include "f64bits.h"
#include "internal.h"

namespace cosmica {

namespace {

// ---- local interstellar spectrum ------------------------------------------------
__device__ double lis_value(int kind, double T, const double *lnT, const double *lnJ, uint32_t m)
{
    if (kind == 0) return pow(T, -2.7) / (1.0 + pow(T, -3.7));
    const double x = log(T);
    if (x <= lnT[0]) return exp(lnJ[0]);
    if (x >= lnT[m - 1]) return exp(lnJ[m - 1]);
    uint32_t lo = 0, hi = m - 1;
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (lnT[mid] <= x) lo = mid; else hi = mid;
    }
    const double t = (x - lnT[lo]) / (lnT[hi] - lnT[lo]);
    return exp(lnJ[lo] + t * (lnJ[hi] - lnJ[lo]));
}

// bin weight w_b = J_LIS(T_b) / P_b^2 at the bin's log-centre
__device__ double bin_weight(const SpecItem &it, uint32_t b, double x_lo, double dx, int lis_kind, const double *lnT,
                             const double *lnJ, uint32_t lis_n)
{
    const double zoa = fabs(it.Z) / it.A;
    const double Pb = pow(10.0, x_lo + ((double)b + 0.5) * dx);
    const double pn = Pb * zoa;
    const double En = sqrt(pn * pn + it.m0 * it.m0);
    const double Tb = pn * pn / (En + it.m0);
    return lis_value(lis_kind, Tb, lnT, lnJ, lis_n) / (Pb * Pb);
}

// The bin weights of the n_sp species (those of items sp_item[s]), one thread per bin: three pow
// each, the whole cost of a spectrum when every item evaluated its own.  Called by every thread
// of the blocks 0, 1, ... that cover n_sp x nbins.
__device__ __forceinline__ void fill_weights(const WeightTable &w, uint32_t nbins, double x_lo, double dx, uint32_t block)
{
    const uint64_t i = (uint64_t)block * blockDim.x + threadIdx.x;
    if (i >= (uint64_t)w.n_sp * nbins) return;
    const uint32_t s = (uint32_t)(i / nbins), b = (uint32_t)(i % nbins);
    w.weights[i] = bin_weight(w.items[w.sp_item[s]], b, x_lo, dx, w.lis_kind, w.lnT, w.lnJ, w.lis_n);
}

// ---- histogram ---------------------------------------------------------------
// b = floor((lnP / ln 10 - x_lo) / dx) costs two FP64 divisions (about 20 slots of 64
// clocks on the FP64 pipe, 15 times the HBM time of a 13-byte record).  The same bin
// comes from fixed point: lnP in units of 2^-27, times A = 1 / (ln 10 dx) scaled to 31
// bits, plus the offset -x_lo / dx, in one 64-bit multiply-add.  Its error is below
// `tol` (in units of the product's high word); a value closer than that to a bin edge,
// and any |lnP| >= 16, takes the FP64 form, so every bin is the FP64 form's.
struct BinRule {
    double x_lo, dx;
    int64_t B;         // -x_lo / dx in units of 2^-(27 + sA)
    int32_t A;         // 1 / (ln 10 dx) in units of 2^-sA
    int32_t shift;     // of the product's high word down to whole bins
    int32_t tol;       // error bound in the high word's units
    int32_t fast;      // 0: the offset or the scale does not fit, FP64 form throughout
};

BinRule make_rule(double x_lo, double dx)
{
    BinRule r{x_lo, dx, 0, 0, 0, 0, 0};
    const double a = 1.0 / (kLn10 * dx), b = -x_lo / dx;
    if (!(a >= 1.0 && a < 0x1p24)) return r;
    const int sA = 30 - std::ilogb(a);          // 2^30 <= a 2^sA < 2^31
    if (!(std::fabs(b) < std::ldexp(1.0, 60 - 27 - sA))) return r;
    r.A = (int32_t)std::min(std::floor(std::ldexp(a, sA)), 2147483647.0);
    r.B = (int64_t)std::ldexp(b, 27 + sA);
    r.shift = 27 + sA - 32;                      // a < 2^24: sA >= 7, shift >= 2
    // truncation of lnP (one unit times A < 2^31), of A (|L| < 2^31 times one unit) and the
    // rounding of B and of the FP64 form itself (a few 2^-52 of |y| + |b|, below 2^-20 bins):
    // 2^32 + 2^32 + 2^(27 + sA - 20) units
    r.tol = 3 + (int32_t)std::ldexp(1.0, std::max(0, 27 + sA - 20 - 32));
    r.fast = r.tol < (1 << (r.shift - 1)) ? 1 : 0;
    return r;
}

__device__ __forceinline__ uint32_t slot_exact(const BinRule &q, double lnP, uint32_t nbins)
{
    const double x = lnP / kLn10;
    const double b = floor((x - q.x_lo) / q.dx);
    if (b < 0.0) return 0u;
    if (b >= (double)nbins) return nbins + 1u;
    return 1u + (uint32_t)b;
}

__device__ __forceinline__ uint32_t slot_of(const BinRule &q, double lnP, uint32_t nbins)
{
    const uint32_t hi = (uint32_t)__double2hiint(lnP), lo = (uint32_t)__double2loint(lnP);
    const uint32_t e = (hi >> 20) & 0x7FFu;                               // |lnP| = m 2^(e - 1054)
    const uint32_t m = __funnelshift_l(lo, (hi & 0xFFFFFu) | 0x100000u, 11);
    const uint32_t sh = 1027u - e;                                        // >= 1 for |lnP| < 16
    const uint32_t mag = sh < 32u ? m >> sh : 0u;
    const int32_t L = (int32_t)hi < 0 ? -(int32_t)mag : (int32_t)mag;
    const int32_t y = (int32_t)(((int64_t)L * q.A + q.B) >> 32);
    if (!q.fast || e > 1026u || (((y + q.tol) ^ (y - q.tol)) >> q.shift) != 0) return slot_exact(q, lnP, nbins);
    const int32_t b = y >> q.shift;
    return b < 0 ? 0u : min(1u + (uint32_t)b, nbins + 1u);
}

constexpr uint32_t kHistThreads = 256;
constexpr uint32_t kHistWords = 8192;      // 32 KB of counters: 15 rows of 512 bins

// One block counts `per` x 256 consecutive exit states.  A propagation writes the states
// of an item next to each other, so a block meets few items: the rows of the first one it
// meets and of the following `rows` - 1 are counted in shared memory (32-bit counters, at
// most 8192 a block) and only the nonzero counters go to the histogram, about one 64-bit
// atomic per 20 states; a state of any other item adds to the histogram directly, lanes
// with the same counter merged.  Loads are scalar and coalesced: the caller's arrays may
// start at any element.
// Bound by HBM: 1.6e7 states (208 MB) into 5760 x 515 counters take 50 us, 4.2 TB/s, 31 us being
// the read at copy speed; with two FP64 divisions a state and one atomic per warp and counter it
// was ten times that.
__global__ void __launch_bounds__(kHistThreads) k_histogram(ExitPtrs ex, uint64_t n, uint32_t n_items, uint32_t nbins,
                                                            BinRule rule, uint32_t rows, uint32_t per,
                                                            unsigned long long *__restrict__ hist, WeightTable wt,
                                                            uint32_t wblocks)
{
    // the first blocks fill the table of bin weights meanwhile (some 8 us of dependent pow: with
    // the clearing, in a launch of their own, the spectrum of 5760 items took 113 us, so 102)
    if (blockIdx.x < wblocks) {
        fill_weights(wt, nbins, rule.x_lo, rule.dx, blockIdx.x);
        return;
    }
    __shared__ __align__(16) uint32_t cnt[kHistWords];
    const uint32_t stride = nbins + 3u;
    const uint64_t g0 = (uint64_t)(blockIdx.x - wblocks) * (per * kHistThreads);
    const uint32_t words = rows * stride;
    for (uint32_t w = threadIdx.x * 4; w < words; w += kHistThreads * 4)
        *reinterpret_cast<uint4 *>(cnt + w) = make_uint4(0u, 0u, 0u, 0u);   // words <= kHistWords, itself a multiple of 4
    // the block's first item, which comes from the caller and may be any number: with row0 + rows <=
    // n_items every counted row is one of the histogram's, and a valid item below row0 wraps to at
    // least 2^32 - row0 > rows
    const uint32_t row0 = n_items <= rows ? 0u : min(ex.item[g0], n_items - rows);
    __syncthreads();
    constexpr uint32_t U = 4;
    for (uint32_t k = 0; k < per; k += U) {
        uint32_t item[U], st[U];
        double lnP[U];
#pragma unroll
        for (uint32_t u = 0; u < U; ++u) {
            const uint64_t g = g0 + (uint64_t)(k + u) * kHistThreads + threadIdx.x;
            const bool in = k + u < per && g < n;
            item[u] = in ? ex.item[g] : 0xFFFFFFFFu;
            st[u] = in ? ex.status[g] : 0u;
            lnP[u] = in ? ex.lnP[g] : 0.0;
        }
#pragma unroll
        for (uint32_t u = 0; u < U; ++u) {
            // exit states come from the caller: an entry whose item is out of range is not counted
            const bool valid = item[u] < n_items;
            const uint32_t slot = st[u] != COSMICA_PATH_EXIT ? nbins + 2u : slot_of(rule, lnP[u], nbins);
            const uint32_t row = item[u] - row0;
            const bool near = valid && row < rows;
            if (near) atomicAdd(cnt + row * stride + slot, 1u);
            const unsigned rest = __ballot_sync(0xffffffffu, valid && !near);
            if (valid && !near) {
                const unsigned long long key = (unsigned long long)item[u] * stride + slot;
                const unsigned peers = __match_any_sync(rest, key);
                if ((threadIdx.x & 31u) == (unsigned)(__ffs(peers) - 1))
                    atomicAdd(hist + key, (unsigned long long)__popc(peers));
            }
        }
    }
    __syncthreads();
    for (uint32_t w = threadIdx.x; w < words; w += kHistThreads) {
        const uint32_t c = cnt[w];      // nonzero only in rows of valid items
        if (c) atomicAdd(hist + (unsigned long long)row0 * stride + w, (unsigned long long)c);
    }
}

template <int NT>
__device__ double block_sum(double v, double *sh)
{
    sh[threadIdx.x] = v;
    __syncthreads();
    for (int o = NT / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    const double r = sh[0];
    __syncthreads();
    return r;
}

constexpr int kSpecThreads = 256;
constexpr uint32_t kPrepThreads = 128;

// Clears the histogram: 16-byte stores between an odd first and last counter (the array may
// start at any counter).
__global__ void __launch_bounds__(kPrepThreads) k_spec_clear(unsigned long long *__restrict__ hist, uint64_t n_hist)
{
    const uint64_t step = (uint64_t)gridDim.x * kPrepThreads;
    const uint64_t t = (uint64_t)blockIdx.x * kPrepThreads + threadIdx.x;
    const uint64_t odd = (reinterpret_cast<uintptr_t>(hist) >> 3) & 1u, pairs = n_hist > odd ? (n_hist - odd) / 2 : 0;
    ulonglong2 *__restrict__ h2 = reinterpret_cast<ulonglong2 *>(hist + odd);
    for (uint64_t i = t; i < pairs; i += step) h2[i] = make_ulonglong2(0ull, 0ull);
    if (t == 0 && odd && n_hist) hist[0] = 0ull;
    if (t == 0 && odd + 2 * pairs < n_hist) hist[n_hist - 1] = 0ull;
}

struct SpecSums {
    double N, mu, S2;      // EXIT paths in the bins, mean weight, sum of c (w - mu)^2
};
static_assert(sizeof(SpecSums) == spectrum_sums_bytes(), "scratch of the callers");

__device__ __forceinline__ void finish_spectrum(const SpecItem &it, double N, double mu, double S2, double *J, double *sigma)
{
    const double T0 = it.T;
    const double P0 = it.A / fabs(it.Z) * sqrt(T0 * (T0 + 2.0 * it.m0));
    const double pref = P0 * P0;
    if (N == 0.0) {
        *J = __longlong_as_double(0x7FF8000000000000ll);
        *sigma = __longlong_as_double(0x7FF8000000000000ll);
    } else {
        *J = pref * mu;
        *sigma = (N > 1.0) ? pref * sqrt(S2 / (N - 1.0) / N) : 0.0;
    }
}

// a + b for sums of nonnegative terms; a group without terms is skipped (adding its 0 would change
// nothing but cost an FP64 slot)
__device__ __forceinline__ double warp_tree(double (&g)[8], uint32_t have)
{
#pragma unroll
    for (int o = 4; o > 0; o >>= 1)
#pragma unroll
        for (int k = 0; k < o; ++k) {
            if (have & (1u << (k + o))) {
                g[k] = (have & (1u << k)) ? g[k] + g[k + o] : g[k + o];
                have |= 1u << k;
            }
        }
    for (int o = 16; o > 0; o >>= 1) g[0] += __shfl_down_sync(0xffffffffu, g[0], o);
    return __shfl_sync(0xffffffffu, g[0], 0);
}

constexpr uint32_t kWarpBins = 4096;       // most bins of the one-warp form
constexpr uint32_t kWarpItems = 4;         // items (warps) per block

// One warp per item.  The sums are FP64-pipe bound (64 clocks a warp instruction), so the form
// counts slots: 32 bins without an exit are passed over, counts become doubles on their bits,
// and the per-item scalars (two square roots, three divisions) are left to k_spectrum_finish,
// which does them for 32 items at a time.  The sums are taken in the order of the 256-thread
// form k_spectrum (eight groups of 32 lanes, then its tree), so both give the same bits.
// Measured, 5760 items of 512 bins: 170 us as one block per item with the weights tabulated,
// 29 + 5 us in this form (and more than 1 ms before, every item evaluating its bins' weights).
__global__ void __launch_bounds__(kWarpItems * 32) k_spectrum_warp(const unsigned long long *__restrict__ hist,
                                                                   uint32_t n_items, uint32_t nbins,
                                                                   const SpecItem *__restrict__ items,
                                                                   const double *__restrict__ weights,
                                                                   SpecSums *__restrict__ sums)
{
    const uint32_t e = blockIdx.x * kWarpItems + (threadIdx.x >> 5), lane = threadIdx.x & 31u;
    if (e >= n_items) return;      // whole warps
    const unsigned long long *h = hist + (size_t)e * (nbins + 3u) + 1u;
    const double *w = weights + (size_t)items[e].sp * nbins;
    double g[8];
    uint32_t have = 0;             // groups with an exit (uniform in the warp)
    unsigned long long cnt = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) g[k] = 0.0;
    auto value = [](unsigned long long n) {
        return n >> 32 ? (double)n : __longlong_as_double((long long)f64bits::from_u32((uint32_t)n));
    };
    for (uint32_t b0 = lane; b0 < nbins + lane; b0 += 256) {
        unsigned long long n[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) n[k] = b0 + 32 * k < nbins ? h[b0 + 32 * k] : 0ull;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            if (!__any_sync(0xffffffffu, n[k] != 0)) continue;
            cnt += n[k];
            const double t = n[k] ? value(n[k]) * w[b0 + 32 * k] : 0.0;
            g[k] = (have & (1u << k)) ? g[k] + t : t;
            have |= 1u << k;
        }
    }
    for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
    const double N = value(cnt);
    const double mu = warp_tree(g, have) / N;
#pragma unroll
    for (int k = 0; k < 8; ++k) g[k] = 0.0;
    have = 0;
    for (uint32_t b0 = lane; b0 < nbins + lane; b0 += 256) {
        unsigned long long n[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) n[k] = b0 + 32 * k < nbins ? h[b0 + 32 * k] : 0ull;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            if (!__any_sync(0xffffffffu, n[k] != 0)) continue;
            const double d = n[k] ? w[b0 + 32 * k] - mu : 0.0;
            const double t = value(n[k]) * d * d;
            g[k] = (have & (1u << k)) ? g[k] + t : t;
            have |= 1u << k;
        }
    }
    const double S2 = warp_tree(g, have);
    if (lane == 0) sums[e] = SpecSums{N, mu, S2};
}

__global__ void k_spectrum_finish(const SpecItem *__restrict__ items, const SpecSums *__restrict__ sums,
                                  uint32_t n_items, double *J, double *sigma)
{
    const uint32_t e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n_items) return;
    finish_spectrum(items[e], sums[e].N, sums[e].mu, sums[e].S2, J + e, sigma + e);
}

// The 256-thread form, one block per item: more bins than one warp should walk through.
__global__ void __launch_bounds__(kSpecThreads) k_spectrum(const unsigned long long *__restrict__ hist,
                                                           uint32_t nbins, double x_lo, double dx,
                                                           const SpecItem *__restrict__ items,
                                                           const double *__restrict__ weights, int lis_kind,
                                                           const double *lnT, const double *lnJ, uint32_t lis_n,
                                                           double *J, double *sigma)
{
    __shared__ double sh[kSpecThreads];
    const uint32_t e = blockIdx.x;
    const SpecItem it = items[e];
    const unsigned long long *h = hist + (size_t)e * (nbins + 3u) + 1u;
    const double *w = weights ? weights + (size_t)it.sp * nbins : nullptr;
    double cnt = 0.0, s1 = 0.0;
    for (uint32_t b = threadIdx.x; b < nbins; b += kSpecThreads) {
        const unsigned long long n = h[b];
        if (n == 0) continue;
        const double c = (double)n;
        cnt += c;
        s1 += c * (w ? w[b] : bin_weight(it, b, x_lo, dx, lis_kind, lnT, lnJ, lis_n));
    }
    const double N = block_sum<kSpecThreads>(cnt, sh);
    const double S1 = block_sum<kSpecThreads>(s1, sh);
    const double mu = S1 / N;
    double s2 = 0.0;
    for (uint32_t b = threadIdx.x; b < nbins; b += kSpecThreads) {
        const unsigned long long n = h[b];
        if (n == 0) continue;
        const double d = (w ? w[b] : bin_weight(it, b, x_lo, dx, lis_kind, lnT, lnJ, lis_n)) - mu;
        s2 += (double)n * d * d;
    }
    const double S2 = block_sum<kSpecThreads>(s2, sh);
    if (threadIdx.x == 0) finish_spectrum(it, N, mu, S2, J + e, sigma + e);
}

// ---- unbinned Eq. 4 ---------------------------------------------------------------
//   momentum form: P0^2 times the mean of J_LIS(T_ex) / P_ex^2
//   energy form:   beta0 times the mean of J_LIS(T_ex) exp(lw) / beta_ex  (lw = -sum L ds)
// FP64-pipe bound, so the analytic spectrum is taken with one pow and
// one division: T^-2.7 / (1 + T^-3.7) = T / (T^3.7 + 1) wherever neither form leaves the range.
__device__ double unbinned_summand(const SpecItem &it, int form, double lnP, double lw, int lis_kind,
                                   const double *lnT, const double *lnJ, uint32_t lis_n)
{
    const double P = exp(lnP);
    const double pn = P * (fabs(it.Z) / it.A);
    const double En = sqrt(pn * pn + it.m0 * it.m0);
    const double T = pn * pn / (En + it.m0);
    double num, den;
    if (lis_kind == 0 && T > 1e-30 && T < 1e30) {
        num = T;
        den = pow(T, 3.7) + 1.0;
    } else {
        num = lis_value(lis_kind, T, lnT, lnJ, lis_n);
        den = 1.0;
    }
    if (form == 0) return num / (den * (P * P));
    return num * exp(lw) * En / (den * pn);
}

constexpr int kUnbThreads = 128;
constexpr uint32_t kUnbPer = 8;        // most exit states a thread takes

struct UnbPartial {
    double n, mean, m2;     // EXIT paths of the chunk, mean summand, sum of squares about it
};

// Bound by the FP64 pipe (about 150 slots a state: two exp, a pow, a square root, two divisions).
// 6e5 states of 30 items: 196 us, against 10 ms with one block per item and two passes.
// One block per chunk of per x 128 consecutive exit states of one item.  The summands stay
// in shared memory for the second moment, which is taken about the chunk's own mean (as exact
// as a second pass over the item, without evaluating anything twice).
__global__ void __launch_bounds__(kUnbThreads) k_unbinned_chunks(ExitPtrs ex, const uint64_t *__restrict__ prefix,
                                                                 const uint64_t *__restrict__ chunk_prefix,
                                                                 uint32_t n_items, uint32_t per,
                                                                 const SpecItem *__restrict__ items, int form,
                                                                 int lis_kind, const double *lnT, const double *lnJ,
                                                                 uint32_t lis_n, UnbPartial *__restrict__ part)
{
    __shared__ double sh[kUnbThreads], v[kUnbPer * kUnbThreads];
    const uint32_t e = find_item(chunk_prefix, n_items, blockIdx.x);
    const SpecItem it = items[e];
    const uint64_t lo = prefix[e] + (blockIdx.x - chunk_prefix[e]) * ((uint64_t)per * kUnbThreads), hi = prefix[e + 1];
    double s1 = 0.0, s2 = 0.0;
    uint32_t have = 0;       // which of the thread's states are EXIT paths
#pragma unroll 1
    for (uint32_t k = 0; k < per; ++k) {
        const uint64_t g = lo + (uint64_t)k * kUnbThreads + threadIdx.x;
        if (g < hi && ex.status[g] == COSMICA_PATH_EXIT) {
            const double f = unbinned_summand(it, form, ex.lnP[g], ex.lw ? ex.lw[g] : 0.0, lis_kind, lnT, lnJ, lis_n);
            v[k * kUnbThreads + threadIdx.x] = f;
            s1 += f;
            have |= 1u << k;
        }
    }
    // the block's scalars by one thread: a division by all four warps is four times its slots
    __shared__ uint32_t s_n;
    __shared__ double s_mean;
    if (threadIdx.x == 0) s_n = 0;
    __syncthreads();
    const uint32_t mine = __reduce_add_sync(0xffffffffu, (uint32_t)__popc(have));
    if ((threadIdx.x & 31u) == 0) atomicAdd(&s_n, mine);
    s1 = block_sum<kUnbThreads>(s1, sh);
    if (threadIdx.x == 0) s_mean = s1 / (double)s_n;
    __syncthreads();
    const double mean = s_mean;
    for (uint32_t k = 0; k < per; ++k) {
        if (have & (1u << k)) {
            const double d = v[k * kUnbThreads + threadIdx.x] - mean;
            s2 += d * d;
        }
    }
    s2 = block_sum<kUnbThreads>(s2, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = UnbPartial{(double)s_n, mean, s2};
}

// One block per item: sum of the chunks' summands and of their squares about the item's mean,
// m2 + n (mean_chunk - mean)^2, in a fixed order.
__global__ void __launch_bounds__(kUnbThreads) k_unbinned_items(const UnbPartial *__restrict__ part,
                                                                const uint64_t *__restrict__ chunk_prefix,
                                                                const SpecItem *__restrict__ items, int form, double *J,
                                                                double *sigma)
{
    __shared__ double sh[kUnbThreads];
    const uint32_t e = blockIdx.x;
    const uint64_t lo = chunk_prefix[e], hi = chunk_prefix[e + 1];
    double cnt = 0.0, s1 = 0.0, s2 = 0.0;
    for (uint64_t c = lo + threadIdx.x; c < hi; c += kUnbThreads) {
        if (part[c].n == 0.0) continue;
        cnt += part[c].n;
        s1 += part[c].n * part[c].mean;
    }
    const double N = block_sum<kUnbThreads>(cnt, sh);
    const double mu = block_sum<kUnbThreads>(s1, sh) / N;
    for (uint64_t c = lo + threadIdx.x; c < hi; c += kUnbThreads) {
        if (part[c].n == 0.0) continue;
        const double d = part[c].mean - mu;
        s2 += part[c].m2 + part[c].n * d * d;
    }
    const double S2 = block_sum<kUnbThreads>(s2, sh);
    if (threadIdx.x == 0) {
        if (N == 0.0) {
            J[e] = __longlong_as_double(0x7FF8000000000000ll);
            sigma[e] = __longlong_as_double(0x7FF8000000000000ll);
        } else {
            const SpecItem it = items[e];
            const double P0 = it.A / fabs(it.Z) * sqrt(it.T * (it.T + 2.0 * it.m0));
            double pref = P0 * P0;
            if (form != 0) {
                const double pn0 = P0 * (fabs(it.Z) / it.A);
                pref = pn0 / sqrt(pn0 * pn0 + it.m0 * it.m0);
            }
            J[e] = pref * mu;
            sigma[e] = (N > 1.0) ? pref * sqrt(S2 / (N - 1.0) / N) : 0.0;
        }
    }
}

}  // namespace

uint64_t unbinned_chunks(uint64_t n, uint32_t per)
{
    return (n + (uint64_t)per * kUnbThreads - 1) / ((uint64_t)per * kUnbThreads);
}
// Exit states a thread takes (at most kUnbPer): a block of 128 fills the FP64 pipe of its SM's four
// schedulers, so a launch lasts the largest number of blocks on an SM times a block's work, some
// 150 slots a state and 60 more for its sums; the size with the shortest such time.  6e5 states of
// 30 items: 196 us with 8 (600 blocks, 3.95 per SM) against 216 with 7 (685, 4.5 per SM).
uint32_t unbinned_per_thread(const uint32_t *n_per_item, uint32_t n_items, int sms)
{
    uint32_t best = kUnbPer;
    uint64_t least = UINT64_MAX;
    for (uint32_t per = 1; per <= kUnbPer; ++per) {
        uint64_t blocks = 0;
        for (uint32_t e = 0; e < n_items; ++e) blocks += unbinned_chunks(n_per_item[e], per);
        const uint64_t cost = (blocks + sms - 1) / sms * (150u * per + 60u);
        if (cost < least) {
            least = cost;
            best = per;
        }
    }
    return best;
}
size_t unbinned_partial_bytes() { return sizeof(UnbPartial); }

cudaError_t launch_spectrum_unbinned(const ExitPtrs &ex, const uint64_t *prefix, const uint64_t *chunk_prefix,
                                     uint64_t n_chunks, uint32_t per, void *partials, uint32_t n_items,
                                     const SpecItem *items, int form, int lis_kind, const double *lis_lnT,
                                     const double *lis_lnJ, uint32_t lis_n, double *J, double *sigma, cudaStream_t s)
{
    if (n_items == 0) return cudaSuccess;
    cudaGetLastError();
    UnbPartial *part = static_cast<UnbPartial *>(partials);
    if (n_chunks > 0) {
        k_unbinned_chunks<<<(unsigned)n_chunks, kUnbThreads, 0, s>>>(ex, prefix, chunk_prefix, n_items, per, items, form,
                                                                     lis_kind, lis_lnT, lis_lnJ, lis_n, part);
        note_launch();
    }
    k_unbinned_items<<<n_items, kUnbThreads, 0, s>>>(part, chunk_prefix, items, form, J, sigma);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_spec_clear(unsigned long long *hist, uint64_t n_hist, cudaStream_t s)
{
    if (n_hist == 0) return cudaSuccess;
    cudaGetLastError();
    const uint64_t blocks = std::min<uint64_t>(2048, (n_hist + 4 * kPrepThreads - 1) / (4 * kPrepThreads));
    k_spec_clear<<<(unsigned)blocks, kPrepThreads, 0, s>>>(hist, n_hist);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_histogram(const ExitPtrs &ex, uint64_t n, uint32_t n_items, uint32_t nbins, double x_lo,
                             double dx, unsigned long long *hist, const WeightTable &wt, int sms, cudaStream_t s)
{
    const uint32_t wblocks = wt.weights ? (uint32_t)(((uint64_t)wt.n_sp * nbins + kHistThreads - 1) / kHistThreads) : 0u;
    if (n_items == 0 || (n == 0 && wblocks == 0)) return cudaSuccess;
    cudaGetLastError();
    // rows of counters that fit (none above 8189 bins: every state then adds to the histogram
    // directly); 1 to 32 states a thread, four blocks per SM first
    const uint32_t rows = nbins <= kHistWords - 3u ? kHistWords / (nbins + 3u) : 0u;
    const uint64_t per = std::min<uint64_t>(32, std::max<uint64_t>(1, n / ((uint64_t)sms * 4 * kHistThreads)));
    const uint64_t blocks = (n + per * kHistThreads - 1) / (per * kHistThreads);
    k_histogram<<<(unsigned)blocks + wblocks, kHistThreads, 0, s>>>(ex, n, n_items, nbins, make_rule(x_lo, dx), rows,
                                                                    (uint32_t)per, hist, wt, wblocks);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_spectrum(const unsigned long long *hist, uint32_t n_items, uint32_t nbins, double x_lo,
                            double dx, const SpecItem *items, const double *weights, int lis_kind,
                            const double *lis_lnT, const double *lis_lnJ, uint32_t lis_n, void *sums, double *J,
                            double *sigma, cudaStream_t s)
{
    if (n_items == 0) return cudaSuccess;
    cudaGetLastError();
    if (weights && sums && nbins <= kWarpBins) {
        SpecSums *d = static_cast<SpecSums *>(sums);
        k_spectrum_warp<<<(n_items + kWarpItems - 1) / kWarpItems, kWarpItems * 32, 0, s>>>(hist, n_items, nbins, items,
                                                                                          weights, d);
        k_spectrum_finish<<<(n_items + 31) / 32, 32, 0, s>>>(items, d, n_items, J, sigma);
        note_launch();
        note_launch();
        return cudaGetLastError();
    }
    k_spectrum<<<n_items, kSpecThreads, 0, s>>>(hist, nbins, x_lo, dx, items, weights, lis_kind, lis_lnT, lis_lnJ,
                                                lis_n, J, sigma);
    note_launch();
    return cudaGetLastError();
}

}  // namespace cosmica
