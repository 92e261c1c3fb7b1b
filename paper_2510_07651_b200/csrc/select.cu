// Pooling + per-head top-budget selection + ordered index emission (Algorithm 2: the num_hh best
// candidates below the cutoff, their indices ascending), and the row gather that builds the compacted cache.
//
//   select_cluster_kernel  one thread-block cluster per (batch item, KV head).  Every CTA pools
//                     its contiguous share of the candidates into order-preserving uint32 keys
//                     held in shared memory; a histogram of their top 11 bits, summed over the
//                     cluster, leaves a few hundred keys, on which every CTA finds the key of the
//                     n_hh-th largest candidate and how many of its ties are kept; the CTAs emit
//                     the kept indices in ascending order.  Bound by the chain of its phases, not
//                     by memory (1 MB of scores at 8 heads of 32768): what a phase costs is barrier
//                     latency and issue slots that all 16 warps spend on the same scalar work, so
//                     sums go through warp reductions, scans run in the one warp that needs them,
//                     four candidates travel per shared-memory access and the last 10 bits are
//                     settled by ranking the few keys left.  8 heads of 32768: 12.0 -> 8.4 us, one
//                     of 1024: 8.8 -> 5.4 (against scans in all warps, one candidate per access
//                     and a third histogram)
//   pool_key_kernel + select_kernel   the same selection with one CTA per head and the keys in
//                     global memory: the path for sequences too long for a cluster's shared memory
//   gather_kernel     16-byte vector copy of the kept K/V rows (and optionally their scores)
#include "obc_common.cuh"

#include <cooperative_groups.h>
#include <mutex>
namespace cg = cooperative_groups;

namespace obc {

namespace {

// fp32 -> uint32 whose unsigned order equals the float order; -0.0 is folded onto +0.0
__device__ __forceinline__ uint32_t float_key(float x) {
    uint32_t u = __float_as_uint(x + 0.0f);          // -0.0 + 0.0 = +0.0
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__device__ __forceinline__ int seq_len(const SelectShape& s, int b) { return s.seq_lens ? s.seq_lens[b] : s.Nmax; }
__device__ __forceinline__ int budget_of(const SelectShape& s, int b) { return s.budgets ? s.budgets[b] : s.budget; }

// key of token p of a head with scores sc: the pooled score of a candidate (lo <= p < hi), 0 (below every candidate) elsewhere
__device__ __forceinline__ uint32_t pooled_key(const SelectShape& s, const float* __restrict__ sc, int p, int lo, int hi) {
    if (p < lo || p >= hi) return 0u;
    const int half = s.pool_kernel / 2;
    float val;
    if (s.pool_mode == OBC_POOL_NONE || s.pool_kernel == 1) {
        val = sc[p];
    } else if (s.pool_mode == OBC_POOL_MAX) {
        val = -INFINITY;
        for (int t = p - half; t <= p + half; ++t)
            if (t >= lo && t < hi) val = fmaxf(val, sc[t]);
    } else {
        val = 0.f;
        for (int t = p - half; t <= p + half; ++t)
            if (t >= lo && t < hi) val = __fadd_rn(val, sc[t]);
        val = __fdiv_rn(val, (float)s.pool_kernel);
    }
    return float_key(val);
}

// Four consecutive pooled values from the twelve staged scores f that begin with the first value's first tap; 2 H + 1 taps
template <int H>
__device__ __forceinline__ float4 pool4(const float (&f)[12], int mode, float kernel) {
    float v[4];
    if (mode == OBC_POOL_MAX) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            v[j] = -INFINITY;
#pragma unroll
            for (int t = 0; t <= 2 * H; ++t) v[j] = fmaxf(v[j], f[j + t]);     // padding taps are -inf
        }
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) {                                          // ascending index order; padding adds +0
            v[j] = 0.f;
#pragma unroll
            for (int t = 0; t <= 2 * H; ++t) v[j] = __fadd_rn(v[j], f[j + t]);
            v[j] = __fdiv_rn(v[j], kernel);
        }
    }
    return make_float4(v[0], v[1], v[2], v[3]);
}

// The same for stage[i ..], i a multiple of four, with three reads of four scores each; kernels up to 7 (half <= 3).
// stage[i] holds the first tap of value i, and is readable up to stage[i + 11].
__device__ __forceinline__ float4 pool4_staged(const float* stage, int half, int mode, int kernel) {
    float f[12];
    *reinterpret_cast<float4*>(&f[0]) = *reinterpret_cast<const float4*>(stage);
    if (half > 0) *reinterpret_cast<float4*>(&f[4]) = *reinterpret_cast<const float4*>(stage + 4);
    if (half > 2) *reinterpret_cast<float4*>(&f[8]) = *reinterpret_cast<const float4*>(stage + 8);
    if (half == 0) return make_float4(f[0], f[1], f[2], f[3]);
    if (half == 1) return pool4<1>(f, mode, (float)kernel);
    if (half == 2) return pool4<2>(f, mode, (float)kernel);
    return pool4<3>(f, mode, (float)kernel);
}

__global__ void __launch_bounds__(256)
pool_key_kernel(SelectShape s, const float* __restrict__ scores, uint32_t* __restrict__ keys) {
    pdl_wait();
    const int unit = blockIdx.y, b = unit / s.Hkv;
    const int N = seq_len(s, b), lo = s.n_sink, hi = N - s.n_recent;
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= s.Nmax) return;
    keys[(size_t)unit * s.Nmax + p] = pooled_key(s, scores + (size_t)unit * s.Nmax, p, lo, hi);
}

// ---- head-adaptive budgets --------------------------------------------------------------------------------
// Every head keeps its n_safe best candidates; the other rem = H (n_hh - n_safe) slots of a batch item go to the best
// remaining candidates of all its heads.  With cnt_h(x) = candidates of head h whose key is at least x, the heads keep
// F(x) = sum_h max(0, cnt_h(x) - n_safe) tokens beyond their guaranteed ones if x is the threshold, so the threshold T is
// the largest key with F(T) >= rem, and what a head keeps is its own best max(n_safe, cnt_h(T + 1)) + (its share of the
// candidates equal to T) tokens: only the COUNTS have to be found across heads, and the per-head selection does the rest.
// T comes out of three histogram levels per head (11 + 11 + 10 bits) over the whole chip:
//   adaptive_pool_kernel   pooled keys, level-1 histograms
//   adaptive_hist_kernel   (levels 2 and 3) every CTA finds the digit of the level before, then counts its keys below it,
//                          the first of which it asked for before the search
//   the selection kernels  last digit, tie shares, scored tokens of the head
// Every histogram row comes with 32 sums over equal runs of its bins, so that a digit is found in two round trips to L2
// (32 runs of every head, then the bins of one run) by any CTA that needs it.
// Latency bound: 8 heads x 32k keys 3.5 + 4.2 + 4.7 us and 7.7 us in the selection, which asks for its keys before the search
// as well (with the keys asked for behind the searches, and one candidate pooled at a time from global memory instead of four
// from shared memory, 5.4 + 4.6 + 5.2 and 8.4 us).  (Ranking
// all heads' keys as one sequence in one 16-CTA cluster took 20 us for the former and, where the keys did not fit one, by
// one CTA, 1.07 ms for the latter.)
constexpr int AD_NT = 512;
constexpr int AD_EARLY = 4;                                    // keys per thread that a histogram kernel asks for first
constexpr int AD_BINS = 2048;                 // bins of levels 1 and 2; level 3 has half of them
constexpr int AD_ROW = AD_BINS + 32;          // a head's row: bins, then the sums over 32 runs of them

struct AdaptiveLevels {                       // in the workspace; scores across heads are ranked when hist != null
    uint32_t* hist;                           // [3 levels][units][AD_ROW]
    uint32_t* above;                          // [2][units]: candidates above the digits of level 1, of levels 1 and 2
    uint32_t* digit;                          // [B][2]: level-1 and level-2 digit of T
    int32_t* counts;                          // [units]: tokens kept per head, or -1 (the caller's)
    uint32_t n_safe;
    int chunk;                                // keys per CTA of the passes
    int units;
    __device__ __forceinline__ uint32_t* row(int level, int unit) const { return hist + ((size_t)level * units + unit) * AD_ROW; }
};

struct AdaptiveFind { uint32_t run_sum[32], bin_sum[64], run, digit; };     // shared memory of the search

__device__ __forceinline__ uint32_t warp_suffix(uint32_t x) {               // sum over the lanes >= lane
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_down_sync(0xffffffffu, x, o);
        if (lane + o < 32) x += t;
    }
    return x;
}

// Largest bin d of level LEVEL (0..2) with sum_h max(0, above[h] + (candidates of head h in bins >= d) - n_safe) >= rem,
// over the H heads from unit u0 on.  All threads of the block call it.
template <int LEVEL>
__device__ uint32_t adaptive_find(const AdaptiveLevels& lv, int u0, int H, uint32_t rem, AdaptiveFind& sh) {
    constexpr int PER = LEVEL == 2 ? 32 : 64;                  // bins per run
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, warps = (int)blockDim.x >> 5;
    const uint32_t* above = LEVEL == 0 ? nullptr : lv.above + (size_t)(LEVEL - 1) * lv.units + u0;
    auto beyond = [&](uint32_t c) { return c > lv.n_safe ? c - lv.n_safe : 0u; };
    if (tid < 32) sh.run_sum[tid] = 0;
    if (tid < 64) sh.bin_sum[tid] = 0;
    if (tid == 0) { sh.run = 0; sh.digit = 0; }
    __syncthreads();
    for (int h = warp; h < H; h += warps) {
        const uint32_t c = warp_suffix(lv.row(LEVEL, u0 + h)[AD_BINS + lane]) + (above ? above[h] : 0u);
        if (beyond(c)) atomicAdd(&sh.run_sum[lane], beyond(c));
    }
    __syncthreads();
    if (tid < 32 && sh.run_sum[tid] >= rem && (tid == 31 || sh.run_sum[tid + 1] < rem)) sh.run = (uint32_t)tid;
    __syncthreads();
    const int run = (int)sh.run;
    for (int h = warp; h < H; h += warps) {
        const uint32_t* row = lv.row(LEVEL, u0 + h);
        const uint32_t runs = row[AD_BINS + lane];
        const uint32_t x0 = row[run * PER + lane], x1 = PER == 64 ? row[run * PER + 32 + lane] : 0u;
        uint32_t up = warp_suffix(lane > run ? runs : 0u);     // candidates in the runs above, in lane 0
        up = __shfl_sync(0xffffffffu, up, 0) + (above ? above[h] : 0u);
        const uint32_t s1 = warp_suffix(x1), s0 = warp_suffix(x0) + __shfl_sync(0xffffffffu, s1, 0);
        if (beyond(up + s0)) atomicAdd(&sh.bin_sum[lane], beyond(up + s0));
        if (PER == 64 && beyond(up + s1)) atomicAdd(&sh.bin_sum[32 + lane], beyond(up + s1));
    }
    __syncthreads();
    if (tid < PER && sh.bin_sum[tid] >= rem && (tid == PER - 1 || sh.bin_sum[tid + 1] < rem)) sh.digit = (uint32_t)(run * PER + tid);
    __syncthreads();
    return sh.digit;
}

// candidates of the unit above the digits found so far, level LEVEL's being d (called by a whole warp, same result in every lane)
template <int LEVEL>
__device__ __forceinline__ uint32_t adaptive_above(const AdaptiveLevels& lv, int unit, uint32_t d) {
    constexpr int PER = LEVEL == 2 ? 32 : 64;
    const int lane = threadIdx.x & 31, run = (int)d / PER, at = (int)d % PER;
    const uint32_t* row = lv.row(LEVEL, unit);
    uint32_t x = lane > run ? row[AD_BINS + lane] : 0u;
    if (lane > at) x += row[run * PER + lane];
    if (PER == 64 && lane + 32 > at) x += row[run * PER + 32 + lane];
    x = __shfl_sync(0xffffffffu, warp_suffix(x), 0);
    return x + (LEVEL == 0 ? 0u : lv.above[(size_t)(LEVEL - 1) * lv.units + unit]);
}

// slots of a batch item's heads beyond the guaranteed ones; -1 when the budget does not fit the sequence
__device__ __forceinline__ int adaptive_rem(const SelectShape& s, int b, uint32_t n_safe) {
    const int N = seq_len(s, b), lo = s.n_sink, hi = N - s.n_recent, n_hh = s.budget - s.n_sink - s.n_recent;
    if (N > s.Nmax || hi < lo || n_hh < 0 || n_hh > hi - lo) return -1;
    return s.Hkv * (n_hh - (int)n_safe);
}

// What head `unit` keeps: n_hh scored tokens (-1: the budget does not fit), found from the last digit of T and the tie
// shares.  Where the head has n_safe candidates at or above T they are those above T and the first k_eq equal to T, and
// the head needs no search of its own (`known`).  All threads of the block call it.
struct HeadShare { int n_hh; bool known; uint32_t T, k_eq; };
__device__ HeadShare adaptive_share(const SelectShape& s, const AdaptiveLevels& lv, int unit, AdaptiveFind& sh) {
    const int b = unit / s.Hkv, u0 = b * s.Hkv, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = (int)blockDim.x >> 5;
    const int rem = adaptive_rem(s, b, lv.n_safe);
    if (rem <= 0) return HeadShare{rem < 0 ? -1 : (int)lv.n_safe, false, 0u, 0u};
    const uint32_t d = adaptive_find<2>(lv, u0, s.Hkv, (uint32_t)rem, sh);
    auto beyond = [&](uint32_t c) { return c > lv.n_safe ? c - lv.n_safe : 0u; };
    // sums over the heads: slots that the candidates above T take, and candidates equal to T of the heads before this one
    if (threadIdx.x < 2) sh.run_sum[threadIdx.x] = 0;
    __syncthreads();
    for (int h = warp; h < s.Hkv; h += warps) {
        const uint32_t up = adaptive_above<2>(lv, u0 + h, d), ties = beyond(up + lv.row(2, u0 + h)[d]) - beyond(up);
        if (lane == 0) {
            atomicAdd(&sh.run_sum[0], beyond(up));
            if (u0 + h < unit) atomicAdd(&sh.run_sum[1], ties);
            if (u0 + h == unit) { sh.bin_sum[0] = up; sh.bin_sum[1] = ties; sh.bin_sum[2] = lv.row(2, unit)[d]; }
        }
    }
    __syncthreads();
    const uint32_t left = (uint32_t)rem - sh.run_sum[0], before = sh.run_sum[1], up = sh.bin_sum[0], ties = sh.bin_sum[1];
    const uint32_t hh = max(lv.n_safe, up) + (before < left ? min(ties, left - before) : 0u);           // ties: lowest head first
    const uint32_t T = lv.digit[b * 2] << 21 | lv.digit[b * 2 + 1] << 10 | d;
    const bool known = up + sh.bin_sum[2] >= lv.n_safe;
    return HeadShare{(int)hh, known, known ? T : 0u, known ? hh - up : 0u};
}

// adds a CTA's histogram of `bins` bins to the unit's row, with the sums over its 32 runs
__device__ __forceinline__ void adaptive_flush(const uint32_t* hist, int bins, uint32_t* row) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, per = bins / 32;
    for (int i = tid; i < bins; i += AD_NT)
        if (hist[i]) atomicAdd(&row[i], hist[i]);
    for (int r = warp; r < 32; r += AD_NT / 32) {
        uint32_t x = hist[r * per + lane];
        if (per == 64) x += hist[r * per + 32 + lane];
        x = warp_suffix(x);
        if (lane == 0 && x) atomicAdd(&row[AD_BINS + r], x);
    }
}

// (a kernel instead of a memset, which would keep the kernels before and after it from overlapping its ends)
__global__ void __launch_bounds__(AD_NT)
adaptive_clear_kernel(uint4* hist, long long n) {
    pdl_wait();
    const long long i = (long long)blockIdx.x * AD_NT + threadIdx.x;
    if (i < n) hist[i] = make_uint4(0u, 0u, 0u, 0u);
}

__global__ void __launch_bounds__(AD_NT)
adaptive_pool_kernel(SelectShape s, const float* __restrict__ scores, uint32_t* __restrict__ keys, AdaptiveLevels lv) {
    __shared__ uint32_t hist[AD_BINS];
    const int unit = blockIdx.y, b = unit / s.Hkv, c0 = blockIdx.x * lv.chunk, c1 = min(c0 + lv.chunk, s.Nmax);
    for (int d = threadIdx.x; d < AD_BINS; d += AD_NT) hist[d] = 0;
    __syncthreads();
    pdl_wait();
    const int lo = s.n_sink, hi = min(seq_len(s, b), s.Nmax) - s.n_recent;
    const float* sc = scores + (size_t)unit * s.Nmax;
    uint32_t* out = keys + (size_t)unit * s.Nmax;
    const int half = s.pool_mode == OBC_POOL_NONE ? 0 : s.pool_kernel / 2, tid = threadIdx.x;
    if (half <= 3) {                                           // four values per thread out of staged scores
        constexpr int BLOCK = 4 * AD_NT;
        __shared__ __align__(16) float stage[BLOCK + 8];
        const float pad = s.pool_mode == OBC_POOL_MAX ? -INFINITY : 0.f;
        for (int base = c0; base < c1; base += BLOCK) {
            float val[5];
#pragma unroll
            for (int u = 0; u < 5; ++u) {
                const int i = u * AD_NT + tid, p = base + i - half;
                val[u] = i < BLOCK + 2 * half && p >= lo && p < hi ? sc[p] : pad;
            }
#pragma unroll
            for (int u = 0; u < 5; ++u)
                if (u * AD_NT + tid < BLOCK + 2 * half) stage[u * AD_NT + tid] = val[u];
            __syncthreads();
            const int p0 = base + tid * 4;
            const float4 v = pool4_staged(stage + tid * 4, half, s.pool_mode, s.pool_kernel);
            const float v4[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int p = p0 + j;
                if (p >= c1) continue;
                const uint32_t key = p >= lo && p < hi ? float_key(v4[j]) : 0u;
                out[p] = key;
                if (key) atomicAdd(&hist[key >> 21], 1u);
            }
            __syncthreads();
        }
    } else {
        for (int p = c0 + tid; p < c1; p += AD_NT) {
            const uint32_t key = pooled_key(s, sc, p, lo, hi);
            out[p] = key;
            if (key) atomicAdd(&hist[key >> 21], 1u);
        }
    }
    __syncthreads();
    adaptive_flush(hist, AD_BINS, lv.row(0, unit));
}

// level 2 or 3: the digit that the level before settles, then the histogram of the keys that share the digits so far
template <int LEVEL>
__global__ void __launch_bounds__(AD_NT)
adaptive_hist_kernel(SelectShape s, const uint32_t* __restrict__ keys, AdaptiveLevels lv) {
    __shared__ uint32_t hist[AD_BINS];
    __shared__ AdaptiveFind sh;
    constexpr int BINS = LEVEL == 2 ? 2048 : 1024;
    for (int d = threadIdx.x; d < BINS; d += AD_NT) hist[d] = 0;
    pdl_wait();
    const int unit = blockIdx.y, b = unit / s.Hkv, u0 = b * s.Hkv, c0 = blockIdx.x * lv.chunk, c1 = min(c0 + lv.chunk, s.Nmax);
    const uint32_t* kin = keys + (size_t)unit * s.Nmax;
    uint32_t early[AD_EARLY];                                  // these keys travel while the digit is looked for
#pragma unroll
    for (int u = 0; u < AD_EARLY; ++u) {
        const int p = c0 + u * AD_NT + threadIdx.x;
        early[u] = p < c1 ? kin[p] : 0u;
    }
    const int rem = adaptive_rem(s, b, lv.n_safe);
    if (rem <= 0) return;                                      // nothing to share out (adaptive_share sees to it)
    const uint32_t d = adaptive_find<LEVEL - 2>(lv, u0, s.Hkv, (uint32_t)rem, sh);
    if (unit == u0 && blockIdx.x == 0) {                       // one CTA per batch item leaves the result for the next level
        for (int h = threadIdx.x >> 5; h < s.Hkv; h += AD_NT / 32) {
            const uint32_t up = adaptive_above<LEVEL - 2>(lv, u0 + h, d);
            if ((threadIdx.x & 31) == 0) lv.above[(size_t)(LEVEL - 2) * lv.units + u0 + h] = up;
        }
        if (threadIdx.x == 0) lv.digit[b * 2 + (LEVEL - 2)] = d;
    }
    const uint32_t prefix = LEVEL == 2 ? d : lv.digit[b * 2] << 11 | d;
    constexpr int SHIFT = LEVEL == 2 ? 21 : 10, NEXT = LEVEL == 2 ? 10 : 0;
#pragma unroll
    for (int u = 0; u < AD_EARLY; ++u)
        if (c0 + u * AD_NT + (int)threadIdx.x < c1 && early[u] >> SHIFT == prefix) atomicAdd(&hist[(early[u] >> NEXT) & (BINS - 1)], 1u);
#pragma unroll 8
    for (int p = c0 + AD_EARLY * AD_NT + threadIdx.x; p < c1; p += AD_NT) {
        const uint32_t key = kin[p];
        if (key >> SHIFT == prefix) atomicAdd(&hist[(key >> NEXT) & (BINS - 1)], 1u);
    }
    __syncthreads();
    adaptive_flush(hist, BINS, lv.row(LEVEL - 1, unit));
}

constexpr int SEL_NT = 1024;

__global__ void __launch_bounds__(SEL_NT)
select_kernel(SelectShape s, const uint32_t* __restrict__ keys_all, int32_t* __restrict__ idx_all, AdaptiveLevels ad) {
    pdl_wait();
    __shared__ uint32_t hist[256];
    __shared__ uint32_t sh_prefix, sh_remaining;
    __shared__ uint32_t warp_gt[32], warp_eq[32];

    const int unit = blockIdx.x, b = unit / s.Hkv;
    const int N = seq_len(s, b);
    const int lo = s.n_sink, hi = N - s.n_recent, n = hi - lo;
    __shared__ AdaptiveFind ad_sh;
    HeadShare share{budget_of(s, b) - s.n_sink - s.n_recent, false, 0u, 0u};
    if (ad.hist) share = adaptive_share(s, ad, unit, ad_sh);
    const int n_hh = share.n_hh;
    const int budget = n_hh + s.n_sink + s.n_recent;
    const uint32_t* keys = keys_all + (size_t)unit * s.Nmax;
    int32_t* idx = idx_all + (size_t)unit * s.idx_stride;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    if (n_hh < 0 || n_hh > n || budget > s.idx_stride || N > s.Nmax || hi < lo) {   // bad per-sequence budget
        for (int j = tid; j < s.idx_stride; j += SEL_NT) idx[j] = -1;
        if (ad.hist && tid == 0) ad.counts[unit] = -1;
        return;
    }
    if (ad.hist && tid == 0) ad.counts[unit] = budget;
    // protected ranges and padding
    for (int j = tid; j < s.n_sink; j += SEL_NT) idx[j] = j;
    for (int j = tid; j < s.n_recent; j += SEL_NT) idx[s.n_sink + n_hh + j] = hi + j;
    for (int j = budget + tid; j < s.idx_stride; j += SEL_NT) idx[j] = -1;
    if (n_hh == 0) return;

    // ---- radix search for the key T of the n_hh-th largest candidate -----------------------
    uint32_t prefix = share.T, mask = 0, remaining = share.known ? share.k_eq : (uint32_t)n_hh;
    for (int shift = 24; shift >= 0 && !share.known; shift -= 8) {
        if (tid < 256) hist[tid] = 0;
        __syncthreads();
        for (int base = 0; base < n; base += SEL_NT) {
            const int i = base + tid;
            const bool in = i < n;
            const uint32_t key = in ? keys[lo + i] : 0u;
            const bool pred = in && ((key & mask) == prefix);
            const unsigned act = __ballot_sync(0xffffffffu, pred);
            if (pred) {
                const uint32_t dgt = (key >> shift) & 255u;
                const unsigned peers = __match_any_sync(act, dgt);
                if (lane == __ffs(peers) - 1) atomicAdd(&hist[dgt], (uint32_t)__popc(peers));
            }
        }
        __syncthreads();
        if (warp == 0) {
            // lane owns bins [8*lane, 8*lane+8); find the highest bin D with
            // count(bins > D) < remaining <= count(bins >= D)
            uint32_t loc[8], tot = 0;
#pragma unroll
            for (int j = 0; j < 8; ++j) { loc[j] = hist[lane * 8 + j]; tot += loc[j]; }
            uint32_t above = 0;                                  // sum over lanes > lane
            uint32_t incl = tot;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                uint32_t t = __shfl_down_sync(0xffffffffu, incl, o);
                if (lane + o < 32) incl += t;
            }
            above = incl - tot;
            if (above < remaining && remaining <= above + tot) {
                uint32_t run = above;
#pragma unroll
                for (int j = 7; j >= 0; --j) {
                    if (run < remaining && remaining <= run + loc[j]) {
                        sh_prefix = prefix | ((uint32_t)(lane * 8 + j) << shift);
                        sh_remaining = remaining - run;
                        run = 0xffffffffu;                       // found: stop matching
                    } else if (run != 0xffffffffu) {
                        run += loc[j];
                    }
                }
            }
        }
        __syncthreads();
        prefix = sh_prefix; remaining = sh_remaining; mask |= 255u << shift;
        __syncthreads();
    }
    const uint32_t T = prefix, k_eq = remaining;      // keep all keys > T and the first k_eq keys == T

    // ---- ordered emission: each warp owns a contiguous segment of the candidates -----------
    const int seg = ((n + 31) / 32 + 31) / 32 * 32;
    const int s0 = warp * seg, s1 = min(s0 + seg, n);
    uint32_t cgt = 0, ceq = 0;
    for (int i = s0 + lane; i < s1; i += 32) {
        const uint32_t key = keys[lo + i];
        cgt += key > T; ceq += key == T;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        cgt += __shfl_xor_sync(0xffffffffu, cgt, o);
        ceq += __shfl_xor_sync(0xffffffffu, ceq, o);
    }
    if (lane == 0) { warp_gt[warp] = cgt; warp_eq[warp] = ceq; }
    __syncthreads();
    uint32_t gt_before = 0, eq_before = 0;
    for (int w = 0; w < warp; ++w) { gt_before += warp_gt[w]; eq_before += warp_eq[w]; }
    uint32_t eq_run = eq_before;
    uint32_t out = s.n_sink + gt_before + min(eq_before, k_eq);
    const unsigned lt_mask = (1u << lane) - 1u;
    for (int base = s0; base < s1; base += 32) {
        const int i = base + lane;
        const uint32_t key = i < s1 ? keys[lo + i] : 0u;
        const bool is_eq = i < s1 && key == T;
        const unsigned beq = __ballot_sync(0xffffffffu, is_eq);
        const bool sel = i < s1 && (key > T || (is_eq && eq_run + __popc(beq & lt_mask) < k_eq));
        const unsigned bsel = __ballot_sync(0xffffffffu, sel);
        if (sel) idx[out + __popc(bsel & lt_mask)] = lo + i;
        out += __popc(bsel);
        eq_run += __popc(beq);
    }
}

// ---- cluster path ----------------------------------------------------------------------------
constexpr int CL_NT = 512;                    // threads per CTA
constexpr int CL_BINS = 2048;                 // 11-bit digits
constexpr int CL_MAX_SEG = 20 * 1024;         // candidates per CTA (two 4-byte shared arrays of this size)

constexpr int CL_GATHER = 2 * CL_BINS;        // survivors of the first pass that every CTA can hold (all CTAs' lists together):
                                              // they lie over the histograms of passes 1 and 2, which are used only when the lists do not fit

struct ClusterShared {                        // fixed part of the CTA's shared memory
    uint32_t sum[3][CL_BINS];                 // per radix pass: histogram of the whole head (every CTA adds into every copy)
    uint32_t local[CL_BINS];                  // this CTA's histogram of the current pass
    uint32_t found[3];                        // result of a pass: digit, remaining, keys that share the digit
    uint32_t n_list, n_above;                 // candidates of this CTA that survive the first pass, and that lie in higher bins
    uint32_t n_few, few[32];                  // keys that share all but the last 10 bits of T, if there are no more than 32
    uint32_t rank_gt[16], rank_eq[16];        // kept-candidate counts of every CTA of the cluster
    uint32_t rank_list[16], rank_above[16];   // per CTA: survivors of the first pass, candidates in higher bins
    uint32_t before[2];                       // kept candidates (greater, equal) in the CTAs before this one
    uint32_t warp_gt[CL_NT / 32], warp_eq[CL_NT / 32];
    uint32_t scan[CL_NT / 32];
    // slot r of the gathered lists: the survivors of CTA r (CL_GATHER / C keys each), in the space of sum[1] and sum[2]
    __device__ __forceinline__ uint32_t* gathered() { return &sum[1][0]; }
};

// The highest bin D of hist[0 .. CL_BINS) with count(bins > D) < remaining <= count(bins >= D), found by the
// whole CTA (thread t owns bins [4t, 4t+4)); found = D, remaining - count(bins > D), count(bin D).  Only the warp that
// owns D looks further than its total: with all of them scanning, issue slots were what this step waited for.
__device__ __forceinline__ void find_bin(const uint32_t* hist, uint32_t remaining, uint32_t* scan, uint32_t* found) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint4 q = reinterpret_cast<const uint4*>(hist)[tid];
    const uint32_t tot = q.x + q.y + q.z + q.w, wtot = __reduce_add_sync(0xffffffffu, tot);
    if (lane == 0) scan[warp] = wtot;
    __syncthreads();
    const uint32_t above_w = __reduce_add_sync(0xffffffffu, lane > warp && lane < CL_NT / 32 ? scan[lane] : 0u);
    if (above_w < remaining && remaining <= above_w + wtot) {
        uint32_t run = above_w + warp_suffix(tot) - tot;           // keys in the bins above this thread's
        if (run < remaining && remaining <= run + tot) {
            int d = 3;
            uint32_t c = q.w;
            if (remaining > run + c) { run += c; d = 2; c = q.z; }
            if (d == 2 && remaining > run + c) { run += c; d = 1; c = q.y; }
            if (d == 1 && remaining > run + c) { run += c; d = 0; c = q.x; }
            found[0] = (uint32_t)(tid * 4 + d);
            found[1] = remaining - run;
            found[2] = c;
        }
    }
    __syncthreads();
}

// ADAPTIVE: the budgets are shared out across the heads, and the pooled keys are there already (keys_in, [units][Nmax])
template <bool ADAPTIVE>
__global__ void __launch_bounds__(CL_NT)
select_cluster_kernel(SelectShape s, const float* __restrict__ scores, int32_t* __restrict__ idx_all, int seg_cap,
                      const uint32_t* __restrict__ keys_in, AdaptiveLevels ad) {
    extern __shared__ __align__(16) uint8_t sel_smem[];
    ClusterShared& sh = *reinterpret_cast<ClusterShared*>(sel_smem);
    uint32_t* keys = reinterpret_cast<uint32_t*>(sel_smem + ((sizeof(ClusterShared) + 15) & ~(size_t)15));   // 16-byte aligned
    float* stage = reinterpret_cast<float*>(keys + seg_cap);          // seg_cap + pool_kernel - 1 floats, and room to read four more
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    cg::cluster_group cluster = cg::this_cluster();
    const int C = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const int lC = __ffs(C) - 1;                   // C is a power of two, up to the number of warps
    auto clear = [&](uint32_t* hist) { reinterpret_cast<uint4*>(hist)[tid] = make_uint4(0u, 0u, 0u, 0u); };
    static_assert(CL_BINS == 4 * CL_NT, "four bins per thread");
    auto reset = [&]() {
        clear(sh.sum[0]);
        clear(sh.local);
        if (tid == 0) { sh.n_list = 0; sh.n_above = 0; sh.n_few = 0; sh.before[0] = 0; sh.before[1] = 0; }
    };
    if (!ADAPTIVE) reset();
    pdl_wait();
    const int unit = blockIdx.x >> lC, b = unit / s.Hkv;
    const int N = seq_len(s, b);
    const int lo = s.n_sink, hi = N - s.n_recent, n = hi - lo;
    // this CTA's share of the candidates: [c0, c1) of [0, n)
    const int seg = (((n + C - 1) >> lC) + 31) / 32 * 32;
    const int c0 = min(rank * seg, n), c1 = min(c0 + seg, n), m = c1 - c0;
    if (ADAPTIVE && N <= s.Nmax) {                 // the keys travel while the head's share is looked for
        const uint32_t* kin = keys_in + (size_t)unit * s.Nmax + lo + c0;
        for (int i = tid; i < m; i += CL_NT)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(keys + i)), "l"(kin + i) : "memory");
    }
    // (the search across heads borrows the space of a histogram that is cleared behind it)
    HeadShare share{budget_of(s, b) - s.n_sink - s.n_recent, false, 0u, 0u};
    if (ADAPTIVE) {
        share = adaptive_share(s, ad, unit, *reinterpret_cast<AdaptiveFind*>(&sh.local[0]));
        __syncthreads();
        reset();
    }
    if (ADAPTIVE) asm volatile("cp.async.wait_all;" ::: "memory");  // (before any way out of the kernel)
    const int n_hh = share.n_hh;
    const int budget = n_hh + s.n_sink + s.n_recent;
    int32_t* idx = idx_all + (size_t)unit * s.idx_stride;
    const int gtid = rank * CL_NT + tid, gthreads = C * CL_NT;

    // these tests depend on the unit only, so all CTAs of the cluster leave together
    if (n_hh < 0 || n_hh > n || budget > s.idx_stride || N > s.Nmax || hi < lo) {   // bad per-sequence budget
        for (int j = gtid; j < s.idx_stride; j += gthreads) idx[j] = -1;
        if (ADAPTIVE && gtid == 0) ad.counts[unit] = -1;
        return;
    }
    if (ADAPTIVE && gtid == 0) ad.counts[unit] = budget;
    for (int j = gtid; j < s.n_sink; j += gthreads) idx[j] = j;
    for (int j = gtid; j < s.n_recent; j += gthreads) idx[s.n_sink + n_hh + j] = hi + j;
    for (int j = budget + gtid; j < s.idx_stride; j += gthreads) idx[j] = -1;
    if (n_hh == 0) return;

    if (ADAPTIVE) {
        __syncthreads();
        cluster.barrier_arrive();
        if (!share.known)
            for (int i = tid; i < m; i += CL_NT) atomicAdd(&sh.local[keys[i] >> 21], 1u);
    } else {
        // pooled keys: stage the scores with their halo, then pool out of shared memory
        const float* sc = scores + (size_t)unit * s.Nmax;
        const int half = (s.pool_mode == OBC_POOL_NONE) ? 0 : s.pool_kernel / 2;
        const float pad = s.pool_mode == OBC_POOL_MAX ? -INFINITY : 0.f;
        // nine loads in flight per thread: a share of 4096 candidates and its halo travel in one round trip
        constexpr int LD = 9;
        for (int base = 0; base < m + 2 * half; base += LD * CL_NT) {
            float val[LD];
    #pragma unroll
            for (int u = 0; u < LD; ++u) {
                const int i = base + u * CL_NT + tid, p = lo + c0 + i - half;
                val[u] = (i < m + 2 * half && p >= lo && p < hi) ? sc[p] : pad;
            }
    #pragma unroll
            for (int u = 0; u < LD; ++u) {
                const int i = base + u * CL_NT + tid;
                if (i < m + 2 * half) stage[i] = val[u];
            }
        }
        __syncthreads();
        cluster.barrier_arrive();                      // this CTA's histograms are clear: others may add to them after their wait
        // wide kernels beforehand, one candidate per thread and step, so that the lanes of a warp read consecutive taps: 64 heads of
        // 65536, 9 / 31 / 101 taps: 36 / 47 / 87 us, against 47 / 97 / 250 with four consecutive candidates per thread (four-way bank
        // conflicts).  (Keys and histogram in the same loop made narrow kernels 0.1 to 0.3 us slower.)
        if (half > 3) {
            float* pooled = reinterpret_cast<float*>(keys);
            for (int i = tid; i < m; i += CL_NT) {
                float val = pad;
                if (s.pool_mode == OBC_POOL_MAX) for (int t = 0; t <= 2 * half; ++t) val = fmaxf(val, stage[i + t]);
                else for (int t = 0; t <= 2 * half; ++t) val = __fadd_rn(val, stage[i + t]);
                pooled[i] = s.pool_mode == OBC_POOL_MAX ? val : __fdiv_rn(val, (float)s.pool_kernel);
            }
            __syncthreads();
        }
        // four candidates per thread and step; the top 11 bits of their keys go straight into the first histogram
        for (int i = tid * 4; i < m; i += CL_NT * 4) {
            const float4 v = half <= 3 ? pool4_staged(stage + i, half, s.pool_mode, s.pool_kernel) : *reinterpret_cast<const float4*>(keys + i);
            const uint4 k4 = make_uint4(float_key(v.x), float_key(v.y), float_key(v.z), float_key(v.w));
            *reinterpret_cast<uint4*>(keys + i) = k4;      // (a share has room for a multiple of 32 keys)
            atomicAdd(&sh.local[k4.x >> 21], 1u);
            if (i + 1 < m) atomicAdd(&sh.local[k4.y >> 21], 1u);
            if (i + 2 < m) atomicAdd(&sh.local[k4.z >> 21], 1u);
            if (i + 3 < m) atomicAdd(&sh.local[k4.w >> 21], 1u);
        }
    }
    __syncthreads();                               // keys and this CTA's histogram of their top bits are complete
    // (the first cluster barrier is split: arrival above, once this CTA's histograms were clear; the wait comes just
    // before the first remote additions, behind the pooling and the first local histogram)
    cluster.barrier_wait();

    // ---- radix search for the key T of the n_hh-th largest candidate ---------------------------
    // The top 11 bits come from the histogram of all keys.  Every CTA adds its non-empty bins into the `sum`
    // copy of every CTA of the cluster, so that after one cluster barrier each CTA finds by itself the bin D that
    // holds the n_hh-th largest key.  The keys of bin D (a few hundred of a 32k-token head) are copied to a list,
    // and every CTA hands its list, and how many of its candidates lie in the bins above D, to all the others:
    // after a second barrier each CTA settles the remaining 21 bits on its own copy of all the lists and knows
    // what the CTAs before it keep, without further exchanges.  Only when the lists do not fit their slots (keys
    // that all but coincide) do passes 1 and 2 run across the cluster as pass 0 did.
    uint32_t* list = reinterpret_cast<uint32_t*>(stage);
    // (A threshold that the ranking across heads has settled needs no search.)
    uint32_t T = share.T, k_eq = share.k_eq;       // keep all keys > T and the first k_eq keys == T
    bool before_known = C == 1;                    // sh.before[] holds what the CTAs before this one keep
    if (!share.known) {
        auto spread = [&](int pass) {              // this CTA's histogram into every copy of the head's
            for (int bin = tid; bin < CL_BINS; bin += CL_NT) {
                const uint32_t c = sh.local[bin];
                if (c) for (int r = 0; r < C; ++r) atomicAdd(cluster.map_shared_rank(&sh.sum[pass][bin], r), c);
            }
            cluster.sync();
        };
        if (C > 1) spread(0);
        find_bin(C > 1 ? sh.sum[0] : sh.local, (uint32_t)n_hh, sh.scan, sh.found);
        const uint32_t digit = sh.found[0];
        T = digit << 21;
        k_eq = sh.found[1];
        // the keys of bin D -> list (any order); candidates of this CTA in the bins above D
        uint32_t above = 0;
        for (int i = tid * 4; i < m; i += CL_NT * 4) {
            const uint4 q = *reinterpret_cast<const uint4*>(keys + i);
            const uint32_t k4[4] = {q.x, q.y, q.z, q.w};
            uint32_t c = 0;
#pragma unroll
            for (int j = 0; j < 4; ++j) { above += i + j < m && k4[j] >> 21 > digit; c += i + j < m && k4[j] >> 21 == digit; }
            if (c) {                               // few threads: one shared-memory atomic each
                uint32_t at = atomicAdd(&sh.n_list, c);
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (i + j < m && k4[j] >> 21 == digit) list[at++] = k4[j];
            }
        }
        above = __reduce_add_sync(0xffffffffu, above);
        if (lane == 0 && above) atomicAdd(&sh.n_above, above);
        __syncthreads();                           // the list and its length are complete
        clear(sh.local);
        const int nl = (int)sh.n_list, slot_cap = C > 1 ? CL_GATHER >> lC : m;
        const int slot = warp & (C - 1), first = (warp >> lC) * 32 + lane, step = (CL_NT / 32 >> lC) * 32;   // warp w serves CTA w mod C
        if (C > 1) {
            if (tid < C) {                         // length and higher-bin count into every CTA
                cluster.map_shared_rank(&sh.rank_list[0], tid)[rank] = (uint32_t)nl;
                cluster.map_shared_rank(&sh.rank_above[0], tid)[rank] = sh.n_above;
            }
            if (nl <= slot_cap) {                  // the keys themselves, into slot `rank` of every CTA
                uint32_t* dst = cluster.map_shared_rank(sh.gathered(), slot) + rank * slot_cap;
                for (int i = first; i < nl; i += step) dst[i] = list[i];
            }
            cluster.sync();                        // lists and counts have arrived everywhere
        } else {
            __syncthreads();
        }
        const uint32_t my_len = C > 1 ? (lane < C ? sh.rank_list[lane] : 0u) : (uint32_t)nl;
        if ((int)__reduce_max_sync(0xffffffffu, my_len) <= slot_cap) {         // (the same answer in every CTA)
            // ---- the remaining 21 bits, on this CTA's copy of all lists (no cluster traffic) ----
            const uint32_t* g = C > 1 ? sh.gathered() + slot * slot_cap : list;
            const int ng = C > 1 ? (int)sh.rank_list[slot] : nl;
            for (int i = first; i < ng; i += step) atomicAdd(&sh.local[(g[i] >> 10) & 2047u], 1u);
            __syncthreads();
            find_bin(sh.local, k_eq, sh.scan, sh.found);
            T |= sh.found[0] << 10;
            k_eq = sh.found[1];
            const int same = (int)sh.found[2];
            if (same <= 32) {                      // all but always: every warp ranks the keys that are left
                for (int i = first; i < ng; i += step)
                    if (g[i] >> 10 == T >> 10) sh.few[atomicAdd(&sh.n_few, 1u)] = g[i];
                __syncthreads();
                const uint32_t key = lane < same ? sh.few[lane] : 0u;
                uint32_t gt = 0, ge = 0;
                for (int j = 0; j < same; ++j) {
                    const uint32_t other = __shfl_sync(0xffffffffu, key, j);
                    gt += other > key;
                    ge += other >= key;
                }
                const int at = __ffs(__ballot_sync(0xffffffffu, lane < same && gt < k_eq && k_eq <= ge)) - 1;
                T = __shfl_sync(0xffffffffu, key, at);
                k_eq -= __shfl_sync(0xffffffffu, gt, at);
            } else {
                clear(sh.local);
                __syncthreads();
                for (int i = first; i < ng; i += step)
                    if (g[i] >> 10 == T >> 10) atomicAdd(&sh.local[g[i] & 1023u], 1u);
                __syncthreads();
                find_bin(sh.local, k_eq, sh.scan, sh.found);
                T |= sh.found[0];
                k_eq = sh.found[1];
            }
            if (C > 1) {
                // what the CTAs before this one keep: their candidates above bin D, and of their lists the keys > T, == T
                uint32_t bg = tid < rank ? sh.rank_above[tid] : 0u, be = 0;
                if (slot < rank)
                    for (int i = first; i < ng; i += step) { bg += g[i] > T; be += g[i] == T; }
                bg = __reduce_add_sync(0xffffffffu, bg);
                be = __reduce_add_sync(0xffffffffu, be);
                if (lane == 0 && (bg | be)) { atomicAdd(&sh.before[0], bg); atomicAdd(&sh.before[1], be); }
                before_known = true;               // published by the barrier behind the counts below
            }
        } else {
            // the exchanged passes 1 and 2 add into the histograms that the lists have overwritten: clear them
            // everywhere before any CTA adds to another's copy
            clear(sh.sum[1]);
            clear(sh.sum[2]);
            cluster.sync();
            for (int pass = 1; pass < 3; ++pass) {
                const int known = pass == 1 ? 21 : 10, shift = pass == 1 ? 10 : 0;
                for (int i = tid; i < nl; i += CL_NT)
                    if (list[i] >> known == T >> known) atomicAdd(&sh.local[(list[i] >> shift) & (pass == 1 ? 2047u : 1023u)], 1u);
                __syncthreads();
                spread(pass);
                clear(sh.local);
                find_bin(sh.sum[pass], k_eq, sh.scan, sh.found);
                T |= sh.found[0] << shift;
                k_eq = sh.found[1];
            }
        }
    }

    // ---- ordered emission: each warp owns a contiguous run of this CTA's candidates ------------------------------
    const int wseg = ((m + CL_NT / 32 - 1) / (CL_NT / 32) + 31) / 32 * 32;
    const int s0 = min(warp * wseg, m), s1 = min(s0 + wseg, m);
    uint32_t cgt = 0, ceq = 0;
#pragma unroll 4
    for (int i = s0 + lane; i < s1; i += 32) {
        const uint32_t key = keys[i];
        cgt += key > T; ceq += key == T;
    }
    cgt = __reduce_add_sync(0xffffffffu, cgt);
    ceq = __reduce_add_sync(0xffffffffu, ceq);
    if (lane == 0) { sh.warp_gt[warp] = cgt; sh.warp_eq[warp] = ceq; }
    __syncthreads();
    const uint32_t wg = lane < CL_NT / 32 ? sh.warp_gt[lane] : 0u, we = lane < CL_NT / 32 ? sh.warp_eq[lane] : 0u;
    if (!before_known) {                           // the CTAs' totals were not derived from the lists: exchange them
        const uint32_t tg = __reduce_add_sync(0xffffffffu, wg), te = __reduce_add_sync(0xffffffffu, we);
        if (tid < C) {                             // this CTA's totals into every CTA of the cluster
            cluster.map_shared_rank(&sh.rank_gt[0], tid)[rank] = tg;
            cluster.map_shared_rank(&sh.rank_eq[0], tid)[rank] = te;
        }
        cluster.sync();
        if (tid == 0) {
            uint32_t bg = 0, be = 0;
            for (int r = 0; r < rank; ++r) { bg += sh.rank_gt[r]; be += sh.rank_eq[r]; }
            sh.before[0] = bg; sh.before[1] = be;
        }
        __syncthreads();
    }
    uint32_t gt_run = sh.before[0] + __reduce_add_sync(0xffffffffu, lane < warp ? wg : 0u);   // kept candidates before the block at hand
    uint32_t eq_run = sh.before[1] + __reduce_add_sync(0xffffffffu, lane < warp ? we : 0u);
    const unsigned lt_mask = (1u << lane) - 1u;
    int32_t* out = idx + s.n_sink;
#pragma unroll 4
    for (int base = s0; base < s1; base += 32) {
        const int i = base + lane;
        const uint32_t key = i < s1 ? keys[i] : 0u;
        const bool is_gt = i < s1 && key > T, is_eq = i < s1 && key == T;
        const unsigned mg = __ballot_sync(0xffffffffu, is_gt), me = __ballot_sync(0xffffffffu, is_eq);
        const uint32_t eq_at = eq_run + __popc(me & lt_mask);       // equal keys before this one: the first k_eq of them are kept
        if (is_gt || (is_eq && eq_at < k_eq)) out[gt_run + __popc(mg & lt_mask) + min(eq_at, k_eq)] = lo + c0 + i;
        gt_run += __popc(mg);
        eq_run += __popc(me);
    }
}

// four 16-byte vectors of K and of V per thread, all loads issued before the first store (`vecs`
// vectors per row; a thread's vectors are a quarter of the unit's vectors apart)
__global__ void __launch_bounds__(256)
gather_kernel(int units, int Hkv, int idx_stride, int vecs, int elem_bytes,
              TensorView k, TensorView v, TensorView ko, TensorView vo,
              const int32_t* __restrict__ idx, const float* __restrict__ s_in, float* __restrict__ s_out, int Nmax, uint32_t zero_rows) {
    pdl_wait();
    const int unit = blockIdx.y, b = unit / Hkv, g = unit % Hkv;
    const int total = idx_stride * vecs, quarter = (total + 3) / 4;
    const int e0 = blockIdx.x * blockDim.x + threadIdx.x;
    if (e0 >= quarter) return;
    const size_t eb = (size_t)elem_bytes;
    const char* kb = (const char*)k.ptr + ((size_t)b * k.sb + (size_t)g * k.sh) * eb;
    const char* vb = (const char*)v.ptr + ((size_t)b * v.sb + (size_t)g * v.sh) * eb;
    char* kob = (char*)ko.ptr + ((size_t)b * ko.sb + (size_t)g * ko.sh) * eb;
    char* vob = (char*)vo.ptr + ((size_t)b * vo.sb + (size_t)g * vo.sh) * eb;
    int src[4], j[4], c[4];
    bool pad[4];                                           // the row exists and its index is negative
    uint4 kv[4], vv[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int e = e0 + u * quarter;
        j[u] = e / vecs; c[u] = e % vecs;
        src[u] = e < total ? idx[(size_t)unit * idx_stride + j[u]] : -1;
        pad[u] = e < total && src[u] < 0;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
        if (src[u] >= 0) {
            kv[u] = __ldg(reinterpret_cast<const uint4*>(kb + (size_t)src[u] * k.st * eb) + c[u]);
            vv[u] = __ldg(reinterpret_cast<const uint4*>(vb + (size_t)src[u] * v.st * eb) + c[u]);
        }
#pragma unroll
    for (int u = 0; u < 4; ++u)
        if (src[u] >= 0) {
            reinterpret_cast<uint4*>(kob + (size_t)j[u] * ko.st * eb)[c[u]] = kv[u];
            reinterpret_cast<uint4*>(vob + (size_t)j[u] * vo.st * eb)[c[u]] = vv[u];
            if (s_in && c[u] == 0) s_out[(size_t)unit * idx_stride + j[u]] = s_in[(size_t)unit * Nmax + src[u]];
        } else if (zero_rows && pad[u]) {            // padding rows of outputs that nobody has cleared
            const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
            if (zero_rows & OBC_ZERO_K) reinterpret_cast<uint4*>(kob + (size_t)j[u] * ko.st * eb)[c[u]] = zero;
            if (zero_rows & OBC_ZERO_V) reinterpret_cast<uint4*>(vob + (size_t)j[u] * vo.st * eb)[c[u]] = zero;
            if ((zero_rows & OBC_ZERO_SCORES) && c[u] == 0) s_out[(size_t)unit * idx_stride + j[u]] = 0.f;
        }
}


// First position of the ascending array a[0, n) whose value is >= v (n if none), found by the whole block: every
// round the threads probe evenly spaced positions of the remaining range at once, so 16384 entries take three
// round trips to memory where a binary search by one thread takes fourteen.  Called by all threads of the block.
template <typename Less>
__device__ __forceinline__ int block_lower_bound(int n, Less value_below) {
    int lo = 0, hi = n;
    while (hi > lo) {
        const int step = (hi - lo + (int)blockDim.x - 1) / (int)blockDim.x;
        const int pos = lo + (int)threadIdx.x * step;
        const int cnt = __syncthreads_count(pos < hi && value_below(pos));   // the probes below v are a prefix
        if (cnt == 0) { hi = lo; }
        else { const int last = lo + (cnt - 1) * step; lo = last + 1; hi = min(last + step, hi); }
    }
    return lo;
}

// A token shard's share of the kept indices: row (b, h) of idx is ascending (padding -1 at the end), so the entries
// in [t0, t0 + n) are one stretch, found by binary search; written relative to the shard, padded with -1.
__global__ void __launch_bounds__(256)
shard_indices_kernel(int idx_stride, int t0, int n, const int32_t* __restrict__ idx_all,
                     int32_t* __restrict__ local_all, int32_t* __restrict__ counts) {
    pdl_wait();
    const int unit = blockIdx.x;
    const int32_t* idx = idx_all + (size_t)unit * idx_stride;
    int32_t* local = local_all + (size_t)unit * idx_stride;
    auto lower_bound = [&](int v) {                       // first entry >= v; the -1 padding counts as past every token
        return block_lower_bound(idx_stride, [&](int i) { const int x = idx[i]; return x >= 0 && x < v; });
    };
    const int seg0 = lower_bound(t0), seg1 = lower_bound(t0 + n), c = seg1 - seg0;
    for (int j = threadIdx.x; j < idx_stride; j += blockDim.x) local[j] = j < c ? idx[seg0 + j] - t0 : -1;
    if (threadIdx.x == 0) counts[unit] = c;
}

}  // namespace

obc_status launch_shard_indices(int units, int idx_stride, int t0, int n, const int32_t* idx, int32_t* local, int32_t* counts,
                                cudaStream_t stream) {
    ProfScope ps("shard_indices", stream);
    OBC_CUDA_TRY(launch_pdl(shard_indices_kernel, dim3((unsigned)units), dim3(256), 0, stream, 1, idx_stride, t0, n, idx, local, counts));
    return OBC_OK;
}

size_t select_workspace_bytes(int B, int Hkv, int Nmax) { return align_up((size_t)B * Hkv * Nmax * 4, 256); }

// Cluster size for the one-cluster-per-head path, or 0 when a head does not fit a cluster's shared memory.  A CTA takes
// 4.3 us and 0.57 us per 1024 candidates, a cluster 1.2 to 1.8 us more, so heads of up to 4096 tokens take one CTA (8 heads:
// 6.2 / 6.7 / 6.5 / 6.4 us for 1 / 2 / 4 / 8 CTAs) and longer ones as many as run side by side, one CTA per SM (8 heads of
// 8192: 8.7 / 7.8 / 6.9 / 6.7; 16 heads: 8.9 / 7.9 / 6.9 / 7.9; 64 heads: 9.0 / 8.1 / 8.8 / 15.6; 128 heads: 9.2 / 10.4 / 16.4 /
// 29.8; 32 heads of 32768: - / 15.5 / 11.0 / 11.6), sixteen only above 2048 candidates per CTA (4 heads of 16384: 7.1 with
// eight, 7.2 with sixteen; of 32768: 8.6 / 8.0).  Above 8192 candidates an SM holds one CTA only: such shares are split
// further whatever runs side by side (256 heads of 32768: 60 us with two CTAs, 56 with four; 16 heads of 65536: 16.1 with
// four, 14.9 with eight; of 131072: 36 with eight, 32 with sixteen; 128 heads of 131072: 163 / 172).
// A pooling kernel so wide that a share and its halo do not fit takes smaller shares.
static size_t select_cluster_smem(int seg, int pool_kernel) { return sizeof(ClusterShared) + (size_t)seg * 8 + (size_t)pool_kernel * 4 + 32; }

// How many clusters of 2, 4, 8 and 16 CTAs, one per SM, the current device runs at once (74, 33, 15 and 7 on 148 SMs), asked once per
// host thread and device.
struct ClustersAtOnce { int dev, of[4]; };
static const ClustersAtOnce& clusters_at_once() {
    thread_local ClustersAtOnce seen{-1, {}};
    int dev = -1, optin = 0;
    if (cudaGetDevice(&dev) == cudaSuccess && dev == seen.dev) return seen;
    const auto kernel = select_cluster_kernel<false>;
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    cfg.blockDim = dim3(CL_NT); cfg.attrs = attr; cfg.numAttrs = 1;
    (void)cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cfg.dynamicSmemBytes = (size_t)optin;                      // all of it (the kernel has no static part): one CTA per SM
    const bool ok = optin > 0 && allow_smem(kernel, cfg.dynamicSmemBytes) == cudaSuccess &&
                    cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
    for (int i = 0; i < 4; ++i) {
        attr[0].val.clusterDim.x = 2u << i;
        cfg.gridDim = dim3(2u << i);
        if (!ok || cudaOccupancyMaxActiveClusters(&seen.of[i], kernel, &cfg) != cudaSuccess) seen.of[i] = 0;
    }
    (void)cudaGetLastError();
    seen.dev = dev;
    return seen;
}

static int select_cluster_size(int units, int Nmax, int pool_kernel, int* seg_cap) {
    constexpr size_t kMost = 227 * 1024;                       // dynamic shared memory of a CTA
    auto seg_of = [&](int C) { return ((Nmax + C - 1) / C + 31) / 32 * 32; };
    int C = 1;
    if (Nmax > 4096) {
        const ClustersAtOnce& at_once = clusters_at_once();
        for (int i = 0; C < 16 && (units <= at_once.of[i] ? C < 8 || seg_of(C) > 2048 : seg_of(C) > 8192 && (C < 8 || units <= 32)); ++i) C *= 2;
    }
    while (C < 16 && (seg_of(C) > CL_MAX_SEG || select_cluster_smem(seg_of(C), pool_kernel) > kMost)) C *= 2;
    if (seg_of(C) > CL_MAX_SEG) return 0;
    *seg_cap = seg_of(C);
    return C;
}

// keys_in: when given, [units][Nmax] keys that take the place of pooling `scores` (which may then be null);
// `ws` is then not written
static obc_status launch_select_impl(const SelectShape& s, const float* scores, const uint32_t* keys_in, AdaptiveLevels ad, int32_t* idx,
                                     void* ws, cudaStream_t stream);
obc_status launch_select(const SelectShape& s, const float* scores, int32_t* idx, void* ws, cudaStream_t stream) {
    return launch_select_impl(s, scores, nullptr, AdaptiveLevels{}, idx, ws, stream);
}
static obc_status launch_select_impl(const SelectShape& s, const float* scores, const uint32_t* keys_in, AdaptiveLevels ad, int32_t* idx,
                                     void* ws, cudaStream_t stream) {
    const int units = s.B * s.Hkv;
    int seg_cap = 0;
    const int C = select_cluster_size(units, s.Nmax, s.pool_kernel, &seg_cap);
    if (C > 0) {
        const size_t smem = select_cluster_smem(seg_cap, s.pool_kernel);
        const bool adaptive = keys_in != nullptr;
        const auto kernel = adaptive ? select_cluster_kernel<true> : select_cluster_kernel<false>;
        OBC_CUDA_TRY(allow_smem(kernel, smem));
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3((unsigned)(units * C)); cfg.blockDim = dim3(CL_NT); cfg.dynamicSmemBytes = smem; cfg.stream = stream;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)C; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr; cfg.numAttrs = 1;
        // whether the device can host such a cluster depends on the cluster size and the shared memory alone: asked once
        // per (kernel, device, size, bytes) and remembered (the query costs as much host time as the launch)
        thread_local struct { bool adaptive; int dev, C; size_t smem; int max_clusters; } seen[8] = {};
        thread_local int seen_next = 0;
        int dev = -1, max_clusters = -1;
        (void)cudaGetDevice(&dev);
        for (const auto& e : seen) if (e.C == C && e.smem == smem && e.dev == dev && e.adaptive == adaptive) max_clusters = e.max_clusters;
        if (max_clusters < 0) {
            if (C > 8) OBC_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
            if (cudaOccupancyMaxActiveClusters(&max_clusters, kernel, &cfg) != cudaSuccess) { max_clusters = 0; (void)cudaGetLastError(); }
            seen[seen_next] = {adaptive, dev, C, smem, max_clusters};
            seen_next = (seen_next + 1) % 8;
        }
        if (max_clusters > 0) {
            { ProfScope ps("select_cluster", stream);
              OBC_CUDA_TRY(launch_pdl(kernel, dim3((unsigned)(units * C)), dim3(CL_NT), smem, stream, C, s, scores, idx, seg_cap, keys_in, ad)); }
            return OBC_OK;
        }
        (void)cudaGetLastError();                  // the device cannot host such a cluster: one CTA per head
    }
    if (keys_in) {
        { ProfScope ps("select", stream); OBC_CUDA_TRY(launch_pdl(select_kernel, dim3(units), dim3(SEL_NT), 0, stream, 1, s, keys_in, idx, ad)); }
        return OBC_OK;
    }
    uint32_t* keys = (uint32_t*)ws;
    { ProfScope ps("pool_key", stream); OBC_CUDA_TRY(launch_pdl(pool_key_kernel, dim3((s.Nmax + 255) / 256, units), dim3(256), 0, stream, 1, s, scores, keys)); }
    { ProfScope ps("select", stream); OBC_CUDA_TRY(launch_pdl(select_kernel, dim3(units), dim3(SEL_NT), 0, stream, 1, s, (const uint32_t*)keys, idx, AdaptiveLevels{})); }
    return OBC_OK;
}

// ---- allocation-free variant: the key scratch is part of the library image -----------------------
// One key per score, shared by every call on the device (see obc_select_noalloc in obcache.h).
static __device__ __align__(256) uint32_t g_select_keys[OBC_SELECT_NOALLOC_MAX_KEYS];

// Device address of g_select_keys on the current device.  In host code the array's name only
// stands for the symbol; the address a kernel can use comes from the runtime, per device.
static obc_status select_static_keys(uint32_t** out) {
    constexpr int kMaxDev = 64;
    static std::mutex mu;
    static uint32_t* ptrs[kMaxDev] = {};
    int dev = 0;
    OBC_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDev) return OBC_ERR_UNSUPPORTED;
    std::lock_guard<std::mutex> lk(mu);
    if (!ptrs[dev]) {
        uint32_t* ptr = nullptr;
        OBC_CUDA_TRY(cudaGetSymbolAddress((void**)&ptr, g_select_keys));
        if (!ptr) return OBC_ERR_CUDA;
        ptrs[dev] = ptr;
    }
    *out = ptrs[dev];
    return OBC_OK;
}

obc_status launch_select_static(const SelectShape& s, const float* scores, int32_t* idx, cudaStream_t stream) {
    const int units = s.B * s.Hkv;
    if ((long long)units * s.Nmax > (long long)OBC_SELECT_NOALLOC_MAX_KEYS) return OBC_ERR_CAPACITY;
    uint32_t* keys = nullptr;
    obc_status st = select_static_keys(&keys);
    if (st != OBC_OK) return st;
    // every key a head reads is written by pool_key_kernel of this call: nothing has to be cleared
    { ProfScope ps("pool_key", stream); OBC_CUDA_TRY(launch_pdl(pool_key_kernel, dim3((s.Nmax + 255) / 256, units), dim3(256), 0, stream, 1, s, scores, keys)); }
    { ProfScope ps("select", stream); OBC_CUDA_TRY(launch_pdl(select_kernel, dim3(units), dim3(SEL_NT), 0, stream, 1, s, (const uint32_t*)keys, idx, AdaptiveLevels{})); }
    return OBC_OK;
}

obc_status launch_gather(int B, int Hkv, int idx_stride, int Nmax, int elem_bytes,
                         TensorView k, TensorView v, TensorView ko, TensorView vo, const int32_t* idx,
                         const float* s_in, float* s_out, uint32_t zero_rows, cudaStream_t stream) {
    const int vecs = kD * elem_bytes / 16;
    const long long total = ((long long)idx_stride * vecs + 3) / 4;    // four vectors per thread
    {
        ProfScope ps("gather", stream);
        OBC_CUDA_TRY(launch_pdl(gather_kernel, dim3((unsigned)((total + 255) / 256), B * Hkv), dim3(256), 0, stream, 1,
                                B * Hkv, Hkv, idx_stride, vecs, elem_bytes, k, v, ko, vo, idx, s_in, s_out, Nmax, zero_rows));
    }
    return OBC_OK;
}

// ---- head-adaptive budgets -------------------------------------------------------------------------------
// workspace: the three histogram levels of every head (cleared by the call) | pooled keys | small results of the search
struct AdaptivePlan { size_t off_hist, off_keys, off_above, off_digit, bytes; };
static AdaptivePlan make_adaptive_plan(const SelectShape& s) {
    AdaptivePlan p{};
    const size_t units = (size_t)s.B * s.Hkv;
    size_t off = 0;
    p.off_hist = off;  off = align_up(off + 3 * units * AD_ROW * 4, 256);
    p.off_keys = off;  off = align_up(off + units * s.Nmax * 4, 256);
    p.off_above = off; off = align_up(off + 2 * units * 4, 256);
    p.off_digit = off; off = align_up(off + (size_t)s.B * 8, 256);
    p.bytes = off;
    return p;
}
size_t select_adaptive_workspace_bytes(const SelectShape& s) { return make_adaptive_plan(s).bytes; }

obc_status launch_select_adaptive(const SelectShape& s, int n_safe, const float* scores, int32_t* idx, int32_t* counts,
                                  void* ws, cudaStream_t stream) {
    const AdaptivePlan plan = make_adaptive_plan(s);
    const int units = s.B * s.Hkv;
    char* w = (char*)ws;
    uint32_t* keys = (uint32_t*)(w + plan.off_keys);
    // about two CTAs per SM: each of them repeats the search through the heads' histograms
    const long long ctas = 2LL * sm_count(), per = ((long long)units * s.Nmax + ctas - 1) / ctas;
    const int chunk = (int)(per < 2048 ? 2048 : (per + AD_NT - 1) / AD_NT * AD_NT);
    const AdaptiveLevels lv{(uint32_t*)(w + plan.off_hist), (uint32_t*)(w + plan.off_above), (uint32_t*)(w + plan.off_digit), counts,
                            (uint32_t)n_safe, chunk, units};
    const dim3 grid((unsigned)((s.Nmax + chunk - 1) / chunk), (unsigned)units);
    const long long n_clear = 3LL * units * AD_ROW / 4;
    { ProfScope ps("adaptive_clear", stream);
      OBC_CUDA_TRY(launch_pdl(adaptive_clear_kernel, dim3((unsigned)((n_clear + AD_NT - 1) / AD_NT)), dim3(AD_NT), 0, stream, 1, (uint4*)lv.hist, n_clear)); }
    { ProfScope ps("adaptive_pool", stream); OBC_CUDA_TRY(launch_pdl(adaptive_pool_kernel, grid, dim3(AD_NT), 0, stream, 1, s, scores, keys, lv)); }
    { ProfScope ps("adaptive_hist", stream); OBC_CUDA_TRY(launch_pdl(adaptive_hist_kernel<2>, grid, dim3(AD_NT), 0, stream, 1, s, (const uint32_t*)keys, lv)); }
    { ProfScope ps("adaptive_hist", stream); OBC_CUDA_TRY(launch_pdl(adaptive_hist_kernel<3>, grid, dim3(AD_NT), 0, stream, 1, s, (const uint32_t*)keys, lv)); }
    return launch_select_impl(s, nullptr, keys, lv, idx, nullptr, stream);
}

}  // namespace obc
