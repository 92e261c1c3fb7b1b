// Tensor-core score path for bf16 caches (sm_100a: TMA + tcgen05 MMA with TMEM accumulators).
//
// Pass 2, the fused score kernel, runs here.  For one tile of 128 cached tokens and one chunk of
// up to 128 window rows it issues two contractions with the TOKENS on the MMA M dimension,
//     Z^T = K_tile . Q_chunk^T          (logits,           Sec. 3)
//     T'^T = V_tile . (-2 O_chunk)^T    (-2 v_p . o_r,     Algorithm 1's "VO" term)
// so that a TMEM lane holds one token and an epilogue thread sums that token's score terms
// (Eq. 4-6 in the expanded form of Algorithm 1) over all rows of the chunk serially in registers:
// the sum over window queries and the GQA group (App. A.5) needs no cross-thread reduction and no
// W x N matrix ever leaves the SM.
//
// Warp roles of the 640-thread CTA (persistent, one CTA per SM):
//   warp 0      TMA producer: K/V tiles into a 2-stage ring, Q / -2O when the unit changes
//   warp 1      MMA issuer (one elected lane), double-buffered TMEM accumulators (2 x 256 columns)
//   warps 2-3   idle when pass 1 ran (its two spare warps computed ||v_p||^2 with the V tile at hand);
//               otherwise (attention outputs supplied by the caller, or the l1 variant) the value norms of every tile
//   warps 4-11  epilogue of the even tiles, warps 12-19 epilogue of the odd tiles.  Each tile has two
//               warpgroups: both hold one token per thread (a warp reads the TMEM lanes 32 (warp mod 4) ..),
//               the first sums the first half of the window rows, the second the other half and hands
//               its sums over through shared memory; the first adds them and stores the token's scores.
//               (One warpgroup per tile spent most of its time waiting on its own dependent instructions:
//               an SM sub-partition then runs two epilogue warps; with four it hides them.)
//
// Every mbarrier wait is bounded: on a timeout the kernel raises the status word in the workspace
// header, stops issuing work, waits (bounded) for its own copies in flight, frees TMEM and returns.
#include "obc_common.cuh"

#include <cuda.h>
#include <cudaTypedefs.h>

namespace obc {
namespace {

constexpr int TILE = 128;                       // tokens per tile = MMA M
constexpr unsigned kObcVariants = OBC_VAR_V | OBC_VAR_K | OBC_VAR_VK;      // Eq. 4-6
constexpr unsigned kAllVariants = OBC_VAR_V | OBC_VAR_K | OBC_VAR_VK | OBC_VAR_ATTN | OBC_VAR_VATP;
constexpr int NSTAGE = 2;
constexpr int MC_ROWS = 64;                     // window rows per chunk of the multi-chunk pass 2
constexpr uint32_t kHalfBytes = 128 * 128;      // [128 rows][64 bf16] = 16 KB, one swizzle-128B block
constexpr uint32_t kOperandBytes = 2 * kHalfBytes;
constexpr int kThreads = 640;                   // single-chunk pass 2: 4 service warps + 4 epilogue warpgroups
constexpr int kThreadsBase = 384;               // the multi-chunk pass 2 keeps two epilogue warpgroups
constexpr unsigned long long kWaitNs = 2000000000ull;   // 2 s per wait

// ---- shared memory map (offsets from a 1024-byte aligned base) ------------------------------
constexpr uint32_t OFF_Q = 0;
constexpr uint32_t OFF_O = OFF_Q + kOperandBytes;
constexpr uint32_t OFF_K = OFF_O + kOperandBytes;                 // NSTAGE x 32 KB
constexpr uint32_t OFF_V = OFF_K + NSTAGE * kOperandBytes;        // NSTAGE x 32 KB
constexpr uint32_t OFF_CONST = OFF_V + NSTAGE * kOperandBytes;    // 16 epilogue warps x 32 float4 (row-pair constants of the warp's half)
constexpr int NSLOT = 4;                                          // ring depth of the per-tile value norms
constexpr uint32_t OFF_NV = OFF_CONST + 16 * 32 * 16;             // NSLOT x 128 x (||v||^2, ||v||_1), own-norm kernels only
constexpr int kNumSums = 7;                                       // running sums a token carries (RowSums)
constexpr uint32_t OFF_XCH = OFF_NV + NSLOT * TILE * 8;           // [tile parity][2][kNumSums][128] floats: the second half's sums
constexpr uint32_t OFF_BAR = OFF_XCH + 2 * 2 * kNumSums * TILE * 4;
constexpr uint32_t kNumBars = 2 * NSTAGE + 2 + 4 + 2 + 2 * NSLOT + 4;
constexpr uint32_t OFF_TMEM = OFF_BAR + kNumBars * 8;
constexpr uint32_t kSmemBytes = OFF_TMEM + 16 + 1024;             // + alignment slack

enum { BAR_FULL = 0, BAR_EMPTY = NSTAGE, BAR_QO_FULL = 2 * NSTAGE, BAR_QO_EMPTY = 2 * NSTAGE + 1,
       BAR_TM_FULL = 2 * NSTAGE + 2,      // [epilogue group][TMEM buffer]
       BAR_TM_EMPTY = 2 * NSTAGE + 6,     // [TMEM buffer]
       BAR_NV = 2 * NSTAGE + 8,           // [epilogue group][slot], own-norm kernels only
       BAR_XCH = 2 * NSTAGE + 8 + 2 * NSLOT };   // [tile parity][2]: the second row half's sums are in shared memory

// ---- PTX wrappers ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
template <bool CLUSTER = false>                    // CLUSTER: what other CTAs of the cluster stored before they arrived is visible, too
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    if (CLUSTER) {
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
        return ok != 0;
    }
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// Device-side extent of a kernel: every CTA folds its first and last clock reading into two words of
// the workspace header (both by atomicMax, the start as its complement, so that zeros mean "no
// reading").  obc_score_kernel_spans() reads and zeroes them.
// (Taken by a thread that has nothing urgent to do at either end: thread 0 issues the first copies.)
__device__ __forceinline__ void span_begin(unsigned long long* span) {
    if (threadIdx.x == 96) atomicMax(span, ~global_ns());
}
__device__ __forceinline__ void span_end(unsigned long long* span) {
    if (threadIdx.x == 96) atomicMax(span + 1, global_ns());
}
// bounded wait: false after kWaitNs without completion
template <bool CLUSTER = false>
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
    if (mbar_try<CLUSTER>(bar, parity)) return true;
    const unsigned long long t0 = global_ns();
    for (;;) {
#pragma unroll 1
        for (int i = 0; i < 64; ++i)
            if (mbar_try<CLUSTER>(bar, parity)) return true;
        if (global_ns() - t0 > kWaitNs) return false;
    }
}

__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, uint32_t bar,
                                            int c0, int c1, int c2, int c3) {
    asm volatile("cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
                 ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3) : "memory");
}
// the same copy with an L2 eviction-priority hint (a policy made by l2_policy_*)
__device__ __forceinline__ void tma_load_4d_hint(uint32_t dst, const CUtensorMap* map, uint32_t bar,
                                                 int c0, int c1, int c2, int c3, uint64_t policy) {
    asm volatile("cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4, %5, %6}], [%2], %7;"
                 ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "l"(policy) : "memory");
}
__device__ __forceinline__ uint64_t l2_policy_evict_first() {
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1) {
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
                 ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1) : "memory");
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1, int c2) {
    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
                 ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2) : "memory");
}
// Pass 2: the window rows from `row` on of a unit (R rows each, one unit after the other).  BY_UNIT, for units whose rows do not
// fill their last chunk: the map has a dimension for the units, so that the rows that fill it up are zeros and not the next unit's
// queries, which need not be finite (their weight of 0 would not help).  Elsewhere the map of plain rows, which is
// the faster one (64 rows x 1024 tokens x 2 heads 13.9 us, 14.0 by unit; 448 rows x 131072 tokens x 4 heads 347.6 and 349.8), and in
// pass 1, where a row of the MMA's M dimension reaches no other.
template <bool BY_UNIT>
__device__ __forceinline__ void load_q(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int row, int unit, int R) {
    if (BY_UNIT) tma_load_3d(dst, map, bar, x, row, unit);
    else tma_load_2d(dst, map, bar, x, unit * R + row);
}

__device__ __forceinline__ void prefetch_tmap(const CUtensorMap* map) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// D[tmem] (+)= A[smem] * B[smem], bf16 inputs, fp32 accumulate
__device__ __forceinline__ void tc_mma(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                 ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void tc_ld16(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                 : "r"(taddr) : "memory");
}
__device__ __forceinline__ float fast_exp2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Shared-memory matrix descriptors: K-major operand with 128-byte swizzle = rows of 64 bf16 (128 B),
// 8-row groups 1024 B apart (the image a swizzle-128B TMA box of 64 elements x rows leaves).
// The MMA thread builds two descriptors per instruction, so they are kept cheap: the high word of a
// descriptor is a constant and the low word is (address >> 4) plus constant fields; shared memory
// addresses are below 256 KB, so adding a byte offset / 16 to the low word cannot carry out of the
// 14-bit address field.
constexpr uint32_t kDescHi = (1024u >> 4) | (1u << 14) | (2u << 29);       // SBO 1024 B, version 1, 128-byte swizzle
__device__ __forceinline__ uint32_t desc_lo_k(uint32_t addr) { return (addr >> 4) | (1u << 16); }                     // K-major
__device__ __forceinline__ uint32_t desc_lo_mn(uint32_t addr) { return (addr >> 4) | ((kHalfBytes >> 4) << 16); }     // MN-major, LBO 16 KB
__device__ __forceinline__ uint64_t desc_make(uint32_t lo) {
    uint64_t d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "r"(lo), "r"(kDescHi));
    return d;
}
__device__ __forceinline__ constexpr uint32_t desc_kstep(int ks, uint32_t half_bytes) {   // K step ks of a [rows][2 x 64] operand
    return (uint32_t)(ks >> 2) * (half_bytes >> 4) + (uint32_t)(ks & 3) * 2u;
}
// kind::f16 instruction descriptor: bf16 x bf16 -> fp32, both operands K-major, M = 128
__host__ __device__ constexpr uint32_t idesc_bf16(int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(TILE >> 4) << 24);
}

struct TcParams {
    int B, Hkv, G, W, R, Nmax;
    const int32_t* seq_lens;
    const int32_t* mask_lens;                 // or nullptr: length the causal mask counts from (token-sharded caches)
    float scale;
    int causal;
    unsigned variants;
    int n_chunks, chunk_rows, rows_out;       // rows_out = n_chunks * chunk_rows
    const float* lse2;                        // [units][rows_out]
    const float4* cpair;                      // [units][rows_out / 2]: (-lse2_0, -lse2_1, |o_0|^2, |o_1|^2) per row pair
    const float* nv;                          // [units][Nmax]: ||v_p||^2 from pass 1
    const float* onorm;                       // [units][rows_out]
    float* scores;                            // [planes][units][Nmax]
    unsigned int* status;                     // device status word (workspace header)
    unsigned long long* span;                 // [2]: ~(earliest CTA start), latest CTA end, in globaltimer ns
    int l2_stream;                            // K/V copies carry the "evict first" L2 hint (their last use)
    int csplit;                               // multi-chunk kernel: the most CTAs that share the row chunks of one tile pair; 1: whole pairs
    float* partial;                           // csplit > 1: [csplit - 1][planes][units][Nmax] scores of every pair's second, third, ... CTA
    int* copies;                              // csplit > 1: [units][pairs of Nmax tokens] how many of them a pair has
    int max_pairs;
};

// (a device-side length is clamped to [0, max_len]: the host cannot check it)
__device__ __forceinline__ int tc_seq_len_raw(const int32_t* lens, int b, int nmax) { return lens ? min(max(lens[b], 0), nmax) : nmax; }
__device__ __forceinline__ int tc_seq_len(const TcParams& p, int b) { return tc_seq_len_raw(p.seq_lens, b, p.Nmax); }
__device__ __forceinline__ int tc_mask_len(const TcParams& p, int b) { return p.mask_lens ? p.mask_lens[b] : tc_seq_len(p, b); }

// Last token that any of the window rows [r0, r1] of a unit sees (row r is query position N - W + r mod W
// of its head): tiles that begin after it contribute nothing to these rows and are not visited.  With a
// short window every chunk of rows reaches the end of the cache; with the whole sequence as the window
// (W = N) about half of the (row chunk, token tile) pairs drop out.
__device__ __forceinline__ int rows_last_token(int r0, int r1, int W, int N, int causal) {
    return (causal && r0 / W == r1 / W) ? N - W + (r1 % W) : N - 1;
}

// Walks the CTA's share of the token tiles.  All non-empty 128-token tiles of all (batch item,
// KV head) units, in (unit, tile) order, are cut into gridDim.x contiguous, equally long runs, so
// that a CTA stays inside one unit for as long as possible (its Q / O operands stay in shared
// memory) and ragged batches are balanced.  Every role of the CTA runs its own copy.
struct TileWalk {
    int unit, tile, tiles_in_unit;            // current position
    long long left;                           // positions still to visit, including the current one
    const TcParams* p;
    __device__ __forceinline__ int tiles_of(int b) const { return (tc_seq_len(*p, b) + TILE - 1) / TILE; }
    __device__ void init(const TcParams& prm) {
        p = &prm;
        long long total = 0;
        if (p->seq_lens) { for (int b = 0; b < p->B; ++b) total += (long long)p->Hkv * tiles_of(b); }
        else total = (long long)p->B * p->Hkv * tiles_of(0);
        const long long lo = total * blockIdx.x / gridDim.x, hi = total * (blockIdx.x + 1) / gridDim.x;
        left = hi - lo;
        unit = 0; tile = 0; tiles_in_unit = 0;
        if (left <= 0) return;
        long long skip = lo;
        int b = 0;
        for (; b < p->B; ++b) {
            const long long blk = (long long)p->Hkv * tiles_of(b);
            if (skip < blk) break;
            skip -= blk;
        }
        tiles_in_unit = tiles_of(b);
        unit = b * p->Hkv + (int)(skip / tiles_in_unit);
        tile = (int)(skip % tiles_in_unit);
    }
    __device__ __forceinline__ bool done() const { return left <= 0; }
    __device__ __forceinline__ void next() {
        --left;
        if (++tile < tiles_in_unit || left <= 0) return;
        tile = 0;
        do { ++unit; tiles_in_unit = tiles_of(unit / p->Hkv); } while (tiles_in_unit == 0);
    }
};

// Walks the CTA's share of the multi-chunk pass 2.  A tile pair's items are the row chunks that see it; the items of all
// pairs of all units, in order, are cut into gridDim.x equal runs, so that a CTA stays with a pair (128 KB of K and V) for
// as long as possible and all do the same work, however many rows see a pair.  Only a CTA's first pair can have been begun
// by another: the CTA's number within that pair is its `slot`, and every slot has its own copy of the score planes.
// With csplit == 1 the runs consist of whole pairs.
// (Dealing the chunks of every pair round to up to eight CTAs loaded each pair eight times and balanced the runs by the order
// of the pairs only.  Pass 2 of the 4k whole-sequence window 268 -> 221 us, of 256 rows x 7043 tokens x 8 heads 32 -> 26, of 448
// rows x 9000 tokens x 4 heads 33.5 -> 21.3.)
template <bool SKIP>
struct ItemWalk {
    const TcParams* p;
    int unit, pair, pairs;                    // current segment: chunks v0 .. v1 - 1 of those that see the pair
    int v0, v1, slot;
    int left;                                 // items still to visit, including the segment's
    int past;                                 // tokens between the first one that not every row sees and the pair's first: > 0 where chunks can be hidden
    __device__ __forceinline__ static int pairs_of(const TcParams& p, int b) { return ((tc_seq_len(p, b) + TILE - 1) / TILE + 1) / 2; }
    __device__ __forceinline__ static int past_of(const TcParams& p, int b, int j) {
        // (chunks of up to 64 rows of a head hold its last query, which sees everything)
        return SKIP && p.causal && p.W > MC_ROWS ? j * 2 * TILE - (tc_mask_len(p, b) - p.W) : 0;
    }
    // a chunk inside head h whose last row lies `past` rows behind the head's first sees nothing of the pair: chunks lo .. hi - 1
    __device__ __forceinline__ static void hidden_run(const TcParams& p, int h, int past, int& lo, int& hi) {
        lo = (h * p.W + MC_ROWS - 1) / MC_ROWS;
        hi = (h * p.W + min(past, p.W - 1)) / MC_ROWS;         // (a head's last query is never hidden)
    }
    __device__ __forceinline__ static int visible(const TcParams& p, int past) {
        int n = p.n_chunks;
        if (past > 0)
            for (int h = 0, lo, hi; h < p.G; ++h) { hidden_run(p, h, past, lo, hi); n -= max(hi - lo, 0); }
        return n;
    }
    // (the lanes of a warp take the pairs side by side: called by whole warps, as run_length and init)
    __device__ __forceinline__ static int items_of(const TcParams& p, int b) {
        const int n = pairs_of(p, b);
        if (p.csplit == 1) return n;
        int t = 0;
        for (int j = threadIdx.x & 31; j < n; j += 32) t += visible(p, past_of(p, b, j));
        return __reduce_add_sync(0xffffffffu, t);
    }
    // items per CTA; a pair is then shared by at most csplit of them
    __device__ __forceinline__ static int run_length(const TcParams& p, int grid) {
        long long total = 0;
        if (p.seq_lens || p.mask_lens) { for (int b = 0; b < p.B; ++b) total += (long long)p.Hkv * items_of(p, b); }
        else total = (long long)p.B * p.Hkv * items_of(p, 0);
        const int run = (int)((total + grid - 1) / grid);
        return max(run, p.csplit == 1 || p.csplit >= p.n_chunks ? 1 : (p.n_chunks + p.csplit - 2) / (p.csplit - 1));
    }
    // the segment that begins at item r of the current pair
    __device__ __forceinline__ void segment(int b, int r) {
        past = past_of(*p, b, pair);
        const int n = visible(*p, past);
        v0 = r;
        v1 = p->csplit == 1 ? n : min(n, r + left);
    }
    __device__ void init(const TcParams& prm) {
        p = &prm; slot = 0; left = 0; unit = pair = pairs = v0 = v1 = past = 0;
        const int run = run_length(prm, (int)gridDim.x);
        long long x = (long long)run * blockIdx.x;
        int b = 0, t = 0;
        for (; b < p->B; ++b) {
            t = items_of(*p, b);
            const long long blk = (long long)p->Hkv * t;
            if (x < blk) break;
            x -= blk;
        }
        if (b == p->B) return;
        long long rest = (long long)p->Hkv * t - x;            // items from here to the end of everything, as far as the run goes
        for (int bb = b + 1; bb < p->B && rest < run; ++bb) rest += (long long)p->Hkv * items_of(*p, bb);
        left = (int)min((long long)run, rest);
        unit = b * p->Hkv + (int)(x / t); pairs = pairs_of(*p, b);
        int r = (int)(x % t);
        if (p->csplit == 1) { pair = r; r = 0; }
        else {
            const int lane = threadIdx.x & 31;
            for (;; pair += 32) {
                const int n = pair + lane < pairs ? visible(*p, past_of(*p, b, pair + lane)) : 0;
                int incl = n;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int up = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += up;
                }
                const unsigned past_r = __ballot_sync(0xffffffffu, incl > r);
                if (past_r) {
                    const int f = __ffs(past_r) - 1;
                    r -= __shfl_sync(0xffffffffu, incl - n, f);
                    pair += f;
                    break;
                }
                r -= __shfl_sync(0xffffffffu, incl, 31);
            }
        }
        segment(b, r);
        if (r > 0) slot = (int)blockIdx.x - (int)(((long long)run * blockIdx.x - r) / run);   // the pair was begun by the CTA of its first item
    }
    __device__ __forceinline__ bool done() const { return left <= 0; }
    __device__ __forceinline__ bool ends_pair() const { return v1 == visible(*p, past); }
    __device__ __forceinline__ void next() {
        left -= p->csplit == 1 ? 1 : v1 - v0;
        slot = 0;
        if (left <= 0) return;
        if (++pair == pairs) {
            pair = 0;
            do { ++unit; pairs = pairs_of(*p, unit / p->Hkv); } while (pairs == 0);
        }
        segment(unit / p->Hkv, 0);
    }
    // the v-th chunk that sees the pair
    __device__ __forceinline__ int chunk(int v) const {
        if (SKIP && past > 0)
            for (int h = 0, lo, hi; h < p->G; ++h) { hidden_run(*p, h, past, lo, hi); if (hi > lo && v >= lo) v += hi - lo; }
        return v;
    }
};

__device__ __forceinline__ float2 bf16x2_to_f32x2(uint32_t w) {
    return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
}
// waits for the TMEM loads of this thread; the registers are operands so that no use is moved above it
__device__ __forceinline__ void tc_wait_ld16x2(uint32_t (&a)[16], uint32_t (&b)[16]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3]), "+r"(a[4]), "+r"(a[5]), "+r"(a[6]), "+r"(a[7]),
                   "+r"(a[8]), "+r"(a[9]), "+r"(a[10]), "+r"(a[11]), "+r"(a[12]), "+r"(a[13]), "+r"(a[14]), "+r"(a[15]),
                   "+r"(b[0]), "+r"(b[1]), "+r"(b[2]), "+r"(b[3]), "+r"(b[4]), "+r"(b[5]), "+r"(b[6]), "+r"(b[7]),
                   "+r"(b[8]), "+r"(b[9]), "+r"(b[10]), "+r"(b[11]), "+r"(b[12]), "+r"(b[13]), "+r"(b[14]), "+r"(b[15])
                 :: "memory");
}

// ||v||^2 (and, with L1, ||v||_1) of row `tok` of a [128 tokens][128 bf16] tile stored as two
// swizzle-128B halves.  Any order of the row's 16-byte pieces gives the same sums; this one is free
// of bank conflicts when consecutive threads take consecutive rows.
template <bool L1>
__device__ __forceinline__ void value_norms(const uint8_t* vt, int tok, float& l2, float& l1) {
    float2 acc0 = make_float2(0.f, 0.f), acc1 = acc0, acc2 = acc0, acc3 = acc0, ab0 = acc0, ab1 = acc0;
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int ch = 0; ch < 8; ++ch) {
            const uint4 u = *reinterpret_cast<const uint4*>(vt + h * kHalfBytes + tok * 128 + ((ch ^ (tok & 7)) << 4));
            const float2 f0 = bf16x2_to_f32x2(u.x), f1 = bf16x2_to_f32x2(u.y);
            const float2 f2 = bf16x2_to_f32x2(u.z), f3 = bf16x2_to_f32x2(u.w);
            acc0 = __ffma2_rn(f0, f0, acc0); acc1 = __ffma2_rn(f1, f1, acc1);
            acc2 = __ffma2_rn(f2, f2, acc2); acc3 = __ffma2_rn(f3, f3, acc3);
            if (L1) {
                ab0 = __fadd2_rn(ab0, __fadd2_rn(make_float2(fabsf(f0.x), fabsf(f0.y)), make_float2(fabsf(f1.x), fabsf(f1.y))));
                ab1 = __fadd2_rn(ab1, __fadd2_rn(make_float2(fabsf(f2.x), fabsf(f2.y)), make_float2(fabsf(f3.x), fabsf(f3.y))));
            }
        }
    const float2 sum = __fadd2_rn(__fadd2_rn(acc0, acc1), __fadd2_rn(acc2, acc3));
    l2 = sum.x + sum.y;
    const float2 sab = __fadd2_rn(ab0, ab1);
    l1 = sab.x + sab.y;
}

// Running sums of one token over the window rows, two rows per packed fp32x2 lane.  With a = A_rp, z the unscaled logit,
// Z = scale z and t' = -2 v.o_r (the expanded norms of Algorithm 1):
//   Eq. 4   sum_r a^2 |v|^2                 = |v|^2 S1
//   Eq. 5   sum_r a^2 Z^2 ||v - o_r||^2     = scale^2 (|v|^2 S3 + S5)
//   Eq. 6   sum_r a^2 ||(1+Z) v - Z o_r||^2 = |v|^2 (S1 + 2 scale S2 + scale^2 S3) + scale S4 + scale^2 S5
// and S6 = sum a (attention-only), with S1 = sum a^2, S2 = sum a^2 z, S3 = sum a^2 z^2, S4 = sum a^2 z t',
// S5 = sum a^2 z^2 (t' + |o_r|^2).  a^2 comes straight out of the exponential, of twice the argument: nine packed
// instructions per row pair and one exponential per row serve Eq. 4-6 together (the sums over u = a z and
// b = a (1 + Z) that they replace took ten for Eq. 5 and 6 and thirteen with the rest: 512 rows per head, four sequences of
// up to 26550 tokens, Eq. 4-6: 265 -> 228 us for pass 2; Eq. 5 and 6 of the 128k layer with 448 rows: 163 -> 157 us).
// The joint score alone is cheaper in u = a z and b = a (1 + Z): s1 = sum b^2, s2 = sum u (b t' + u scale |o_r|^2), and the
// score is |v|^2 s1 + scale s2 with seven instructions per row pair.
// S1 + 2 scale S2 + scale^2 S3 stands for a sum of squares and cancels where Z is near -1 in every row that counts, which
// few rows can bring about (one row: 1e-4 of the token's own score, against 4e-6; no difference from 16 rows on).  Calls with
// fewer than 64 rows (HILO), whose sums are to be those of 32 bits, therefore keep the squares: S1 = sum a^2, S2 = sum b^2,
// S3 = sum u^2, S4 = sum u b t', S5 = sum u^2 t', S7 = sum u^2 |o_r|^2, and
//   Eq. 5   scale^2 (|v|^2 S3 + S5 + S7),   Eq. 6   |v|^2 S2 + scale (S4 + scale S7),
// with one instruction per row pair more.
struct RowSums { float2 s1, s2, s3, s4, s5, s6, s7; };

template <unsigned VARS> constexpr bool kSumsA = (VARS & (OBC_VAR_ATTN | OBC_VAR_VATP)) != 0;
// what the exponent is multiplied with: a^2 alone is wanted, or a
template <unsigned VARS, bool HILO = false> constexpr float kExpFactor = HILO || VARS == OBC_VAR_VK || kSumsA<VARS> ? 1.f : 2.f;

// 16 rows of one token: zr = logits, tr = -2 v.o_r, cst = per row pair (-lse2_0, -lse2_1, |o_0|^2, |o_1|^2), the
// first two times kExpFactor (as sl2); when only the joint score is computed the |o|^2 entries arrive multiplied by scale
template <unsigned VARS, bool MASKED, bool HILO>
__device__ __forceinline__ void score_rows16(const uint32_t (&zr)[16], const uint32_t (&tr)[16], const float4* cst,
                                             float2 sl2, float2 sc, RowSums& S, int ptok, int mask_base, int W, int& wi) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const float4 cp = cst[i];
        const float2 z = make_float2(__uint_as_float(zr[2 * i]), __uint_as_float(zr[2 * i + 1]));
        const float2 t2 = make_float2(__uint_as_float(tr[2 * i]), __uint_as_float(tr[2 * i + 1]));
        float2 e = __ffma2_rn(z, sl2, make_float2(cp.x, cp.y));
        if (MASKED) {                                   // row r sees tokens p <= N - W + (r mod W)
            if (ptok > mask_base + wi) e.x = -INFINITY;
            wi = wi + 1 == W ? 0 : wi + 1;
            if (ptok > mask_base + wi) e.y = -INFINITY;
            wi = wi + 1 == W ? 0 : wi + 1;
        }
        const float2 a = make_float2(fast_exp2(e.x), fast_exp2(e.y));
        if (VARS == OBC_VAR_VK) {
            const float2 u = __fmul2_rn(a, z);
            const float2 b = __ffma2_rn(u, sc, a);
            S.s1 = __ffma2_rn(b, b, S.s1);
            S.s2 = __ffma2_rn(u, __ffma2_rn(u, make_float2(cp.z, cp.w), __fmul2_rn(b, t2)), S.s2);
        } else if (HILO) {
            const float2 u = __fmul2_rn(a, z), b = __ffma2_rn(u, sc, a), w = __fmul2_rn(u, t2);
            S.s1 = __ffma2_rn(a, a, S.s1);
            S.s2 = __ffma2_rn(b, b, S.s2);
            S.s3 = __ffma2_rn(u, u, S.s3);
            S.s4 = __ffma2_rn(b, w, S.s4);
            S.s5 = __ffma2_rn(u, w, S.s5);
            S.s7 = __ffma2_rn(u, __fmul2_rn(u, make_float2(cp.z, cp.w)), S.s7);
            if (kSumsA<VARS>) S.s6 = __fadd2_rn(a, S.s6);
        } else {
            float2 c0 = a;                              // a^2 already
            if (kSumsA<VARS>) { c0 = __fmul2_rn(a, a); S.s6 = __fadd2_rn(a, S.s6); }
            const float2 c1 = __fmul2_rn(c0, z), c2 = __fmul2_rn(c1, z);
            S.s1 = __fadd2_rn(c0, S.s1);
            S.s2 = __fadd2_rn(c1, S.s2);
            S.s3 = __fadd2_rn(c2, S.s3);
            S.s4 = __ffma2_rn(c1, t2, S.s4);
            S.s5 = __ffma2_rn(c2, __fadd2_rn(t2, make_float2(cp.z, cp.w)), S.s5);
        }
    }
}

// stores the planes of one token from its sums (packed lanes folded)
template <unsigned VARS, bool HILO = false>
__device__ __forceinline__ void store_scores(const float (&sum)[kNumSums], float nv, float nv1, float scale, unsigned variants, float* out,
                                             size_t plane, bool live) {
    int pl = 0;
    if (VARS == OBC_VAR_VK) { out[0] = live ? fmaf(nv, sum[0], scale * sum[1]) : 0.f; return; }
    const float s2 = scale * scale;
    if (variants & OBC_VAR_V)    out[(size_t)(pl++) * plane] = live ? nv * sum[0] : 0.f;
    if (variants & OBC_VAR_K)    out[(size_t)(pl++) * plane] = live ? s2 * (fmaf(nv, sum[2], sum[4]) + (HILO ? sum[6] : 0.f)) : 0.f;
    if (variants & OBC_VAR_VK)   out[(size_t)(pl++) * plane] =
        !live ? 0.f : HILO ? fmaf(nv, sum[1], scale * fmaf(scale, sum[6], sum[3]))
                           : fmaf(nv, fmaf(s2, sum[2], fmaf(2.f * scale, sum[1], sum[0])), fmaf(scale, sum[3], s2 * sum[4]));
    if (variants & OBC_VAR_ATTN) out[(size_t)(pl++) * plane] = live ? sum[5] : 0.f;
    if (variants & OBC_VAR_VATP) out[(size_t)(pl++) * plane] = live ? nv1 * sum[5] : 0.f;
}

// One (tile, chunk) item of one token: all rows of the chunk, one batch of 16 rows in registers at a time.  (Loading
// the next batch ahead of the math, which doubles the registers, was slower in both kernels: the other epilogue
// warps of the SM sub-partition cover the wait for a batch.)
// HILO: the columns of T' come twice, `lo` columns apart (from the high and from the low part of -2 O): their sum is T'.
template <unsigned VARS, bool MASKED, bool HILO = false>
__device__ __forceinline__ void score_chunk(uint32_t zt, uint32_t tt, int chunk_rows, const float4* cst,
                                                 float2 sl2, float2 sc, RowSums& S, int ptok, int mask_base, int W, int wi, int lo = 0) {
    uint32_t z0[16], t0[16];
#pragma unroll 1
    for (int c0 = 0; c0 < chunk_rows; c0 += 16) {
        tc_ld16(tt + c0, t0);
        if (HILO) {
            tc_ld16(tt + lo + c0, z0);
            tc_wait_ld16x2(z0, t0);
#pragma unroll
            for (int i = 0; i < 16; ++i) t0[i] = __float_as_uint(__uint_as_float(t0[i]) + __uint_as_float(z0[i]));
        }
        tc_ld16(zt + c0, z0);
        tc_wait_ld16x2(z0, t0);
        score_rows16<VARS, MASKED, HILO>(z0, t0, cst + (c0 >> 1), sl2, sc, S, ptok, mask_base, W, wi);
    }
}

// VARS: variants this instantiation computes (a superset of p.variants).  OWN_NV: no pass 1 ran (the
// caller supplied the attention outputs), so warps 2-3 compute the value norms from the V tiles here.
// HILO: fewer than 64 window rows.  Such a call is summed in 32 bits throughout: -2 O enters as the sum of two bf16
// parts, which stand side by side on the MMA's N dimension (at most 2 x 64 rows) and meet in the epilogue.  The
// kernel stays bound by the K/V tiles it streams, with half of the epilogue's rows idle.  Scores against 64 bits, thirteen
// shapes of 1 to 63 rows: 0.9e-6 of the norm and 2.6e-6 of the largest, as on CUDA cores.  (The parts leave out 2^-17 of
// O, which shows where |v - o|^2 is a small difference of large terms: 3 rows x 64 tokens with logits of up to 10, 3.7e-6 of the norm
// against 1.2e-6.  A third part, 192 columns of T', brought that to 1.9e-6 and cost calls of 63 rows 3 to 6 %.)
template <unsigned VARS, bool OWN_NV, bool HILO, bool BY_UNIT>
__global__ void __launch_bounds__(kThreads, 1)
tc_pass2_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_o,
                const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                const __grid_constant__ TcParams p) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const uint32_t sbase = smem_u32(smem);
    const uint32_t bars = sbase + OFF_BAR;
    auto bar = [&](int i) { return bars + 8u * (uint32_t)i; };
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem + OFF_TMEM);
    float4* sConst = reinterpret_cast<float4*>(smem + OFF_CONST);   // [16 epilogue warps][32 row pairs]
    float2* sNv = reinterpret_cast<float2*>(smem + OFF_NV);         // [NSLOT][128] (||v||^2, ||v||_1)
    float* sXch = reinterpret_cast<float*>(smem + OFF_XCH);         // [tile parity][2][kNumSums][128]

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    span_begin(p.span);
    const int units = p.B * p.Hkv;

    if (threadIdx.x == 0) {
        prefetch_tmap(&map_k); prefetch_tmap(&map_v); prefetch_tmap(&map_q); prefetch_tmap(&map_o);
        // a K/V stage is released by the MMA commit and, when the norms are computed here, by warps 2-3
        for (int i = 0; i < NSTAGE; ++i) { mbar_init(bar(BAR_FULL + i), 1); mbar_init(bar(BAR_EMPTY + i), OWN_NV ? 3 : 1); }
        if (OWN_NV) for (int i = 0; i < 2 * NSLOT; ++i) mbar_init(bar(BAR_NV + i), 2);
        mbar_init(bar(BAR_QO_FULL), 1); mbar_init(bar(BAR_QO_EMPTY), 1);
        for (int i = 0; i < 4; ++i) mbar_init(bar(BAR_TM_FULL + i), 1);
        for (int i = 0; i < 2; ++i) mbar_init(bar(BAR_TM_EMPTY + i), 8);
        for (int i = 0; i < 4; ++i) mbar_init(bar(BAR_XCH + i), 4);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sbase + OFF_TMEM), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;

    bool failed = false;
    int fail_site = 0;                             // source line of the wait that gave up (status word)
    const uint32_t qo_bytes = (uint32_t)p.chunk_rows * 256u * (HILO ? 3u : 2u);   // Q and O chunks, two halves each (O: high and low part)

    // Every role walks the same tiles (TileWalk); all window rows of a unit (at most 128) are one chunk.
    // Tiles go to the two epilogue groups alternately.  What an epilogue group waits for (accumulators
    // ready) is signalled on barriers of its own, so that each waiter sees every phase of the barriers
    // it uses; a parity wait must never fall two phases behind.  ||v_p||^2 comes from pass 1 (or, with
    // OWN_NV, from warps 2-3 through a ring of NSLOT slots) and the per-row constants from the combine kernel.
    // `item` counts the (tile, chunk) pairs processed so far and indexes the smem stage, TMEM
    // buffer and constant-slot rings.
    TileWalk tw;
    tw.init(p);
    if (!(warp == 0 && lane == 0)) pdl_wait();       // the producer thread waits after its first K/V copies
    if (warp == 0) {
        // ===================================== TMA producer =====================================
        if (lane == 0) {
            uint32_t item = 0, qo_loads = 0;
            int qo_unit = -1;
            const uint64_t pol_stream = l2_policy_evict_first();
            for (; !tw.done() && !failed; tw.next()) {
                const int unit = tw.unit, b = unit / p.Hkv, g = unit % p.Hkv, t0 = tw.tile * TILE;
                const uint32_t st = item % NSTAGE, use = item / NSTAGE;
                if (!mbar_wait(bar(BAR_EMPTY + st), (use & 1) ^ 1)) { failed = true; fail_site = __LINE__; break; }
                mbar_expect_tx(bar(BAR_FULL + st), 2 * kOperandBytes);
                const uint32_t dk = sbase + OFF_K + st * kOperandBytes, dv = sbase + OFF_V + st * kOperandBytes;
                if (p.l2_stream) {                             // last use of the tile: it may leave the cache first
                    tma_load_4d_hint(dk, &map_k, bar(BAR_FULL + st), 0, t0, g, b, pol_stream);
                    tma_load_4d_hint(dk + kHalfBytes, &map_k, bar(BAR_FULL + st), 64, t0, g, b, pol_stream);
                    tma_load_4d_hint(dv, &map_v, bar(BAR_FULL + st), 0, t0, g, b, pol_stream);
                    tma_load_4d_hint(dv + kHalfBytes, &map_v, bar(BAR_FULL + st), 64, t0, g, b, pol_stream);
                } else {
                    tma_load_4d(dk, &map_k, bar(BAR_FULL + st), 0, t0, g, b);
                    tma_load_4d(dk + kHalfBytes, &map_k, bar(BAR_FULL + st), 64, t0, g, b);
                    tma_load_4d(dv, &map_v, bar(BAR_FULL + st), 0, t0, g, b);
                    tma_load_4d(dv + kHalfBytes, &map_v, bar(BAR_FULL + st), 64, t0, g, b);
                }
                // K, V and the sequence lengths were read by pass 1 of this call, so the first tile
                // may be fetched while the preceding kernel drains; -2 O is that kernel's output
                if (item == 0) pdl_wait();
                if (unit != qo_unit) {
                    if (!mbar_wait(bar(BAR_QO_EMPTY), (qo_loads & 1) ^ 1)) { failed = true; fail_site = __LINE__; break; }
                    mbar_expect_tx(bar(BAR_QO_FULL), qo_bytes);
                    const int orow = unit * p.rows_out * (HILO ? 2 : 1);
                    load_q<BY_UNIT>(sbase + OFF_Q, &map_q, bar(BAR_QO_FULL), 0, 0, unit, p.R);
                    load_q<BY_UNIT>(sbase + OFF_Q + kHalfBytes, &map_q, bar(BAR_QO_FULL), 64, 0, unit, p.R);
                    tma_load_2d(sbase + OFF_O, &map_o, bar(BAR_QO_FULL), 0, orow);
                    tma_load_2d(sbase + OFF_O + kHalfBytes, &map_o, bar(BAR_QO_FULL), 64, orow);
                    qo_unit = unit; ++qo_loads;
                }
                ++item;
            }
            // drain: every copy this thread issued must have landed before the CTA may exit
            for (uint32_t back = 0; back < NSTAGE && back < item; ++back) {
                const uint32_t it = item - 1 - back;
                (void)mbar_wait(bar(BAR_FULL + it % NSTAGE), (it / NSTAGE) & 1);
            }
            if (qo_loads) (void)mbar_wait(bar(BAR_QO_FULL), (qo_loads - 1) & 1);
        }
    } else if (warp == 1) {
        // ===================================== MMA issuer =======================================
        if (lane == 0) {
            const uint32_t idesc = idesc_bf16(p.chunk_rows), idesc_t = idesc_bf16(HILO ? 2 * p.chunk_rows : p.chunk_rows);
            uint32_t item = 0, qo_loads = 0, tile_seq = 0;
            int qo_unit = -1;
            for (; !tw.done() && !failed; tw.next(), ++tile_seq) {
                const int unit = tw.unit;
                const uint32_t owner = tile_seq & 1;               // epilogue group of this tile
                const bool new_qo = unit != qo_unit;
                if (new_qo) {
                    if (!mbar_wait(bar(BAR_QO_FULL), qo_loads & 1)) { failed = true; fail_site = __LINE__; break; }
                    qo_unit = unit; ++qo_loads;
                }
                const uint32_t st = item % NSTAGE, buf = item & 1;
                if (!mbar_wait(bar(BAR_FULL + st), (item / NSTAGE) & 1)) { failed = true; fail_site = __LINE__; break; }
                if (!mbar_wait(bar(BAR_TM_EMPTY + buf), ((item >> 1) & 1) ^ 1)) { failed = true; fail_site = __LINE__; break; }
                tc_fence_after();
                const uint32_t zt = tmem_base + buf * 256u, tt = zt + 128u;
                const uint32_t ak = desc_lo_k(sbase + OFF_K + st * kOperandBytes), av = desc_lo_k(sbase + OFF_V + st * kOperandBytes);
                const uint32_t bq = desc_lo_k(sbase + OFF_Q), bo = desc_lo_k(sbase + OFF_O);
#pragma unroll
                for (int ks = 0; ks < 8; ++ks)                 // d = 128 = 8 steps of K = 16
                    tc_mma(zt, desc_make(ak + desc_kstep(ks, kHalfBytes)), desc_make(bq + desc_kstep(ks, kHalfBytes)), idesc, ks > 0);
#pragma unroll
                for (int ks = 0; ks < 8; ++ks)
                    tc_mma(tt, desc_make(av + desc_kstep(ks, kHalfBytes)), desc_make(bo + desc_kstep(ks, kHalfBytes)), idesc_t, ks > 0);
                tc_commit(bar(BAR_TM_FULL + owner * 2 + buf)); // accumulators ready for the tile's epilogue group
                tc_commit(bar(BAR_EMPTY + st));                // K/V stage no longer read by the MMA
                // Q / O may be overwritten once these MMAs are done, if the next item needs others
                const bool last_of_unit = tw.left > 1 && tw.tile + 1 == tw.tiles_in_unit;
                if (last_of_unit) tc_commit(bar(BAR_QO_EMPTY));
                ++item;
            }
        }
    } else if (warp < 4) {
        // ================= value norms of every tile (only when no pass 1 supplied them) ===========
        if (OWN_NV) {
            const int t64 = threadIdx.x - 64;                      // 0..63
            uint32_t item = 0;
            for (; !tw.done() && !failed; tw.next(), ++item) {
                const uint32_t st = item % NSTAGE, slot = item % NSLOT, owner = item & 1;
                if (!mbar_wait(bar(BAR_FULL + st), (item / NSTAGE) & 1)) { failed = true; fail_site = __LINE__; break; }
                const uint8_t* vt = smem + OFF_V + st * kOperandBytes;
                // slot `slot` was last read for the tile four back, whose owner took it into registers before
                // releasing the accumulators that the MMA of the tile two back (whose commit freed this stage) needed
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const int tok = t64 + 64 * j;
                    float l2, l1;
                    value_norms<(VARS & OBC_VAR_VATP) != 0>(vt, tok, l2, l1);
                    sNv[slot * TILE + tok] = make_float2(l2, l1);
                }
                __syncwarp();
                if (lane == 0) { mbar_arrive(bar(BAR_NV + owner * NSLOT + slot)); mbar_arrive(bar(BAR_EMPTY + st)); }
            }
        }
    } else {
        // ======================================= epilogue =======================================
        const int wg = (warp - 4) >> 3;                            // 0: even tiles, 1: odd tiles
        const int half = ((warp - 4) >> 2) & 1;                    // 0: first half of the window rows (and the stores), 1: the rest
        const int lane_grp = warp & 3;                             // TMEM lanes 32*lane_grp .. +31
        const int tok = lane_grp * 32 + lane;                      // token within the tile
        // the chunk's rows in two runs of whole 16-row batches
        const int rows0 = min(p.chunk_rows, (p.chunk_rows / 2 + 15) / 16 * 16);
        const int r_begin = half ? rows0 : 0, r_count = half ? p.chunk_rows - rows0 : rows0;
        const float ksl = p.scale * kLog2e * kExpFactor<VARS, HILO>;
        const float2 sl2 = make_float2(ksl, ksl), sc = make_float2(p.scale, p.scale);
        const size_t plane = (size_t)units * p.Nmax;
        uint32_t item = 0, tile_seq = 0, mine_seq = 0;
        uint32_t full_par = 0, nv_par = 0;                         // phase parity of this group's barriers, one bit each
        float4* my_const = sConst + (warp - 4) * 32;               // this warp's copy of its rows' constants
        int const_unit = -1;
        for (; !tw.done() && !failed; tw.next()) {
            const bool mine = (tile_seq & 1) == (uint32_t)wg;
            ++tile_seq;
            if (!mine) { ++item; continue; }
            const int unit = tw.unit, b = unit / p.Hkv;
            const int N = tc_seq_len(p, b), t0 = tw.tile * TILE;
            float* out = p.scores + (size_t)unit * p.Nmax;
            const int ptok = t0 + tok;
            // rows of the window that do not see this tile's last token need the causal mask
            const int Nm = tc_mask_len(p, b);
            const bool masked_tile = p.causal && (t0 + TILE - 1 > Nm - p.W);
            RowSums S;
            S.s1 = S.s2 = S.s3 = S.s4 = S.s5 = S.s6 = S.s7 = make_float2(0.f, 0.f);
            const uint32_t buf = item & 1;
            float nv = 0.f, nv1 = 0.f;                             // used after the row loop
            if (!OWN_NV && half == 0 && ptok < N) nv = p.nv[(size_t)unit * p.Nmax + ptok];
            if (unit != const_unit) {                              // at most once per unit: (-lse2, |o|^2) of the warp's row pairs
                __syncwarp();
                {
                    const int rp = (r_begin >> 1) + lane;          // row pair of the chunk
                    float4 c4 = lane * 2 < r_count ? p.cpair[(((size_t)unit * p.rows_out) >> 1) + rp] : make_float4(-INFINITY, -INFINITY, 0.f, 0.f);
                    if (VARS == OBC_VAR_VK) { c4.z *= p.scale; c4.w *= p.scale; }
                    c4.x *= kExpFactor<VARS, HILO>; c4.y *= kExpFactor<VARS, HILO>;
                    my_const[lane] = c4;
                }
                __syncwarp();
                const_unit = unit;
            }
            if (!mbar_wait(bar(BAR_TM_FULL + wg * 2 + buf), (full_par >> buf) & 1)) { failed = true; fail_site = __LINE__; break; }
            full_par ^= 1u << buf;
            tc_fence_after();
            if (OWN_NV && half == 0) {                             // the norms of this tile (ready long before the accumulators)
                const uint32_t slot = item % NSLOT;
                if (!mbar_wait(bar(BAR_NV + wg * NSLOT + slot), (nv_par >> slot) & 1)) { failed = true; fail_site = __LINE__; break; }
                nv_par ^= 1u << slot;
                const float2 n21 = sNv[slot * TILE + tok];
                nv = n21.x; nv1 = n21.y;
            }
            const float4* cst = my_const;
            const uint32_t zt = tmem_base + ((uint32_t)(lane_grp * 32) << 16) + buf * 256u + (uint32_t)r_begin, tt = zt + 128u;
            if (r_count > 0) {
                if (masked_tile)
                    score_chunk<VARS, true, HILO>(zt, tt, r_count, cst, sl2, sc, S, ptok, Nm - p.W, p.W, r_begin % p.W, p.chunk_rows);
                else
                    score_chunk<VARS, false, HILO>(zt, tt, r_count, cst, sl2, sc, S, ptok, 0, 0, 0, p.chunk_rows);
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(BAR_TM_EMPTY + buf));
            ++item;
            // the two row halves of the token meet: the sums of RowSums, packed lanes folded
            float sum[kNumSums] = {S.s1.x + S.s1.y, S.s2.x + S.s2.y, S.s3.x + S.s3.y, S.s4.x + S.s4.y, S.s5.x + S.s5.y, S.s6.x + S.s6.y, S.s7.x + S.s7.y};
            // slot xs was last used two of this group's tiles ago; the first half read it before it released the
            // accumulators of the tile after that one, without which the tile at hand could not have been computed
            const uint32_t xs = mine_seq & 1;
            float* xch = sXch + ((wg * 2 + xs) * kNumSums) * TILE + tok;
            if (half == 1) {
#pragma unroll
                for (int j = 0; j < kNumSums; ++j) {
                    const bool used = VARS == OBC_VAR_VK ? j < 2 : j < 5 || (j == 5 ? kSumsA<VARS> : HILO);
                    if (used) xch[j * TILE] = sum[j];
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(BAR_XCH + wg * 2 + xs));
                ++mine_seq;
                continue;
            }
            if (!mbar_wait(bar(BAR_XCH + wg * 2 + xs), (mine_seq >> 1) & 1)) { failed = true; fail_site = __LINE__; break; }
            ++mine_seq;
#pragma unroll
            for (int j = 0; j < kNumSums; ++j) {
                const bool used = VARS == OBC_VAR_VK ? j < 2 : j < 5 || (j == 5 ? kSumsA<VARS> : HILO);
                if (used) sum[j] += xch[j * TILE];
            }
            if (ptok < p.Nmax) store_scores<VARS, HILO>(sum, nv, nv1, p.scale, p.variants, out + ptok, plane, ptok < N);
        }
        // padding beyond the last tile of a shorter sequence: zeros
        if (p.seq_lens) {
            const int et = threadIdx.x - 128;                      // 0..511
            const int n_planes = __popc(p.variants);
            for (int unit = blockIdx.x; unit < units; unit += gridDim.x) {
                const int first = (tc_seq_len(p, unit / p.Hkv) + TILE - 1) / TILE * TILE;
                for (int pl = 0; pl < n_planes; ++pl)
                    for (int i = first + et; i < p.Nmax; i += 512) p.scores[(size_t)pl * plane + (size_t)unit * p.Nmax + i] = 0.f;
            }
        }
    }

    if (failed) atomicCAS(p.status, 0u, (unsigned)(fail_site > 0 ? fail_site : 1));   // the first failure is kept
    tc_fence_before();
    __syncthreads();
    span_end(p.span);
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
    }
}

// =================================================================================================
// Pass 2 for more than 128 window rows per KV head (e.g. GQA 7 x W 64 = 448).  The rows are cut
// into chunks of 64.  A CTA holds TWO consecutive token tiles of a unit in its two K/V stages and
// sweeps the row chunks over both: every Q / -2 O chunk (two buffers) is fetched once per tile pair
// and used by two MMA pairs with N = 64 (four TMEM buffers of Z 64 + T' 64 columns), so the fetch
// of the next chunk hides behind twice the tensor work.  Epilogue warpgroup j owns tile j of the
// pair: it sums all chunks of its 128 tokens in registers and stores their scores itself.
// =================================================================================================
constexpr uint32_t kHalfB64 = 64 * 128;                           // B operand block: [64 rows][64 bf16]
constexpr uint32_t kQoBuf = 4 * kHalfB64;                         // Q chunk (2 x 8 KB) + -2 O chunk (2 x 8 KB)
constexpr uint32_t MC_OFF_QO = 0;                                 // 2 buffers x 32 KB
constexpr uint32_t MC_OFF_K = MC_OFF_QO + 2 * kQoBuf;             // 2 tiles x 32 KB
constexpr uint32_t MC_OFF_V = MC_OFF_K + 2 * kOperandBytes;
constexpr uint32_t MC_OFF_NV = MC_OFF_V + 2 * kOperandBytes;      // [pair parity][tile of the pair][128] x (||v||^2, ||v||_1)
constexpr uint32_t MC_OFF_CONST = MC_OFF_NV + 4 * TILE * 8;       // 4 slots x 32 float4 (per chunk)
constexpr uint32_t MC_OFF_BAR = MC_OFF_CONST + 4 * 32 * 16;
enum { MC_FULL = 0, MC_EMPTY = 2, MC_QO_FULL = 4, MC_QO_EMPTY = 6, MC_TM_FULL = 8, MC_TM_EMPTY = 12,
       MC_NV = 16, MC_CONST = 18, MC_NBARS = 22 };
constexpr uint32_t MC_OFF_TMEM = MC_OFF_BAR + MC_NBARS * 8;
constexpr int kThreadsMulti = kThreadsBase + 32;                      // + warp 12: the second MMA-issuing thread
constexpr uint32_t kSmemMulti = MC_OFF_TMEM + 16 + 1024;

// SPLIT: the general walk (row chunks of a pair shared by several CTAs, hidden tile pairs skipped); without
// it every CTA takes whole pairs and every chunk, which is all a short window over a long cache needs.
template <unsigned VARS, bool SPLIT, bool BY_UNIT>
__global__ void __launch_bounds__(kThreadsMulti, 1)
tc_pass2_multi_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_o,
                      const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                      const __grid_constant__ TcParams p) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const uint32_t sbase = smem_u32(smem);
    const uint32_t bars = sbase + MC_OFF_BAR;
    auto bar = [&](int i) { return bars + 8u * (uint32_t)i; };
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem + MC_OFF_TMEM);
    float2* sNv = reinterpret_cast<float2*>(smem + MC_OFF_NV);
    float* sConst = reinterpret_cast<float*>(smem + MC_OFF_CONST);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    span_begin(p.span);
    const int units = p.B * p.Hkv;

    if (threadIdx.x == 0) {
        prefetch_tmap(&map_k); prefetch_tmap(&map_v); prefetch_tmap(&map_q); prefetch_tmap(&map_o);
        // two threads issue the MMAs (see below), so what an MMA commit signals takes two arrivals
        for (int i = 0; i < 2; ++i) { mbar_init(bar(MC_FULL + i), 1); mbar_init(bar(MC_EMPTY + i), 4); }
        for (int i = 0; i < 2; ++i) { mbar_init(bar(MC_QO_FULL + i), 1); mbar_init(bar(MC_QO_EMPTY + i), 2); }
        for (int i = 0; i < 4; ++i) { mbar_init(bar(MC_TM_FULL + i), 2); mbar_init(bar(MC_TM_EMPTY + i), 4); }
        for (int i = 0; i < 2; ++i) mbar_init(bar(MC_NV + i), 2);
        for (int i = 0; i < 4; ++i) mbar_init(bar(MC_CONST + i), 2);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sbase + MC_OFF_TMEM), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;

    bool failed = false;
    int fail_site = 0;                             // source line of the wait that gave up (status word)
    const uint32_t qo_bytes = MC_ROWS * 128u * 2u * 2u;

    // A position of the walk is a pair of tiles (2 * tw.pair + j, j = 0, 1; the second one may lie past
    // the end of a unit with an odd tile count: it is computed all the same and stores only zeros) and a run of row chunks.
    // `pitem` counts positions, `citem` row chunks over all positions; the chunk's two MMA pairs are
    // items 2 * citem + j.  Rings: K/V stage j; Q/O buffer citem & 1; constant slot citem & 3; TMEM
    // buffer item & 3, so that epilogue group j always sees buffers j and j + 2.
    ItemWalk<SPLIT> tw;
    tw.init(p);
    if (!(warp == 0 && lane == 0)) pdl_wait();       // the producer thread waits after its first K/V copies
    if (warp == 0) {
        // ===================================== TMA producer =====================================
        if (lane == 0) {
            uint32_t pitem = 0, citem = 0;
            for (; !tw.done() && !failed; tw.next(), ++pitem) {
                const int unit = tw.unit, b = unit / p.Hkv, g = unit % p.Hkv;
                for (int j = 0; j < 2 && !failed; ++j) {
                    if (!mbar_wait(bar(MC_EMPTY + j), (pitem & 1) ^ 1)) { failed = true; fail_site = __LINE__; break; }
                    const int t0 = (tw.pair * 2 + j) * TILE;
                    mbar_expect_tx(bar(MC_FULL + j), 2 * kOperandBytes);
                    const uint32_t dk = sbase + MC_OFF_K + j * kOperandBytes, dv = sbase + MC_OFF_V + j * kOperandBytes;
                    tma_load_4d(dk, &map_k, bar(MC_FULL + j), 0, t0, g, b);
                    tma_load_4d(dk + kHalfBytes, &map_k, bar(MC_FULL + j), 64, t0, g, b);
                    tma_load_4d(dv, &map_v, bar(MC_FULL + j), 0, t0, g, b);
                    tma_load_4d(dv + kHalfBytes, &map_v, bar(MC_FULL + j), 64, t0, g, b);
                }
                if (pitem == 0) pdl_wait();                        // K and V were read by pass 1; -2 O is the preceding kernel's output
                for (int v = tw.v0; v < tw.v1 && !failed; ++v) {
                    const int c = tw.chunk(v);
                    const uint32_t qb = citem & 1;
                    if (!mbar_wait(bar(MC_QO_EMPTY + qb), ((citem >> 1) & 1) ^ 1)) { failed = true; fail_site = __LINE__; break; }
                    mbar_expect_tx(bar(MC_QO_FULL + qb), qo_bytes);
                    const int orow = unit * p.rows_out + c * MC_ROWS;
                    const uint32_t dq = sbase + MC_OFF_QO + qb * kQoBuf, dob = dq + 2 * kHalfB64;
                    load_q<BY_UNIT>(dq, &map_q, bar(MC_QO_FULL + qb), 0, c * MC_ROWS, unit, p.R);
                    load_q<BY_UNIT>(dq + kHalfB64, &map_q, bar(MC_QO_FULL + qb), 64, c * MC_ROWS, unit, p.R);
                    tma_load_2d(dob, &map_o, bar(MC_QO_FULL + qb), 0, orow);
                    tma_load_2d(dob + kHalfB64, &map_o, bar(MC_QO_FULL + qb), 64, orow);
                    ++citem;
                }
            }
            // drain: every copy this thread issued must have landed before the CTA may exit
            if (pitem > 0) {
                (void)mbar_wait(bar(MC_FULL + 0), (pitem - 1) & 1);
                (void)mbar_wait(bar(MC_FULL + 1), (pitem - 1) & 1);
            }
            for (uint32_t back = 0; back < 2 && back < citem; ++back) {
                const uint32_t it = citem - 1 - back;
                (void)mbar_wait(bar(MC_QO_FULL + (it & 1)), (it >> 1) & 1);
            }
        }
    } else if (warp == 1 || warp == 12) {
        // ===================================== MMA issuers ======================================
        // One thread gets a tcgen05.mma out about every 88 cycles here (it shares its scheduler with two epilogue
        // warps), and a 128x64x16 MMA keeps the tensor pipe busy for 32: so two threads issue, warp 1 the logits
        // Z = K Q^T and warp 12 the cross terms T' = V (-2 O)^T.  Each commits what it issued; the barriers that
        // an MMA commit signals count two arrivals.
        const bool z_side = warp == 1;
        if (lane == 0) {
            const uint32_t idesc = idesc_bf16(MC_ROWS);
            uint32_t pitem = 0, citem = 0;
            for (; !tw.done() && !failed; tw.next(), ++pitem) {
                if (!mbar_wait(bar(MC_FULL + 0), pitem & 1) || !mbar_wait(bar(MC_FULL + 1), pitem & 1)) { failed = true; fail_site = __LINE__; break; }
                for (int v = tw.v0; v < tw.v1 && !failed; ++v) {
                    const uint32_t qb = citem & 1;
                    if (!mbar_wait(bar(MC_QO_FULL + qb), (citem >> 1) & 1)) { failed = true; fail_site = __LINE__; break; }
                    const uint32_t bq = desc_lo_k(sbase + MC_OFF_QO + qb * kQoBuf), bo = bq + ((2 * kHalfB64) >> 4);
                    for (int j = 0; j < 2; ++j) {
                        const uint32_t item = 2 * citem + j, buf = item & 3;
                        if (!mbar_wait(bar(MC_TM_EMPTY + buf), ((item >> 2) & 1) ^ 1)) { failed = true; fail_site = __LINE__; break; }
                        tc_fence_after();
                        const uint32_t zt = tmem_base + buf * 128u, tt = zt + 64u;
                        const uint32_t ak = desc_lo_k(sbase + MC_OFF_K + j * kOperandBytes), av = desc_lo_k(sbase + MC_OFF_V + j * kOperandBytes);
                        if (z_side) {
#pragma unroll
                            for (int ks = 0; ks < 8; ++ks)         // d = 128 = 8 steps of K = 16
                                tc_mma(zt, desc_make(ak + desc_kstep(ks, kHalfBytes)), desc_make(bq + desc_kstep(ks, kHalfB64)), idesc, ks > 0);
                        } else {
#pragma unroll
                            for (int ks = 0; ks < 8; ++ks)
                                tc_mma(tt, desc_make(av + desc_kstep(ks, kHalfBytes)), desc_make(bo + desc_kstep(ks, kHalfB64)), idesc, ks > 0);
                        }
                        tc_commit(bar(MC_TM_FULL + buf));          // this thread's accumulator of the item is ready
                    }
                    if (failed) break;
                    tc_commit(bar(MC_QO_EMPTY + qb));              // this Q / O buffer may be refilled
                    ++citem;
                }
                if (!failed) { tc_commit(bar(MC_EMPTY + 0)); tc_commit(bar(MC_EMPTY + 1)); }   // both tiles no longer read
            }
        }
    } else if (warp < 4) {
        // ==================== ||v_p||^2 per tile, per-row constants per chunk ===================
        // At a new position the constants of the first chunk go out before the norms are computed: the epilogue needs
        // them as soon as the first accumulators are ready, the norms only when the position's last chunk is summed.
        const int t64 = threadIdx.x - 64;                          // 0..63
        uint32_t pitem = 0, citem = 0;
        for (; !tw.done() && !failed; tw.next(), ++pitem) {
            const int unit = tw.unit;
            auto norms = [&]() -> bool {
                for (int j = 0; j < 2; ++j) {
                    if (!mbar_wait(bar(MC_FULL + j), pitem & 1)) { fail_site = __LINE__; return false; }
                    const uint8_t* vt = smem + MC_OFF_V + j * kOperandBytes;
                    float2* nvdst = sNv + ((pitem & 1) * 2 + j) * TILE;
#pragma unroll
                    for (int jj = 0; jj < 2; ++jj) {
                        const int tok = t64 + 64 * jj;
                        float l2, l1;
                        value_norms<(VARS & OBC_VAR_VATP) != 0>(vt, tok, l2, l1);
                        nvdst[tok] = make_float2(l2, l1);
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar(MC_EMPTY + j));
                }
                if (lane == 0) mbar_arrive(bar(MC_NV + (pitem & 1)));
                return true;
            };
            bool norms_done = false;
            for (int v = tw.v0; v < tw.v1 && !failed; ++v) {
                const int c = tw.chunk(v);
                const uint32_t cs = citem & 3;
                const size_t crow = (size_t)unit * p.rows_out + (size_t)c * MC_ROWS + t64;
                const float2 cst = make_float2(-kExpFactor<VARS> * p.lse2[crow], p.onorm[crow] * (VARS == OBC_VAR_VK ? p.scale : 1.f));
                // slot cs was last read by the chunk four back; the chunk two back has been summed once
                // the TMEM buffers this chunk is going to use are free again
                const uint32_t i0 = 2 * citem, i1 = i0 + 1;
                if (!mbar_wait(bar(MC_TM_EMPTY + (i0 & 3)), ((i0 >> 2) & 1) ^ 1) ||
                    !mbar_wait(bar(MC_TM_EMPTY + (i1 & 3)), ((i1 >> 2) & 1) ^ 1)) { failed = true; fail_site = __LINE__; break; }
                float* cdst = sConst + cs * 128 + (t64 >> 1) * 4 + (t64 & 1);      // row pair: (-lse2_0, -lse2_1, |o_0|^2, |o_1|^2)
                cdst[0] = cst.x; cdst[2] = cst.y;
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(MC_CONST + cs));
                ++citem;
                if (!norms_done) { norms_done = true; if (!norms()) { failed = true; break; } }
            }
            if (!failed && !norms_done && !norms()) failed = true;
        }
    } else if (warp < 12) {
        // ======================================= epilogue =======================================
        const int wg = (warp - 4) >> 2;                            // owns tile wg of every pair
        const int lane_grp = warp & 3;                             // TMEM lanes 32*lane_grp .. +31
        const int tok = lane_grp * 32 + lane;                      // token within the tile
        const float ksl = p.scale * kLog2e * kExpFactor<VARS>;
        const float2 sl2 = make_float2(ksl, ksl), sc = make_float2(p.scale, p.scale);
        const size_t plane = (size_t)units * p.Nmax;
        uint32_t pitem = 0, citem = 0;
        for (; !tw.done() && !failed; tw.next(), ++pitem) {
            const int unit = tw.unit, b = unit / p.Hkv;
            const int N = tc_seq_len(p, b), Nm = tc_mask_len(p, b), t0 = (tw.pair * 2 + wg) * TILE;
            const int ptok = t0 + tok;
            const bool masked_tile = p.causal && (t0 + TILE - 1 > Nm - p.W);
            RowSums S;
            S.s1 = S.s2 = S.s3 = S.s4 = S.s5 = S.s6 = S.s7 = make_float2(0.f, 0.f);
            for (int v = tw.v0; v < tw.v1; ++v) {
                const int c = tw.chunk(v);
                const uint32_t item = 2 * citem + wg, buf = item & 3, cs = citem & 3;
                if (!mbar_wait(bar(MC_CONST + cs), (citem >> 2) & 1)) { failed = true; fail_site = __LINE__; break; }
                if (!mbar_wait(bar(MC_TM_FULL + buf), (item >> 2) & 1)) { failed = true; fail_site = __LINE__; break; }
                tc_fence_after();
                const float4* cst = reinterpret_cast<const float4*>(sConst + cs * 128);
                const uint32_t zt = tmem_base + ((uint32_t)(lane_grp * 32) << 16) + buf * 128u, tt = zt + 64u;
                // a chunk whose rows lie in one head sees the whole tile as soon as its first row does (with the whole
                // sequence as the window that is every item off the diagonal)
                bool use_mask = masked_tile;
                if (use_mask) {
                    const int wfirst = (c * MC_ROWS) % p.W;
                    if (wfirst + MC_ROWS <= p.W && t0 + TILE - 1 <= Nm - p.W + wfirst) use_mask = false;
                }
                if (use_mask)
                    score_chunk<VARS, true>(zt, tt, MC_ROWS, cst, sl2, sc, S, ptok, Nm - p.W, p.W, (c * MC_ROWS) % p.W);
                else
                    score_chunk<VARS, false>(zt, tt, MC_ROWS, cst, sl2, sc, S, ptok, 0, 0, 0);
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(MC_TM_EMPTY + buf));
                ++citem;
            }
            if (failed) break;
            if (!mbar_wait(bar(MC_NV + (pitem & 1)), (pitem >> 1) & 1)) { failed = true; fail_site = __LINE__; break; }
            const float2 nv21 = sNv[((pitem & 1) * 2 + wg) * TILE + tok];
            const float nv = nv21.x, nv1 = nv21.y;
            if (ptok < p.Nmax) {
                // with the chunks of the pair shared by several CTAs each writes its part of the sums (the scores are
                // linear in them), the first into the scores, the others into copies that tc_partial_sum_kernel adds in order
                if (SPLIT && p.csplit > 1 && threadIdx.x == 128 && tw.ends_pair()) p.copies[(size_t)unit * p.max_pairs + tw.pair] = tw.slot;
                float* out = (tw.slot > 0 ? p.partial + (size_t)(tw.slot - 1) * __popc(p.variants) * plane : p.scores) + (size_t)unit * p.Nmax;
                const float sum[kNumSums] = {S.s1.x + S.s1.y, S.s2.x + S.s2.y, S.s3.x + S.s3.y, S.s4.x + S.s4.y, S.s5.x + S.s5.y, S.s6.x + S.s6.y, S.s7.x + S.s7.y};
                store_scores<VARS>(sum, nv, nv1, p.scale, p.variants, out + ptok, plane, ptok < N);
            }
        }
        // padding beyond the last tile of a shorter sequence: zeros
        if (p.seq_lens) {
            const int et = threadIdx.x - 128;                      // 0..255
            const int n_planes = __popc(p.variants);
            for (int unit = blockIdx.x; unit < units; unit += gridDim.x) {
                const int first = (tc_seq_len(p, unit / p.Hkv) + TILE - 1) / TILE * TILE;
                for (int pl = 0; pl < n_planes; ++pl)
                    for (int i = first + et; i < p.Nmax; i += 256) p.scores[(size_t)pl * plane + (size_t)unit * p.Nmax + i] = 0.f;
            }
        }
    }

    if (failed) atomicCAS(p.status, 0u, (unsigned)(fail_site > 0 ? fail_site : 1));   // the first failure is kept
    tc_fence_before();
    __syncthreads();
    span_end(p.span);
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
    }
}

// Adds to the scores of every tile pair that several CTAs shared what its second, third, ... CTA left in its copy, in that
// order.  One block per pair.
__global__ void __launch_bounds__(2 * TILE)
tc_partial_sum_kernel(TcParams p, int n_planes) {
    pdl_wait();
    const int unit = blockIdx.y, j = blockIdx.x, tok = j * 2 * TILE + threadIdx.x;
    if (j * 2 * TILE >= tc_seq_len(p, unit / p.Hkv) || tok >= p.Nmax) return;
    // (bounded: after a wait that gave up nobody may have written the count)
    const int copies = min(p.copies[(size_t)unit * p.max_pairs + j], p.csplit - 1);
    if (copies <= 0) return;
    const size_t plane = (size_t)p.B * p.Hkv * p.Nmax;
    for (int pl = 0; pl < n_planes; ++pl) {
        const size_t at = (size_t)pl * plane + (size_t)unit * p.Nmax + tok;
        float sum = p.scores[at];
#pragma unroll 4
        for (int cp = 0; cp < copies; ++cp) sum += p.partial[(size_t)cp * n_planes * plane + at];
        p.scores[at] = sum;
    }
}

// =================================================================================================
// Pass 1 on tensor cores: streaming softmax statistics and window outputs (Sec. 3: A = softmax(Z),
// O = A V over the perturbation window, Eq. 9), split over the cached tokens.
//
// Rows of the window (one chunk of up to 128) sit on the MMA M dimension, so a TMEM lane holds one
// row and the softmax thread that owns it reduces along the tile without cross-thread traffic.
// Two softmax warpgroups take alternate token tiles; each keeps its own running statistics and its
// own output accumulator; at the end the CTA merges the two and writes one partial result per
// token split, which the combine kernel merges across splits.  For tile t and warpgroup w = t mod 2:
//     S_w  = Q_chunk . K_tile^T                    (tcgen05, accumulator in TMEM)
//     P_w  = exp2(S_w * scale*log2e - m_used)      (registers -> bf16 -> TMEM, over S_w's columns)
//     O_w += P_w . V_tile                          (tcgen05: A operand from TMEM, V as MN-major B)
// m_used is the exponent reference of the row; it is only moved up (and O_w, l rescaled) when the
// tile maximum exceeds it by more than 8 (a factor 256), which keeps P within bf16/fp32 range.
// MMAs issued by one thread execute in order, so S_w of tile t+2 cannot overwrite P_w before
// P_w . V of tile t has read it, and a commit after S_w(t) also covers P_w . V of tile t-2.
//
//   warp 0      TMA producer (Q chunk once, K/V tiles into a 3-stage ring)
//   warp 1      MMA issuer
//   warps 4-7   softmax warpgroup 0 (even tiles), warps 8-11 softmax warpgroup 1 (odd tiles)
// TMEM columns: S_0 [0,128)  S_1 [128,256)  O_0 [256,384)  O_1 [384,512)
// =================================================================================================
constexpr int kThreadsP1 = 384;
constexpr int P1_NSTAGE = 3;
constexpr uint32_t P1_OFF_Q = 0;
constexpr uint32_t P1_OFF_K = P1_OFF_Q + kOperandBytes;
constexpr uint32_t P1_OFF_V = P1_OFF_K + P1_NSTAGE * kOperandBytes;
constexpr uint32_t P1_OFF_BAR = P1_OFF_V + P1_NSTAGE * kOperandBytes;
enum { P1_FULL = 0, P1_EMPTY = P1_NSTAGE, P1_QFULL = 2 * P1_NSTAGE, P1_SFULL = 2 * P1_NSTAGE + 1,
       P1_PFULL = 2 * P1_NSTAGE + 3, P1_ODONE = 2 * P1_NSTAGE + 5, P1_NBARS = 2 * P1_NSTAGE + 6 };
constexpr uint32_t P1_OFF_TMEM = P1_OFF_BAR + P1_NBARS * 8;
constexpr uint32_t kSmemP1 = P1_OFF_TMEM + 16 + 1024;
constexpr float kRescaleThreshold = 8.f;                   // log2 units

struct P1Params {
    int B, Hq, Hkv, G, W, R, Nmax;
    const int32_t* seq_lens;
    const int32_t* mask_lens;                              // or nullptr: length the causal mask counts from
    float scale;
    int causal;
    int n_chunks, chunk_rows;
    int head_chunks;                                       // whole row chunks (pairs of them) that a head's W rows fill, under a causal window; else 0
    int n_splits, tiles_per_split;                         // CTAs per (unit, chunk); each writes one partial
    int l2_stream;                                         // K/V copies carry the "evict first" L2 hint
    float* part_m; float* part_l; float* part_o;           // [units][n_splits][R] (x d for part_o)
    float* nv;                                             // [units][Nmax]: ||v_p||^2, written by the CTAs of the last row chunk; null: not wanted
    unsigned int* status;
    unsigned long long* span;                              // [2]: ~(earliest CTA start), latest CTA end, in globaltimer ns
    // One CTA per (unit, row chunk): the CTA writes the merged results itself (what the combine kernel would make of its
    // single partial), the last chunk's also the padding rows, and no combine kernel runs.  Null out_o: partial results as above.
    int rows_out;
    float* out_o; __nv_bfloat16* out_obf;                  // [units][rows_out][d]: O; -2 O (HILO: a high and a low part per unit)
    float* out_lse2; float* out_onorm; float* out_cpair;   // [units][rows_out]; row-pair constants as float4 per pair
};

__device__ __forceinline__ void tc_ld32(uint32_t taddr, uint32_t* r) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
                 "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
                   "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
                   "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
                 : "r"(taddr) : "memory");
}
// waits for this thread's TMEM loads; the registers are operands so that no use is moved above it
__device__ __forceinline__ void tc_wait_ld32(uint32_t* r) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]),
                   "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]),
                   "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
                 :: "memory");
}
__device__ __forceinline__ void tc_st32(uint32_t taddr, const uint32_t* r) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
                 "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};"
                 ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
                   "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]),
                   "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]),
                   "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
                 : "memory");
}
__device__ __forceinline__ void tc_st16(uint32_t taddr, const uint32_t* r) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
                 ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
                   "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
                 : "memory");
}
__device__ __forceinline__ void tc_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
// D[tmem] (+)= A[tmem] * B[smem]: the A operand (rows on lanes, K packed two bf16 per column) is read from TMEM
__device__ __forceinline__ void tc_mma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
                 ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}

// (V as the MN-major B operand of P.V: 64 contiguous head-dim elements per 128-byte row, 8 tokens per
// 1024-byte group = stride byte offset, the next 64 head-dim elements one 16 KB block further = leading
// byte offset: the image of a [tokens][head_dim] tile loaded as two 64-wide boxes; see desc_lo_mn.)
__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
__device__ __forceinline__ float fmax3(float a, float b, float c) {
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// zeroes the calling thread's row of a V tile, for the MMAs that follow, if it is row `first` or a later one
__device__ __forceinline__ void zero_rows_from(uint8_t* tile, int row, int first) {
    if (row < first) return;
    uint8_t* at = tile + row * 128;
#pragma unroll
    for (int ch = 0; ch < 8; ++ch) {
        *reinterpret_cast<uint4*>(at + (ch << 4)) = make_uint4(0, 0, 0, 0);
        *reinterpret_cast<uint4*>(at + kHalfBytes + (ch << 4)) = make_uint4(0, 0, 0, 0);
    }
    fence_async_smem();
}

// The softmax of one 128-token tile of pass 1, by the thread that owns the row (tc_short_kernel has one of its own: half a tile per warpgroup,
// and no running reference, since it has a single tile): logits at tS in, P over their first 64 columns out, the running
// reference m_used and sum l moved on; `has_o`: the warpgroup's accumulator tO holds earlier tiles and follows the reference.
__device__ __forceinline__ void softmax_tile(uint32_t tS, uint32_t tO, int nvis, bool masked, float sl2, bool valid, bool low_part, bool has_o,
                                             float& m_used, float& l) {
    // sweep 1: tile maximum of the row (raw logits; the scale is positive)
    float mt = -INFINITY;
    {
        uint32_t sa[32], sb[32];
        tc_ld32(tS, sa);
#pragma unroll
        for (int pc = 0; pc < 4; pc += 2) {
            tc_wait_ld32(sa);
            tc_ld32(tS + (pc + 1) * 32, sb);
            if (masked) {
#pragma unroll
                for (int j = 0; j < 32; ++j) if (pc * 32 + j >= nvis) sa[j] = 0xff800000u;
            }
#pragma unroll
            for (int j = 0; j < 32; j += 2) mt = fmax3(mt, __uint_as_float(sa[j]), __uint_as_float(sa[j + 1]));
            tc_wait_ld32(sb);
            if (pc + 2 < 4) tc_ld32(tS + (pc + 2) * 32, sa);
            if (masked) {
#pragma unroll
                for (int j = 0; j < 32; ++j) if ((pc + 1) * 32 + j >= nvis) sb[j] = 0xff800000u;
            }
#pragma unroll
            for (int j = 0; j < 32; j += 2) mt = fmax3(mt, __uint_as_float(sb[j]), __uint_as_float(sb[j + 1]));
        }
    }
    mt *= sl2;
    const bool need = mt > m_used + kRescaleThreshold;               // also true for the first visible tile
    const float factor = need ? fast_exp2(m_used - mt) : 1.f;        // m_used = -inf -> 0
    if (has_o && __any_sync(0xffffffffu, valid && need && m_used != -INFINITY)) {
        // P.V of this warpgroup's previous tile is complete (the commit that signalled S covers it)
#pragma unroll 1
        for (int q4 = 0; q4 < 4; ++q4) {
            uint32_t ov[32];
            tc_ld32(tO + q4 * 32, ov);
            tc_wait_ld32(ov);
#pragma unroll
            for (int j = 0; j < 32; ++j) ov[j] = __float_as_uint(__uint_as_float(ov[j]) * factor);
            tc_st32(tO + q4 * 32, ov);
        }
    }
    l *= factor;
    if (need) m_used = mt;
    const float m_eff = m_used == -INFINITY ? 0.f : m_used;
    const float2 sl2v = make_float2(sl2, sl2), negm = make_float2(-m_eff, -m_eff);

    // sweep 2: P = exp2(S * scale*log2e - m_used) as bf16 over the first 64 columns of S_w
    float2 lsum = make_float2(0.f, 0.f);
    {
        uint32_t sa[32], sb[32];
        auto piece = [&](uint32_t* sv, int pc) {
            uint32_t pk[16];
#pragma unroll
            for (int j = 0; j < 32; j += 2) {
                float2 x = make_float2(__uint_as_float(sv[j]), __uint_as_float(sv[j + 1]));
                x = __ffma2_rn(x, sl2v, negm);
                if (masked) {
                    if (pc * 32 + j >= nvis) x.x = -INFINITY;
                    if (pc * 32 + j + 1 >= nvis) x.y = -INFINITY;
                }
                const float2 e = make_float2(fast_exp2(x.x), fast_exp2(x.y));
                lsum = __fadd2_rn(lsum, e);
                pk[j >> 1] = pack_bf16x2(e.x, e.y);
                if (low_part) {                                      // P = bf16(P) + bf16(P - bf16(P)): the second term
                    const float2 h = bf16x2_to_f32x2(pk[j >> 1]);
                    pk[j >> 1] = pack_bf16x2(e.x - h.x, e.y - h.y);
                }
            }
            tc_st16(tS + pc * 16, pk);
        };
        tc_ld32(tS, sa);
#pragma unroll
        for (int pc = 0; pc < 4; pc += 2) {
            tc_wait_ld32(sa);
            tc_ld32(tS + (pc + 1) * 32, sb);
            piece(sa, pc);
            tc_wait_ld32(sb);
            if (pc + 2 < 4) tc_ld32(tS + (pc + 2) * 32, sa);
            piece(sb, pc + 1);
        }
    }
    l += lsum.x + lsum.y;
    tc_wait_st();
}

// Row chunk of a block (PAIR: pair of consecutive row chunks, in place of a chunk below).  Under a causal window a chunk of rows visits the tiles up to its last row's position, and all
// of them if it holds the end of a head and the start of the next.  With more CTAs than SMs the chunks that visit most
// tiles are handed out first: where a head has several chunks, blocks are ordered by the chunk's place counted back from
// the chunk of its head's last row.  (Heads need not end where chunks do: by chunk number alone pass 1 took 63 instead
// of 46 us for 2 KV heads x 4 heads x 3500 queries, 136 instead of 126 us for 8 x 4 x 3001.)  Otherwise by chunk, last first.
template <bool PAIR>
__device__ __forceinline__ void p1_chunk_of_block(const P1Params& p, int vu, int& unit, int& c) {
    const int rows = PAIR ? 2 * p.chunk_rows : p.chunk_rows, n = PAIR ? (p.n_chunks + 1) / 2 : p.n_chunks;
    const int base = p.head_chunks;                         // a head has this many chunks or one more; 0: by chunk number
    if (base) {
        auto end = [&](int h) { return ((h + 1) * p.W - 1) / rows; };       // the chunk of head h's last row
        const int heads = p.B * p.Hkv * p.G, place = vu / heads;
        if (place < base) {
            const int rest = vu % heads;
            unit = rest / p.G;
            c = end(rest % p.G) - place;
        } else {                                            // the first chunk of every head that has one more
            const int rest = vu - base * heads, extra = n - base * p.G;
            int e = rest % extra, h = 0, before = -1;       // before: the end of the head before h
            for (; h < p.G; ++h) {
                const int at = end(h);
                if (at - before > base && e-- == 0) break;
                before = at;
            }
            unit = rest / extra;
            c = before + 1;
        }
        return;
    }
    unit = vu / n;
    c = n - 1 - vu % n;
}

// HILO: fewer than 64 window rows; MMA rows 64.. repeat rows 0.. and carry the low part of P.
// PAIR: the CTA takes two row chunks, one per softmax warpgroup, and each warpgroup sees every tile: a tile is fetched for
// both, there are half as many CTAs to set up and to drain, and nothing to merge between the warpgroups.  Warpgroup 0 has the
// chunk that visits more tiles.  Two K/V stages make room for the second Q chunk; a tile lasts twice as long.
template <bool HILO, bool PAIR>
__global__ void __launch_bounds__(kThreadsP1, 1)
tc_pass1_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                const __grid_constant__ CUtensorMap map_v, const __grid_constant__ P1Params p) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const uint32_t sbase = smem_u32(smem);
    const uint32_t bars = sbase + P1_OFF_BAR;
    auto bar = [&](int i) { return bars + 8u * (uint32_t)i; };
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem + P1_OFF_TMEM);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    span_begin(p.span);

    const int split = blockIdx.x;
    constexpr int NST = PAIR ? 2 : P1_NSTAGE;
    constexpr uint32_t OFF_K1 = PAIR ? P1_OFF_Q + 2 * kOperandBytes : P1_OFF_K, OFF_V1 = OFF_K1 + NST * kOperandBytes;
    static_assert(OFF_V1 + NST * kOperandBytes <= P1_OFF_BAR && !(HILO && PAIR), "layout");
    int unit, c;
    p1_chunk_of_block<PAIR>(p, blockIdx.y, unit, c);
    const int b = unit / p.Hkv, g = unit % p.Hkv;
    const bool nv_job = !PAIR && p.nv != nullptr && c == p.n_chunks - 1;     // this CTA also writes ||v_p||^2 of the tiles it visits
    if (threadIdx.x == 0) {
        prefetch_tmap(&map_q); prefetch_tmap(&map_k); prefetch_tmap(&map_v);
        // a K/V stage is released by the MMA commit and, where they are at work, by the two ||v||^2 warps
        for (int i = 0; i < NST; ++i) { mbar_init(bar(P1_FULL + i), 1); mbar_init(bar(P1_EMPTY + i), nv_job ? 3 : 1); }
        mbar_init(bar(P1_QFULL), 1); mbar_init(bar(P1_ODONE), 1);
        for (int i = 0; i < 2; ++i) { mbar_init(bar(P1_SFULL + i), 1); mbar_init(bar(P1_PFULL + i), 4); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sbase + P1_OFF_TMEM), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    bool failed = false;
    int fail_site = 0;                             // source line of the wait that gave up (status word)
    pdl_wait();                                    // above, only the span words of the workspace header were touched (atomically)
    // the status word starts at 0: no wait of this call can have given up yet (each lasts seconds)
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *p.status = 0u;
    const int N = tc_seq_len_raw(p.seq_lens, b, p.Nmax);
    // a split past the end of a shorter sequence has nothing to do and the merge does not read its partial result
    // (the lengths may be the preceding kernel's output, so they are read after the wait)
    const bool idle_split = split > 0 && split * p.tiles_per_split * TILE >= N;
    const int tile_lo = split * p.tiles_per_split;
    // tiles past the last token that any row of this chunk sees are not visited
    const int Nm = p.mask_lens ? p.mask_lens[b] : N;       // a shard of a longer sequence: its distance to that sequence's end
    auto tiles_of_chunk = [&](int ch) -> int {
        if (ch >= p.n_chunks) return 0;
        const int chunk_last = rows_last_token(ch * p.chunk_rows, min((ch + 1) * p.chunk_rows, p.R) - 1, p.W, Nm, p.causal);
        return max(min(min(tile_lo + p.tiles_per_split, (N + TILE - 1) / TILE), chunk_last / TILE + 1) - tile_lo, 0);
    };
    int c0 = c, c1 = c, n_tiles, n1 = 0;                   // chunks of the two warpgroups; tiles of the first (PAIR: and of the second)
    if (PAIR) {
        c0 = 2 * c + 1; c1 = 2 * c;
        n_tiles = tiles_of_chunk(c0); n1 = tiles_of_chunk(c1);
        if (n1 > n_tiles) { c0 = 2 * c; c1 = 2 * c + 1; const int t = n1; n1 = n_tiles; n_tiles = t; }
    } else {
        n_tiles = tiles_of_chunk(c);
    }

    if (idle_split) {
        // nothing to compute and nothing to store
    } else if (warp == 0) {
        // ===================================== TMA producer =====================================
        if (lane == 0 && n_tiles > 0) {
            mbar_expect_tx(bar(P1_QFULL), (uint32_t)p.chunk_rows * (HILO || (PAIR && n1 > 0) ? 512u : 256u));
            const int qrow = (b * p.Hq + g * p.G) * p.W + c0 * p.chunk_rows;
            tma_load_2d(sbase + P1_OFF_Q, &map_q, bar(P1_QFULL), 0, qrow);
            tma_load_2d(sbase + P1_OFF_Q + kHalfBytes, &map_q, bar(P1_QFULL), 64, qrow);
            if (HILO) {
                tma_load_2d(sbase + P1_OFF_Q + kHalfBytes / 2, &map_q, bar(P1_QFULL), 0, qrow);
                tma_load_2d(sbase + P1_OFF_Q + kHalfBytes + kHalfBytes / 2, &map_q, bar(P1_QFULL), 64, qrow);
            }
            if (PAIR && n1 > 0) {
                const int qrow1 = (b * p.Hq + g * p.G) * p.W + c1 * p.chunk_rows;
                tma_load_2d(sbase + P1_OFF_Q + kOperandBytes, &map_q, bar(P1_QFULL), 0, qrow1);
                tma_load_2d(sbase + P1_OFF_Q + kOperandBytes + kHalfBytes, &map_q, bar(P1_QFULL), 64, qrow1);
            }
            int issued = 0;
            const uint64_t pol_stream = l2_policy_evict_first();
            for (int i = 0; i < n_tiles; ++i) {
                const uint32_t st = i % NST;
                if (!mbar_wait(bar(P1_EMPTY + st), ((i / NST) & 1) ^ 1)) { failed = true; fail_site = __LINE__; break; }
                mbar_expect_tx(bar(P1_FULL + st), 2 * kOperandBytes);
                const uint32_t dk = sbase + OFF_K1 + st * kOperandBytes, dv = sbase + OFF_V1 + st * kOperandBytes;
                const int t0 = (tile_lo + i) * TILE;
                if (p.l2_stream) {                             // the cache cannot hold K and V until pass 2 anyway
                    tma_load_4d_hint(dk, &map_k, bar(P1_FULL + st), 0, t0, g, b, pol_stream);
                    tma_load_4d_hint(dk + kHalfBytes, &map_k, bar(P1_FULL + st), 64, t0, g, b, pol_stream);
                    tma_load_4d_hint(dv, &map_v, bar(P1_FULL + st), 0, t0, g, b, pol_stream);
                    tma_load_4d_hint(dv + kHalfBytes, &map_v, bar(P1_FULL + st), 64, t0, g, b, pol_stream);
                } else {
                    tma_load_4d(dk, &map_k, bar(P1_FULL + st), 0, t0, g, b);
                    tma_load_4d(dk + kHalfBytes, &map_k, bar(P1_FULL + st), 64, t0, g, b);
                    tma_load_4d(dv, &map_v, bar(P1_FULL + st), 0, t0, g, b);
                    tma_load_4d(dv + kHalfBytes, &map_v, bar(P1_FULL + st), 64, t0, g, b);
                }
                ++issued;
            }
            for (int back = 0; back < NST && back < issued; ++back) {         // drain own copies
                const int it = issued - 1 - back;
                (void)mbar_wait(bar(P1_FULL + it % NST), (it / NST) & 1);
            }
            (void)mbar_wait(bar(P1_QFULL), 0);
        }
    } else if (warp == 1) {
        // ===================================== MMA issuer =======================================
        if (lane == 0 && n_tiles > 0) {
            const uint32_t idesc_s = idesc_bf16(TILE);
            const uint32_t idesc_pv = idesc_bf16(kD) | (1u << 16);           // B operand (V) is MN-major
            // Item i: tile i, warpgroup i mod 2; in pairs tile i / 2 (items of warpgroup 1 past its tiles are left out).
            auto tile_at = [&](int i) { return PAIR ? i >> 1 : i; };
            auto is_item = [&](int i) { return PAIR ? (i >> 1) < ((i & 1) ? n1 : n_tiles) : i < n_tiles; };
            auto issue_s = [&](int j) -> bool {                              // S_w = Q . K_j^T
                const uint32_t tl = tile_at(j), st = tl % NST;
                if (!mbar_wait(bar(P1_FULL + st), (tl / NST) & 1)) return false;
                tc_fence_after();
                const uint32_t ak = desc_lo_k(sbase + OFF_K1 + st * kOperandBytes);
                const uint32_t aq = desc_lo_k(sbase + P1_OFF_Q + (PAIR ? (j & 1) * kOperandBytes : 0u));
#pragma unroll
                for (int ks = 0; ks < 8; ++ks)
                    tc_mma(tmem_base + (j & 1) * 128u, desc_make(aq + desc_kstep(ks, kHalfBytes)), desc_make(ak + desc_kstep(ks, kHalfBytes)), idesc_s, ks > 0);
                tc_commit(bar(P1_SFULL + (j & 1)));
                return true;
            };
            failed = !mbar_wait(bar(P1_QFULL), 0);
            if (!failed) failed = !issue_s(0);
            if (!failed && is_item(1)) failed = !issue_s(1);
            if (failed) fail_site = __LINE__;
            const int n_items = PAIR ? 2 * n_tiles : n_tiles;
            for (int i = 0; i < n_items && !failed; ++i) {
                const uint32_t w = i & 1, tl = tile_at(i);
                if (PAIR && !is_item(i)) continue;
                if (!mbar_wait(bar(P1_PFULL + w), (i >> 1) & 1)) { failed = true; fail_site = __LINE__; break; }
                tc_fence_after();
                const uint32_t av = desc_lo_mn(sbase + OFF_V1 + (tl % NST) * kOperandBytes);
                const uint32_t first = i > 1;                                // the warpgroup's first tile initialises O_w
#pragma unroll
                for (int ks = 0; ks < 8; ++ks)                               // 128 tokens = 8 steps of K = 16 (2048 bytes of V each)
                    tc_mma_ts(tmem_base + 256u + w * 128u, tmem_base + w * 128u + ks * 8, desc_make(av + ks * (2048 >> 4)),
                              idesc_pv, ks > 0 ? 1u : first);
                if (!PAIR || w == 1 || !is_item(i + 1))
                    tc_commit(bar(P1_EMPTY + (tl % NST)));                   // S(i) and P.V(i) have read the stage (in pairs: both warpgroups')
                if (is_item(i + 2) && !issue_s(i + 2)) { failed = true; fail_site = __LINE__; break; }
            }
            if (!failed) tc_commit(bar(P1_ODONE));
        }
    } else if (warp < 4) {
        // ============ ||v_p||^2 of every cached token (CTAs of the last row chunk) ===============
        // Pass 2 needs it per token; the V tile is in shared memory here anyway, and these two warps
        // have nothing else to do, whereas in pass 2 every issue slot next to the epilogue counts.
        // (The last chunk holds the last window row, which sees every token, so its CTAs visit every tile.  The
        // pass-2 kernel for more than 128 window rows computes the norms itself: p.nv is null then.)
        if (nv_job) {
            const int t64 = threadIdx.x - 64;                                // 0..63
            for (int i = 0; i < n_tiles && !failed; ++i) {
                const uint32_t st = i % NST;
                if (!mbar_wait(bar(P1_FULL + st), (i / NST) & 1)) { failed = true; fail_site = __LINE__; break; }
                const uint8_t* vt = smem + OFF_V1 + st * kOperandBytes;
                const int t0 = (tile_lo + i) * TILE;
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const int tok = t64 + 64 * j;
                    float2 acc0 = make_float2(0.f, 0.f), acc1 = acc0, acc2 = acc0, acc3 = acc0;
#pragma unroll
                    for (int h = 0; h < 2; ++h)
#pragma unroll
                        for (int ch = 0; ch < 8; ++ch) {
                            const uint4 u = *reinterpret_cast<const uint4*>(vt + h * kHalfBytes + tok * 128 + ((ch ^ (tok & 7)) << 4));
                            const float2 f0 = bf16x2_to_f32x2(u.x), f1 = bf16x2_to_f32x2(u.y);
                            const float2 f2 = bf16x2_to_f32x2(u.z), f3 = bf16x2_to_f32x2(u.w);
                            acc0 = __ffma2_rn(f0, f0, acc0); acc1 = __ffma2_rn(f1, f1, acc1);
                            acc2 = __ffma2_rn(f2, f2, acc2); acc3 = __ffma2_rn(f3, f3, acc3);
                        }
                    const float2 sum = __fadd2_rn(__fadd2_rn(acc0, acc1), __fadd2_rn(acc2, acc3));
                    if (t0 + tok < p.Nmax) p.nv[(size_t)unit * p.Nmax + t0 + tok] = sum.x + sum.y;
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(P1_EMPTY + st));
            }
        }
    } else {
        // ======================================= softmax ========================================
        const int w = (warp - 4) >> 2;                                       // warpgroup: tiles w, w+2, ...
        const int lane_grp = warp & 3;
        const int row = lane_grp * 32 + lane;                                // row within the chunk
        const int cw = PAIR && w == 1 ? c1 : c0;                             // this warpgroup's row chunk
        const int rows_valid = min(p.chunk_rows, p.R - cw * p.chunk_rows);
        const bool low_part = HILO && lane_grp >= 2;                       // this warp's rows are the second copies of rows 0..63
        const int row_q = HILO ? row & 63 : row;
        const int r = cw * p.chunk_rows + row_q;
        const bool valid = row_q < rows_valid;
        const int last = valid ? (p.causal ? min(Nm - p.W + (r % p.W), N - 1) : N - 1) : -1;   // last visible token
        const int first_masked = min(p.causal ? Nm - p.W + 1 : N, N);        // tiles reaching it need the mask
        const float sl2 = p.scale * kLog2e;
        const uint32_t lane_addr = (uint32_t)(lane_grp * 32) << 16;
        const uint32_t tS = tmem_base + lane_addr + w * 128u, tO = tmem_base + lane_addr + 256u + w * 128u;
        float m_used = -INFINITY, l = 0.f;
        int my_tiles = 0;

        const int i_end = PAIR && w == 1 ? n1 : n_tiles;
        for (int i = PAIR ? 0 : w; i < i_end && !failed; i += PAIR ? 1 : 2, ++my_tiles) {
            const int t0 = (tile_lo + i) * TILE;
            if (!mbar_wait(bar(P1_SFULL + w), my_tiles & 1)) { failed = true; fail_site = __LINE__; break; }
            tc_fence_after();
            const int nvis = last - t0 + 1;                                  // columns j < nvis are visible
            // (a warp whose rows all see the whole tile skips the mask: under a whole-sequence window that is every tile off the diagonal)
            const bool masked = t0 + TILE > first_masked && __any_sync(0xffffffffu, nvis < TILE);

            softmax_tile(tS, tO, nvis, masked, sl2, valid, low_part, my_tiles > 0, m_used, l);
            if (t0 + TILE > N) zero_rows_from(smem + OFF_V1 + (i % NST) * kOperandBytes, row, N - t0);   // V rows past the sequence must not reach the MMA
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(P1_PFULL + w));
        }

        // ---- the CTA's partial result: merge the two warpgroups, then store whole 512-byte rows ----
        // A warp may read its 32 TMEM lanes in any column, so the thread of row r in either
        // warpgroup can read both accumulators of that row.  The warpgroups exchange (m, l) through
        // shared memory (the Q region, which the MMAs no longer read), then warpgroup w merges
        // head-dim columns [64 w, 64 w + 64) into a [128 rows][32 x 16 B] tile in the first K/V stage
        // (16-byte chunks XOR-swizzled by the row), and all eight warps store 512-byte rows.
        float* xm = reinterpret_cast<float*>(smem + P1_OFF_Q);               // [2][128]
        float* xl = xm + 256;                                                // [2][128]
        uint8_t* xo = smem + OFF_K1;
        bool have = my_tiles > 0 && !failed;
        if (n_tiles > 0) {                                                   // all MMAs done: accumulators final, smem free
            if (!mbar_wait(bar(P1_ODONE), 0)) { failed = true; fail_site = __LINE__; have = false; }
            tc_fence_after();
        }
        if constexpr (PAIR) {
            // every row is this thread's alone: normalised, turned through shared memory (the K stages are warpgroup 0's,
            // the V stages warpgroup 1's) and stored in whole rows
            xo += w * 2 * kOperandBytes;
            const bool fin = p.out_o != nullptr;
            const float M = have ? m_used : -INFINITY;
            const float o_scale = fin ? (l > 0.f ? 1.f / l : 0.f) : 1.f;
            float sq = 0.f;
#pragma unroll 1
            for (int q = 0; q < 4; ++q) {
                uint32_t oa[32];
                if (my_tiles > 0) { tc_ld32(tO + q * 32, oa); tc_wait_ld32(oa); }
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (my_tiles > 0)
                        o = make_float4(__uint_as_float(oa[4 * j]) * o_scale, __uint_as_float(oa[4 * j + 1]) * o_scale,
                                        __uint_as_float(oa[4 * j + 2]) * o_scale, __uint_as_float(oa[4 * j + 3]) * o_scale);
                    sq = fmaf(o.x, o.x, fmaf(o.y, o.y, fmaf(o.z, o.z, fmaf(o.w, o.w, sq))));
                    *reinterpret_cast<float4*>(xo + row * 512 + (((q * 8 + j) ^ (row & 31)) << 4)) = o;
                }
            }
            const size_t out0 = (size_t)unit * p.rows_out + (size_t)cw * p.chunk_rows;                          // row 0 of the chunk
            const size_t prow0 = ((size_t)unit * p.n_splits + split) * p.R + (size_t)cw * p.chunk_rows;
            if (valid && fin) {
                const float lse2 = M + log2f(l);
                p.out_lse2[out0 + row] = lse2; p.out_onorm[out0 + row] = sq;
                float* cp = p.out_cpair + ((out0 + row) >> 1) * 4 + ((out0 + row) & 1);
                cp[0] = -lse2; cp[2] = sq;
            } else if (valid) {
                p.part_m[prow0 + row] = M; p.part_l[prow0 + row] = l;
            }
            __syncwarp();                                                    // a warp stores the 32 rows it has turned
            __nv_bfloat16* obf = p.out_obf + out0 * kD + lane * 4;
#pragma unroll 1
            for (int h = 0; h < 2; ++h) {
                float4 rowv[16];
#pragma unroll
                for (int rr = 0; rr < 16; ++rr) {
                    const int orow = lane_grp * 32 + h * 16 + rr;
                    rowv[rr] = *reinterpret_cast<const float4*>(xo + orow * 512 + ((lane ^ (orow & 31)) << 4));
                }
#pragma unroll
                for (int rr = 0; rr < 16; ++rr) {
                    const int orow = lane_grp * 32 + h * 16 + rr;
                    if (orow >= rows_valid) continue;
                    const float4 o = rowv[rr];
                    if (!fin) { *reinterpret_cast<float4*>(p.part_o + (prow0 + orow) * kD + lane * 4) = o; continue; }
                    *reinterpret_cast<float4*>(p.out_o + (out0 + orow) * kD + lane * 4) = o;
                    *reinterpret_cast<uint2*>(obf + (size_t)orow * kD) =
                        make_uint2(pack_bf16x2(-2.f * o.x, -2.f * o.y), pack_bf16x2(-2.f * o.z, -2.f * o.w));
                }
            }
            if (fin && cw == p.n_chunks - 1)                                 // padding rows: O = 0, weight 0
                for (int r0 = p.R - cw * p.chunk_rows + lane_grp; r0 < p.rows_out - cw * p.chunk_rows; r0 += 4) {
                    *reinterpret_cast<float4*>(p.out_o + (out0 + r0) * kD + lane * 4) = make_float4(0.f, 0.f, 0.f, 0.f);
                    *reinterpret_cast<uint2*>(obf + (size_t)r0 * kD) = make_uint2(0u, 0u);
                    if (lane == 0) {
                        p.out_lse2[out0 + r0] = INFINITY; p.out_onorm[out0 + r0] = 0.f;
                        float* cp = p.out_cpair + ((out0 + r0) >> 1) * 4 + ((out0 + r0) & 1);
                        cp[0] = -INFINITY; cp[2] = 0.f;
                    }
                }
        } else {
        xm[w * 128 + row] = have ? m_used : -INFINITY;
        xl[w * 128 + row] = l;
        asm volatile("bar.sync 1, 256;" ::: "memory");                       // both softmax warpgroups
        {
            const float m0 = xm[row], m1 = xm[128 + row];
            const float M = fmaxf(m0, m1);
            const float f0 = m0 == -INFINITY ? 0.f : fast_exp2(m0 - M), f1 = m1 == -INFINITY ? 0.f : fast_exp2(m1 - M);
            const uint32_t tO0 = tmem_base + lane_addr + 256u + w * 64u, tO1 = tO0 + 128u;   // this half of O_0 and O_1
            const size_t prow0 = ((size_t)unit * p.n_splits + split) * p.R + (size_t)c * p.chunk_rows;   // row 0 of the chunk
            const bool fin = p.out_o != nullptr;
            const float Lrow = fmaf(xl[row], f0, xl[128 + row] * f1);
            // (L = 0: the row saw no token, which only a shard of a longer sequence can show)
            const float o_scale = fin ? (Lrow > 0.f ? 1.f / Lrow : 0.f) : 1.f;
            const float g0 = f0 * o_scale, g1 = f1 * o_scale;
            float sq = 0.f;                                                  // squared norm of this thread's 64 output columns
            if (w == 0 && valid && !fin && !low_part) { p.part_m[prow0 + row] = M; p.part_l[prow0 + row] = Lrow; }
#pragma unroll 1
            for (int q = 0; q < 2; ++q) {
                // CTA-uniform: warpgroup 0 owns tiles iff the split has any, warpgroup 1 iff it has two or more
                // (an accumulator that no MMA wrote is never read; one whose row saw no token holds zeros)
                uint32_t oa[32], ob[32];
                if (n_tiles > 0) { tc_ld32(tO0 + q * 32, oa); tc_wait_ld32(oa); }
                if (n_tiles > 1) { tc_ld32(tO1 + q * 32, ob); tc_wait_ld32(ob); }
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (n_tiles > 0)
                        o = make_float4(__uint_as_float(oa[4 * j]) * g0, __uint_as_float(oa[4 * j + 1]) * g0,
                                        __uint_as_float(oa[4 * j + 2]) * g0, __uint_as_float(oa[4 * j + 3]) * g0);
                    if (n_tiles > 1) {
                        o.x = fmaf(__uint_as_float(ob[4 * j]), g1, o.x);     o.y = fmaf(__uint_as_float(ob[4 * j + 1]), g1, o.y);
                        o.z = fmaf(__uint_as_float(ob[4 * j + 2]), g1, o.z); o.w = fmaf(__uint_as_float(ob[4 * j + 3]), g1, o.w);
                    }
                    sq = fmaf(o.x, o.x, fmaf(o.y, o.y, fmaf(o.z, o.z, fmaf(o.w, o.w, sq))));
                    const int chunk = w * 16 + q * 8 + j;
                    *reinterpret_cast<uint4*>(xo + row * 512 + ((chunk ^ (row & 31)) << 4)) =
                        make_uint4(__float_as_uint(o.x), __float_as_uint(o.y), __float_as_uint(o.z), __float_as_uint(o.w));
                }
            }
            float* xs = xl + 256;                                            // [2][128]: the two halves of ||o||^2; then [128] log2-sum-exp
            if (fin) {
                xs[w * 128 + row] = sq;
                if (w == 0) xs[256 + row] = M + log2f(Lrow);
            }
            asm volatile("bar.sync 2, 256;" ::: "memory");                   // the merged tile is complete
            const int row_lo = (warp - 4) * 16;                              // 8 warps x 16 rows
            uint4 rowv[16];
#pragma unroll
            for (int rr = 0; rr < 16; ++rr) {
                const int orow = row_lo + rr;
                rowv[rr] = *reinterpret_cast<const uint4*>(xo + orow * 512 + ((lane ^ (orow & 31)) << 4));
            }
            if (HILO) {                                                    // rows 64.. hold what the low part of P added to rows 0..
#pragma unroll
                for (int rr = 0; rr < 16; ++rr) {
                    const int orow = (row_lo + rr) | 64;
                    const float4 lo = *reinterpret_cast<const float4*>(xo + orow * 512 + ((lane ^ (orow & 31)) << 4));
                    rowv[rr] = make_uint4(__float_as_uint(__uint_as_float(rowv[rr].x) + lo.x), __float_as_uint(__uint_as_float(rowv[rr].y) + lo.y),
                                          __float_as_uint(__uint_as_float(rowv[rr].z) + lo.z), __float_as_uint(__uint_as_float(rowv[rr].w) + lo.w));
                }
            }
            if (fin) {
                // O, -2 O in bf16, and per row the log2-sum-exp, ||o||^2 and the row's half of its pair's constants
                const size_t out0 = (size_t)unit * p.rows_out + (size_t)c * p.chunk_rows;
                __nv_bfloat16* obf = p.out_obf + ((size_t)unit * p.rows_out * (HILO ? 2 : 1) + (size_t)c * p.chunk_rows) * kD + lane * 4;
                float on = 0.f;                                              // of row row_lo + lane
                if (!HILO && lane < 16) on = xs[row_lo + lane] + xs[128 + row_lo + lane];
#pragma unroll
                for (int rr = 0; rr < 16; ++rr) {
                    const int orow = row_lo + rr;
                    if (orow < rows_valid) {
                        const float4 o = make_float4(__uint_as_float(rowv[rr].x), __uint_as_float(rowv[rr].y), __uint_as_float(rowv[rr].z), __uint_as_float(rowv[rr].w));
                        *reinterpret_cast<float4*>(p.out_o + (out0 + orow) * kD + lane * 4) = o;
                        const uint32_t b0 = pack_bf16x2(-2.f * o.x, -2.f * o.y), b1 = pack_bf16x2(-2.f * o.z, -2.f * o.w);
                        *reinterpret_cast<uint2*>(obf + (size_t)orow * kD) = make_uint2(b0, b1);
                        if (HILO) {                                          // what the high part leaves out; the norm of both parts of O
                            const float2 h0 = bf16x2_to_f32x2(b0), h1 = bf16x2_to_f32x2(b1);
                            *reinterpret_cast<uint2*>(obf + (size_t)(p.rows_out + orow) * kD) =
                                make_uint2(pack_bf16x2(fmaf(-2.f, o.x, -h0.x), fmaf(-2.f, o.y, -h0.y)), pack_bf16x2(fmaf(-2.f, o.z, -h1.x), fmaf(-2.f, o.w, -h1.y)));
                            const float n = warp_sum((o.x * o.x + o.y * o.y) + (o.z * o.z + o.w * o.w));
                            if (lane == rr) on = n;
                        }
                    }
                }
                if (lane < 16 && row_lo + lane < rows_valid) {
                    const size_t gr = out0 + row_lo + lane;
                    const float lse2 = xs[256 + row_lo + lane];
                    p.out_lse2[gr] = lse2; p.out_onorm[gr] = on;
                    float* cp = p.out_cpair + (gr >> 1) * 4 + (gr & 1);
                    cp[0] = -lse2; cp[2] = on;
                }
                if (c == p.n_chunks - 1)                                     // padding rows: O = 0, weight 0
                    for (int r0 = p.R - c * p.chunk_rows + warp - 4; r0 < p.rows_out - c * p.chunk_rows; r0 += 8) {
                        *reinterpret_cast<float4*>(p.out_o + (out0 + r0) * kD + lane * 4) = make_float4(0.f, 0.f, 0.f, 0.f);
                        *reinterpret_cast<uint2*>(obf + (size_t)r0 * kD) = make_uint2(0u, 0u);
                        if (HILO) *reinterpret_cast<uint2*>(obf + (size_t)(p.rows_out + r0) * kD) = make_uint2(0u, 0u);
                        if (lane == 0) {
                            const size_t gr = out0 + r0;
                            p.out_lse2[gr] = INFINITY; p.out_onorm[gr] = 0.f;
                            float* cp = p.out_cpair + (gr >> 1) * 4 + (gr & 1);
                            cp[0] = -INFINITY; cp[2] = 0.f;
                        }
                    }
            } else {
#pragma unroll
                for (int rr = 0; rr < 16; ++rr) {                            // one coalesced 512-byte row per instruction
                    const int orow = row_lo + rr;
                    if (orow < rows_valid) *reinterpret_cast<uint4*>(p.part_o + (prow0 + orow) * kD + lane * 4) = rowv[rr];
                }
            }
        }
        }
        tc_fence_before();
    }

    if (failed) atomicCAS(p.status, 0u, (unsigned)(fail_site > 0 ? fail_site : 1));   // the first failure is kept
    tc_fence_before();
    __syncthreads();
    span_end(p.span);
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
    }
}

// =================================================================================================
// A short cache in one kernel: both passes and the merge between them, for a unit whose tiles have a cluster of CTAs, one
// tile each (CTAs beyond the tiles, where the cluster has some, take their share of the merge).  As three kernels such a call is mostly
// their beginnings and ends and the second trip of K and V.  A CTA forms the logits, P and its part of O as pass 1 does; row slices of the partial outputs go to the CTA that owns the slice, which adds them
// in the order of the tiles and hands -2 O (HILO: both parts), as the operand image, and the row constants to every CTA of the
// cluster; the scores of the tile follow from the K and V tiles that are still there (Z from before K and Q made room for the staged O).
// Partial outputs cross the cluster as bulk copies of runs of staged rows, the merged rows as plain stores; both arrive on the
// receiver's mbarriers, and a CTA that has seen its image complete has neither copies out of its memory nor stores into it under way
// (its owners have merged what it sent, and all that it receives is counted).  A warp whose wait gives up arrives nowhere any more and
// copies and stores nothing more, so that nobody takes what is missing for complete; its CTA stays until the cluster's other CTAs are
// done with it (end of the kernel).
// The code runs once per launch, from a cold instruction cache: loops are kept short rather than unrolled.
//   warps 0-7  softmax (64 tokens of the tile per warpgroup), merge, score epilogue (half of the rows per warpgroup)
//   warp 8  copies     warp 9  MMAs     warps 10-11  value norms
// TMEM columns: S and P [0, 128)  O [128, 256)  Z^T [256, 384)  T'^T [384, 512)
// Bound by that chain, not by bytes: at 64 rows x 8 CTAs, cycles of set-up 2.1 k, copies and logits 2.1 k, softmax 2.5 k, P.V 1.3 k, the
// exchange of partial outputs 2.3 k, merge and hand-out 5.1 k, T' 0.9 k, scores 1.7 k.  Per call, three kernels / this one: 8 heads on 2 of
// 1024 tokens x 16 queries 13.9 / 10.7 us, 32 on 8 x 32 queries 16.7 / 13.8, one head of 128 tokens 14.8 / 8.8, of 2048 14.5 / 11.8, 7 KV heads of 2048
// 18.2 / 14.6, 32 of 512 19.3 / 14.9, 74 of 256 19.4 / 12.3.  (Partial outputs and -2 O through the workspace instead, with a device-wide
// fence before each arrival: 11.7, 14.2, 11.2, 12.5, 14.3, 16.5, 14.8; -2 O alone: 10.9, 14.0, 9.6, 11.9, 14.6, 15.3, 12.6.)
// =================================================================================================
constexpr int kThreadsShort = 384;
constexpr int SH_MAXC = 16;
constexpr uint32_t SH_PITCH = 528;                                 // a staged row: 128 floats of O, m, l of either half of the tile; no bank conflicts by row or by column
constexpr uint32_t SH_OFF_Q = 0;
constexpr uint32_t SH_OFF_K = SH_OFF_Q + kOperandBytes;
constexpr uint32_t SH_OFF_STAGE = SH_OFF_Q;                        // [128 accumulator rows], over Q and K once the MMAs have read them
constexpr uint32_t SH_OFF_XCH = SH_OFF_Q;                          // [kNumSums][128]: the second row half's sums, once the staged rows are with their owners
constexpr uint32_t SH_OFF_V = SH_OFF_STAGE + 128 * SH_PITCH;
constexpr uint32_t SH_OFF_O = SH_OFF_V + kOperandBytes;            // -2 O of the unit's rows
constexpr uint32_t SH_OFF_RX = SH_OFF_O + kOperandBytes;           // [source][row of the slice]
constexpr uint32_t SH_RX_ROWS = 160;                               // sources x slice rows: at most 128 + C - 1, or 2 x (63 + C - 1) with low parts
constexpr uint32_t SH_OFF_ROWS = SH_OFF_RX + SH_RX_ROWS * SH_PITCH; // [128] (-lse2, |o|^2, -, -)
constexpr uint32_t SH_OFF_CONST = SH_OFF_ROWS + 128 * 16;          // 8 epilogue warps x 32 float4: row-pair constants of the warp's rows
constexpr uint32_t SH_OFF_MAX = SH_OFF_CONST + 8 * 32 * 16;        // [2][128]: row maxima of the tile's halves
constexpr uint32_t SH_OFF_NV = SH_OFF_MAX + 2 * 128 * 4;           // [128] (||v||^2, ||v||_1)
constexpr uint32_t SH_OFF_BAR = SH_OFF_NV + TILE * 8;
enum { SH_QK = 0, SH_V, SH_S, SH_P, SH_ODONE, SH_STAGED, SH_RX, SH_IMG, SH_NORMS, SH_T, SH_DRAIN, SH_NBARS };
constexpr uint32_t SH_OFF_TMEM = SH_OFF_BAR + SH_NBARS * 8;
constexpr uint32_t kSmemShort = SH_OFF_TMEM + 16 + 1024;
static_assert(SH_OFF_V % 1024 == 0 && kSmemShort <= 227 * 1024, "layout");
static_assert(SH_RX_ROWS >= 128 + SH_MAXC - 1 && SH_RX_ROWS >= 2 * (63 + SH_MAXC - 1), "partial outputs of a slice");

__device__ __forceinline__ uint32_t cluster_addr(uint32_t addr, int rank) {      // the same place in another CTA of the cluster
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void st_cluster2(uint32_t addr, uint32_t a, uint32_t b) {
    asm volatile("st.shared::cluster.v2.b32 [%0], {%1, %2};" ::"r"(addr), "r"(a), "r"(b) : "memory");
}
__device__ __forceinline__ void arrive_at_cta(uint32_t remote_bar) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(remote_bar) : "memory");
}
// own shared memory -> another CTA's; the bytes arrive on that CTA's mbarrier
__device__ __forceinline__ void copy_to_cta(uint32_t dst, uint32_t src, uint32_t bytes, uint32_t dst_bar) {
    asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "r"(src), "r"(bytes), "r"(dst_bar) : "memory");
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

template <unsigned VARS, bool HILO, bool BY_UNIT>
__global__ void __launch_bounds__(kThreadsShort, 1)
tc_short_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                const __grid_constant__ CUtensorMap map_v, const __grid_constant__ TcParams p, int C) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const uint32_t sbase = smem_u32(smem), dbase = sbase & 0x3ffffu;   // (in a cluster the address carries the CTA's rank, which a matrix descriptor has no room for)
    auto bar = [&](int i) { return sbase + SH_OFF_BAR + 8u * (uint32_t)i; };
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem + SH_OFF_TMEM);
    float4* sRows = reinterpret_cast<float4*>(smem + SH_OFF_ROWS);
    float2* sNv = reinterpret_cast<float2*>(smem + SH_OFF_NV);
    float* sXch = reinterpret_cast<float*>(smem + SH_OFF_XCH);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    span_begin(p.span);
    const int unit = blockIdx.x / C, rank = blockIdx.x % C, b = unit / p.Hkv, g = unit % p.Hkv, t0 = rank * TILE;
    const int slice = (p.R + C - 1) / C;                               // rows [rank slice, rank slice + slice) are this CTA's to merge
    const int my_rows = max(min(slice, p.R - rank * slice), 0);
    const int mergers = p.R / slice * min(slice, 8) + min(p.R % slice, 8);     // warps of the cluster that merge rows: one at least, eight at most per slice
    constexpr uint32_t kParts = HILO ? 2 : 1;                          // of a partial output, and of -2 O

    if (threadIdx.x == 0) {
        prefetch_tmap(&map_k); prefetch_tmap(&map_v); prefetch_tmap(&map_q);
        for (int i = 0; i < SH_NBARS; ++i)
            mbar_init(bar(i), i == SH_P || i == SH_STAGED ? 8 : i == SH_NORMS ? 2 : i == SH_IMG ? (uint32_t)mergers : 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    cluster_arrive();                                                  // (waited for before the first copy to another CTA: its mbarriers are set up)
    if (warp == 8) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sbase + SH_OFF_TMEM), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // padding rows: O = 0, weight 0
    const int pad = p.chunk_rows - p.R;
    for (int i = threadIdx.x; i < pad * 16 * (int)kParts; i += kThreadsShort) {
        const int at = i >> 4, r = p.R + at + (at < pad ? 0 : p.chunk_rows - pad), ch = i & 15;
        *reinterpret_cast<uint4*>(smem + SH_OFF_O + (ch >> 3) * kHalfBytes + r * 128 + ((ch & 7) << 4)) = make_uint4(0, 0, 0, 0);
    }
    if ((int)threadIdx.x < pad) sRows[p.R + threadIdx.x] = make_float4(-INFINITY, 0.f, 0.f, 0.f);
    fence_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    bool failed = false;
    int fail_site = 0;                                                 // source line of the wait that gave up (status word)
    pdl_wait();
    if (blockIdx.x == 0 && threadIdx.x == 0) *p.status = 0u;           // no wait of this call can have given up yet (each lasts seconds)
    const int N = tc_seq_len(p, b), Nm = tc_mask_len(p, b);
    const bool empty = t0 >= N;                                        // a CTA past the end merges its slice and writes zeros
    const int n_src = min(C, (N + TILE - 1) / TILE);                   // tiles of the unit = partial outputs of a row
    const uint32_t tS = tmem_base, tO = tmem_base + 128u, tZ = tmem_base + 256u, tT = tmem_base + 384u;
    auto wait = [&](int i, int line) {
        if (!failed && !(i == SH_IMG ? mbar_wait<true>(bar(i), 0) : mbar_wait(bar(i), 0))) { failed = true; fail_site = line; }
        return !failed;
    };
    auto none_failed = [&] { __syncwarp(); return __all_sync(0xffffffffu, !failed) != 0; };   // in the calling warp
    auto arrive = [&](int i) { if (none_failed() && lane == 0) mbar_arrive(bar(i)); };         // for a whole warp

    if (warp == 8 && lane == 0) {
        mbar_expect_tx(bar(SH_RX), (uint32_t)(my_rows * (empty ? n_src : n_src - 1)) * kParts * SH_PITCH);   // (its own part stays where it is)
        if (!empty) {
            mbar_expect_tx(bar(SH_QK), kOperandBytes + (uint32_t)p.chunk_rows * 256u * kParts);
            for (int h = 0; h < 2; ++h) {
                load_q<BY_UNIT>(sbase + SH_OFF_Q + h * kHalfBytes, &map_q, bar(SH_QK), h * 64, 0, unit, p.R);
                tma_load_4d(sbase + SH_OFF_K + h * kHalfBytes, &map_k, bar(SH_QK), h * 64, t0, g, b);
                if (HILO) load_q<BY_UNIT>(sbase + SH_OFF_Q + h * kHalfBytes + kHalfBytes / 2, &map_q, bar(SH_QK), h * 64, 0, unit, p.R);
            }
            mbar_expect_tx(bar(SH_V), kOperandBytes);
            for (int h = 0; h < 2; ++h) tma_load_4d(sbase + SH_OFF_V + h * kHalfBytes, &map_v, bar(SH_V), h * 64, t0, g, b);
        }
    }
    __syncwarp();
    cluster_wait();                                                    // (behind the copies' start)

    if (warp == 8) {
        // ============================================ copies ================================================
        if (!empty) {
            wait(SH_QK, __LINE__); wait(SH_V, __LINE__);
            const int rows = min(slice, p.R - lane * slice);           // of owner `lane`
            if (wait(SH_STAGED, __LINE__) && lane < C && lane != rank && rows > 0)
                for (uint32_t part = 0; part < kParts; ++part)         // (the low part's accumulators are rows 64 ..)
                    copy_to_cta(cluster_addr(sbase + SH_OFF_RX + (rank * kParts + part) * slice * SH_PITCH, lane),
                                sbase + SH_OFF_STAGE + (part * 64u + lane * slice) * SH_PITCH, (uint32_t)rows * SH_PITCH, cluster_addr(bar(SH_RX), lane));
        }
    } else if (warp == 9) {
        // ============================================= MMAs =================================================
        if (lane == 0 && !empty) {
            const uint32_t aq = desc_lo_k(dbase + SH_OFF_Q), ak = desc_lo_k(dbase + SH_OFF_K);
            if (wait(SH_QK, __LINE__)) {
                tc_fence_after();
#pragma unroll
                for (int ks = 0; ks < 8; ++ks)
                    tc_mma(tS, desc_make(aq + desc_kstep(ks, kHalfBytes)), desc_make(ak + desc_kstep(ks, kHalfBytes)), idesc_bf16(TILE), ks > 0);
                tc_commit(bar(SH_S));
#pragma unroll
                for (int ks = 0; ks < 8; ++ks)
                    tc_mma(tZ, desc_make(ak + desc_kstep(ks, kHalfBytes)), desc_make(aq + desc_kstep(ks, kHalfBytes)), idesc_bf16(p.chunk_rows), ks > 0);
            }
            if (wait(SH_V, __LINE__) && wait(SH_P, __LINE__)) {
                tc_fence_after();
                const uint32_t av = desc_lo_mn(dbase + SH_OFF_V);
#pragma unroll
                for (int ks = 0; ks < 8; ++ks)                         // (P of tokens 64 .. stands over the logits of those)
                    tc_mma_ts(tO, tS + (ks >> 2) * 64 + (ks & 3) * 8, desc_make(av + ks * (2048 >> 4)), idesc_bf16(kD) | (1u << 16), ks > 0);
                tc_commit(bar(SH_ODONE));
            }
            if (wait(SH_IMG, __LINE__)) {
                asm volatile("fence.proxy.async;" ::: "memory");       // (the image was written by plain stores)
                tc_fence_after();
                const uint32_t av = desc_lo_k(dbase + SH_OFF_V), bo = desc_lo_k(dbase + SH_OFF_O);
#pragma unroll
                for (int ks = 0; ks < 8; ++ks)
                    tc_mma(tT, desc_make(av + desc_kstep(ks, kHalfBytes)), desc_make(bo + desc_kstep(ks, kHalfBytes)), idesc_bf16((int)kParts * p.chunk_rows), ks > 0);
                tc_commit(bar(SH_T));
            }
        }
    } else if (warp >= 10) {
        // ========================================== value norms =============================================
        if (!empty && wait(SH_V, __LINE__)) {
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int tok = (int)threadIdx.x - 320 + 64 * j;
                float l2, l1;
                value_norms<(VARS & OBC_VAR_VATP) != 0>(smem + SH_OFF_V, tok, l2, l1);
                sNv[tok] = make_float2(l2, l1);
            }
        }
        arrive(SH_NORMS);
    } else {
        const int w = warp >> 2, lane_grp = warp & 3, row = lane_grp * 32 + lane;
        const uint32_t lane_addr = (uint32_t)(lane_grp * 32) << 16;
        // ================= the tile's softmax and partial output: warpgroup w takes tokens [64 w, 64 w + 64) =================
        if (!empty) {
            const bool low_part = HILO && lane_grp >= 2;               // this warp's rows are the second copies of rows 0..63
            const int r = HILO ? row & 63 : row;
            const float sl2 = p.scale * kLog2e;
            float* sMax = reinterpret_cast<float*>(smem + SH_OFF_MAX);
            uint32_t z[32];
            float mt = -INFINITY, l = 0.f;
            const int last = r < p.R ? (p.causal ? min(Nm - p.W + (r % p.W), N - 1) : N - 1) : -1;   // last visible token
            const int nvis = last - t0 - w * 64 + 1;                   // columns j < nvis are visible
            const bool masked = __any_sync(0xffffffffu, nvis < 64);
            const uint32_t tSw = tS + lane_addr + w * 64u;
            auto load_logits = [&](int pc) {
                tc_ld32(tSw + pc * 32, z);
                tc_wait_ld32(z);
                if (masked) {
#pragma unroll
                    for (int j = 0; j < 32; ++j) if (pc * 32 + j >= nvis) z[j] = 0xff800000u;
                }
            };
            if (wait(SH_S, __LINE__)) {
                tc_fence_after();
#pragma unroll 1
                for (int pc = 0; pc < 2; ++pc) {
                    load_logits(pc);
#pragma unroll
                    for (int j = 0; j < 32; j += 2) mt = fmax3(mt, __uint_as_float(z[j]), __uint_as_float(z[j + 1]));
                }
            }
            sMax[w * 128 + row] = mt;
            asm volatile("bar.sync 1, 256;" ::: "memory");             // both warpgroups
            mt = fmaxf(mt, sMax[(w ^ 1) * 128 + row]);
            const float m = mt == -INFINITY ? mt : mt * sl2;
            if (!failed) {
                const float m_eff = m == -INFINITY ? 0.f : m;
                const float2 sl2v = make_float2(sl2, sl2), negm = make_float2(-m_eff, -m_eff);
                float2 lsum = make_float2(0.f, 0.f);
#pragma unroll 1
                for (int pc = 0; pc < 2; ++pc) {
                    uint32_t pk[16];
                    load_logits(pc);
#pragma unroll
                    for (int j = 0; j < 32; j += 2) {
                        const float2 x = __ffma2_rn(make_float2(__uint_as_float(z[j]), __uint_as_float(z[j + 1])), sl2v, negm);
                        const float2 e = make_float2(fast_exp2(x.x), fast_exp2(x.y));
                        lsum = __fadd2_rn(lsum, e);
                        pk[j >> 1] = pack_bf16x2(e.x, e.y);
                        if (low_part) {                                // P = bf16(P) + bf16(P - bf16(P)): the second term
                            const float2 h = bf16x2_to_f32x2(pk[j >> 1]);
                            pk[j >> 1] = pack_bf16x2(e.x - h.x, e.y - h.y);
                        }
                    }
                    tc_st16(tSw + pc * 16, pk);
                }
                l = low_part ? 0.f : lsum.x + lsum.y;                  // (the low part of P adds to O alone)
                tc_wait_st();
            }
            if (w == 1 && t0 + TILE > N && wait(SH_V, __LINE__)) zero_rows_from(smem + SH_OFF_V, row, N - t0);   // V rows past the sequence must not reach the MMA
            tc_fence_before();
            arrive(SH_P);
            if (wait(SH_ODONE, __LINE__)) {
                tc_fence_after();
                uint8_t* dst = smem + SH_OFF_STAGE + row * SH_PITCH;   // warpgroup w: head-dim columns [64 w, 64 w + 64)
#pragma unroll 1
                for (int pc = 0; pc < 2; ++pc) {
                    tc_ld32(tO + lane_addr + w * 64u + pc * 32u, z);
                    tc_wait_ld32(z);
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        *reinterpret_cast<uint4*>(dst + w * 256 + pc * 128 + j * 16) = make_uint4(z[4 * j], z[4 * j + 1], z[4 * j + 2], z[4 * j + 3]);
                }
                float* ml = reinterpret_cast<float*>(dst + 512);       // (m, l of the first half, l of the second, -)
                if (w == 0) { ml[0] = m; ml[1] = l; } else { ml[2] = l; }
                tc_fence_before();
            }
            fence_async_smem();
            arrive(SH_STAGED);
        }
        // ==================== the slice's rows: merged, row by row of a warp, two at a time ====================
        if ((empty || wait(SH_STAGED, __LINE__)) && wait(SH_RX, __LINE__)) {
            const int parts = n_src * (int)kParts;
            auto part_row = [&](int sp, int local) {
                const int mine = HILO ? sp - 2 * rank : sp - rank;     // 0 (and 1: the low part): this CTA's own
                return smem + (mine >= 0 && mine < (int)kParts ? SH_OFF_STAGE + (uint32_t)(mine * 64 + rank * slice + local) * SH_PITCH
                                                               : SH_OFF_RX + (uint32_t)(sp * slice + local) * SH_PITCH);
            };
#pragma unroll 1
            for (int local = warp; local < my_rows; local += 8) {
                const int r = rank * slice + local;
                const float4 ml = lane < parts ? *reinterpret_cast<const float4*>(part_row(lane, local) + 512) : make_float4(-INFINITY, 0.f, 0.f, 0.f);
                const float M = warp_max(ml.x), wt = ml.x == -INFINITY ? 0.f : exp2f(ml.x - M), L = warp_sum((ml.y + ml.z) * wt);
                float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 2
                for (int sp = 0; sp < parts; ++sp) {
                    const float f = __shfl_sync(0xffffffffu, wt, sp);
                    const float4 x = *reinterpret_cast<const float4*>(part_row(sp, local) + lane * 16);
                    o.x = fmaf(x.x, f, o.x); o.y = fmaf(x.y, f, o.y); o.z = fmaf(x.z, f, o.z); o.w = fmaf(x.w, f, o.w);
                }
                const float inv = L > 0.f ? 1.f / L : 1.f;
                o.x *= inv; o.y *= inv; o.z *= inv; o.w *= inv;
                const float onorm = warp_sum((o.x * o.x + o.y * o.y) + (o.z * o.z + o.w * o.w));
                const uint32_t h0 = pack_bf16x2(-2.f * o.x, -2.f * o.y), h1 = pack_bf16x2(-2.f * o.z, -2.f * o.w);
                const float2 f0 = bf16x2_to_f32x2(h0), f1 = bf16x2_to_f32x2(h1);   // HILO: and what the high part leaves out
                const uint32_t e0 = pack_bf16x2(fmaf(-2.f, o.x, -f0.x), fmaf(-2.f, o.y, -f0.y)), e1 = pack_bf16x2(fmaf(-2.f, o.z, -f1.x), fmaf(-2.f, o.w, -f1.y));
                // elements 4 lane .. of the row in the 128-byte swizzle of the operand
                auto place = [&](int at) { return sbase + SH_OFF_O + (uint32_t)((lane >> 4) * kHalfBytes + at * 128 + ((((lane & 15) >> 1) ^ (at & 7)) << 4) + (lane & 1) * 8); };
                const uint32_t hi = place(r), lo = place(p.chunk_rows + r);
#pragma unroll 2
                for (int d = 0; d < C; ++d) {
                    st_cluster2(cluster_addr(hi, d), h0, h1);
                    if (HILO) st_cluster2(cluster_addr(lo, d), e0, e1);
                }
                if (lane < C) st_cluster2(cluster_addr(sbase + SH_OFF_ROWS + (uint32_t)r * 16u, lane), __float_as_uint(-(M + log2f(L))), __float_as_uint(onorm));
            }
        }
        if (warp < my_rows) {
            asm volatile("fence.proxy.async;" ::: "memory");
            if (none_failed() && lane < C) arrive_at_cta(cluster_addr(bar(SH_IMG), lane));
        }
        // ========================================= the tile's scores =========================================
        const size_t plane = (size_t)p.B * p.Hkv * p.Nmax;
        const int tok = row, ptok = t0 + tok;
        if (empty) {
            if (w == 0 && ptok < p.Nmax)
                for (int pl = 0; pl < __popc(p.variants); ++pl) p.scores[(size_t)pl * plane + (size_t)unit * p.Nmax + ptok] = 0.f;
            wait(SH_IMG, __LINE__);
        } else {
            const int rows0 = min(p.chunk_rows, (p.chunk_rows / 2 + 15) / 16 * 16);    // two runs of whole 16-row batches
            const int r_begin = w ? rows0 : 0, r_count = w ? p.chunk_rows - rows0 : rows0;
            const float ksl = p.scale * kLog2e * kExpFactor<VARS, HILO>;
            const float2 sl2 = make_float2(ksl, ksl), sc = make_float2(p.scale, p.scale);
            const bool masked_tile = p.causal && (t0 + TILE - 1 > Nm - p.W);
            RowSums S;
            S.s1 = S.s2 = S.s3 = S.s4 = S.s5 = S.s6 = S.s7 = make_float2(0.f, 0.f);
            float4* my_const = reinterpret_cast<float4*>(smem + SH_OFF_CONST) + warp * 32;
            if (wait(SH_IMG, __LINE__) && lane * 2 < r_count) {
                const float4 c0 = sRows[r_begin + 2 * lane], c1 = sRows[r_begin + 2 * lane + 1];
                constexpr float kx = kExpFactor<VARS, HILO>;
                const float ko = VARS == OBC_VAR_VK ? p.scale : 1.f;
                my_const[lane] = make_float4(c0.x * kx, c1.x * kx, c0.y * ko, c1.y * ko);
            }
            __syncwarp();
            if (wait(SH_T, __LINE__) && r_count > 0) {
                tc_fence_after();
                const uint32_t zt = tZ + lane_addr + (uint32_t)r_begin, tt = zt + 128u;
                if (masked_tile) score_chunk<VARS, true, HILO>(zt, tt, r_count, my_const, sl2, sc, S, ptok, Nm - p.W, p.W, r_begin % p.W, p.chunk_rows);
                else score_chunk<VARS, false, HILO>(zt, tt, r_count, my_const, sl2, sc, S, ptok, 0, 0, 0, p.chunk_rows);
                tc_fence_before();
            }
            float sum[kNumSums] = {S.s1.x + S.s1.y, S.s2.x + S.s2.y, S.s3.x + S.s3.y, S.s4.x + S.s4.y, S.s5.x + S.s5.y, S.s6.x + S.s6.y, S.s7.x + S.s7.y};
            if (w == 1 && !failed) {
#pragma unroll
                for (int j = 0; j < kNumSums; ++j) sXch[j * TILE + tok] = sum[j];
            }
            asm volatile("bar.sync 1, 256;" ::: "memory");             // both warpgroups
            if (w == 0 && wait(SH_NORMS, __LINE__)) {
                const float2 nv = sNv[tok];
#pragma unroll
                for (int j = 0; j < kNumSums; ++j) sum[j] += sXch[j * TILE + tok];
                if (ptok < p.Nmax)
                    store_scores<VARS, HILO>(sum, nv.x, nv.y, p.scale, p.variants, p.scores + (size_t)unit * p.Nmax + ptok, plane, ptok < N);
            }
        }
    }
    if (failed) atomicCAS(p.status, 0u, (unsigned)(fail_site > 0 ? fail_site : 1));   // the first failure is kept
    tc_fence_before();
    if (__syncthreads_or(failed)) {
        // Copies into this CTA or out of it may be under way or still to come from CTAs that are only late.  Those where no wait gave up need
        // none of this: they saw their image complete, and a thread that has left counts as arrived.  Every wait of the others is bounded.
        cluster_arrive(); cluster_wait();                              // nobody issues anything more
        if (threadIdx.x == 0) {                                        // what was issued lands: rows of other CTAs, tiles
            (void)mbar_wait(bar(SH_RX), 0);
            if (!empty) { (void)mbar_wait(bar(SH_QK), 0); (void)mbar_wait(bar(SH_V), 0); }
        } else if (threadIdx.x == 288) {                               // the thread that issued the MMAs
            tc_commit(bar(SH_DRAIN));
            (void)mbar_wait(bar(SH_DRAIN), 0);
        }
        cluster_arrive(); cluster_wait();                              // ... in every CTA, so that what went out of this one has been read
    }
    span_end(p.span);
    if (warp == 8) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
    }
}

// ---- host side ----------------------------------------------------------------------------------
// Row chunks.  Pass 1 cuts the R window rows into n_chunks pieces of chunk_rows <= 128 (its MMA M
// dimension).  Pass 2 takes the rows whole when R <= 128 and in pieces of 64 otherwise; rows_out is
// the padded row count of the combined arrays it reads.
struct TcChunks { int n_chunks, chunk_rows, rows_out; };
TcChunks tc_chunks(int R) {
    TcChunks c;
    c.n_chunks = (R + 127) / 128;
    c.chunk_rows = ((R + c.n_chunks - 1) / c.n_chunks + 15) / 16 * 16;
    c.rows_out = c.n_chunks > 1 ? (R + MC_ROWS - 1) / MC_ROWS * MC_ROWS : c.chunk_rows;
    return c;
}

size_t l2_bytes() {
    static size_t n = 0;
    if (!n) {
        int dev = 0, v = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&v, cudaDevAttrL2CacheSize, dev) != cudaSuccess || v <= 0) v = 126 << 20;
        n = (size_t)v;
    }
    return n;
}

}  // namespace

// Fewer than 64 window rows fill half of the MMA's M dimension at most.  Pass 1 then runs every row twice, the second
// copy with the low part of P, and pass 2 takes -2 O as two parts on its N dimension, so that such a call keeps the 32-bit
// sums of the CUDA-core kernels at the tensor cores' rate (32 heads x 8191 tokens x 32 rows: one score call 489 us on CUDA cores, 63 us here, of which K and V twice
// through HBM are 41; 8 heads x 2547 tokens x 32 rows: 87 against 26 us).
static bool tc_hilo(const ScoreShape& s) { return s.R < 64; }

bool tc_supported(const ScoreShape& s, int dtype, const TensorView& q) {
    if (dtype != OBC_BF16) return false;
    // the window rows of a KV head's group must be one uniformly strided run of rows
    return q.sh == (long long)s.W * q.st && q.sb == (long long)s.Hq * q.sh;
}

// Multi-chunk pass 2: with fewer tile pairs than about two per SM (a short cache scored over a long window) the row chunks
// of a pair may be shared by several CTAs (see ItemWalk): as many as an equal share of the items allows, where at least half
// of all (pair, chunk) items are visible.  With more pairs whole ones balance well enough and no partial scores have to be
// added up.
static int tc_chunk_split(const ScoreShape& s, const TcChunks& ch) {
    if (ch.n_chunks <= 1) return 1;
    const long long pairs = (long long)s.B * s.Hkv * (((s.Nmax + TILE - 1) / TILE + 1) / 2);
    if (pairs >= 2LL * sm_count()) return 1;
    const int nc = ch.rows_out / MC_ROWS;
    const int run = (int)(pairs * nc / (2 * sm_count())), c = (nc + run) / (run > 1 ? run : 1) + 1;
    return c < 2 ? 2 : c > 32 ? 32 : c > nc ? nc : c;
}

// Pass 1 takes the row chunks of a unit two by two (tc_pass1_kernel, PAIR) where the pairs alone give every SM a CTA and
// the cache is longer than ten tiles.  Whole-sequence windows of 8 KV heads x 4 heads, chunks / pairs: 1100 queries (144
// pairs) 31 / 35 us, 1300 (168) 42 / 39, 2048 68 / 57, 3001 126 / 120, 4096 188 / 174; 2 x 4 x 4096 (128 pairs) 49 / 79; 8 x 4 x 1024
// (eight tiles) 26.5 / 28.2.  With several splits per pair (few rows, a long cache) the gain in pass 1 (56691 to 93869 tokens: from 10 %
// faster to 16 % slower) went to the merge of twice as many partial results.
static bool p1_pairs(const ScoreShape& s, const TcChunks& ch) {
    return ch.n_chunks > 1 && (long long)s.B * s.Hkv * ((ch.n_chunks + 1) / 2) >= sm_count() && s.Nmax > 10 * TILE;
}

// Workspace plan of the tensor-core path: the SIMT plan's layout with splits counted in 128-token tiles.
static SimtPlan make_tc_plan(const ScoreShape& s) {
    const TcChunks ch = tc_chunks(s.R);
    const int units = s.B * s.Hkv, vus = units * ch.n_chunks;
    const int tiles = (s.Nmax + TILE - 1) / TILE;
    int n = sm_count() / vus;                          // one wave of CTAs when the sequences are equal
    // (48 tiles per CTA: with 32 the ragged batch of 8 spent 6 % more in pass 1 on prologues and tails, with 64 the last wave ran half empty)
    if (s.seq_lens) { const int cap = (tiles + 47) / 48; if (cap > n) n = cap; }   // ragged: bound the work per CTA
    if (n < 1) n = 1;
    if (n > tiles) n = tiles;
    SimtPlan p{};
    p.tiles_per_split = (tiles + n - 1) / n;                                   // per pass-1 CTA
    p.n_splits = (tiles + p.tiles_per_split - 1) / p.tiles_per_split;          // CTAs, and partial results, per unit
    p.tile_tokens = TILE;
    p.rows_out = ch.rows_out;
    p.want_obf = tc_hilo(s) ? 2 : 1;
    const size_t rows = (size_t)units * s.R, prow = rows * p.n_splits, orow = (size_t)units * ch.rows_out;
    size_t off = 0;
    p.off_flag = off;   off = 256;
    p.off_part_m = off; off = align_up(off + prow * 4, 256);
    p.off_part_l = off; off = align_up(off + prow * 4, 256);
    p.off_part_o = off; off = align_up(off + prow * kD * 4, 256);
    p.off_lse2 = off;   off = align_up(off + orow * 4, 256);
    p.off_onorm = off;  off = align_up(off + orow * 4, 256);
    p.off_o = off;      off = align_up(off + orow * kD * 4, 256);
    p.off_obf = off;    off = align_up(off + orow * kD * 2 * p.want_obf, 1024);
    p.off_cpair = off;  off = align_up(off + orow * 8, 256);
    p.off_nv = off;     off = align_up(off + (size_t)units * s.Nmax * 4, 256);
    p.bytes = off;
    return p;
}

// the partial score planes of a shared multi-chunk pass 2 follow the plan's arrays
static size_t tc_partial_bytes(const ScoreShape& s) {
    const int cs = tc_chunk_split(s, tc_chunks(s.R));
    const size_t units = (size_t)s.B * s.Hkv;
    return cs > 1 ? (size_t)(cs - 1) * s.n_planes * units * s.Nmax * 4 + units * ((s.Nmax + 2 * TILE - 1) / (2 * TILE)) * 4 : 0;
}

size_t tc_workspace_bytes(const ScoreShape& s) { return make_tc_plan(s).bytes + tc_partial_bytes(s); }

// How many clusters of 2, 4, 8 or 16 CTAs of tc_short_kernel the current device runs at once, asked once per host thread and device (the first
// kDevices of them); a query that fails is not remembered
static int short_clusters(int C) {
    if (C == 1) return sm_count();
    constexpr int kDevices = 16;
    thread_local struct { bool known; int n; } seen[kDevices][4] = {};
    int dev = -1, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    const int at = C == 2 ? 0 : C == 4 ? 1 : C == 8 ? 2 : 3;
    if (dev < kDevices && seen[dev][at].known) return seen[dev][at].n;
    const auto kernel = tc_short_kernel<OBC_VAR_VK, false, false>;                 // (one CTA per SM, whatever the instantiation)
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)C; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)C); cfg.blockDim = dim3(kThreadsShort); cfg.attrs = attr; cfg.numAttrs = 1; cfg.dynamicSmemBytes = kSmemShort;
    if (allow_smem(kernel, kSmemShort, true) != cudaSuccess || cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) {
        (void)cudaGetLastError();
        return 0;
    }
    if (dev < kDevices) seen[dev][at] = {true, n};
    return n;
}
// Cluster size for a call that one kernel serves (tc_short_kernel), or 0: up to 128 window rows, a tile per CTA, all units side by side.
// With a second wave of clusters three kernels are the faster ones, us three / one: 8 heads of 2048 x 32 rows 17.2 / 22.9, x 128 rows 19.0 / 27.4, 16 of
// 1024 x 16 rows 17.1 / 19.1, x 128 rows 18.5 / 26.5, 30 of 1000 x 64 rows 20.0 / 22.3, 34 of 512 x 32 rows 18.4 / 19.3, 148 of 256 x 64 rows 21.9 / 24.5
// (of single CTAs not always, 149 of 128 x 32 rows 29.3 / 20.4, 160 of 100 x 128 rows 30.6 / 36.8: no line was measured there).
// Within one wave the CTAs without a tile that a power of two leaves do not cost what they look like: 1100 tokens (9 tiles of 16 CTAs) x 16 rows, one head 14.7 / 10.8,
// 7 heads 16.1 / 11.2, x 128 rows 18.1 / 14.0; 600 (5 of 8) x 128 rows, 14 heads 17.7 / 13.9.
// Each CTA merges its share of the rows (0.08 us per row), so where the chip has room the cluster has more CTAs than tiles, until a share is
// 32 rows at most: one head of 128 tokens x 128 rows 14.3 us by three kernels, 17.8 with one CTA, 14.5 with two, 12.9 with four; of 256 tokens 14.7, 15.0
// with two, 12.9 with four; 74 heads of 128 tokens x 128 rows 17.3, 18.2, 15.3 with two.  Where each unit has one CTA all the same, three kernels
// are faster for few units and many rows (their time grows by 0.045 us per unit): 90 heads of 128 tokens x 128 rows 17.9 / 18.4 us, 110 19.0 / 18.5; x 112
// rows 74 17.1 / 17.3, 90 17.7 / 17.4; x 96 rows 90 17.1 / 16.0.
static int short_cluster_size(const ScoreShape& s, const TcChunks& ch) {
    const int tiles = (s.Nmax + TILE - 1) / TILE, units = s.B * s.Hkv;
    if (ch.n_chunks > 1 || tiles > SH_MAXC) return 0;
    int C = 1;
    while (C < tiles) C *= 2;
    if (units > short_clusters(C)) return 0;
    while (C < SH_MAXC && s.R > 32 * C && units <= short_clusters(2 * C)) C *= 2;
    return C == 1 && s.R > 32 && s.R > units + 28 ? 0 : C;
}

obc_status launch_attention_tc(const ScoreShape& s, TensorView q, TensorView k, TensorView v, void* ws, cudaStream_t stream,
                               SimtPlan* plan_out) {
    return launch_score_tc(s, q, k, v, nullptr, ws, stream, nullptr, plan_out);
}

obc_status launch_score_tc(const ScoreShape& s, TensorView q, TensorView k, TensorView v,
                           float* scores, void* ws, cudaStream_t stream, const GivenAttention* given,
                           SimtPlan* attention_only) {
    const TcChunks ch = tc_chunks(s.R);
    const SimtPlan plan = make_tc_plan(s);
    char* wsb = (char*)ws;
    const int units = s.B * s.Hkv;
    const bool hilo = tc_hilo(s);
    const int short_c = given || attention_only ? 0 : short_cluster_size(s, ch);
    CUtensorMap mq, mo, mk, mv;
    {
        const uint64_t qd[2] = {(uint64_t)kD, (uint64_t)s.B * s.Hq * s.W};
        const uint64_t qs[1] = {(uint64_t)q.st * 2};
        const uint64_t od[2] = {(uint64_t)kD, (uint64_t)units * ch.rows_out * plan.want_obf};
        const uint64_t os[1] = {(uint64_t)kD * 2};
        const uint64_t kd[4] = {(uint64_t)kD, (uint64_t)s.Nmax, (uint64_t)s.Hkv, (uint64_t)s.B};
        const uint64_t ks[3] = {(uint64_t)k.st * 2, (uint64_t)(s.Hkv > 1 ? k.sh : k.st * s.Nmax) * 2,
                                (uint64_t)(s.B > 1 ? k.sb : (s.Hkv > 1 ? k.sh * s.Hkv : k.st * s.Nmax)) * 2};
        const uint64_t vs[3] = {(uint64_t)v.st * 2, (uint64_t)(s.Hkv > 1 ? v.sh : v.st * s.Nmax) * 2,
                                (uint64_t)(s.B > 1 ? v.sb : (s.Hkv > 1 ? v.sh * s.Hkv : v.st * s.Nmax)) * 2};
        if ((!short_c && (!make_map(&mq, q.ptr, 2, qd, qs, (uint32_t)ch.chunk_rows) ||
                          !make_map(&mo, wsb + plan.off_obf, 2, od, os, (uint32_t)(ch.chunk_rows * plan.want_obf)))) ||
            !make_map(&mk, k.ptr, 4, kd, ks, TILE) || !make_map(&mv, v.ptr, 4, kd, vs, TILE)) {
            set_last_cuda_error((int)cudaErrorInvalidValue);
            return OBC_ERR_CUDA;
        }
    }
    // A cache that cannot hold K and V from pass 1 to pass 2 is better streamed through: with the "evict
    // first" hint on the K/V copies pass 1 ran 2 us faster on the 32k Llama layer (134 MB against 126 MB of L2).
    // Smaller caches keep the default policy, so that pass 2 finds in L2 what pass 1 read.
    const bool l2_stream = ch.n_chunks == 1 && !given &&
        (double)units * s.Nmax * kD * 2 * 2 > 0.75 * (double)l2_bytes();
    if (short_c) {
        // everything in one kernel (below)
    } else if (given) {   // the caller's O and LSE take the place of pass 1 + combine; pass 2 computes the value norms itself
        obc_status st = launch_given_prep(s, plan, *given, ws, stream);
        if (st != OBC_OK) return st;
    } else {       // pass 1 + combine
        const bool pairs = p1_pairs(s, ch);
        P1Params p1{};
        p1.B = s.B; p1.Hq = s.Hq; p1.Hkv = s.Hkv; p1.G = s.G; p1.W = s.W; p1.R = s.R; p1.Nmax = s.Nmax;
        p1.seq_lens = s.seq_lens; p1.mask_lens = s.mask_lens; p1.scale = s.scale; p1.causal = s.causal;
        p1.n_chunks = ch.n_chunks; p1.chunk_rows = ch.chunk_rows;
        p1.head_chunks = s.causal && ch.n_chunks > 1 ? s.W / (pairs ? 2 * ch.chunk_rows : ch.chunk_rows) : 0;
        p1.n_splits = plan.n_splits; p1.tiles_per_split = plan.tiles_per_split;
        p1.l2_stream = l2_stream ? 1 : 0;
        p1.part_m = (float*)(wsb + plan.off_part_m); p1.part_l = (float*)(wsb + plan.off_part_l);
        p1.part_o = (float*)(wsb + plan.off_part_o);
        // only the single-chunk pass 2 without the l1 plane reads the norms that pass 1 leaves
        const bool want_nv = ch.n_chunks == 1 && !attention_only && !(s.variants & OBC_VAR_VATP);
        p1.nv = want_nv ? (float*)(wsb + plan.off_nv) : nullptr;
        p1.status = (unsigned int*)(wsb + plan.off_flag);
        p1.span = (unsigned long long*)(wsb + plan.off_flag + kSpanOffset);
        // with one CTA per (unit, row chunk) there is nothing to merge: pass 1 writes the results itself
        const bool direct = plan.n_splits == 1;
        if (direct) {
            p1.rows_out = plan.rows_out;
            p1.out_o = (float*)(wsb + plan.off_o); p1.out_obf = (__nv_bfloat16*)(wsb + plan.off_obf);
            p1.out_lse2 = (float*)(wsb + plan.off_lse2); p1.out_onorm = (float*)(wsb + plan.off_onorm);
            p1.out_cpair = (float*)(wsb + plan.off_cpair);
        }
        const auto pass1 = hilo ? tc_pass1_kernel<true, false> : pairs ? tc_pass1_kernel<false, true> : tc_pass1_kernel<false, false>;
        OBC_CUDA_TRY(allow_smem(pass1, kSmemP1));
        { ProfScope ps("tc_pass1", stream);
          OBC_CUDA_TRY(launch_pdl(pass1, dim3(plan.n_splits, units * (pairs ? (ch.n_chunks + 1) / 2 : ch.n_chunks)), dim3(kThreadsP1), kSmemP1, stream, 1, mq, mk, mv, p1)); }
        if (!direct) {
            obc_status st = launch_combine(s, plan, ws, stream);
            if (st != OBC_OK) return st;
        }
    }
    if (attention_only) { *attention_only = plan; return OBC_OK; }      // the workspace holds the window attention
    TcParams p{};
    p.B = s.B; p.Hkv = s.Hkv; p.G = s.G; p.W = s.W; p.R = s.R; p.Nmax = s.Nmax; p.seq_lens = s.seq_lens; p.mask_lens = s.mask_lens;
    p.scale = s.scale; p.causal = s.causal; p.variants = s.variants;
    p.n_chunks = ch.n_chunks; p.chunk_rows = ch.chunk_rows; p.rows_out = ch.rows_out;
    p.lse2 = (const float*)(wsb + plan.off_lse2);
    p.onorm = (const float*)(wsb + plan.off_onorm);
    p.scores = scores;
    p.status = (unsigned int*)(wsb + plan.off_flag);
    p.span = (unsigned long long*)(wsb + plan.off_flag + kSpanOffset) + 2;
    p.cpair = (const float4*)(wsb + plan.off_cpair);
    p.nv = (const float*)(wsb + plan.off_nv);
    p.l2_stream = l2_stream ? 1 : 0;
    p.csplit = 1; p.partial = nullptr;
    const long long n_tiles = (long long)units * ((s.Nmax + TILE - 1) / TILE);
    const int grid = (int)(n_tiles < sm_count() ? n_tiles : sm_count());

    // the queries of pass 2, by unit where its rows do not fill their last chunk (see load_q)
    const bool by_unit = s.R % (ch.n_chunks > 1 ? MC_ROWS : ch.chunk_rows) != 0;
    auto map_queries = [&](CUtensorMap* m, int rows) {
        const uint64_t rows_of_all[2] = {(uint64_t)kD, (uint64_t)units * s.R}, per_unit[3] = {(uint64_t)kD, (uint64_t)s.R, (uint64_t)units};
        const uint64_t strides[2] = {(uint64_t)q.st * 2, (uint64_t)s.R * q.st * 2};
        return make_map(m, q.ptr, by_unit ? 3 : 2, by_unit ? per_unit : rows_of_all, strides, (uint32_t)rows);
    };
    auto flag = [](bool f, auto g) { return f ? g(std::true_type{}) : g(std::false_type{}); };
    if (short_c) {
        CUtensorMap ms;
        if (!map_queries(&ms, ch.chunk_rows)) { set_last_cuda_error((int)cudaErrorInvalidValue); return OBC_ERR_CUDA; }
        auto launch_short = [&](auto kernel) -> obc_status {
            OBC_CUDA_TRY(allow_smem(kernel, kSmemShort, short_c > 8));
            ProfScope ps("tc_short", stream);
            OBC_CUDA_TRY(launch_pdl(kernel, dim3(units * short_c), dim3(kThreadsShort), kSmemShort, stream, short_c, ms, mk, mv, p, short_c));
            return OBC_OK;
        };
        return flag(hilo, [&](auto hl) { return flag(by_unit, [&](auto bu) {
            if (s.variants == OBC_VAR_VK) return launch_short(tc_short_kernel<OBC_VAR_VK, hl.value, bu.value>);
            if (!(s.variants & ~kObcVariants)) return launch_short(tc_short_kernel<kObcVariants, hl.value, bu.value>);
            return launch_short(tc_short_kernel<kAllVariants, hl.value, bu.value>);
        }); });
    }
    if (ch.n_chunks > 1) {                               // more than 128 window rows: chunks of 64, K/V tile kept
        CUtensorMap mq64, mo64;
        const uint64_t od[2] = {(uint64_t)kD, (uint64_t)units * ch.rows_out};
        const uint64_t os[1] = {(uint64_t)kD * 2};
        if (!map_queries(&mq64, MC_ROWS) || !make_map(&mo64, wsb + plan.off_obf, 2, od, os, MC_ROWS)) {
            set_last_cuda_error((int)cudaErrorInvalidValue);
            return OBC_ERR_CUDA;
        }
        p.n_chunks = ch.rows_out / MC_ROWS; p.chunk_rows = MC_ROWS;
        p.csplit = tc_chunk_split(s, ch);
        p.partial = (float*)(wsb + plan.bytes);
        const int pairs = (s.Nmax + 2 * TILE - 1) / (2 * TILE);
        p.max_pairs = pairs;
        p.copies = (int*)(p.partial + (size_t)(p.csplit - 1) * s.n_planes * units * s.Nmax);
        const long long positions = (long long)units * pairs * (p.csplit > 1 ? p.n_chunks : 1);
        const int mgrid = (int)(positions < sm_count() ? positions : sm_count());
        auto launch_multi = [&](auto kernel) -> obc_status {
            OBC_CUDA_TRY(allow_smem(kernel, kSmemMulti));
            { ProfScope ps("tc_pass2", stream); OBC_CUDA_TRY(launch_pdl(kernel, dim3(mgrid), dim3(kThreadsMulti), kSmemMulti, stream, 1, mq64, mo64, mk, mv, p)); }
            if (p.csplit > 1) {
                ProfScope ps("partial_sum", stream);
                OBC_CUDA_TRY(launch_pdl(tc_partial_sum_kernel, dim3(pairs, units), dim3(2 * TILE), 0, stream, 1, p, s.n_planes));
            }
            return OBC_OK;
        };
        const bool split = p.csplit > 1 || (s.causal && s.W > MC_ROWS);
        return flag(split, [&](auto sp) { return flag(by_unit, [&](auto bu) {
            if (s.variants == OBC_VAR_VK) return launch_multi(tc_pass2_multi_kernel<OBC_VAR_VK, sp.value, bu.value>);
            if (!(s.variants & ~kObcVariants)) return launch_multi(tc_pass2_multi_kernel<kObcVariants, sp.value, bu.value>);
            return launch_multi(tc_pass2_multi_kernel<kAllVariants, sp.value, bu.value>);
        }); });
    }

    auto launch = [&](auto kernel) -> obc_status {
        OBC_CUDA_TRY(allow_smem(kernel, kSmemBytes));
        { ProfScope ps("tc_pass2", stream); OBC_CUDA_TRY(launch_pdl(kernel, dim3(grid), dim3(kThreads), kSmemBytes, stream, 1, mq, mo, mk, mv, p)); }
        return OBC_OK;
    };
    // pass 1 leaves only ||v||^2; without it, and for the l1 variant, the norms come from the V tiles in pass 2
    const bool own_nv = given || (s.variants & OBC_VAR_VATP);
    if (by_unit && !map_queries(&mq, ch.chunk_rows)) { set_last_cuda_error((int)cudaErrorInvalidValue); return OBC_ERR_CUDA; }
    return flag(own_nv, [&](auto own) { return flag(hilo, [&](auto hl) { return flag(by_unit, [&](auto bu) {
        if (s.variants == OBC_VAR_VK) return launch(tc_pass2_kernel<OBC_VAR_VK, own.value, hl.value, bu.value>);
        if (!(s.variants & ~kObcVariants)) return launch(tc_pass2_kernel<kObcVariants, own.value, hl.value, bu.value>);
        return launch(tc_pass2_kernel<own.value ? kAllVariants : kAllVariants & ~OBC_VAR_VATP, own.value, hl.value, bu.value>);
    }); }); });
}

}  // namespace obc
