// Batched-serving head (33 to 256 hidden rows; which of 33 to 64 see head_stream_takes): the projection is a real dense contraction
// and runs on the 5th-generation tensor cores (Algorithm 2, the drafter-forward and index-mapping steps, with many sequences and
// tree nodes drafted at once).
//
//   D[b, j] = sum_i h[b, i] * W_trim[j, i]      M = hidden rows (the TMEM lanes), N = vocabulary rows
//                                               of a tile (TMEM columns), K-loop over d in 64-column steps
//
// B <= 128: one persistent CTA per SM walks vocabulary tiles (M = 128, tcgen05.mma.cta_group::1).
// B  > 128: the two CTAs of a cluster act as one MMA of M = 256 (cta_group::2).  Each CTA stages its
// own 128 hidden rows and HALF of the tile's vocabulary rows; the tensor cores of both SMs read the
// two halves of the B operand from both shared memories.  Per SM and flop this halves the operand
// bytes staged and read compared with two M tiles in one CTA, which is what bounded that form.
//
// Warp 0 feeds a shared-memory ring with TMA tensor copies (128-byte swizzle, every CTA fetches its own tiles); in a pair
// both CTAs' copies count their bytes on the leader's barrier.  A ring stage holds one or two 64-column steps of d
// (two where three such stages fit): the two threads that drive the ring wait and release once per stage, and their
// turn-around is on its critical path, so they also move their cursors by additions only.  One thread of warp 1 (of the leader)
// issues the MMAs (bf16 x bf16 -> fp32) with the operands described in place by shared-memory
// descriptors and the accumulators in tensor memory: two accumulator stages of up to 256 columns, so
// the epilogue of tile t overlaps the MMAs of tile t+1.  tcgen05.commit releases ring stages and
// publishes accumulators (to both CTAs of a pair).  Eight epilogue warps read the accumulators back
// with tcgen05.ld -- TMEM lane = hidden row; the two warps of a lane quadrant take one half of a tile's
// columns each (up to 64 rows a wide tile is computed in two halves, on lanes of their own) -- 16 columns at a time: running max /
// sum-exp of z = logit / T_b, Gumbel-max candidate from the caller's uniforms, and a sorted top-k list kept in registers.
// Logits never go to HBM.  The column shares of a row are merged through shared memory (a pair's two shares leave a record
// each); per CTA and hidden row one record goes to scratch; a second small kernel (six warps per hidden row) merges the
// records, applies the index mapper and writes the outputs.  Every wait is bounded; on expiry the CTA raises
// VT_FLAG_TIMEOUT and leaves after releasing its tensor memory.
//
// What bounds it: W_trim and the uniforms stream in at 6 TB/s while MMAs and all but the last tile's epilogue run; then the last
// epilogue and the merge are exposed, while HBM idles.  So that epilogue is kept short: the Gumbel noise of the last
// tile is made while its MMAs run, and over a CTA's only tile the top-k list is found by sorting networks.  The epilogue issues
// at half the schedulers' rate at most (two warps on each, selects and minima at half rate).  us per chained step before
// any of this / now (the merge's share included): 40 rows of 20001 x 3072 41.3 / 31.9, 64 rows 42.7 / 33.5, 100 rows 46.2 / 34.8,
// 90 rows of 10000 x 4096 with top-10 43.7 / 27.2, 256 rows of 32768 x 4096 74.5 / 72.2.
#include <cfloat>
#include <cmath>

#include "vt_common.cuh"
#include "vt_head_common.cuh"
#include "vt_tc.cuh"
#include "vt_tree_common.cuh"

namespace vt {

namespace {

constexpr int kBM = 128;                  // hidden rows per CTA (TMEM lanes)
constexpr int kMaxBN = 256;               // vocabulary rows per tile at most (TMEM columns per accumulator)
constexpr int kMaxSub = 2;                // d-steps of kBK columns one ring stage holds at most
constexpr int kMaxStages = 8;
constexpr int kCh = 16;                   // accumulator columns per epilogue step (keeps the row state in registers)
constexpr int kParts = 2;                  // epilogue warps per TMEM lane quadrant
constexpr int kTmemCols = 512;            // 2 accumulator stages x kMaxBN columns
constexpr int kMaxTopk = 16;              // the list's values live in registers
constexpr unsigned long long kWaitLimitNs = 2000000000ull;
constexpr size_t kSmemBudget = 225 * 1024;   // ring and candidate entries at most (227 KB per CTA less alignment slack and statics)
// What of it a pair leaves to L1 where the uniforms come one by one (K no multiple of four, or an unaligned pointer).  Sixteen loads then
// share the 256 lines of the eight epilogue warps, 32 KB; beside more than 196 KB of shared memory L1 has 28 KB, and 60 beside this.
// Over a long d a single narrow tile has its noise made behind its MMAs, and the shorter ring costs more than that (us per call, 28 / 60
// KB: 256 rows of 33001 x 2048 69.3 / 49.5, of 16573 x 1536 41.6 / 28.8, of 9109 x 3072 30.9 / 28.8, of 18941 x 4096 54.9 / 50.4; of 4735 x
// 4096 24.9 / 27.5, of 11801 x 4096 36.4 / 37.6; up to 128 rows no difference).
constexpr size_t kL1Room = 32 * 1024;

// Phase stamps (-DVT_STAMPS builds only): one thread per role writes %globaltimer into a region behind the
// records; bench.py --case stamps reads them back.  Slots per CTA: 0 entry, 1 set up (barriers, tensor
// memory), 2 producer released by the launch dependency, 3 first stage landed (MMA issuer), 4 / 5 MMAs of the
// CTA's first / last tile issued, 6 / 7 accumulators of the first / last tile complete (epilogue warp 0),
// 8 / 9 first / last tile's epilogue done, 10 record written, 11 leaving; CTA 0 also carries the merge
// kernel's 12 start (records complete) and 13 end for hidden row 0.
#ifdef VT_STAMPS
#define VT_DSTAMP(slot) do { stamps[(size_t)blockIdx.x * kStampSlots + (slot)] = global_ns(); } while (0)
#else
#define VT_DSTAMP(slot) do {} while (0)
#endif

// ---- PTX wrappers ----------------------------------------------------------------------------------
__device__ __forceinline__ bool mbar_wait(uint64_t* b, uint32_t parity, volatile int* abort_flag) {
    if (mbar_try(b, parity)) return true;
    const unsigned long long t0 = global_ns();
    for (;;) {
#pragma unroll 1
        for (int i = 0; i < 128; ++i)
            if (mbar_try(b, parity)) return true;
        if (*abort_flag) return false;
        if (global_ns() - t0 > kWaitLimitNs) { *abort_flag = 1; return false; }
    }
}
// Same, called by all 32 lanes of a warp that expects to wait long (a whole tile of MMAs): lane 0
// polls with pauses -- 256 spinning threads cost issue slots and power the tensor pipe wants -- then
// every lane observes the completed phase itself.  The outcome is voted on so the lanes never part
// ways before a warp-collective instruction.
__device__ __forceinline__ bool mbar_wait_warp(uint64_t* b, uint32_t parity, volatile int* abort_flag) {
    bool ok = true;
    if ((threadIdx.x & 31) == 0 && !mbar_try(b, parity)) {
        const unsigned long long t0 = global_ns();
        for (;;) {
            __nanosleep(128);
            if (mbar_try(b, parity)) break;
            if (*abort_flag) { ok = false; break; }
            if (global_ns() - t0 > kWaitLimitNs) { *abort_flag = 1; ok = false; break; }
        }
    }
    ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
    if (ok) ok = mbar_try(b, parity) || mbar_wait(b, parity, abort_flag);
    return __all_sync(0xffffffffu, ok);
}
// 16 consecutive columns of this thread's TMEM lane.  (The wait sits in the same statement: nothing that uses the values can be
// moved in front of it.)
__device__ __forceinline__ void tc_ld16(uint32_t taddr, float (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=&f"(r[0]), "=&f"(r[1]), "=&f"(r[2]), "=&f"(r[3]), "=&f"(r[4]), "=&f"(r[5]), "=&f"(r[6]), "=&f"(r[7]), "=&f"(r[8]),
          "=&f"(r[9]), "=&f"(r[10]), "=&f"(r[11]), "=&f"(r[12]), "=&f"(r[13]), "=&f"(r[14]), "=&f"(r[15])
        : "r"(taddr) : "memory");
}
// 16 consecutive columns written; complete when it returns
__device__ __forceinline__ void tc_st16(uint32_t taddr, const float (&r)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%16], {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15};\n\t"
        "tcgen05.wait::st.sync.aligned;"
        ::"f"(r[0]), "f"(r[1]), "f"(r[2]), "f"(r[3]), "f"(r[4]), "f"(r[5]), "f"(r[6]), "f"(r[7]), "f"(r[8]), "f"(r[9]), "f"(r[10]),
          "f"(r[11]), "f"(r[12]), "f"(r[13]), "f"(r[14]), "f"(r[15]), "r"(taddr) : "memory");
}

// ---- CTA-pair forms (cta_group::2): two CTAs of a cluster act as one 256-row MMA ---------------------
__device__ __forceinline__ uint32_t cluster_ctarank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// shared::cluster address of the same variable in CTA `rank` of this cluster
__device__ __forceinline__ uint32_t mapa_u32(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_addr) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
// tensor copy into THIS CTA's shared memory whose bytes are counted on a barrier of either CTA of the pair
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* tm, int x, int y, uint32_t bar_cluster) {
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
        ::"r"(dst), "l"(tm), "r"(bar_cluster), "r"(x), "r"(y) : "memory");
}
// arrives on the barrier at this shared-memory offset in both CTAs once the MMAs issued so far are done:
// one commit per CTA of the pair (the peer's barrier by its shared::cluster address)
__device__ __forceinline__ void tc_commit_pair(uint64_t* bar) {
    const uint32_t own = smem_u32(bar);
    const uint32_t peer = mapa_u32(own, 1);
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(own) : "memory");
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(peer) : "memory");
}
// D[tmem of both CTAs] (+)= A * B^T, 256 x N x 16: each CTA supplies 128 rows of A and N/2 rows of B
__device__ __forceinline__ void tc_mma_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t acc) {
    const uint32_t z = 0;
    asm volatile(
        "{ .reg .pred p; setp.ne.b32 p, %4, 0;"
        " tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, {%5, %5, %5, %5, %5, %5, %5, %5}, p; }"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(acc), "r"(z) : "memory");
}

struct DenseGeo {
    int n_tiles;      // vocabulary tiles of bn rows
    int n_kc;         // ring steps per tile: ceil(d / kBK)
    int bn;           // vocabulary rows per tile (per CTA pair when paired); a multiple of 16, <= kMaxBN
    int n_stages;     // ring depth
    int stage_bytes;  // bytes one CTA stages per step: hidden rows + its share of the vocabulary rows
    int n_groups;     // CTAs (or CTA pairs) walking the tiles round-robin
    int h_rows;       // hidden rows a copy brings (the rest of the MMA's 128 is whatever lies there: lanes nobody looks at)
    int h_bytes;      // shared memory of a step's hidden rows (a multiple of 1024); its vocabulary rows lie behind them
    int ring_bytes;
    int bn0;          // SPLIT: columns of a tile's first half (a multiple of 16, <= kHalfCols; the second has no more)
    int tail_bytes;   // behind the ring, for operand rows that the last stage's MMAs read beyond it
    int sub;          // d-steps per ring stage (1 or 2): one wait and one release per stage, so two steps per stage halve
                      // what the two single threads that drive the ring spend per MMA; taken when three such stages fit
};

// Rows of uniforms that 16-byte loads can read.
__host__ __device__ __forceinline__ bool uniforms_aligned(const float* u, int K) {
    return (K & 3) == 0 && (reinterpret_cast<uintptr_t>(u) & 15) == 0;
}

// Per-thread state of one hidden row over the columns the thread has seen.
template <int KT>
struct RowState {
    float m, s;               // running max and sum of exp(z - m)
    float gb_s, gb_z;         // best Gumbel score and its z
    int gb_j;
    float tv[KT];             // top-k list at the END of the arrays (slots KT-topk .. KT-1, descending)
    int tj[KT];               // behind +inf sentinels: the insertion threshold is always slot KT-1; -1: no entry
};

// Insert (cv, cj) into the sorted list with selects only; equal values keep the entry already there.
template <int KT>
__device__ __forceinline__ void list_insert(float (&tv)[KT], int (&tj)[KT], float cv, int cj) {
    bool gt[KT];
#pragma unroll
    for (int p = 0; p < KT; ++p) gt[p] = cv > tv[p];
#pragma unroll
    for (int p = KT - 1; p >= 1; --p) {
        tv[p] = gt[p] ? (gt[p - 1] ? tv[p - 1] : cv) : tv[p];
        tj[p] = gt[p] ? (gt[p - 1] ? tj[p - 1] : cj) : tj[p];
    }
    tv[0] = gt[0] ? cv : tv[0];
    tj[0] = gt[0] ? cj : tj[0];
}

// ---- sorting networks (descending, everything in registers) ------------------------------------------
__device__ __forceinline__ void order2(float& a, float& b) {
    const float hi = fmaxf(a, b), lo = fminf(a, b);
    a = hi;
    b = lo;
}
__device__ __forceinline__ void order2(unsigned long long& a, unsigned long long& b) {
    const bool sw = b > a;
    const unsigned long long hi = sw ? b : a, lo = sw ? a : b;
    a = hi;
    b = lo;
}
__device__ __forceinline__ float larger(float a, float b) { return fmaxf(a, b); }
__device__ __forceinline__ unsigned long long larger(unsigned long long a, unsigned long long b) { return b > a ? b : a; }
// Batcher's odd-even merge sort of v[O .. O + N), N a power of two (the indices are template arguments: they have to be constants)
template <int O, int N, int R, class T, int A>
__device__ __forceinline__ void odd_even_merge(T (&v)[A]) {
    if constexpr (2 * R < N) {
        odd_even_merge<O, N, 2 * R>(v);
        odd_even_merge<O + R, N, 2 * R>(v);
#pragma unroll
        for (int i = O + R; i + R < O + N; i += 2 * R) order2(v[i], v[i + R]);
    } else {
        order2(v[O], v[O + R]);
    }
}
template <int O, int N, class T, int A>
__device__ __forceinline__ void sort_desc(T (&v)[A]) {
    if constexpr (N > 1) {
        sort_desc<O, N / 2>(v);
        sort_desc<O + N / 2, N / 2>(v);
        odd_even_merge<O, N, 1>(v);
    }
}
// list <- the N largest of list and v[O .. O + N), both descending: the larger ones of opposite ends are those, in bitonic
// order, which half-cleaners sort
template <int O, int N, class T, int A>
__device__ __forceinline__ void merge_desc(T (&list)[N], const T (&v)[A]) {
#pragma unroll
    for (int i = 0; i < N; ++i) list[i] = larger(list[i], v[O + N - 1 - i]);
#pragma unroll
    for (int k = N / 2; k >= 1; k >>= 1)
#pragma unroll
        for (int i = 0; i < N; ++i)
            if ((i & k) == 0) order2(list[i], list[i + k]);
}

// KT: capacity of the list (8 or kMaxTopk).  PAIR: two CTAs of a cluster form one MMA.  Two epilogue warps per TMEM lane
// quadrant, each with a contiguous share of the quadrant's 16-column chunks.  Warps whose lanes hold no hidden row leave at once.
// SPLIT (up to 64 hidden rows, tiles of kSplitCols columns and more): an MMA's first 64 rows are the hidden rows and its second 64 nobody's, and a quadrant's warps sit on
// one scheduler, so half of them would do the whole epilogue.  So a tile's columns are computed in two halves: one with the
// hidden rows as rows 0-63, the other with the operand's start 64 rows earlier, which makes them rows 64-127; each half
// of the lanes then has half of the columns (in TMEM kHalfCols apart) and all eight warps work.  (40 rows of 20001 x 3072, four
// warps on each of two quadrants / this: 34.2 / 31.9 us.)
constexpr int kHalfCols = kMaxBN / 2;
template <int KT, bool PAIR, bool SPLIT>
__global__ void __launch_bounds__((2 + 4 * kParts) * 32, 1)
k_head_dense(const HeadArgs a, Ctrl* ctrl, float* __restrict__ recs, const DenseGeo geo,
             const __grid_constant__ CUtensorMap tm_h, const __grid_constant__ CUtensorMap tm_w) {
    extern __shared__ uint8_t s_dyn[];
    __shared__ uint64_t s_full[kMaxStages], s_empty[kMaxStages], s_acc_full[2], s_acc_empty[2];
    __shared__ uint32_t s_tmem_base;
    __shared__ int s_abort;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#ifdef VT_STAMPS
    unsigned long long* stamps = reinterpret_cast<unsigned long long*>(
        reinterpret_cast<uint8_t*>(recs) + align_up_dev((size_t)kMaxGrid * a.B * rec_fields(a.topk) * 4, 256));
    if (threadIdx.x == 0) VT_DSTAMP(0);
#endif
    // identical in both CTAs of a pair: the MMA addresses the peer's operands by the leader's offsets
    // (the candidate entries lie in front of the ring)
    constexpr int kShares = SPLIT ? 2 * kParts : kParts;           // column shares of a hidden row
    constexpr int kRows = SPLIT ? kBM / 2 : kBM, kEntStride = kShares * kRows;
    uint8_t* entries = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(s_dyn) + 1023) & ~(uintptr_t)1023);
    uint8_t* ring = entries + KT * kEntStride * sizeof(float2);
    const uint32_t ring_u32 = smem_u32(ring);
    const int B = a.B, K = a.K, topk = a.topk;
    const uint32_t rank = PAIR ? cluster_ctarank() : 0u;          // 0 = leader: issues the MMAs, owns the full barriers
    const int group = PAIR ? (int)(blockIdx.x >> 1) : (int)blockIdx.x;
    const int bn = geo.bn, n_stages = geo.n_stages;
    const int w_rows = PAIR ? bn / 2 : bn;                         // vocabulary rows this CTA stages per step
    // epilogue warps of a CTA with this many of the hidden rows that have any of them to look after
    auto live_warps = [&](int rows) { return (min(max(rows, 0), kBM) + 31) / 32 * kShares; };

    if (threadIdx.x == 0) {
        // the two tensor maps are fetched now, not by the first copy that needs them
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tm_h)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tm_w)) : "memory");
        for (int s = 0; s < kMaxStages; ++s) { mbar_init(&s_full[s], 1); mbar_init(&s_empty[s], 1); }
        for (int p = 0; p < 2; ++p) { mbar_init(&s_acc_full[p], 1); mbar_init(&s_acc_empty[p], live_warps(B) + (PAIR ? live_warps(B - kBM) : 0)); }
        s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {   // tensor memory: all 512 columns of the SM (one CTA per SM by shared-memory size)
        if (PAIR) {
            asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;"
                         ::"r"(smem_u32(&s_tmem_base)), "r"((uint32_t)kTmemCols) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
        } else {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                         ::"r"(smem_u32(&s_tmem_base)), "r"((uint32_t)kTmemCols) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        }
    }
    tc_fence_before();
    if (PAIR) cluster_sync_all(); else __syncthreads();           // barriers initialised in both CTAs before any signal
    tc_fence_after();
    const uint32_t tmem_base = s_tmem_base;
    volatile int* abort_flag = &s_abort;
    griddep_launch_dependents();                                  // the merge kernel may take its seats
#ifdef VT_STAMPS
    if (threadIdx.x == 0) VT_DSTAMP(1);
#endif

    if (warp == 0) {
        // ================= TMA producer (both CTAs of a pair) ==========================================
        if (elect_one()) {
            // fills are numbered g = 0 .. total-1 over (tile, step in d); fill g uses stage g % n_stages
            const int my_tiles = (geo.n_tiles - group + geo.n_groups - 1) / geo.n_groups;
            const int sub = geo.sub;
            const int n_ks = (geo.n_kc + sub - 1) / sub;               // ring stages per tile
            const int total = my_tiles * n_ks;
            const uint32_t sub_bytes = (uint32_t)geo.stage_bytes / (uint32_t)sub, h_bytes = (uint32_t)geo.h_bytes;
            const uint32_t full0 = PAIR ? mapa_u32(smem_u32(&s_full[0]), 0) : 0u;      // the leader's full barriers
            auto subs_of = [&](int g) { return min(sub, geo.n_kc - (g % n_ks) * sub); };
            auto load_w = [&](int g) {
                const int s = g % n_stages, tile = group + (g / n_ks) * geo.n_groups;
                for (int u = 0; u < subs_of(g); ++u) {
                    const int kc = (g % n_ks) * sub + u;
                    const uint32_t dst = ring_u32 + (uint32_t)s * (uint32_t)geo.stage_bytes + (uint32_t)u * sub_bytes + h_bytes;
                    if (PAIR) tma_load_2d_pair(dst, &tm_w, kc * kBK, tile * bn + (int)rank * w_rows, full0 + (uint32_t)(s * sizeof(uint64_t)));
                    else tma_load_2d(dst, &tm_w, kc * kBK, tile * bn, &s_full[s]);
                }
            };
            auto load_h = [&](int g) {
                const int s = g % n_stages;
                for (int u = 0; u < subs_of(g); ++u) {
                    const int kc = (g % n_ks) * sub + u;
                    const uint32_t dst = ring_u32 + (uint32_t)s * (uint32_t)geo.stage_bytes + (uint32_t)u * sub_bytes;
                    if (PAIR) tma_load_2d_pair(dst, &tm_h, kc * kBK, (int)rank * kBM, full0 + (uint32_t)(s * sizeof(uint64_t)));
                    else tma_load_2d(dst, &tm_h, kc * kBK, 0, &s_full[s]);
                }
            };
            // what lands per step: the hidden rows of the copy and this CTA's share of the vocabulary rows
            const uint32_t step_tx = (uint32_t)(geo.h_rows + w_rows) * (kBK * 2);
            auto bytes_of = [&](int g) { return (uint32_t)(PAIR ? 2 : 1) * step_tx * (uint32_t)subs_of(g); };
            // The weights are static: the first ring of them is requested before the work this launch
            // depends on has finished; everything that work may have produced is touched after the wait.
            const int pre = min(n_stages, total);
            for (int g = 0; g < pre; ++g) {
                if (rank == 0) mbar_expect_tx(&s_full[g], bytes_of(g));
                load_w(g);
            }
            griddep_wait();
            VT_DSTAMP(2);
            for (int g = 0; g < pre; ++g) load_h(g);
            int done = pre;
            {
                // steady state: the cursor over (stage, step in d, tile) moves by additions only -- this thread's
                // turn-around between "stage free" and "copies asked for" is on the ring's critical path
                int sc = pre % n_stages, ks = pre % n_ks, tl = pre / n_ks;
                uint32_t par = (uint32_t)((pre / n_stages) & 1) ^ 1u;
                const uint32_t pair_mul = PAIR ? 2u : 1u;
                for (int g = pre; g < total; ++g, ++done) {
                    if (!mbar_wait(&s_empty[sc], par, abort_flag)) break;
                    const int subs = min(sub, geo.n_kc - ks * sub);
                    if (rank == 0) mbar_expect_tx(&s_full[sc], pair_mul * step_tx * (uint32_t)subs);
                    const uint32_t dst0 = ring_u32 + (uint32_t)sc * (uint32_t)geo.stage_bytes;
                    const uint32_t bar = full0 + (uint32_t)(sc * sizeof(uint64_t));
                    const int row_w = (group + tl * geo.n_groups) * bn + (PAIR ? (int)rank * w_rows : 0);
#pragma unroll
                    for (int u = 0; u < kMaxSub; ++u) {
                        if (u < subs) {
                            const int x = (ks * sub + u) * kBK;
                            if (PAIR) {
                                tma_load_2d_pair(dst0 + (uint32_t)u * sub_bytes, &tm_h, x, (int)rank * kBM, bar);
                                tma_load_2d_pair(dst0 + (uint32_t)u * sub_bytes + h_bytes, &tm_w, x, row_w, bar);
                            } else {
                                tma_load_2d(dst0 + (uint32_t)u * sub_bytes, &tm_h, x, 0, &s_full[sc]);
                                tma_load_2d(dst0 + (uint32_t)u * sub_bytes + h_bytes, &tm_w, x, row_w, &s_full[sc]);
                            }
                        }
                    }
                    if (++sc == n_stages) { sc = 0; par ^= 1u; }
                    if (++ks == n_ks) { ks = 0; ++tl; }
                }
            }
            if (done == total && !*abort_flag) {
                // every fill consumed: all copies have landed and every commit aimed at this CTA's
                // barriers has arrived before the CTA may leave
                for (int g = max(0, total - n_stages); g < total; ++g)
                    if (!mbar_wait(&s_empty[g % n_stages], (uint32_t)((g / n_stages) & 1), abort_flag)) break;
            }
            if (*abort_flag) {
                // something timed out: give copies still in flight time to land before the memory goes away
                const unsigned long long t0 = global_ns();
                while (global_ns() - t0 < 200000ull) {}
            }
        }
    } else if (warp == 1) {
        // ================= MMA issuer (leader CTA only) ================================================
        if (rank == 0 && elect_one()) {
            const int bn0 = SPLIT ? geo.bn0 : bn;                               // columns of the (first) MMA
            const uint32_t idesc = make_idesc(PAIR ? 2 * kBM : kBM, bn0), idesc1 = make_idesc(kBM, SPLIT ? bn - bn0 : 16);
            const uint64_t desc_a0 = make_desc(ring_u32);                       // (the ring is 1024-byte aligned and under 256 KB:
            const uint64_t sub16 = (uint64_t)(((uint32_t)geo.stage_bytes / (uint32_t)geo.sub) >> 4);   //  adding byte offsets >> 4 stays inside the address field)
            int s = 0, t_local = 0;
            uint32_t ph = 0;
            bool alive = true;
            for (int tile = group; tile < geo.n_tiles && alive; tile += geo.n_groups, ++t_local) {
                const int as = t_local & 1;
                const uint32_t use = (uint32_t)(t_local >> 1);
                if (t_local >= 2 && !mbar_wait(&s_acc_empty[as], (use - 1) & 1, abort_flag)) { alive = false; break; }
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + (uint32_t)(as * kMaxBN);
                const int n_ks = (geo.n_kc + geo.sub - 1) / geo.sub;
                for (int ks = 0; ks < n_ks; ++ks) {
                    const int kc = ks * geo.sub;
                    if (!mbar_wait(&s_full[s], ph, abort_flag)) { alive = false; break; }
#ifdef VT_STAMPS
                    if (t_local == 0 && kc == 0) VT_DSTAMP(3);
#endif
                    tc_fence_after();
                    const int subs = min(geo.sub, geo.n_kc - kc);
                    const uint64_t da0 = desc_a0 + (uint64_t)(((uint32_t)s * (uint32_t)geo.stage_bytes) >> 4);
                    const uint64_t db0 = da0 + (uint64_t)(geo.h_bytes >> 4);
#pragma unroll
                    for (int u = 0; u < kMaxSub; ++u) {
                        if (u < subs) {
#pragma unroll
                            for (int k = 0; k < kBK / 16; ++k) {
                                const uint64_t step = (uint64_t)u * sub16 + (uint64_t)(k * 2);
                                if (PAIR) tc_mma_pair(d_tmem, da0 + step, db0 + step, idesc, (kc | u | k) != 0 ? 1u : 0u);
                                else tc_mma(d_tmem, da0 + step, db0 + step, idesc, (kc | u | k) != 0 ? 1u : 0u);
                                if (SPLIT)
                                    tc_mma(d_tmem + kHalfCols, da0 + step - (uint64_t)(kRows * kBK * 2 >> 4),
                                           db0 + step + (uint64_t)(bn0 * kBK * 2 >> 4), idesc1, (kc | u | k) != 0 ? 1u : 0u);
                            }
                        }
                    }
                    // the stage is free (in both CTAs) once these MMAs have read it
                    if (PAIR) tc_commit_pair(&s_empty[s]); else tc_commit(&s_empty[s]);
                    if (++s == n_stages) { s = 0; ph ^= 1; }
                }
                if (alive) {                                      // accumulators of this tile are complete
                    if (PAIR) tc_commit_pair(&s_acc_full[as]); else tc_commit(&s_acc_full[as]);
#ifdef VT_STAMPS
                    if (t_local == 0) VT_DSTAMP(4);
                    VT_DSTAMP(5);
#endif
                }
            }
            // the last accumulators have been read (every arrival of the peer has landed) before leaving
            for (int t = max(0, t_local - 2); t < t_local && alive; ++t)
                if (!mbar_wait(&s_acc_empty[t & 1], (uint32_t)((t >> 1) & 1), abort_flag)) break;
        }
    } else {
        // ================= epilogue warps: one hidden row and one share of the tile's columns per thread =
        const int ew = warp - 2;
        const int quad = warp & 3;                            // TMEM lanes this warp may read
        const int half = SPLIT ? quad >> 1 : 0;               // which columns the quadrant has
        const int row0 = SPLIT ? (quad & 1) * 32 : quad * 32; // first of its hidden rows
        const int share = half * kParts + (ew >> 2);          // which of the row's columns this warp takes
        const int rows = min(B - (int)rank * kBM, kBM);       // hidden rows of this CTA
        const int n_ch = bn / kCh, n_ch0 = SPLIT ? geo.bn0 / kCh : n_ch;
        const int ch0 = half ? n_ch0 : 0, n_mine = half ? n_ch - n_ch0 : n_ch0;
        const int ch_lo = ch0 + (ew >> 2) * n_mine / kParts, ch_hi = ch0 + ((ew >> 2) + 1) * n_mine / kParts;
        const int col_off = half ? kHalfCols - geo.bn0 : 0;   // from a column of the tile to its place in the accumulator stage
        const int b = (int)rank * kBM + row0 + lane;
        const bool row_live = b < B;
        if (row0 < rows) {
            griddep_wait();                                   // temp, uniforms and the record scratch belong to earlier work until here
            float invT = 0.f;
            if (row_live) {
                const float T = a.temp[b];
                invT = (T > 0.f && T < CUDART_INF_F) ? 1.f / T : CUDART_NAN_F;
            }
            RowState<KT> st;
            st.m = -CUDART_INF_F; st.s = 0.f; st.gb_s = -CUDART_INF_F; st.gb_z = 0.f; st.gb_j = -1;
#pragma unroll
            for (int i = 0; i < KT; ++i) { st.tv[i] = (i < KT - topk) ? CUDART_INF_F : -CUDART_INF_F; st.tj[i] = -1; }
            float2* ent = reinterpret_cast<float2*>(entries) + share * kRows + row0 + lane;
            const bool vec_u = a.uniforms && uniforms_aligned(a.uniforms, K);
            const bool use_u = row_live && a.uniforms != nullptr;
            const uint32_t acc_empty_bar = PAIR ? mapa_u32(smem_u32(&s_acc_empty[0]), 0) : 0u;
            const uint32_t tmem_row = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)col_off;
            // The warp's chunks one after the other, through all tiles: a chunk's uniforms are requested when the one before it has
            // used its own.
            float u[kCh];
#pragma unroll
            for (int i = 0; i < kCh; ++i) u[i] = 0.5f;
            auto request_u = [&](int j0) {
                if (!use_u || j0 >= K) return;
                const float* up = a.uniforms + (size_t)b * K + j0;
                if (vec_u && j0 + kCh <= K) {
#pragma unroll
                    for (int i = 0; i < kCh / 4; ++i) {
                        const float4 q = reinterpret_cast<const float4*>(up)[i];
                        u[4 * i] = q.x; u[4 * i + 1] = q.y; u[4 * i + 2] = q.z; u[4 * i + 3] = q.w;
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < kCh; ++i) u[i] = (j0 + i < K) ? up[i] : 0.5f;
                }
            };
            // log2(-log u) of the chunk at hand: -log u from a short series in 1-u near 1 (where the fast logarithm's absolute
            // error would dominate), fast logarithms elsewhere; u is clamped to [2^-24, 1 - 2^-24] where each of the two looks at it
            auto noise = [&](float (&g)[kCh]) {
#pragma unroll
                for (int i = 0; i < kCh; ++i) {
                    const float t = fmaxf(1.f - u[i], 0x1p-24f);
                    const float lp = t * (1.f + t * (0.5f + t * (0.33333334f + t * (0.25f + t * 0.2f))));
                    const float L = u[i] > 0.95f ? lp : log2_fast(fmaxf(u[i], 0x1p-24f)) * -kLn2;
                    g[i] = log2_fast(L);
                }
            };
            if (ch_lo < ch_hi) request_u(group * bn + ch_lo * kCh);
            int t_local = 0;
            for (int tile = group; tile < geo.n_tiles; tile += geo.n_groups, ++t_local) {
                const int as = t_local & 1;
                const int jt = tile * bn;                     // first vocabulary row of the tile
                const int ch_end = min(ch_hi, (K - jt + kCh - 1) / kCh);       // (chunks that have columns)
                const uint32_t acc = tmem_row + (uint32_t)(as * kMaxBN);
                // The Gumbel noise of the CTA's last tile is made while its MMAs run, and parked in the accumulator stage that
                // no further tile will use: the only epilogue that nothing hides has neither the loads nor the logarithms.
                const bool last = tile + geo.n_groups >= geo.n_tiles;
                const uint32_t parked = tmem_row + (uint32_t)((as ^ 1) * kMaxBN);
                if (last && a.uniforms) {
#pragma unroll 1
                    for (int ch = ch_lo; ch < ch_end; ++ch) {
                        float g[kCh];
                        noise(g);
                        if (ch + 1 < ch_end) request_u(jt + (ch + 1) * kCh);
                        __syncwarp();
                        tc_st16(parked + (uint32_t)(ch * kCh), g);
                    }
                }
                if (!mbar_wait_warp(&s_acc_full[as], (uint32_t)((t_local >> 1) & 1), abort_flag)) break;
#ifdef VT_STAMPS
                if (warp == 2 && lane == 0) { if (t_local == 0) VT_DSTAMP(6); VT_DSTAMP(7); }
#endif
                tc_fence_after();
                // z of a chunk's columns; columns that do not exist carry -inf
                auto load_z = [&](int ch, float (&z)[kCh]) {
                    float r[kCh];
                    __syncwarp();
                    tc_ld16(acc + (uint32_t)(ch * kCh), r);
                    const int nv = K - (jt + ch * kCh);
#pragma unroll
                    for (int i = 0; i < kCh; ++i) z[i] = r[i] * invT;
                    if (nv < kCh) {
#pragma unroll
                        for (int i = 0; i < kCh; ++i) z[i] = (i < nv) ? z[i] : -CUDART_INF_F;
                    }
                };
                // (Warp-uniform throughout: the lane of a hidden row that does not exist goes along with whatever it has and is
                // never looked at.)
#pragma unroll 1
                for (int ch = ch_lo; ch < ch_end; ++ch) {
                    const int j0 = jt + ch * kCh;

                    float z[kCh];
                    load_z(ch, z);
                    float cmax = z[0];
#pragma unroll
                    for (int i = 1; i < kCh; ++i) cmax = fmaxf(cmax, z[i]);
                    if (a.dbg_logits) {
                        float r[kCh];
                        tc_ld16(acc + (uint32_t)(ch * kCh), r);
#pragma unroll
                        for (int i = 0; i < kCh; ++i)
                            if (row_live && j0 + i < K) a.dbg_logits[(size_t)b * K + j0 + i] = r[i];
                    }
                    // running max / sum-exp: one rescale per chunk, independent exponentials, two sums.  The maximum is
                    // subtracted before the scaling to base 2: z - m is exact or nearly so whatever the size of the logits,
                    // while z * log2e - round(m * log2e) carries half a unit of m * log2e into every exponent of the chunk
                    const float m_new = fmaxf(st.m, cmax);
                    const float m_ref = (m_new == -CUDART_INF_F) ? 0.f : m_new;
                    float acc0 = 0.f, acc1 = 0.f;
#pragma unroll
                    for (int i = 0; i < kCh; i += 2) {
                        acc0 += exp_fast(z[i] - m_ref);
                        acc1 += exp_fast(z[i + 1] - m_ref);
                    }
                    const float add = acc0 + acc1;
                    st.s = st.s * exp_fast(st.m - m_ref) + add;
                    st.m = m_new;

                    if (a.uniforms) {
                        // Gumbel maximum, score z - log(-log u)
                        float g[kCh];
                        if (last) {
                            __syncwarp();
                            tc_ld16(parked + (uint32_t)(ch * kCh), g);
                        } else {
                            noise(g);
                            request_u(ch + 1 < ch_end ? j0 + kCh : jt + geo.n_groups * bn + ch_lo * kCh);
                        }
                        float bs[2] = {-CUDART_INF_F, -CUDART_INF_F}, bz[2] = {0.f, 0.f};       // (two halves side by side)
                        int bj[2] = {-1, -1};
#pragma unroll
                        for (int i = 0; i < kCh; ++i) {
                            const int q = i / (kCh / 2);
                            const float sc = fmaf(g[i], -kLn2, z[i]);
                            const bool win = sc > bs[q];              // columns that do not exist carry z = -inf
                            bs[q] = win ? sc : bs[q];
                            bj[q] = win ? i : bj[q];
                            bz[q] = win ? z[i] : bz[q];
                        }
                        const bool second = bs[1] > bs[0];
                        const float cs = second ? bs[1] : bs[0];
                        if (cs > st.gb_s) {
                            st.gb_s = cs;
                            st.gb_j = j0 + (second ? bj[1] : bj[0]);
                            st.gb_z = second ? bz[1] : bz[0];
                        }
                    }

                    if (t_local == 0) {
                        // Top-k over the first tile, where nearly everything is a candidate at first: the list's values alone, by
                        // sorting networks, whatever a chunk holds; the indices follow below.  (Inserting the candidates one by one,
                        // a warp does as many trips as the one of its 32 rows that has most of them, 9 a chunk.)
                        if (__any_sync(0xffffffffu, add != add)) {
                            // a NaN logit (or an infinite one) somewhere: a NaN is no candidate, and the networks have to be without it
                            // (min and max would drop it and keep its partner twice)
#pragma unroll
                            for (int i = 0; i < kCh; ++i) z[i] = fmaxf(z[i], -CUDART_INF_F);
                        }
                        sort_desc<0, KT>(z);
                        merge_desc<0>(st.tv, z);
                        if (KT < kCh) {
                            sort_desc<kCh - KT, KT>(z);
                            merge_desc<kCh - KT>(st.tv, z);
                        }
                    } else {
                        // Later on a chunk has few candidates, the columns that beat the list's last entry as it stands; they go in
                        // by ascending column (equal values keep the lower column ahead), one per trip of a warp-uniform loop that
                        // runs while any row still has one, everything inside select-based: one row's insertions never make the
                        // other 31 rows branch.  A candidate that has fallen under the entry that moved up meanwhile simply finds no
                        // slot.  (A NaN logit beats nothing.)
                        const float thr = st.tj[KT - 1] >= 0 ? st.tv[KT - 1] : -CUDART_INF_F;  // a threshold only once the list is full
                        uint32_t cand = 0;
#pragma unroll
                        for (int i = 0; i < kCh; ++i) cand |= (z[i] > thr) ? (1u << i) : 0u;
                        while (__any_sync(0xffffffffu, cand != 0)) {
                            const bool take = cand != 0;
                            const int i = take ? __ffs(cand) - 1 : 0;
                            float q8[8], q4[4], q2[2];
#pragma unroll
                            for (int k = 0; k < 8; ++k) q8[k] = (i & 1) ? z[2 * k + 1] : z[2 * k];
#pragma unroll
                            for (int k = 0; k < 4; ++k) q4[k] = (i & 2) ? q8[2 * k + 1] : q8[2 * k];
#pragma unroll
                            for (int k = 0; k < 2; ++k) q2[k] = (i & 4) ? q4[2 * k + 1] : q4[2 * k];
                            const float v = (i & 8) ? q2[1] : q2[0];
                            list_insert<KT>(st.tv, st.tj, take ? v : -CUDART_INF_F, j0 + i);
                            cand &= cand - 1;
                        }
                    }
                }

                if (t_local == 0) {
                    // The threshold is known: the columns at or above it are the list, and go to shared memory with their indices in
                    // ascending order.  More of them than fit means that columns tie at the threshold; then it is done again and of
                    // those only the first are taken, as many as there is room for.
                    const float thr = st.tv[KT - 1];
                    const float least = fmaxf(thr, -FLT_MAX);          // (a list that is not full: every column but -inf)
                    int n = 0;
#pragma unroll 1
                    for (int ch = ch_lo; ch < ch_end; ++ch) {
                        float z[kCh];
                        load_z(ch, z);
#pragma unroll
                        for (int i = 0; i < kCh; ++i) {
                            const bool in = z[i] >= least;
                            if (in) ent[min(n, KT - 1) * kEntStride] = make_float2(z[i], __int_as_float(jt + ch * kCh + i));
                            n += in ? 1 : 0;
                        }
                    }
                    if (__any_sync(0xffffffffu, row_live && n > topk)) {
                        int ties = KT;                        // entries equal to the threshold that there is room for
#pragma unroll
                        for (int i = 0; i < KT; ++i) ties -= st.tv[i] > thr || (i < KT - topk && thr == CUDART_INF_F) ? 1 : 0;
                        n = 0;
#pragma unroll 1
                        for (int ch = ch_lo; ch < ch_end; ++ch) {
                            float z[kCh];
                            load_z(ch, z);
#pragma unroll
                            for (int i = 0; i < kCh; ++i) {
                                const bool tie = z[i] == thr;
                                const bool in = z[i] >= least && (!tie || ties > 0);
                                ties -= in && tie ? 1 : 0;
                                if (in) ent[min(n, KT - 1) * kEntStride] = make_float2(z[i], __int_as_float(jt + ch * kCh + i));
                                n += in ? 1 : 0;
                            }
                        }
                    }

                    unsigned long long key[KT];
                    n = min(n, topk);
#pragma unroll
                    for (int i = 0; i < KT; ++i) {
                        const float2 e = i < n ? ent[i * kEntStride] : make_float2(0.f, 0.f);
                        // (-0 orders as 0; the sentinels in front of everything)
                        key[i] = i < n ? key64(e.x + 0.f, __float_as_int(e.y)) : i < topk ? 0ull : ~0ull;
                    }
                    sort_desc<0, KT>(key);
#pragma unroll
                    for (int i = 0; i < KT; ++i) {
                        st.tj[i] = i < KT - topk || key[i] == 0ull ? -1 : key_idx(key[i]);
                        st.tv[i] = i < KT - topk ? CUDART_INF_F : key[i] == 0ull ? -CUDART_INF_F : key_val(key[i]);
                    }

                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) {
                    if (PAIR) mbar_arrive_cluster(acc_empty_bar + (uint32_t)(as * sizeof(uint64_t)));
                    else mbar_arrive(&s_acc_empty[as]);
                }
#ifdef VT_STAMPS
                if (warp == 2 && lane == 0) { if (t_local == 0) VT_DSTAMP(8); VT_DSTAMP(9); }
#endif
            }

            const bool ok = !*abort_flag;
            unsigned long long key[KT];                       // the list as keys, behind the sentinels
#pragma unroll
            for (int i = 0; i < KT; ++i) key[i] = i < KT - topk ? ~0ull : st.tj[i] >= 0 ? key64(st.tv[i] + 0.f, st.tj[i]) : 0ull;
            if (!PAIR) {
                // the column shares of a row meet in shared memory: lists where the thread's entries were, the rest in the ring
                // (idle by now: the last accumulators were complete, so every MMA has read its operands and every copy has landed)
                unsigned long long* klist = reinterpret_cast<unsigned long long*>(ent);
                float* xch = reinterpret_cast<float*>(ring) + share * kRows + row0 + lane;
#pragma unroll
                for (int o = 1; o < kShares; o <<= 1) {
                    if ((share & (2 * o - 1)) == o && ok) {
#pragma unroll
                        for (int i = 0; i < KT; ++i) klist[((i + topk) & (KT - 1)) * kEntStride] = i < KT - topk ? 0ull : key[i];
                        xch[0] = st.m; xch[kEntStride] = st.s; xch[2 * kEntStride] = st.gb_s;
                        xch[3 * kEntStride] = __int_as_float(st.gb_j); xch[4 * kEntStride] = st.gb_z;
                    }
                    asm volatile("bar.sync 1, %0;" ::"r"(live_warps(rows) * 32) : "memory");
                    if ((share & (2 * o - 1)) == 0 && ok) {
                        const float* x = xch + o * kRows;
                        unsigned long long other[KT];
#pragma unroll
                        for (int i = 0; i < KT; ++i) other[i] = klist[i * kEntStride + o * kRows];
                        lse_merge(st.m, st.s, x[0], x[kEntStride]);
                        const float os = x[2 * kEntStride];
                        const int oj = __float_as_int(x[3 * kEntStride]);
                        if (better(os, oj, st.gb_s, st.gb_j) && oj >= 0) { st.gb_s = os; st.gb_j = oj; st.gb_z = x[4 * kEntStride]; }
                        merge_desc<0>(key, other);
                    }
                }
            }

            if ((PAIR || share == 0) && ok && row_live) {
                // ---- the record of hidden row b: this CTA's, or this share's of the pair's columns (a pair leaves two per row, which
                // the merge takes as well as one)
                unsigned long long* kp = rec_keys(recs, b, topk);
                float* fp = rec_f32(recs, b, topk);
                const int c = PAIR ? group * kParts + share : group;
                fp[c] = st.m;
                fp[kMaxGrid + c] = st.s;
                fp[2 * kMaxGrid + c] = st.gb_z;
                kp[c] = st.gb_j >= 0 ? key64(st.gb_s, st.gb_j) : 0ull;
#pragma unroll
                for (int p = 0; p < KT; ++p)
                    if (p >= KT - topk) kp[(size_t)(1 + p - (KT - topk)) * kMaxGrid + c] = key[p];
            }

        }
#ifdef VT_STAMPS
        if (warp == 2 && lane == 0) VT_DSTAMP(10);
#endif
    }
    tc_fence_before();
    __syncwarp();                                                 // lanes of the single-thread roles rejoin their warps
    if (PAIR) cluster_sync_all(); else __syncthreads();           // nobody leaves while its peer may still signal it
    if (warp == 1) {
        tc_fence_after();
        if (PAIR) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)kTmemCols) : "memory");
        else asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)kTmemCols) : "memory");
    }
    if (threadIdx.x == 0 && s_abort) {
        atomicOr(&ctrl->flags, (uint32_t)VT_FLAG_TIMEOUT);
        atomicOr(&ctrl->head_aborted, 1u);                        // the merge reports every row as missing
    }
#ifdef VT_STAMPS
    if (threadIdx.x == 0) VT_DSTAMP(11);
#endif
}

// A block of six warps per hidden row: merge the CTA records, remap, write the outputs.  After a wait that expired somewhere the records are
// incomplete: every row is reported as missing.  FUSE: tree drafting -- the block that finishes last turns the merged
// candidates into pool nodes and chooses the next frontier, so that a tree depth needs no launch for it.  (Dynamic shared
// memory, sized by the need: the block has to fit beside the head kernel's CTA to take its seat early.)
// Bound by latency: two L2 round trips (records; index mapper, behind the ranking) and about ten short dependent phases.  us per
// chained step, two warps per row and a round trip more / this: one row of 5000 x 1024 9.7 / 8.7, of 32768 x 3072 31.6 / 30.5, 8
// rows of 9973 x 3072 17.6 / 16.7, 100 rows of 20001 x 3072 37.3 / 35.3.
constexpr int kFuseNodes = 64;                                    // new nodes that the last block expands (see launch_head_merge)
// LEAN: 32 registers, with spills, where the head's CTAs have eighteen warps of 96 (9 to 64 rows of the streaming kernel): beside five
// of those in a quarter of the register file there is room for one warp of 32 and none of 48, and a merge that does not find
// its seat early starts 1.5-2 us late (48 / 32 registers, us per step: 12 rows of 4757 x 2048 15.4 / 13.2, 10 rows of 9973 x 3072 19.2 /
// 17.7, 24 rows of 5000 x 2048 17.1 / 15.6; beside the other heads the spills show: 8 rows of 9973 x 3072 16.2 / 16.8).
template <bool LEAN>
__global__ void __launch_bounds__(kMergeThreads, LEAN ? 10 : 1)
k_head_merge(const HeadArgs a, Ctrl* ctrl, float* __restrict__ recs, int G, int fuse) {
    extern __shared__ __align__(16) float s_stage[];              // [kMergeStageWords], and over it the keys of the expansion
    __shared__ float s_xch;
    __shared__ int s_last, s_n, s_deep;
    const int b = blockIdx.x;
    griddep_launch_dependents();                                  // the next step may start fetching its weights
    if (threadIdx.x == 0) { s_n = 0; s_deep = 0; }
    __syncthreads();
    griddep_wait();                                               // the records are complete
#ifdef VT_STAMPS
    unsigned long long* stamps = reinterpret_cast<unsigned long long*>(
        reinterpret_cast<uint8_t*>(recs) + align_up_dev((size_t)kMaxGrid * a.B * rec_fields(a.topk) * 4, 256));
    if (b == 0 && threadIdx.x == 0) stamps[12] = global_ns();
#endif
    // (everything is on its way before the mark is looked at: a round trip to L2 is a fifth of the merge)
    const uint32_t mark = ld_cg_u32(&ctrl->head_aborted);
    const MergeOut mo{a.map, a.out_ids, a.out_logprobs, a.dbg_lse, a.temp, a.topk, a.uniforms != nullptr};
    MergeLoads ld;
    merge_request(mo, recs, b, G, ld);
    const bool aborted = mark != 0u;
    if (aborted) {
        for (int i = threadIdx.x; i < 1 + a.topk; i += kMergeThreads) {
            a.out_ids[(size_t)b * (1 + a.topk) + i] = -1;
            a.out_logprobs[(size_t)b * (1 + a.topk) + i] = CUDART_NAN_F;
        }
    } else {
        if (threadIdx.x < 32 * kMaxOwn) merge_candidates(mo, ctrl, recs, b, G, ld, s_stage, &s_n, &s_deep, &s_xch);
        else merge_stats(mo, ctrl, b, G, ld, &s_xch);
    }
#ifdef VT_STAMPS
    if (b == 0 && threadIdx.x == 0) stamps[13] = global_ns();
#endif
    if (!fuse && !aborted) return;
    __syncthreads();                                              // the row's outputs are written
    if (threadIdx.x == 0) {
        unsigned old;
        asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], %2;" : "=r"(old) : "l"(&ctrl->head_ticket), "r"(1u) : "memory");
        s_last = old == gridDim.x - 1;
        if (s_last) {                                             // every block has looked: ready for the next launch
            ctrl->head_ticket = 0;
            ctrl->head_aborted = 0;
        }
    }
    __syncthreads();
    if (!s_last || !fuse) return;
    tree_expand_block(a.tree, a.out_ids, a.out_logprobs, a.B, a.topk, 1 + a.topk, 1, reinterpret_cast<unsigned long long*>(s_stage),
                      (int)threadIdx.x, kMergeThreads);
}

// ---- host side ----------------------------------------------------------------------------------------
// Tile width: the vocabulary is dealt to `groups` CTAs (pairs) in tiles of bn rows.  A CTA's time is that of its tiles -- what it takes
// from HBM (its rows of W, and the uniforms of its columns) or, where that is longer, what it stages through L2 (those and all hidden
// rows again, per tile), and the turn-around of a tile and of its steps -- and of the last tile's epilogue, which nothing hides.  The
// rates are a CTA's share with all SMs at work, fitted to 2500 timed widths of 183 shapes (3000 to 111000 rows, d = 512 to 4096, 33 to 256
// hidden rows): the width they choose is the fastest one for half of the shapes and within 6 % of it for nine in ten.  Evening out the
// rows per CTA alone, as this did before, takes 16 columns for one K in five, and each such tile brings the hidden rows again (us per
// call, even rows / this, with uniforms: 100 hidden rows of 40000 x 3072 150 / 52, of 95000 x 3072 346 / 105, 40 of 40000 x 2048 137 / 37;
// pairs: 200 of 95000 x 3072 306 / 141, 256 of 40000 x 1024 72 / 47).  On equal terms the wider tile.  Multiples of 16, for a pair of 32:
// the columns of an MMA over two CTAs come in those.
struct TileCost {
    double hbm, staged;                   // bytes / ns
    double tile, step, column;            // ns per tile, per 64-column step, per column of the last epilogue
};
constexpr TileCost kCostSplit{41., 90., 200., 10., 10.}, kCostNarrow{41., 90., 800., 10., 20.}, kCostSingle{44., 90., 400., 10., 20.},
    kCostPair{44., 160., 1800., 5., 20.};
// Columns from which a tile of up to 64 hidden rows is computed in two halves.  Its MMAs are twice as many, and one takes some 40 cycles
// however few its columns; what the second set of lanes saves is epilogue, by the column (us per call, one / two halves: 40 rows of
// 3000 x 3072 in tiles of 32 16.7 / 21.9, of 9973 x 4096 in 80 24.3 / 28.8, of 14000 x 1024 in 96 16.5 / 17.6, in 112 16.3 / 16.2, of
// 16668 x 3072 in 128 29.1 / 28.2, of 20001 x 2048 in 160 25.4 / 24.3, of 60000 x 1024 in 208 41.7 / 34.4).
constexpr int kSplitCols = 112;

int tile_width(int32_t B, int32_t K, int32_t d, bool sampled, int max_groups) {
    const bool pair = B > kBM;
    const int by = pair ? 32 : 16, h_rows = pair ? kBM : B, n_kc = (d + kBK - 1) / kBK;
    int best_bn = kMaxBN;
    double best = -1.;
    for (int bn = kMaxBN; bn >= by; bn -= by) {
        const TileCost& c = pair ? kCostPair : B > kBM / 2 ? kCostSingle : bn >= kSplitCols ? kCostSplit : kCostNarrow;
        const int tiles = (K + bn - 1) / bn, own = (tiles + max_groups - 1) / max_groups, w_rows = pair ? bn / 2 : bn;
        const double hbm = 2. * w_rows * d + (sampled ? 4. * bn * h_rows : 0.), staged = 2. * (h_rows + w_rows) * d;
        const double ns = own * (fmax(hbm / c.hbm, staged / c.staged) + c.tile + c.step * n_kc) + c.column * bn;
        if (best < 0. || ns < best) { best = ns; best_bn = bn; }
    }
    return best_bn;
}

DenseGeo make_geo(int32_t K, int32_t d, bool pair, int h_rows, int bn, int max_groups, size_t ring_budget) {
    DenseGeo g{};
    g.bn = bn;
    g.n_tiles = (K + g.bn - 1) / g.bn;
    g.n_kc = (d + kBK - 1) / kBK;
    g.n_groups = g.n_tiles < max_groups ? g.n_tiles : max_groups;
    g.h_rows = h_rows;
    // (the MMA reads 128 hidden rows from here: beyond those that exist whatever follows)
    g.h_bytes = (int)align_up((size_t)h_rows * kBK * 2, 1024);
    const int step_bytes = g.h_bytes + (pair ? g.bn / 2 : g.bn) * kBK * 2;
    g.bn0 = (g.bn / 2 + 15) / 16 * 16;
    g.tail_bytes = kBM * kBK * 2 > step_bytes ? kBM * kBK * 2 - step_bytes : 0;
    ring_budget -= (size_t)g.tail_bytes;
    g.sub = (3 * kMaxSub * (size_t)step_bytes <= ring_budget && g.n_kc >= kMaxSub) ? kMaxSub : 1;
    g.stage_bytes = step_bytes * g.sub;
    g.n_stages = (int)(ring_budget / (size_t)g.stage_bytes);
    if (g.n_stages > kMaxStages) g.n_stages = kMaxStages;
    g.ring_bytes = g.n_stages * g.stage_bytes;
    return g;
}

// shared memory of the candidate entries (in front of the ring: also what a split tile's second operand reads before it)
template <int KT>
constexpr size_t entry_bytes() { return (size_t)KT * kParts * kBM * sizeof(float2); }
static_assert(entry_bytes<8>() >= (size_t)kBM / 2 * kBK * 2 && entry_bytes<8>() % 1024 == 0, "64 operand rows before the ring lie inside");

template <int KT, bool PAIR, bool SPLIT>
cudaError_t launch_variant(const HeadArgs& a, Ctrl* ctrl, float* recs, int bn, int max_groups, int* records, cudaStream_t s) {
    constexpr size_t kEntries = entry_bytes<KT>();
    const bool one_by_one = a.uniforms && !uniforms_aligned(a.uniforms, a.K) && (a.d <= 3072 || bn >= 224 || a.K > bn * max_groups);
    const DenseGeo geo = make_geo(a.K, a.d, PAIR, PAIR ? kBM : a.B, bn, max_groups, kSmemBudget - kEntries - (PAIR && one_by_one ? kL1Room : 0));
    CUtensorMap tm_h, tm_w;
    if (!encode_map(&tm_h, a.h, a.B, a.d, geo.h_rows) || !encode_map(&tm_w, a.W, a.K, a.d, PAIR ? geo.bn / 2 : geo.bn))
        return cudaErrorInvalidValue;
    static int attr_done[64] = {0};
    const size_t smem = (size_t)geo.ring_bytes + kEntries + geo.tail_bytes + 1024;   // + slack to align the ring to 1024 bytes
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64 || !attr_done[dev]) {
        cudaError_t e = cudaFuncSetAttribute(k_head_dense<KT, PAIR, SPLIT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)(kSmemBudget + 1024));
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) attr_done[dev] = 1;
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(PAIR ? 2 * geo.n_groups : geo.n_groups));
    cfg.blockDim = dim3((2 + 4 * kParts) * 32);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = PAIR ? 2 : 1;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = a.overlap ? 2 : 1;
    *records = PAIR ? geo.n_groups * kParts : geo.n_groups;
    return cudaLaunchKernelEx(&cfg, k_head_dense<KT, PAIR, SPLIT>, a, ctrl, recs, geo, tm_h, tm_w);
}

}  // namespace

bool head_dense_supported(int32_t B, int32_t K, int32_t d) {
    return B >= 1 && B <= 2 * kBM && K >= 1 && d >= 8 && (d & 7) == 0;
}

bool head_dense_topk_ok(int32_t topk) { return topk >= 1 && topk <= kMaxTopk; }

size_t head_dense_scratch_bytes(int32_t B, int32_t K, int32_t topk) {
    (void)K;
    return align_up((size_t)kMaxGrid * B * rec_fields(topk) * 4, 256) + kStampBytes;
}

#ifdef VT_STAMPS
size_t head_stamps_offset(int32_t B, int32_t topk) {
    return align_up((size_t)kMaxGrid * B * rec_fields(topk) * 4, 256);
}
#endif

cudaError_t launch_head_dense(const HeadArgs& a, Ctrl* ctrl, uint8_t* scratch, cudaStream_t s) {
    if (!head_dense_supported(a.B, a.K, a.d) || !head_dense_topk_ok(a.topk)) return cudaErrorInvalidValue;
    const bool pair = a.B > kBM;                       // more than one MMA's worth of hidden rows: CTA pairs
    int max_groups = pair ? num_sms() / 2 : num_sms();
    const int most = pair ? kMaxGrid / 2 : kMaxGrid;   // (a pair leaves two records per row)
    if (max_groups > most) max_groups = most;
    if (max_groups < 1) return cudaErrorInvalidValue;
    float* recs = reinterpret_cast<float*>(scratch);
    cudaError_t e;
    int records = 0;
    const int bn = tile_width(a.B, a.K, a.d, a.uniforms != nullptr, max_groups);
    const bool split = a.B <= kBM / 2 && bn >= kSplitCols;
    if (a.topk <= 8) e = pair  ? launch_variant<8, true, false>(a, ctrl, recs, bn, max_groups, &records, s)
                       : split ? launch_variant<8, false, true>(a, ctrl, recs, bn, max_groups, &records, s)
                               : launch_variant<8, false, false>(a, ctrl, recs, bn, max_groups, &records, s);
    else e = pair  ? launch_variant<kMaxTopk, true, false>(a, ctrl, recs, bn, max_groups, &records, s)
           : split ? launch_variant<kMaxTopk, false, true>(a, ctrl, recs, bn, max_groups, &records, s)
                   : launch_variant<kMaxTopk, false, false>(a, ctrl, recs, bn, max_groups, &records, s);
    if (e != cudaSuccess) return e;
    count_launch();
    return launch_head_merge(a, ctrl, recs, records, false, s);
}

// The records of G CTAs (pairs) -> outputs; with a tree, its expansion as one more launch (it needs every row's merge).
cudaError_t launch_head_merge(const HeadArgs& a, Ctrl* ctrl, float* recs, int G, bool lean, cudaStream_t s) {
    // the merge always follows its own producer closely: it takes its seats early and waits on the device
    const int n_new = a.B * a.topk;
    // The expansion inside the merge saves a launch; as a kernel of its own it has more threads, and the blocks need not meet.  Up to
    // 64 new nodes the one wins, from there to 170 neither, beyond the other (us per depth of a tree over 9973 x 3072, fused /
    // kernel: 64 nodes 19.0 / 19.9, 100 nodes 22.9 / 22.7, 144 nodes 23.5 / 23.8, 169 nodes 25.1 / 24.8, 256 nodes 29.6 / 28.2).
    const bool fuse = a.tree.pool_token && n_new <= kFuseNodes;
    size_t smem = (size_t)kMergeStageWords * 4;
    if (fuse && (size_t)padded_keys(n_new) * 8 > smem) smem = (size_t)padded_keys(n_new) * 8;
    // (in front of an expansion kernel the early seat does not pay: 10 rows of 32768 x 4096 six depths deep 305 us without, 312 with it)
    lean = lean && (!a.tree.pool_token || fuse);
    const cudaError_t e = lean ? launch_dependent(k_head_merge<true>, (unsigned)a.B, kMergeThreads, smem, s, a, ctrl, recs, G, fuse ? 1 : 0)
                               : launch_dependent(k_head_merge<false>, (unsigned)a.B, kMergeThreads, smem, s, a, ctrl, recs, G, fuse ? 1 : 0);
    if (e != cudaSuccess || !a.tree.pool_token || fuse) return e;
    return launch_tree_expand(a.out_ids, a.out_logprobs, a.B, a.topk, 1 + a.topk, 1, a.tree, s);
}

}  // namespace vt
