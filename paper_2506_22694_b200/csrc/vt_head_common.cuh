// Pieces shared by the two head kernels (streaming and dense): ordering helpers, the per-CTA record
// layout and the cross-CTA merge that turns the records into out_ids / out_logprobs.
#pragma once
#include <math_constants.h>

#include "vt_common.cuh"

namespace vt {
namespace {

constexpr int kMaxGrid = 160;                    // merge: each lane owns at most kMaxOwn CTA records
constexpr int kMaxOwn = kMaxGrid / 32;
constexpr int kMergeDepth = 4;                   // list entries per CTA staged on chip by the merge
constexpr int kSelCap = 128;                     // entries the merge's direct selection can rank
// staging words (32-bit) of a merging block: the staged list heads, or before it comes to that the selection's buffers
constexpr int kMergeStageWords = 2 * kMergeDepth * kMaxGrid;
constexpr int kStampSlots = 16;                  // phase stamps per CTA (-DVT_STAMPS builds)
#ifdef VT_STAMPS
constexpr size_t kStampBytes = (size_t)kMaxGrid * kStampSlots * 8;
#else
constexpr size_t kStampBytes = 0;
#endif

__device__ __forceinline__ bool better(float v, int j, float bv, int bj) {
    return v > bv || (v == bv && j < bj);
}

// (m, s) <- (m, s) (+) (m2, s2) for running max / sum of exponentials.  (A NaN is left out of the maximum and lives in the sum, also
// where neither side has a maximum: 0 + 0 stays 0, NaN stays NaN.)
__device__ __forceinline__ void lse_merge(float& m, float& s, float m2, float s2) {
    const float M = fmaxf(m, m2);
    if (M == -CUDART_INF_F) { m = M; s = s + s2; return; }
    s = s * __expf(m - M) + s2 * __expf(m2 - M);
    m = M;
}


// Order-preserving map of a float onto unsigned integers (and back); no NaN ever reaches it.
__device__ __forceinline__ unsigned f2ord(float f) {
    const unsigned u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float ord2f(unsigned k) {
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

// (value, index) as one unsigned 64-bit key: larger key = better candidate (higher value, then lower
// index).  Comparing keys needs no data-dependent branch; per-lane branches inside a warp cost far
// more than the arithmetic they skip.  No real candidate has key 0, which marks an empty slot.
__device__ __forceinline__ unsigned long long key64(float v, int j) {
    return ((unsigned long long)f2ord(v) << 32) | (unsigned)(~j);
}
__device__ __forceinline__ float key_val(unsigned long long k) { return ord2f((unsigned)(k >> 32)); }
__device__ __forceinline__ int key_idx(unsigned long long k) { return (int)~(unsigned)k; }

// exp and log of the epilogue: one multiplication and the hardware's base-2 function, results and arguments under
// 2^-126 flushed to zero (the arguments of the logarithm are at least 2^-25; an exponential is added to a sum that
// holds 1).
constexpr float kLog2e = 1.4426950408889634f, kLn2 = 0.6931471805599453f;
__device__ __forceinline__ float exp2_fast(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float log2_fast(float x) {
    float y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float exp_fast(float x) { return exp2_fast(x * kLog2e); }
__device__ __forceinline__ float log_fast(float x) { return log2_fast(x) * kLn2; }

// rk[i] += number of the N keys in shared memory that are greater than ek[i]; the buffer is 16-byte aligned and
// zero-padded to a multiple of four.
template <int NS>
__device__ __forceinline__ void rank_among(const unsigned long long* keys, int N, const unsigned long long (&ek)[NS], int (&rk)[NS]) {
    const ulonglong2* k2 = reinterpret_cast<const ulonglong2*>(keys);
#pragma unroll 2
    for (int e = 0; e < N; e += 4) {
        const ulonglong2 p = k2[e >> 1], q = k2[(e >> 1) + 1];
#pragma unroll
        for (int i = 0; i < NS; ++i)
            rk[i] += ((p.x > ek[i]) ? 1 : 0) + ((p.y > ek[i]) ? 1 : 0) + ((q.x > ek[i]) ? 1 : 0) + ((q.y > ek[i]) ? 1 : 0);
    }
}

// A lower bound of the k-th largest (k <= 32) of the lanes' values: that value with its low five bits cleared (they
// tell equal lanes apart meanwhile).  Every lane counts the values above its own in shared memory (32 words, 16-byte
// aligned): broadcast reads that overlap, where 32 shuffles took 1500 cycles.
__device__ __forceinline__ unsigned kth_of_lanes(unsigned v, int k, unsigned* s32) {
    const unsigned lane = threadIdx.x & 31;
    const unsigned mine = (v & ~31u) | (31u - lane);
    s32[lane] = mine;
    __syncwarp();
    const uint4* s4 = reinterpret_cast<const uint4*>(s32);
    int rk = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const uint4 o = s4[i];
        rk += ((o.x > mine) ? 1 : 0) + ((o.y > mine) ? 1 : 0) + ((o.z > mine) ? 1 : 0) + ((o.w > mine) ? 1 : 0);
    }
    const unsigned at = __ballot_sync(0xffffffffu, rk == k - 1);
    const unsigned tau = __shfl_sync(0xffffffffu, mine, __ffs(at) - 1) & ~31u;       // (exactly one lane has that rank)
    __syncwarp();                                           // the words may be reused
    return tau;
}

// Records.  Per hidden row b a block of rec_fields(topk) * kMaxGrid 32-bit words, laid out in planes
// with the CTA index fastest, so that a merging warp reads every plane with coalesced loads:
//   64-bit planes: 0 = Gumbel-max candidate as key64(score, j); 1 + r = entry r of the CTA's top-k list
//                  as key64(z, j), best first, 0 = no entry;
//   32-bit planes (behind them): 0 = running max m, 1 = sum of exp(z - m), 2 = z of the Gumbel candidate.
__host__ __device__ inline int rec_fields(int topk) { return 5 + 2 * topk; }
__device__ __forceinline__ unsigned long long* rec_keys(float* recs, int b, int topk) {
    return reinterpret_cast<unsigned long long*>(recs + (size_t)b * rec_fields(topk) * kMaxGrid);
}
__device__ __forceinline__ float* rec_f32(float* recs, int b, int topk) {
    return recs + (size_t)b * rec_fields(topk) * kMaxGrid + (size_t)2 * (1 + topk) * kMaxGrid;
}
__device__ __forceinline__ unsigned long long ld_cg_u64(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.global.cg.b64 %0, [%1];" : "=l"(v) : "l"(p));
    return v;
}

struct MergeOut {
    const int32_t* map;
    int32_t* out_ids;
    float* out_logprobs;
    float* dbg_lse;
    const float* temp;
    int topk;
    int sampled;       // uniforms were given: column 0 is the Gumbel-max draw
};

// What a row without a full result is reported as.  (A row of unusable temperature has NaN for every z and so no candidates: nothing
// else looks at the temperature, which may lie in host memory.)
__device__ __forceinline__ uint32_t merge_flag(const MergeOut& a, int b) {
    const float T = ld_cg_f32(a.temp + b);
    return T > 0.f && T < CUDART_INF_F ? (uint32_t)VT_FLAG_NAN_ROW : (uint32_t)VT_FLAG_BAD_TEMP;
}

// The merge of one hidden row by six warps.  A warp runs dependent code at a few cycles per instruction, and the row's result is what
// the next step waits for, so the work is spread: five warps hold a CTA's list heads per lane, the sixth the
// statistics (log-sum-exp over all CTAs, the Gumbel-max winner).  Everything a warp needs from memory is asked for at once.
// (Two warps, five CTAs to a lane, took 4150 cycles from the records being there to the outputs, a quarter of them one L2 round
// trip for the abort mark in front of the records and the gathers through the index mapper behind the ranking.)
constexpr int kMergeThreads = 32 * (kMaxOwn + 1);

struct MergeLoads {                                // what a thread has asked for
    unsigned long long ek[kMergeDepth];            // candidate warps: the best entries of a CTA's list
    float hm[kMaxOwn], hs[kMaxOwn], hz[kMaxOwn];   // statistics warp: kMaxOwn CTAs to a lane
    unsigned long long hk[kMaxOwn];
};

// (loads of records that do not exist go to one that does and are not looked at: no branch around any of them)
__device__ __forceinline__ void merge_request(const MergeOut& a, float* recs, int b, int G, MergeLoads& ld) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned long long* kp = rec_keys(recs, b, a.topk);
    if (warp < kMaxOwn) {
        const int depth = min(a.topk, kMergeDepth), c = min(warp * 32 + lane, G - 1);
#pragma unroll
        for (int r = 0; r < kMergeDepth; ++r) ld.ek[r] = ld_cg_u64(kp + (size_t)(1 + min(r, depth - 1)) * kMaxGrid + c);
    } else {
        const float* fp = rec_f32(recs, b, a.topk);
#pragma unroll
        for (int o = 0; o < kMaxOwn; ++o) {
            const int c = min(lane + 32 * o, G - 1);
            ld.hm[o] = ld_cg_f32(fp + c);
            ld.hs[o] = ld_cg_f32(fp + kMaxGrid + c);
        }
        if (a.sampled) {
#pragma unroll
            for (int o = 0; o < kMaxOwn; ++o) {
                const int c = min(lane + 32 * o, G - 1);
                ld.hz[o] = ld_cg_f32(fp + 2 * kMaxGrid + c);
                ld.hk[o] = ld_cg_u64(kp + c);
            }
        }
    }
}

__device__ __forceinline__ void merge_stats(const MergeOut& a, Ctrl* ctrl, int b, int G, MergeLoads& ld, volatile float* xch) {
    const int lane = threadIdx.x & 31;
    int* oid = a.out_ids + (size_t)b * (1 + a.topk);
    float* olp = a.out_logprobs + (size_t)b * (1 + a.topk);
    // the row's maximum over this lane's CTAs and by one warp reduction, every CTA's sum rescaled to it once, added in
    // CTA order, a butterfly of additions (a fixed order: the result does not depend on which CTA finished when)
    float M = -CUDART_INF_F, gz = 0.f;
    unsigned long long gk = 0ull;
#pragma unroll
    for (int o = 0; o < kMaxOwn; ++o) {
        const bool on = lane + 32 * o < G;
        ld.hm[o] = on ? ld.hm[o] : -CUDART_INF_F;
        ld.hs[o] = on ? ld.hs[o] : 0.f;
        M = fmaxf(M, ld.hm[o]);
    }
    if (a.sampled) {
#pragma unroll
        for (int o = 0; o < kMaxOwn; ++o) {
            const bool w = lane + 32 * o < G && ld.hk[o] > gk;
            gk = w ? ld.hk[o] : gk;
            gz = w ? ld.hz[o] : gz;
        }
    }
    const float Mall = ord2f(__reduce_max_sync(0xffffffffu, f2ord(M)));
    const float Mref = Mall == -CUDART_INF_F ? 0.f : Mall;
    float sc = 0.f;
#pragma unroll
    for (int o = 0; o < kMaxOwn; ++o) sc += ld.hs[o] * exp_fast(ld.hm[o] - Mref);     // (hm = -inf: nothing but a NaN sum counts)
#pragma unroll
    for (int o = 16; o; o >>= 1) sc += __shfl_xor_sync(0xffffffffu, sc, o);
    const float lse = Mall + logf(sc);
    if (lane == 0) *xch = lse;                              // the ranking warp is waiting for it
    __syncwarp();
    asm volatile("bar.arrive 2, 64;" ::: "memory");
    unsigned long long gwin = 0ull;
    float gzw = 0.f;
    if (a.sampled) {
        const unsigned hi = (unsigned)(gk >> 32);
        const unsigned kmax = __reduce_max_sync(0xffffffffu, hi);
        const unsigned lomax = __reduce_max_sync(0xffffffffu, hi == kmax ? (unsigned)gk : 0u);
        const unsigned who = __ballot_sync(0xffffffffu, hi == kmax && (unsigned)gk == lomax);
        gzw = __shfl_sync(0xffffffffu, gz, __ffs(who) - 1);
        gwin = ((unsigned long long)kmax << 32) | lomax;
    }
    if (lane == 0) {
        bool bad = !(lse == lse);                           // a NaN logit somewhere in the row, or an unusable temperature
        if (a.sampled) {
            const bool ok = gwin != 0ull;
            const int gj = key_idx(gwin);
            oid[0] = ok ? (a.map ? ld_cg_s32(a.map + gj) : gj) : -1;
            olp[0] = ok ? gzw - lse : CUDART_NAN_F;
            bad = bad || !ok;
        }
        if (a.dbg_lse) a.dbg_lse[b] = lse;
        if (bad) atomicOr(&ctrl->flags, merge_flag(a, b));
    }
}

// Entry `key` of the merged list is the r-th best (r < topk): id and log-probability.  The id is asked for before the ranking.
__device__ __forceinline__ void merge_emit(const MergeOut& a, int b, int r, int id, unsigned long long key, float lse) {
    int* oid = a.out_ids + (size_t)b * (1 + a.topk);
    float* olp = a.out_logprobs + (size_t)b * (1 + a.topk);
    const bool ok = key != 0ull;
    id = ok ? id : -1;
    const float lp = ok ? key_val(key) - lse : CUDART_NAN_F;
    oid[1 + r] = id;
    olp[1 + r] = lp;
    if (r == 0 && !a.sampled) { oid[0] = id; olp[0] = lp; }
}
__device__ __forceinline__ int merge_id(const MergeOut& a, unsigned long long key) {
    const int j = key != 0ull ? key_idx(key) : 0;
    return a.map ? ld_cg_s32(a.map + j) : j;
}

// Ranks the n keys in sel (NS to a lane) and writes the topk best of them.
template <int NS>
__device__ __forceinline__ void merge_rank(const MergeOut& a, const unsigned long long* sel, int n, int b, volatile float* xch) {
    const int lane = threadIdx.x & 31;
    unsigned long long mine[NS];
    int rk[NS], id[NS];
#pragma unroll
    for (int i = 0; i < NS; ++i) {
        mine[i] = lane + 32 * i < n ? sel[lane + 32 * i] : 0ull;
        rk[i] = 0;
    }
#pragma unroll
    for (int i = 0; i < NS; ++i) id[i] = merge_id(a, mine[i]);
    rank_among<NS>(sel, n, mine, rk);
    asm volatile("bar.sync 2, 64;" ::: "memory");
    const float lse = *xch;
#pragma unroll
    for (int i = 0; i < NS; ++i)
        if (lane + 32 * i < n && rk[i] < a.topk) merge_emit(a, b, rk[i], id[i], mine[i], lse);
    for (int r = n + lane; r < a.topk; r += 32) merge_emit(a, b, r, -1, 0ull, lse);          // fewer than topk candidates
}

__device__ __forceinline__ void merge_candidates(const MergeOut& a, Ctrl* ctrl, float* recs, int b, int G, MergeLoads& ld,
                                                 float* stage, int* s_n, int* s_deep, volatile float* xch) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int topk = a.topk, depth = min(topk, kMergeDepth), c = warp * 32 + lane;
    unsigned long long* sel = reinterpret_cast<unsigned long long*>(stage);                    // [kSelCap] and padding
    unsigned* heads = reinterpret_cast<unsigned*>(stage) + 2 * (kSelCap + 8);                  // [kMaxGrid]
    unsigned* kth = heads + kMaxGrid + warp * 32;
    static_assert(2 * (kSelCap + 8) + 2 * kMaxGrid <= kMergeStageWords, "the selection's words fit");
#pragma unroll
    for (int r = 0; r < kMergeDepth; ++r) ld.ek[r] = c < G && r < depth ? ld.ek[r] : 0ull;
    bool direct = topk <= 32;
    if (direct) {
        // Direct selection.  tau = the topk-th largest of 32 maxima over five list heads each is a lower bound of the topk-th
        // best entry overall, so only staged entries >= tau can matter: a few dozen at most.  They are compacted into shared
        // memory and every one finds its output position as its rank -- no sequential rounds.  Falls back to the rounds below
        // when a list might hold qualifying entries beyond the staged ones, or when too many qualify.
        heads[c] = (unsigned)(ld.ek[0] >> 32);
        asm volatile("bar.sync 1, %0;" ::"n"(32 * kMaxOwn) : "memory");
        unsigned lh = heads[lane];
#pragma unroll
        for (int o = 1; o < kMaxOwn; ++o) lh = max(lh, heads[lane + 32 * o]);
        const unsigned tau = kth_of_lanes(lh, topk, kth);
        unsigned m[kMergeDepth];
        int total = 0;
        bool deep = false;
#pragma unroll
        for (int r = 0; r < kMergeDepth; ++r) {
            const bool in = ld.ek[r] != 0ull && (unsigned)(ld.ek[r] >> 32) >= tau;
            m[r] = __ballot_sync(0xffffffffu, in);
            total += __popc(m[r]);
            deep = deep || (r == depth - 1 && depth < topk && m[r] != 0u);
        }
        if (total) {                                        // (warp-uniform; the order among the warps does not matter, ranks decide)
            int base = 0;
            if (lane == 0) {
                base = atomicAdd(s_n, total);
                if (deep) *s_deep = 1;
            }
            base = __shfl_sync(0xffffffffu, base, 0);
#pragma unroll
            for (int r = 0; r < kMergeDepth; ++r) {
                const int pos = base + __popc(m[r] & lanemask_lt());
                if (((m[r] >> lane) & 1u) && pos < kSelCap) sel[pos] = ld.ek[r];
                base += __popc(m[r]);
            }
        }
        asm volatile("bar.sync 1, %0;" ::"n"(32 * kMaxOwn) : "memory");
        const int n = *s_n;
        direct = n <= kSelCap && !*s_deep;
        if (direct) {
            if (warp != 0) return;
            if (lane < 4) sel[n + lane] = 0ull;                                    // (read in groups of four)
            __syncwarp();
            if (n <= 32) merge_rank<1>(a, sel, n, b, xch);
            else merge_rank<kSelCap / 32>(a, sel, n, b, xch);
            if (lane == 0 && n < topk) atomicOr(&ctrl->flags, merge_flag(a, b));
            return;
        }
        asm volatile("bar.sync 1, %0;" ::"n"(32 * kMaxOwn) : "memory");            // (the words are given up)
    }
    // heads of the lists: entry r of CTA c at stk[r * kMaxGrid + c]
    unsigned long long* stk = sel;
#pragma unroll
    for (int r = 0; r < kMergeDepth; ++r) stk[r * kMaxGrid + c] = ld.ek[r];
    asm volatile("bar.sync 1, %0;" ::"n"(32 * kMaxOwn) : "memory");
    if (warp != 0) return;
    // k rounds of one warp; every lane keeps the current head of each of its lists in registers, a round is two
    // warp reductions, and the winner alone advances (from the staged entries, else from global memory)
    const unsigned long long* kp = rec_keys(recs, b, topk);
    unsigned long long res_k[2] = {0ull, 0ull};
    int head[kMaxOwn];
    unsigned long long ck[kMaxOwn];
#pragma unroll
    for (int o = 0; o < kMaxOwn; ++o) {
        head[o] = 0;
        ck[o] = stk[lane + 32 * o];
    }
    for (int r = 0; r < topk; ++r) {
        unsigned long long lk = ck[0];
#pragma unroll
        for (int o = 1; o < kMaxOwn; ++o) lk = ck[o] > lk ? ck[o] : lk;
        const unsigned hi = (unsigned)(lk >> 32);
        const unsigned kmax = __reduce_max_sync(0xffffffffu, hi);
        const unsigned lomax = __reduce_max_sync(0xffffffffu, hi == kmax ? (unsigned)lk : 0u);
        if (kmax == 0u) break;                                // every list is exhausted
        const unsigned long long win = ((unsigned long long)kmax << 32) | lomax;
        if (lk == win) {                                      // one lane: advance the list it came from
#pragma unroll
            for (int o = 0; o < kMaxOwn; ++o)
                if (ck[o] == win) {
                    const int hd = ++head[o];
                    unsigned long long nk = 0ull;
                    if (hd < depth) nk = stk[hd * kMaxGrid + lane + 32 * o];
                    else if (hd < topk) nk = ld_cg_u64(kp + (size_t)(1 + hd) * kMaxGrid + lane + 32 * o);
                    ck[o] = nk;
                }
        }
        if (lane == r) res_k[0] = win;
        if (lane + 32 == r) res_k[1] = win;
    }
    const int ids[2] = {merge_id(a, res_k[0]), merge_id(a, res_k[1])};
    asm volatile("bar.sync 2, 64;" ::: "memory");
    const float lse = *xch;
    bool miss = false;
#pragma unroll
    for (int sl = 0; sl < 2; ++sl) {
        const int r = lane + 32 * sl;
        if (r < topk) {
            merge_emit(a, b, r, ids[sl], res_k[sl], lse);
            miss = miss || res_k[sl] == 0ull;
        }
    }
    const bool any_missing = __any_sync(0xffffffffu, miss);
    if (lane == 0 && any_missing) atomicOr(&ctrl->flags, merge_flag(a, b));
}

}  // namespace
}  // namespace vt
