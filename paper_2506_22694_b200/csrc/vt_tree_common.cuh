// Draft-tree expansion as a block-wide device function, shared by the stand-alone kernel and by the
// head kernel that runs it right after its merge (Settings: tree construction following EAGLE-2).
#pragma once
#include "vt_common.cuh"

namespace vt {
namespace {

__device__ __forceinline__ uint32_t score_ord(float s) {
    if (s != s) s = __int_as_float(0xff800000);      // NaN ranks with -inf
    if (s == 0.0f) s = 0.0f;                         // one zero
    const uint32_t u = __float_as_uint(s);
    return u ^ ((u >> 31) ? 0xffffffffu : 0x80000000u);
}

__device__ __forceinline__ unsigned long long node_key(float s, int i) {
    return ((unsigned long long)score_ord(s) << 32) | (uint32_t)~(uint32_t)i;     // greater key = preferred
}

// rank among keys[0..n): number of strictly greater keys (keys are distinct).  All lanes read the same words, two keys
// to a 128-bit broadcast and eight loads in flight: keys is 16-byte aligned and padded with zeros to a multiple of
// kKeyGroup (a key of a node is never 0).
constexpr int kKeyGroup = 16;
__host__ __device__ inline int padded_keys(int n) { return (n + kKeyGroup - 1) / kKeyGroup * kKeyGroup; }
__device__ __forceinline__ int rank_of(const unsigned long long* keys, int n, unsigned long long mine) {
    const ulonglong2* k2 = reinterpret_cast<const ulonglong2*>(keys);
    int r = 0;
    for (int j = 0; j < n; j += kKeyGroup) {
#pragma unroll
        for (int q = 0; q < kKeyGroup / 2; ++q) {
            const ulonglong2 k = k2[j / 2 + q];
            r += (k.x > mine ? 1 : 0) + (k.y > mine ? 1 : 0);
        }
    }
    return r;
}

// One depth of the expansion by the `nthreads` threads `tid` of a CTA that all call it; s_key holds
// B * topk keys, padded to a multiple of kKeyGroup.  Contains a CTA barrier.
__device__ __forceinline__ void tree_expand_block(const TreeArgs& t, const int32_t* cand_ids,
                                                  const float* cand_lp, int32_t B, int32_t topk,
                                                  int32_t ld, int32_t col0, unsigned long long* s_key, int tid,
                                                  int nthreads) {
    const int n_new = B * topk;
    for (int i = tid; i < n_new; i += nthreads) {
        const int b = i / topk, j = i - b * topk;
        int32_t par = t.frontier ? ld_cg_s32(t.frontier + b) : -1;
        if (par < -1 || par >= t.pool_base) par = -1;                   // memory safety; callers pass earlier nodes
        const float base = par < 0 ? 0.0f : ld_cg_f32(t.pool_score + par);         // earlier depth: not written by this launch
        const float lp = ld_cg_f32(cand_lp + (int64_t)b * ld + col0 + j);    // (written by other blocks of this launch)
        const float step = (lp != lp) ? lp : fminf(lp, 0.0f);          // a log-probability is never positive
        const float s = base + step;
        const int node = t.pool_base + i;
        t.pool_token[node] = ld_cg_s32(cand_ids + (int64_t)b * ld + col0 + j);
        t.pool_parent[node] = par;
        t.pool_score[node] = s;
        s_key[i] = node_key(s, i);
    }
    if (n_new + tid < padded_keys(n_new)) s_key[n_new + tid] = 0ull;
    __syncthreads();
    for (int i = tid; i < n_new; i += nthreads) {
        const int r = rank_of(s_key, n_new, s_key[i]);
        if (r < t.n_front) t.next_frontier[r] = t.pool_base + i;
    }
}

}  // namespace
}  // namespace vt
