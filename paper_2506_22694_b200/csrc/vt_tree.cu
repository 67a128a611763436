// Draft-tree construction around the head (Section 4.1, Settings: the EAGLE-2 tree procedure with
// depth 3 / top-K 8 / 32 draft tokens; Table 4: 60 draft tokens in the depth ablation).  Two on-chip selections over at most
// a few thousand values: the frontier of the next depth, and the final rerank of the node pool.
// Scores are cumulative log-probabilities in fp32; ties go to the lower node index; NaN ranks last.
#include "vt_common.cuh"
#include "vt_tree_common.cuh"

namespace vt {
namespace {

constexpr int kTreeThreads = 1024;
constexpr int kTreeMax = 4096;                       // nodes one call ranks (VT_TREE_MAX_NODES)

__global__ void __launch_bounds__(kTreeThreads, 1)
k_tree_expand(const int32_t* cand_ids, const float* cand_lp, int32_t B, int32_t topk,
              int32_t ld, int32_t col0, const TreeArgs t) {
    __shared__ __align__(16) unsigned long long s_key[kTreeMax];
    griddep_launch_dependents();
    griddep_wait();
    tree_expand_block(t, cand_ids, cand_lp, B, topk, ld, col0, s_key, (int)threadIdx.x, kTreeThreads);
}

__global__ void __launch_bounds__(kTreeThreads, 1)
k_tree_rerank(const int32_t* pool_token, const int32_t* pool_parent, const float* pool_score, int32_t n,
              int32_t budget, int32_t* __restrict__ out_nodes, int32_t* __restrict__ out_token, int32_t* __restrict__ out_parent) {
    __shared__ __align__(16) unsigned long long s_key[kTreeMax];
    __shared__ uint32_t s_sel[kTreeMax / 32];        // bit i: node i is kept
    __shared__ int s_before[kTreeMax / 32];          // kept nodes in earlier words
    static_assert(kTreeMax % kKeyGroup == 0, "the padded keys fit");
    griddep_launch_dependents();
    griddep_wait();                                  // (the pool comes from the kernels before)
    const int words = (n + 31) / 32;
    for (int i = threadIdx.x; i < n; i += (int)blockDim.x) s_key[i] = node_key(ld_cg_f32(pool_score + i), i);
    if (n + (int)threadIdx.x < padded_keys(n)) s_key[n + threadIdx.x] = 0ull;
    for (int w = threadIdx.x; w < words; w += (int)blockDim.x) s_sel[w] = 0;
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += (int)blockDim.x)
        if (rank_of(s_key, n, s_key[i]) < budget) atomicOr(&s_sel[i >> 5], 1u << (i & 31));
    __syncthreads();
    if (threadIdx.x < 32) {                          // kept nodes before each word: a warp scan, 32 words at a time
        int run = 0;
        for (int w0 = 0; w0 < words; w0 += 32) {
            const int w = w0 + (int)threadIdx.x;
            const int c = w < words ? __popc(s_sel[w]) : 0;
            int incl = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, o);
                if ((int)threadIdx.x >= o) incl += y;
            }
            if (w < words) s_before[w] = run + incl - c;
            run += __shfl_sync(0xffffffffu, incl, 31);
        }
    }
    __syncthreads();
    const int m = min(budget, n);
    for (int i = threadIdx.x; i < n; i += (int)blockDim.x) {
        const uint32_t bit = 1u << (i & 31);
        if (!(s_sel[i >> 5] & bit)) continue;
        const int pos = s_before[i >> 5] + __popc(s_sel[i >> 5] & (bit - 1));
        const int32_t par = ld_cg_s32(pool_parent + i);
        int32_t ppos = -1;
        if (par >= 0) {
            const bool ok = par < n && (s_sel[par >> 5] >> (par & 31) & 1u);
            ppos = ok ? s_before[par >> 5] + __popc(s_sel[par >> 5] & ((1u << (par & 31)) - 1)) : -2;
        }
        out_nodes[pos] = i;
        out_token[pos] = ld_cg_s32(pool_token + i);
        out_parent[pos] = ppos;
    }
    for (int64_t k = m + threadIdx.x; k < budget; k += blockDim.x) {
        out_nodes[k] = -1;
        out_token[k] = -1;
        out_parent[k] = -1;
    }
}

}  // namespace

int tree_max_nodes() { return kTreeMax; }

cudaError_t launch_tree_expand(const int32_t* cand_ids, const float* cand_lp, int32_t B, int32_t topk, int32_t ld,
                               int32_t col0, const TreeArgs& t, cudaStream_t st) {
    return launch_dependent(k_tree_expand, 1, kTreeThreads, 0, st, cand_ids, cand_lp, B, topk, ld, col0, t);
}

cudaError_t launch_tree_rerank(const int32_t* pool_token, const int32_t* pool_parent, const float* pool_score,
                               int32_t n, int32_t budget, int32_t* out_nodes, int32_t* out_token,
                               int32_t* out_parent, cudaStream_t st) {
    // as many threads as there are nodes to place (a quarter of the CTA for a tree of depth 3): the rest would only meet
    // at the barriers
    const int most = n > budget ? n : budget;
    const int threads = most < kTreeThreads ? (most + 31) & ~31 : kTreeThreads;
    return launch_dependent(k_tree_rerank, 1, (unsigned)threads, 0, st, pool_token, pool_parent, pool_score, n, budget, out_nodes, out_token,
                            out_parent);
}

}  // namespace vt
