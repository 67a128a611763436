// Shared declarations of the CUDA side: control block layout, launch bookkeeping, small
// device helpers.  Nothing here is seen by the CPU oracle.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "vocabtrim.h"

namespace vt {

// First VT_CTRL_BYTES of every workspace.  Cleared once by vt_workspace_init; every kernel
// leaves `ticket` words at zero when it finishes.
struct Ctrl {
    uint32_t flags;               // sticky VT_FLAG_* bits
    uint32_t head_ticket;         // "last block" ticket of the head's merge kernel (wraps to 0)
    unsigned long long n_bad;     // ids skipped by the histogram
    unsigned long long wait_ns;   // bound of a device-side wait in nanoseconds (0 = the built-in default)
    uint32_t head_aborted;        // a CTA of the head kernel gave up on a wait: its call's merge reports and clears it
    uint32_t pad[57];
};
static_assert(sizeof(Ctrl) == VT_CTRL_BYTES, "control block size");

constexpr int kNumSMsFallback = 148;

int num_sms();                    // SM count of the current device (cached per device)
void count_launch(int n = 1);     // host-side launch counter behind vt_launch_count

// A launch that may take its seats before the kernel in front of it on the stream has finished (programmatic stream
// serialization): every kernel launched this way executes griddepcontrol.wait before it touches global memory.
template <class Kernel, class... Args>
inline cudaError_t launch_dependent(Kernel k, unsigned grid, unsigned block, size_t smem, cudaStream_t s, Args... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    count_launch();
    return cudaLaunchKernelEx(&cfg, k, args...);
}

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }
#ifdef __CUDACC__
__device__ __forceinline__ size_t align_up_dev(size_t x, size_t a) { return (x + a - 1) / a * a; }
#endif

// ---- launchers implemented in the .cu files (host functions) --------------------------------
struct HistPlan {
    bool small;            // all bins fit in one CTA's shared memory
    int parts;             // id ranges the packed kernel deals to different CTAs (0: not packed)
    size_t off_sample;     // uint32 [V]   sampled counts
    size_t off_packed;     // uint32 [V]   what the packed kernel counted (only when three bins per word fit)
    size_t off_gate;       // uint32 [4]   {recount, CTAs that have recounted, skipped ids (64 bits)}
    size_t clear_bytes;    // the scratch prefix every call zeroes
    size_t off_table;      // uint2  [ceil(V/32)] hot-bin table {bitmap word, slot base}
    size_t bytes;          // scratch after the control block
};
// scratch_bytes: what the caller has; a vocabulary that needs several id ranges is counted the packed way only
// when the scratch holds the packed counts too (hist_min_bytes does not include them)
HistPlan hist_plan(int32_t V, int64_t n, size_t scratch_bytes);
size_t hist_min_bytes(int32_t V);
bool hist_supported(int32_t V);   // V the counting kernels take (bins or lookup table fit shared memory)
cudaError_t launch_histogram(const int32_t* ids, int64_t n, int32_t V, uint32_t* counts,
                             int accumulate, Ctrl* ctrl, uint8_t* scratch, size_t scratch_bytes, cudaStream_t s);

cudaError_t launch_hist_fold(const int32_t* ids, int64_t n, int32_t V, int32_t bins, uint32_t* counts, cudaStream_t s);

size_t select_scratch_bytes(int32_t V);
cudaError_t launch_select_topk(const uint32_t* counts, int32_t V, int32_t K, int32_t* map,
                               int32_t* inv_map, uint8_t* scratch, cudaStream_t s);

size_t select_cut_scratch_bytes(int32_t V);
cudaError_t launch_select_cut(const uint32_t* counts, int32_t V, int mode, double pfrac, uint32_t min_count,
                              int32_t* map, int32_t* inv_map, int32_t* k_out, uint8_t* scratch, cudaStream_t s);

cudaError_t launch_verify_greedy(const int32_t* token, const int32_t* parent, const int32_t* target, int32_t S,
                                 int32_t N, int32_t* n_accept, int32_t* path, int32_t* emitted,
                                 unsigned long long* tokens_total, cudaStream_t st);

// One depth of the draft-tree expansion (vt_tree_expand's arguments); pool_token == nullptr: none.
struct TreeArgs {
    const int32_t* frontier;      // [B] pool index of each hidden row's node, or nullptr (the prefix)
    int32_t* pool_token;
    int32_t* pool_parent;
    float* pool_score;
    int32_t pool_base, n_front;
    int32_t* next_frontier;       // [n_front]
};

int tree_max_nodes();
cudaError_t launch_tree_expand(const int32_t* cand_ids, const float* cand_lp, int32_t B, int32_t topk, int32_t ld,
                               int32_t col0, const TreeArgs& t, cudaStream_t st);
cudaError_t launch_tree_rerank(const int32_t* pool_token, const int32_t* pool_parent, const float* pool_score,
                               int32_t n, int32_t budget, int32_t* out_nodes, int32_t* out_token,
                               int32_t* out_parent, cudaStream_t st);

cudaError_t launch_gather_rows(const uint16_t* W_full, const int32_t* map, uint16_t* W_trim,
                               int32_t V, int32_t K, int32_t d, Ctrl* ctrl, cudaStream_t s);

struct HeadArgs {
    const uint16_t* h;
    const uint16_t* W;
    const int32_t* map;
    int32_t B, K, d;
    const float* temp;
    int32_t topk;
    const float* uniforms;
    int32_t* out_ids;
    float* out_logprobs;
    float* dbg_logits;
    float* dbg_lse;
    int32_t overlap;       // launch with programmatic stream serialization (weights may be fetched early)
    TreeArgs tree;         // expansion to run on the merged top-k (pool_token == nullptr: none)
};
bool head_skinny_supported(int32_t B, int32_t d);   // shapes whose candidate lists may be VT_MAX_TOPK long
bool head_stream_takes(int32_t B, int32_t K, int32_t d);      // calls the streaming kernel is launched for
size_t head_skinny_scratch_bytes(int32_t B, int32_t K, int32_t topk);
cudaError_t launch_head_skinny(const HeadArgs& a, Ctrl* ctrl, uint8_t* scratch, cudaStream_t s);
#ifdef VT_STAMPS
size_t head_stamps_offset(int32_t B, int32_t topk);   // offset of the phase stamps in the scratch of either head
#endif

cudaError_t launch_head_merge(const HeadArgs& a, Ctrl* ctrl, float* recs, int G, bool lean, cudaStream_t s);

bool head_dense_supported(int32_t B, int32_t K, int32_t d);
bool head_dense_topk_ok(int32_t topk);
size_t head_dense_scratch_bytes(int32_t B, int32_t K, int32_t topk);
cudaError_t launch_head_dense(const HeadArgs& a, Ctrl* ctrl, uint8_t* scratch, cudaStream_t s);

// ---- device helpers ----------------------------------------------------------------------------
#ifdef __CUDACC__
// Programmatic dependent launch: let the next launch on the stream become resident / wait until the
// work this launch depends on has completed and its writes are visible (no-ops in a plain launch).
__device__ __forceinline__ void griddep_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void griddep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Streaming 128-bit load: read-only path, do not keep the line in L1 (data is used once).
__device__ __forceinline__ uint4 ld_stream_u4(const void* p) {
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.L2::128B.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p));
    return v;
}
// The same by an ordinary (coherent) load, for data that a kernel in front may have written while this one was resident.
__device__ __forceinline__ uint4 ld_once_u4(const void* p) {
    uint4 v;
    asm volatile("ld.global.L1::no_allocate.L2::128B.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p)
                 : "memory");
    return v;
}
__device__ __forceinline__ void st_stream_u4(void* p, uint4 v) {
    asm volatile("st.global.cs.v4.u32 [%0], {%1,%2,%3,%4};" ::"l"(p), "r"(v.x), "r"(v.y),
                 "r"(v.z), "r"(v.w)
                 : "memory");
}
// Loads through L2: what other CTAs of the same grid have written, and in a dependent launch the results of the kernels in
// front of it.  Such a launch may be resident while they still write, so their results are neither constant during the
// kernel (which the non-coherent path of __ldg and of const __restrict__ pointers takes for granted) nor to be read
// before griddep_wait (volatile, as that is: the two keep their order).
__device__ __forceinline__ uint32_t ld_cg_u32(const uint32_t* p) {
    uint32_t v;
    asm volatile("ld.global.cg.u32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ uint2 ld_cg_u2(const uint2* p) {
    uint2 v;
    asm volatile("ld.global.cg.v2.u32 {%0,%1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
    return v;
}
__device__ __forceinline__ float ld_cg_f32(const float* p) {
    float v;
    asm volatile("ld.global.cg.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ int ld_cg_s32(const int* p) {
    int v;
    asm volatile("ld.global.cg.s32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ unsigned lanemask_lt() {
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}
#endif

}  // namespace vt
