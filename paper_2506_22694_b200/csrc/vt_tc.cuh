// Tensor-core plumbing shared by the two head kernels: mbarrier and TMA wrappers, tcgen05 operand and
// instruction descriptors, and the host-side encoding of the tensor maps.
#pragma once
#include <cuda.h>

#include <mutex>

#include "vt_common.cuh"

namespace vt {
namespace {

constexpr int kBK = 64;                   // columns of d per tensor copy: 128 bytes, one swizzle row

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint64_t* b, int count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* b, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(b)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* b) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(b)) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint64_t* b, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
        : "=r"(ok) : "r"(smem_u32(b)), "r"(parity) : "memory");
    return ok != 0;
}
__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// One lane of a converged warp.  The single-thread roles (copy producer, MMA issuer) are entered through this and
// not through `lane == 0`: behind elect.sync the compiler knows that one thread is active and hands tcgen05 and
// copy instructions their operands in uniform registers; behind a comparison it guards every one of them against
// a divergent warp (measured: 70-105 cycles to issue an MMA of M = 128, N = 16 instead of the 40 it takes).
__device__ __forceinline__ bool elect_one() {
    uint32_t r;
    asm volatile("{ .reg .pred p; elect.sync _|p, 0xffffffff; selp.u32 %0, 1, 0, p; }" : "=r"(r));
    return r != 0;
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* tm, int x, int y, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
        ::"r"(dst), "l"(tm), "r"(x), "r"(y), "r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* tm, int x, int y, int z, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(dst), "l"(tm), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// D[tmem] (+)= A[smem] * B[smem]^T, 128 x N x 16, bf16 inputs, fp32 accumulation
__device__ __forceinline__ void tc_mma(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{ .reg .pred p; setp.ne.b32 p, %4, 0; tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p; }"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(acc) : "memory");
}

// The same with the descriptors as their lower words (what the operands' addresses change) and one common upper word: 32-bit
// additions between MMAs, which a single thread issues one after the other
__device__ __forceinline__ void tc_mma_lo(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t hi, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{ .reg .pred p; .reg .b64 a, b; mov.b64 a, {%1, %3}; mov.b64 b, {%2, %3}; setp.ne.b32 p, %5, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %4, p; }"
        ::"r"(d_tmem), "r"(a_lo), "r"(b_lo), "r"(hi), "r"(idesc), "r"(acc) : "memory");
}

// Shared-memory operand descriptor: K-major tile of 128-byte rows, 128-byte swizzle, 8-row groups
// 1024 bytes apart (the layout a TMA tensor copy with SWIZZLE_128B and a 64-column bf16 box writes).
// Fields: start address >> 4 [0,14); leading byte offset >> 4 [16,30) (unused for swizzled K-major: 1);
// stride byte offset >> 4 [32,46); descriptor version 1 at [46,48); layout type 2 = 128B swizzle at [61,64).
__device__ __forceinline__ uint64_t make_desc(uint32_t smem_addr) {
    return (uint64_t)((smem_addr >> 4) & 0x3fffu) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}
// Instruction descriptor of kind::f16: fp32 accumulator (1 at [4,6)), A and B bf16 (1 at [7,10) and
// [10,13)), both K-major (0 at bits 15 and 16), N >> 3 at [17,23), M >> 4 at [24,29).
__host__ __device__ constexpr uint32_t make_idesc(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// ---- host side ------------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

typedef CUresult (*ReplaceAddressFn)(CUtensorMap*, void*);

struct MapFns {
    EncodeTiledFn encode;
    ReplaceAddressFn replace;
};

const MapFns& map_fns() {
    static std::mutex mu;
    static MapFns fns{nullptr, nullptr};
    std::lock_guard<std::mutex> lock(mu);
    if (!fns.encode) {
        void *e = nullptr, *r = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapReplaceAddress", &r, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fns.replace = reinterpret_cast<ReplaceAddressFn>(r);
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &e, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess && fns.replace)
            fns.encode = reinterpret_cast<EncodeTiledFn>(e);
    }
    return fns;
}

// bf16 matrix [rows, cols] row-major -> boxes of kBK columns x box_rows rows, 128-byte swizzle; with steps > 0 boxes of
// `steps` of those behind one another, as a third dimension (cols a multiple of kBK).  Encoding a map
// takes the host about 2.5 us, two of them 5 of a call's 12; the last few shapes of a thread are kept encoded (a
// shape, not a matrix: the address is put in on every call, which costs a tenth of that).
bool encode_map(CUtensorMap* tm, const void* base, int rows, int cols, int box_rows, int steps = 0) {
    struct Shape {
        int rows, cols, box_rows, steps;
        CUtensorMap map;
    };
    constexpr int kShapes = 8;
    static thread_local Shape kept[kShapes] = {};
    static thread_local int next = 0;
    const MapFns& fn = map_fns();
    if (!fn.encode) return false;
    for (int i = 0; i < kShapes; ++i)
        if (kept[i].rows == rows && kept[i].cols == cols && kept[i].box_rows == box_rows && kept[i].steps == steps) {
            *tm = kept[i].map;
            return fn.replace(tm, const_cast<void*>(base)) == CUDA_SUCCESS;
        }
    cuuint64_t gdim[3] = {(cuuint64_t)(steps ? kBK : cols), (cuuint64_t)rows, (cuuint64_t)(cols / kBK)};
    cuuint64_t gstr[2] = {(cuuint64_t)cols * 2, (cuuint64_t)kBK * 2};
    cuuint32_t box[3] = {(cuuint32_t)kBK, (cuuint32_t)box_rows, (cuuint32_t)steps};
    cuuint32_t estr[3] = {1, 1, 1};
    if (fn.encode(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, steps ? 3 : 2, const_cast<void*>(base), gdim, gstr, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return false;
    kept[next] = Shape{rows, cols, box_rows, steps, *tm};
    next = (next + 1) % kShapes;
    return true;
}

}  // namespace
}  // namespace vt
