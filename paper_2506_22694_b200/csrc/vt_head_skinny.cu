// Trimmed LM head for up to 64 hidden rows, fused with its sampling epilogue (Algorithm 2, the
// drafter-forward and index-mapping steps: drafter head over the trimmed vocabulary, then the index mapper).
//
// HBM-bound: the only large operand is W_trim [K,d] bf16, read exactly once.  Every CTA owns a contiguous
// slab of vocabulary rows (K / grid of them, equal to within one row) and walks it in tiles of at most 128
// rows.  The contraction runs on the 5th-generation tensor cores with the VOCABULARY rows as the M operand:
//
//   D[j, b] = sum_i W_trim[j, i] * h[b, i]     M = vocabulary rows of a tile (the TMEM lanes),
//                                              N = hidden rows (TMEM columns), K-loop over d in 64-column steps
//
// so a weight is moved once (TMA into a shared-memory ring, 128-byte swizzle, where the MMA reads it in place)
// and no register, no shuffle and no partial tile of another warp ever sees it.  Warp 0 feeds the ring (a
// stage = up to four 64-column steps of the tile's rows and of h), one thread of warp 1 issues the MMAs (up to eight
// hidden rows: it and one of the last warp, every other stage each).
// fp32 accumulation inside the tensor core is a long serial sum, so d is cut into phases of eight steps and a
// phase's 32 MMAs go to up to eight accumulators in turn (TMEM columns are plentiful); the epilogue adds the
// accumulators up in fp32 registers, phase by phase, while the next phase's MMAs fill the other set.
//
// Epilogue warps read their TMEM lanes (lane = vocabulary row) and turn the finished tile around in shared
// memory; then warp w owns hidden rows w, w + EW, ...: its lanes walk the tile's rows, updating running
// max / sum-exp of z = logit / T, the Gumbel-max candidate from the caller's uniforms and the row's sorted
// top-k list.  Logits never go to HBM.  Each CTA leaves one small record per hidden row; a second kernel, one
// block per row, merges them in CTA order, remaps trimmed indices through `map` and writes the outputs
// (vt_head_dense.cu).  It takes its seats while this one runs, and a CTA here is gone as soon as its record is
// written, which lets the next step's weights in; the merge by the last CTA to finish (atomic ticket) kept them
// out for its 4-6 us (us per chained step, one CTA / second kernel: 1 row of 5000 x 2048 14.8 / 11.7, 10 rows of
// 32768 x 4096 46.1 / 43.5; one launch more on the host).
//
// What bounds it: the HBM read of W_trim (201 MB, cold: 35.0-36.7 us per chained step by box = 0.84-0.88 of the measured
// copy rate; the warp-level MMA kernel before it 38.3-39.8) and, for small heads, a fixed chain of about 8 us: h by TMA
// 0.5, two threads' issue of the MMAs (about 45 cycles each), epilogue 2, merge and two launch dependencies 5.
//
// Every wait is bounded: on expiry the CTA raises VT_FLAG_TIMEOUT, lets its own copies and MMAs finish and leaves.
#include <math_constants.h>

#include <type_traits>

#include "vt_common.cuh"
#include "vt_head_common.cuh"
#include "vt_tc.cuh"

namespace vt {

namespace {

constexpr int kBM = 128;                         // vocabulary rows per tile at most (TMEM lanes)
constexpr int kMaxStages = 16;
constexpr int kMaxSub = 4;                       // 64-column steps of d one ring stage holds at most
constexpr int kPhase = 8;                        // 64-column steps of d accumulated in one accumulator set
constexpr int kSetCols = 128;                    // TMEM columns of an accumulator set (two sets)
constexpr uint32_t kTmemCols = 2 * kSetCols;     // (half of the SM's: two CTAs of consecutive launches may be resident together)
constexpr int kMaxB = 64;
// Dynamic shared memory at most: what an SM has less 1 KB per block, the static part and a block of the merge kernel, which
// has its seat while the next step's CTAs come in.  Where it did not fit beside them, the CTAs of the SMs it sits on
// started 2-3 us after all others (one row, L2: 5000 x 3072 12.9 -> 11.7 us, 5000
// x 4096 14.6 -> 13.2).
constexpr size_t kSmemLimit = 228 * 1024 - (1024 + 512) - (kMergeStageWords * 4 + 1024 + 128);
constexpr unsigned long long kWaitLimitNs = 2000000000ull;   // default bound of a device-side wait (Ctrl::wait_ns overrides)

// Phase stamps (-DVT_STAMPS builds only): one thread per role writes %globaltimer at fixed points into
// a region behind the records; bench.py --case stamps reads them back.  Slots: 0 entry, 1 ring fill
// requested, 2 released by the launch dependency, 3 first stage landed, 4 last accumulators complete,
// 5 record written, 6 all warps done, 11 SM id; CTA 0 also carries the merge
// kernel's 12 start and 13 end for hidden row 0.
#ifdef VT_STAMPS
#define VT_STAMP(slot) do { stamps[(size_t)blockIdx.x * kStampSlots + (slot)] = global_ns(); } while (0)
#else
#define VT_STAMP(slot) do {} while (0)
#endif

struct Geo {
    int grid;          // CTAs
    int n_tiles;       // tiles per CTA
    int rows;          // vocabulary rows of a tile (rows of one W copy)
    int mma_rows;      // M of the MMA: 64 where a tile has no more rows, else 128
    int n_kc;          // 64-column steps of d, rounded up to a multiple of comb
    int comb;          // steps an MMA takes side by side (see make_geo)
    int pitch;         // vocabulary rows from one step's W part to the next one's
    int h_steps;       // steps of h one copy brings: a whole stage's, or one
    int sub;           // steps per ring stage
    int spp;           // ring stages accumulated in one accumulator set: a phase
    int issuers;       // warps that issue MMAs, stages dealt to them in turn (see make_geo)
    int n_stages;      // ring depth
    int h_bytes;       // shared memory of a step's h part (a multiple of 1024)
    int step_bytes;    // ... of a step: W part + h part; a stage holds its W parts and behind them its h parts
    int ring_bytes;
    int buf_bytes;     // selection buffers of the epilogue warps
    uint32_t keep;     // bit g & 31: the weights of fill g keep their L2 lines
};

// ---- bounded waits ---------------------------------------------------------------------------------
// non-blocking probe of a phase (try_wait may suspend the thread for a system-chosen time before it answers)
__device__ __forceinline__ bool mbar_test(uint64_t* b, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{ .reg .pred p; mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
        : "=r"(ok) : "r"(smem_u32(b)), "r"(parity) : "memory");
    return ok != 0;
}
// The bound of a wait is kept with the SM's cycle counter (reading the nanosecond timer costs far more
// than a probe): two cycles per nanosecond, i.e. at least the time asked for at any SM clock up to
// 2 GHz.  It lives in shared memory and is looked at only once a wait has to spin.  Bounds under a
// millisecond spin on non-blocking probes only: try_wait may park the thread for a system-chosen time before
// it answers, which is what a long wait wants and a short bound cannot afford.
__device__ __forceinline__ long long bound_cycles(unsigned long long ns) {
    return (long long)(ns < (1ull << 61) ? 2 * ns : (1ull << 62));
}
constexpr long long kShortBoundCycles = 2000000;      // 1 ms
// Bounded wait of one thread; false when the CTA is aborting or the bound expired (which starts an abort).  A role that
// waits before the launch dependency is released passes `released`: earlier work on the stream does not count, the clock
// starts when that flag is up (until then the bound is a thousand times the default).
__device__ __forceinline__ bool mbar_wait(uint64_t* b, uint32_t parity, volatile int* abort_flag, const long long* bound,
                                          volatile int* released = nullptr) {
    if (mbar_test(b, parity)) return true;
    bool counts = !released || *released;
    long long t0 = clock64();
    for (;;) {
        const long long lim = counts ? *bound : 1000 * bound_cycles(kWaitLimitNs);
        const bool nb = lim < kShortBoundCycles;
#pragma unroll 1
        for (int i = 0; i < 64; ++i) {
            if (nb ? mbar_test(b, parity) : mbar_try(b, parity)) return true;
            if (nb && clock64() - t0 > lim) break;
        }
        if (*abort_flag) return false;
        if (!counts && *released) { counts = true; t0 = clock64(); continue; }
        if (clock64() - t0 > lim) { *abort_flag = 1; return false; }
    }
}
// Same, called by all 32 lanes of a warp: lane 0 polls (a CTA of polling threads takes shared-memory and issue
// slots from what it waits for), then every lane observes the completed phase itself.  The outcome is voted on,
// so the lanes never part ways before a warp-collective instruction.
__device__ __forceinline__ bool mbar_wait_warp(uint64_t* b, uint32_t parity, volatile int* abort_flag, const long long* bound) {
    int ok = 1;
    if ((threadIdx.x & 31) == 0) ok = mbar_wait(b, parity, abort_flag, bound) ? 1 : 0;
    ok = __shfl_sync(0xffffffffu, ok, 0);
    if (ok) ok = mbar_try(b, parity) ? 1 : 0;
    return __all_sync(0xffffffffu, ok != 0);
}
// before the CTA leaves: what is in flight gets this long to finish
__device__ __forceinline__ void drain_wait(uint64_t* b, uint32_t parity) {
    if (mbar_try(b, parity)) return;                     // (the usual case; reading the timer costs 0.1 us)
    const unsigned long long t0 = global_ns();
    while (!mbar_try(b, parity) && global_ns() - t0 < kWaitLimitNs) {}
}

// eight times four consecutive accumulator columns of this thread's TMEM lane (the wait sits in the same
// statement: nothing that uses the values can be moved in front of it)
__device__ __forceinline__ void tc_ld_8x4(const uint32_t (&ad)[8], float (&r)[8][4]) {
    uint32_t v[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%32];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%4,%5,%6,%7}, [%33];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%8,%9,%10,%11}, [%34];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%12,%13,%14,%15}, [%35];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%16,%17,%18,%19}, [%36];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%20,%21,%22,%23}, [%37];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%24,%25,%26,%27}, [%38];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%28,%29,%30,%31}, [%39];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=&r"(v[0]), "=&r"(v[1]), "=&r"(v[2]), "=&r"(v[3]), "=&r"(v[4]), "=&r"(v[5]), "=&r"(v[6]), "=&r"(v[7]),
          "=&r"(v[8]), "=&r"(v[9]), "=&r"(v[10]), "=&r"(v[11]), "=&r"(v[12]), "=&r"(v[13]), "=&r"(v[14]), "=&r"(v[15]),
          "=&r"(v[16]), "=&r"(v[17]), "=&r"(v[18]), "=&r"(v[19]), "=&r"(v[20]), "=&r"(v[21]), "=&r"(v[22]), "=&r"(v[23]),
          "=&r"(v[24]), "=&r"(v[25]), "=&r"(v[26]), "=&r"(v[27]), "=&r"(v[28]), "=&r"(v[29]), "=&r"(v[30]), "=&r"(v[31])
        : "r"(ad[0]), "r"(ad[1]), "r"(ad[2]), "r"(ad[3]), "r"(ad[4]), "r"(ad[5]), "r"(ad[6]), "r"(ad[7])
        : "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) r[i >> 2][i & 3] = __uint_as_float(v[i]);
}

// ---- top-k list of one hidden row ------------------------------------------------------------------
constexpr int kBufKeys = VT_MAX_TOPK + kBM + 4;       // a warp's selection buffer: list, candidates, padding

// Warp-cooperative selection: buf holds the keys of a sorted list and behind them candidate keys, N in all; the
// best min(topk, N) of them become the new sorted list (descending; keys order by value, then lower index).  Every
// element's final position is its rank -- the number of elements that beat it -- so there are no sequential
// selection rounds: each lane keeps up to NS elements in registers while all of them stream by as broadcast
// 128-bit shared-memory reads, several in flight.
template <int NS>
__device__ __forceinline__ void rank_scatter(unsigned long long* list, const unsigned long long* buf, int N, int topk) {
    const int lane = threadIdx.x & 31;
    unsigned long long ek[NS];
    int rk[NS];
#pragma unroll
    for (int i = 0; i < NS; ++i) {
        ek[i] = lane + 32 * i < N ? buf[lane + 32 * i] : 0ull;
        rk[i] = 0;
    }
    rank_among<NS>(buf, N, ek, rk);
#pragma unroll
    for (int i = 0; i < NS; ++i)
        if (lane + 32 * i < N && rk[i] < topk) list[rk[i]] = ek[i];
}

// One lane's state of one hidden row over the vocabulary rows it has seen.
struct RowState {
    float m, s;        // running max and sum of exp(z - m)
    float gs, gz;      // best Gumbel score and its z
    int gj;
};

// The variant of up to eight hidden rows may have a second warp for the MMAs (the last one; see make_geo).  With sixteen
// epilogue warps one more slows them down by more than it gives (9 rows of 12000 x 2048 13.3 us without, 15.8 with it).
__host__ __device__ constexpr int max_issuers(int ew) { return ew == 8 ? 2 : 1; }

// EW epilogue warps (a multiple of 4: the warps of a lane quadrant share the accumulator columns), at most RPW hidden
// rows per epilogue warp.  COMB: an MMA takes several steps of d side by side (see make_geo).
template <int EW, int RPW, bool COMB>
__global__ void __launch_bounds__((EW + 1 + max_issuers(EW)) * 32, EW == 8 ? 2 : 1)
k_head_stream(const HeadArgs a, Ctrl* ctrl, float* __restrict__ recs, const Geo geo,
              const __grid_constant__ CUtensorMap tm_h, const __grid_constant__ CUtensorMap tm_w) {
    extern __shared__ uint8_t s_dyn[];
    __shared__ uint64_t s_full[kMaxStages], s_empty[kMaxStages], s_acc_full[2], s_acc_empty[2], s_drain;
    __shared__ uint32_t s_tmem_base;
    __shared__ int s_abort;
    __shared__ int s_issued[2];                          // ring stages each issuer has released
    __shared__ int s_released;                           // the launch dependency is
    __shared__ long long s_bound;                        // bound of a wait in SM cycles
    // An accumulator set holds kAccs accumulators of kNpad columns (hidden rows).  The kParts warps of a lane quadrant
    // take kUnits groups of four columns each: always eight loads per warp and phase.
    constexpr int kParts = EW / 4, kUnits = RPW, kAccs = 8 / kUnits, kNpad = 16 * kUnits, kIssuers = max_issuers(EW);
    static_assert(kAccs * kNpad <= kSetCols && kParts * kUnits * 4 <= kNpad, "a set's columns");
    // Steps side by side: a set holds c_accs accumulators of c_cols columns, kNrow of them per step.
    constexpr int kNrow = EW;                            // (8 or 16 hidden rows at most)
    const int c_cols = (geo.comb == 2 ? 2 : 4) * kNrow, c_accs = min(4, kSetCols / c_cols);
    const int B = a.B, K = a.K, topk = a.topk;
    uint8_t* ring = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(s_dyn) + 1023) & ~(uintptr_t)1023);
    const uint32_t ring_u32 = smem_u32(ring);
    float* zt = reinterpret_cast<float*>(ring + geo.ring_bytes);                                  // [B][kBM]: a tile's logits, row by row
    unsigned long long* lists = reinterpret_cast<unsigned long long*>(zt + B * kBM);              // [B][topk]
    unsigned long long* bufs = lists + ((B * topk + 1) & ~1);                                     // [min(EW, B)][kBufKeys]
    RowState* states = reinterpret_cast<RowState*>(reinterpret_cast<uint8_t*>(bufs) + geo.buf_bytes);     // [B][32]
    float* s_invT = reinterpret_cast<float*>(states + B * 32);                                    // [B] 1 / T, NaN for an unusable temperature
    int* s_cnt = reinterpret_cast<int*>(s_invT + B);                                              // [B] entries in the row's list

    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int r0 = (int)((long long)K * blockIdx.x / gridDim.x);
    const int r1 = (int)((long long)K * (blockIdx.x + 1) / gridDim.x);
#ifdef VT_STAMPS
    unsigned long long* stamps = reinterpret_cast<unsigned long long*>(
        reinterpret_cast<uint8_t*>(recs) + align_up_dev((size_t)kMaxGrid * B * rec_fields(topk) * 4, 256));
    if (threadIdx.x == 0) {
        unsigned smid;
        asm volatile("mov.u32 %0, %%smid;" : "=r"(smid));
        stamps[(size_t)blockIdx.x * kStampSlots + 11] = smid;
        VT_STAMP(0);
    }
#endif
    if (threadIdx.x == 0) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tm_w)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tm_h)) : "memory");
        for (int s = 0; s < geo.n_stages; ++s) { mbar_init(&s_full[s], 1); mbar_init(&s_empty[s], 1); }
        for (int p = 0; p < 2; ++p) { mbar_init(&s_acc_full[p], geo.issuers); mbar_init(&s_acc_empty[p], EW); }
        mbar_init(&s_drain, geo.issuers);
        s_abort = 0;
        s_issued[0] = s_issued[1] = 0;
        s_released = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (threadIdx.x == 64) {                             // (beside the barriers' and the tensor memory's set-up, which take as long)
        // the caller's bound, 0 = the default: written with the host waiting for it, so it is final before any later launch
        const unsigned long long ns = *reinterpret_cast<volatile unsigned long long*>(&ctrl->wait_ns);
        s_bound = bound_cycles(ns ? ns : kWaitLimitNs);
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(&s_tmem_base)), "r"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = s_tmem_base;
    volatile int* abort_flag = &s_abort;
    // Programmatic dependent launch (a no-op unless the launch asked for it): the next kernel on the stream
    // may become resident as soon as its resources are free (this CTA has its tensor memory by now), and this
    // kernel goes no further than fetching weights until everything enqueued before it has completed.
    griddep_launch_dependents();

    if (warp == 0) {
        // ================= TMA producer ================================================================
        if (elect_one()) {
            const int sub = geo.sub, S = geo.n_stages;
            const int n_ks = (geo.n_kc + sub - 1) / sub;               // ring stages per tile
            const int total = geo.n_tiles * n_ks;
            // bytes that land: per step, and per stage (h in one copy: all its rows and steps, zeros where there are none)
            const bool h_whole = RPW == 1 && geo.h_steps > 1;
            const uint32_t step_tx = (uint32_t)(geo.rows + (h_whole ? 0 : B)) * (kBK * 2);
            const uint32_t stage_tx = h_whole ? (uint32_t)(geo.h_steps * geo.h_bytes) : 0u;
            const uint32_t w_step = (uint32_t)geo.pitch * (kBK * 2), h_step = (uint32_t)geo.h_bytes;
            const uint32_t stage_bytes = (uint32_t)(sub * geo.step_bytes), h_off = (uint32_t)sub * w_step;
            // W_trim is read once per call: its lines are the first to go when L2 needs room, so that the records, the
            // index mapper, h and the uniforms stay resident from step to step -- except for the share of it that a
            // drafting loop finds in L2 again at its next step (see make_geo)
            uint64_t first_policy, keep_policy;
            asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(first_policy));
            asm("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(keep_policy));
            auto load_w = [&](uint32_t dst, int x, int y, uint64_t* bar, int g) {
                asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint"
                             " [%0], [%1, {%2, %3}], [%4], %5;"
                             ::"r"(dst), "l"(&tm_w), "r"(x), "r"(y), "r"(smem_u32(bar)),
                               "l"(((geo.keep >> (g & 31)) & 1u) ? keep_policy : first_policy) : "memory");
            };
            // The weights are static: the first ring of them is requested before the work this launch
            // depends on has finished; everything that work may have produced is touched after the wait.
            const int pre = min(S, total);
            {
                int ks = 0, y = r0;
                for (int g = 0; g < pre; ++g) {
                    const int subs = min(sub, geo.n_kc - ks * sub);
                    mbar_expect_tx(&s_full[g], stage_tx + step_tx * (uint32_t)subs);
                    for (int u = 0; u < subs; ++u)
                        load_w(ring_u32 + (uint32_t)g * stage_bytes + (uint32_t)u * w_step, (ks * sub + u) * kBK, y, &s_full[g], g);
                    if (++ks == n_ks) { ks = 0; y += geo.rows; }
                }
            }
            VT_STAMP(1);
            griddep_wait();
            *const_cast<volatile int*>(&s_released) = 1;
            VT_STAMP(2);
            {
                int ks = 0;
                for (int g = 0; g < pre; ++g) {
                    if (h_whole) {
                        tma_load_3d(ring_u32 + (uint32_t)g * stage_bytes + h_off, &tm_h, 0, 0, ks * sub, &s_full[g]);
                        if (++ks == n_ks) ks = 0;
                        continue;
                    }
                    const int subs = min(sub, geo.n_kc - ks * sub);
                    for (int u = 0; u < subs; ++u)
                        tma_load_2d(ring_u32 + (uint32_t)g * stage_bytes + h_off + (uint32_t)u * h_step, &tm_h, (ks * sub + u) * kBK, 0, &s_full[g]);
                    if (++ks == n_ks) ks = 0;
                }
            }
            int done = pre;
            {
                // steady state: the cursor over (stage, step in d, tile) moves by additions only
                int sc = pre == S ? 0 : pre, ks = pre % n_ks, y = r0 + (pre / n_ks) * geo.rows;
                uint32_t par = 0;                                   // fill g waits for the release of fill g - S
                for (int g = pre; g < total; ++g, ++done) {
                    if (!mbar_wait(&s_empty[sc], par, abort_flag, &s_bound)) break;
                    const int subs = min(sub, geo.n_kc - ks * sub);
                    mbar_expect_tx(&s_full[sc], stage_tx + step_tx * (uint32_t)subs);
                    const uint32_t dst0 = ring_u32 + (uint32_t)sc * stage_bytes;
                    if (h_whole) tma_load_3d(dst0 + h_off, &tm_h, 0, 0, ks * sub, &s_full[sc]);
#pragma unroll
                    for (int u = 0; u < kMaxSub; ++u) {
                        if (u < subs) {
                            const int x = (ks * sub + u) * kBK;
                            load_w(dst0 + (uint32_t)u * w_step, x, y, &s_full[sc], g);
                            if (!h_whole) tma_load_2d(dst0 + h_off + (uint32_t)u * h_step, &tm_h, x, 0, &s_full[sc]);
                        }
                    }
                    if (++sc == S) { sc = 0; par ^= 1u; }
                    if (++ks == n_ks) { ks = 0; y += geo.rows; }
                }
            }
            // Every copy asked for has landed before the CTA may leave, whatever the other roles do from here on: a wait of
            // theirs may expire after this thread's last request, and then nobody else looks at these stages again.  (The last
            // fill of a stage is its barrier's last phase; in an undisturbed run the MMAs finish later than this.)
            for (int g = max(0, done - S); g < done; ++g) drain_wait(&s_full[g % S], (uint32_t)((g / S) & 1));
        }
    } else if (warp == 1 || (kIssuers == 2 && warp == EW + 2)) {
        // ================= MMA issuers =================================================================
        const int me = warp == 1 ? 0 : 1, ni = geo.issuers;
        if (me < ni && elect_one()) {
            const int comb = geo.comb;
            const uint32_t idesc = make_idesc(geo.mma_rows, COMB ? c_cols : kNpad);
            // (the ring is 1024-byte aligned and under 256 KB: adding byte offsets >> 4 stays inside the address field;
            // rows of an operand beyond the tile's / beyond B are whatever lies behind it: their TMEM lanes and columns
            // are not looked at)
            const uint64_t desc_h0 = make_desc(ring_u32);
            const uint32_t desc_lo = (uint32_t)desc_h0, desc_hi = (uint32_t)(desc_h0 >> 32);
            const uint32_t w16 = (uint32_t)geo.pitch * (kBK * 2 / 16), h16 = (uint32_t)(geo.h_bytes >> 4);      // operand steps >> 4
            const int S = geo.n_stages, sub = geo.sub;
            const int n_ks = (geo.n_kc + sub - 1) / sub, spp = geo.spp;            // ring stages per tile / per phase
            const int total = geo.n_tiles * n_ks;
            // Every MMA of a stage: consecutive ones go to this issuer's N accumulators (from column d on) in turn, the first
            // round of a phase overwrites.  in_phase: this issuer's steps in the phase so far.  Accumulators and flags are
            // constants of the unrolled code (an odd step swaps the halves of eight accumulators).
            auto issue = [&](auto accs, uint32_t d, uint32_t w_lo, uint32_t h_lo, int subs, int in_phase) {
                constexpr int N = decltype(accs)::value;
                const uint32_t odd = N > 4 ? (uint32_t)(in_phase & 1) * (4 * kNpad) : 0u;
                const uint32_t d_even = d + odd, d_odd = N > 4 ? d + 4 * kNpad - odd : d;
                auto steps = [&](auto later) {
#pragma unroll
                    for (int u = 0; u < kMaxSub; ++u)
                        if (u < subs) {
#pragma unroll
                            for (int k = 0; k < kBK / 16; ++k)
                                tc_mma_lo(((u & 1) ? d_odd : d_even) + (uint32_t)((k % N) * kNpad), w_lo + (uint32_t)u * w16 + (uint32_t)(2 * k),
                                          h_lo + (uint32_t)u * h16 + (uint32_t)(2 * k), desc_hi, idesc,
                                          (decltype(later)::value || u * (kBK / 16) + k >= N) ? 1u : 0u);
                        }
                };
                if (in_phase * (kBK / 16) >= N) steps(std::true_type{}); else steps(std::false_type{});
            };
            // The same with `comb` steps side by side: an MMA's vocabulary rows are those of `comb` W parts, its columns those
            // of as many h parts, and of the product only the blocks on the diagonal are looked at.
            const int my_accs = c_accs / ni;
            auto issue_comb = [&](uint32_t d, uint32_t w_lo, uint32_t h_lo, int subs, int in_phase) {
                d += (uint32_t)(me * my_accs * c_cols);
#pragma unroll
                for (int g = 0; g < kMaxSub / 2; ++g) {
                    if (g * comb < subs) {
#pragma unroll
                        for (int k = 0; k < kBK / 16; ++k)
                            tc_mma_lo(d + (uint32_t)((k & (my_accs - 1)) * c_cols), w_lo + (uint32_t)(2 * k), h_lo + (uint32_t)(2 * k), desc_hi, idesc,
                                      in_phase + g > 0 || k >= my_accs ? 1u : 0u);
                        w_lo += (uint32_t)comb * w16;
                        h_lo += (uint32_t)comb * h16;
                    }
                }
            };
            // (no griddep_wait here: h is asked for after it, so no stage is complete before; waking up from it costs 0.3 us
            // that a probe on the stage does not)
            int s = me, own = me, first = 0, set_no = 0;            // own: this issuer's next stage, first: the phase's first
            uint32_t ph = 0;
            bool alive = true;
            for (int t = 0; t < geo.n_tiles && alive; ++t) {
                for (int ks0 = 0; ks0 < n_ks && alive; ks0 += spp) {
                    // a new accumulator set: the epilogue has read what it held
                    if (set_no >= 2 && !mbar_wait(&s_acc_empty[set_no & 1], (uint32_t)(((set_no >> 1) - 1) & 1), abort_flag, &s_bound)) {
                        alive = false;
                        break;
                    }
                    const uint32_t d_tmem = tmem_base + (uint32_t)((set_no & 1) * kSetCols);
                    const int end = first + min(spp, n_ks - ks0);
                    int in_phase = 0;
                    for (; own < end; own += ni) {
                        if (!mbar_wait(&s_full[s], ph, abort_flag, &s_bound, &s_released)) { alive = false; break; }
#ifdef VT_STAMPS
                        if (own == 0) VT_STAMP(3);
#endif
                        tc_fence_after();
                        const int subs = min(sub, geo.n_kc - (ks0 + own - first) * sub);
                        const uint32_t w_lo = desc_lo + ((uint32_t)(s * sub * geo.step_bytes) >> 4), h_lo = w_lo + (uint32_t)sub * w16;
                        if (COMB)
                            issue_comb(d_tmem, w_lo, h_lo, subs, in_phase);
                        else if (kIssuers == 2 && ni == 2)
                            issue(std::integral_constant<int, kAccs / 2>{}, d_tmem + (uint32_t)(me * (kAccs / 2) * kNpad), w_lo, h_lo, subs, in_phase);
                        else
                            issue(std::integral_constant<int, kAccs>{}, d_tmem, w_lo, h_lo, subs, in_phase);
                        in_phase += subs;
                        tc_commit(&s_empty[s]);                     // the stage is free once these MMAs have read it
                        s += ni;
                        if (s >= S) { s -= S; ph ^= 1u; }
                    }
                    if (alive) tc_commit(&s_acc_full[set_no & 1]);  // this issuer's part of the phase's accumulators is complete
                    first = end;
                    ++set_no;
                }
            }
            s_issued[me] = (own - me) / ni;
            // every MMA issued has finished and every commit has arrived before the CTA may leave (a stage's last release: its
            // barrier moves no further)
            tc_commit(&s_drain);
            drain_wait(&s_drain, 0);
            if (alive)
                for (int g = own - ni; g >= max(0, total - S); g -= ni) drain_wait(&s_empty[g % S], (uint32_t)((g / S) & 1));
        }
    } else {
        // ================= epilogue warps ==============================================================
        const int e = warp - 2;
        const int quad = warp & 3;                                  // TMEM lanes this warp may read
        const int qrows = geo.mma_rows / 4;                         // vocabulary rows in them (M = 64 fills the first 16 of 32)
        const int part = e >> 2;                                    // which accumulator columns of the quadrant
        unsigned long long* buf = bufs + (size_t)(e < B ? e : 0) * kBufKeys;     // (used only by warps that own a row: e < B)
        for (int b = e; b < B; b += EW) {
            states[b * 32 + lane] = RowState{-CUDART_INF_F, 0.f, -CUDART_INF_F, 0.f, -1};
            if (lane == 0) s_cnt[b] = 0;
        }
        griddep_wait();                                             // temp, uniforms and the record scratch belong to earlier work until here
        for (int b = e; b < B; b += EW) {
            const float T = a.temp[b];
            if (lane == 0) s_invT[b] = (T > 0.f) && (T < CUDART_INF_F) ? 1.f / T : CUDART_NAN_F;
        }
        __syncwarp();
        const int n_ks = (geo.n_kc + geo.sub - 1) / geo.sub, spp = geo.spp;     // ring stages per tile / per phase
        const int n_ph = (n_ks + spp - 1) / spp;
        // steps side by side: this warp's TMEM lanes belong to one step's rows or to two's
        const int comb = COMB ? geo.comb : 1;
        const int step_a = COMB ? quad * 32 / geo.pitch : 0, step_b = COMB ? min((quad * 32 + 31) / geo.pitch, comb - 1) : 0;
        const bool in_b = quad * 32 + lane >= step_b * geo.pitch;
        int set_no = 0;
        for (int t = 0; t < geo.n_tiles; ++t) {
            const int j0 = r0 + t * geo.rows;                       // first vocabulary row of the tile
            const int nrow = min(geo.rows, r1 - j0);                // rows of it that are this CTA's
            float un[4];                                            // the next row's uniforms; the first row's are requested before the MMAs are waited for
            auto load_u = [&](int b) {
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    un[i] = (a.uniforms && b < B && lane + 32 * i < nrow) ? a.uniforms[(size_t)b * K + j0 + lane + 32 * i] : 0.5f;
            };
            load_u(e);
            // the accumulators of the tile, phase by phase, added up per (vocabulary row = lane, hidden row = column)
            float x[kUnits][4];
#pragma unroll
            for (int i = 0; i < kUnits; ++i)
#pragma unroll
                for (int q = 0; q < 4; ++q) x[i][q] = 0.f;
            bool ok = true;
            for (int p = 0; p < n_ph; ++p, ++set_no) {
                const int set = set_no & 1;
                ok = mbar_wait_warp(&s_acc_full[set], (uint32_t)((set_no >> 1) & 1), abort_flag, &s_bound);
                if (!ok) break;
                tc_fence_after();
                if (COMB) {
                    if (quad * 32 < comb * geo.pitch && part * 4 < B) {
                        const uint32_t base = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(set * kSetCols + part * 4);
                        uint32_t ad[8];
                        float v[8][4];
#pragma unroll
                        for (int i = 0; i < 8; ++i) ad[i] = base + (uint32_t)((i & (c_accs - 1)) * c_cols + (i < 4 ? step_a : step_b) * kNrow);
                        tc_ld_8x4(ad, v);
                        // (a short last phase of one stage: the other issuer's accumulators hold nothing)
                        const bool one = kIssuers == 2 && geo.issuers == 2 && n_ks - p * spp == 1;
                        const int c0 = one && ((p * spp) & 1) ? c_accs / 2 : 0, c1 = one ? c0 + c_accs / 2 : c_accs;
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            float w[4];
#pragma unroll
                            for (int c = 0; c < 4; ++c) w[c] = c >= c0 && c < c1 ? (in_b ? v[4 + c][q] : v[c][q]) : 0.f;
                            x[0][q] += (w[0] + w[2]) + (w[1] + w[3]);
                        }
                    }
                } else if (quad * qrows < nrow && part * 4 < B) {
                    const uint32_t base = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(set * kSetCols + part * 4);
                    uint32_t ad[8];
                    float v[8][4];
#pragma unroll
                    for (int i = 0; i < 8; ++i) ad[i] = base + (uint32_t)((i % kAccs) * kNpad + (i / kAccs) * kParts * 4);
                    tc_ld_8x4(ad, v);
                    // (an accumulator that a short last phase did not get to holds nothing: those beyond its MMAs or, where
                    // it is one stage, the half of the issuer that had no stage; the others pairwise: fewer roundings in a
                    // row than one after the other)
                    int c0 = 0, c1 = min(kPhase, geo.n_kc - p * kPhase) * (kBK / 16);
                    if (kIssuers == 2 && geo.issuers == 2) {
                        const bool one = n_ks - p * spp == 1;
                        c0 = one && ((t * n_ks + p * spp) & 1) ? kAccs / 2 : 0;
                        c1 = one ? c0 + kAccs / 2 : kAccs;
                    }
#pragma unroll
                    for (int q = 0; q < 4; ++q)
#pragma unroll
                        for (int i = 0; i < kUnits; ++i) {
                            float w[kAccs];
#pragma unroll
                            for (int c = 0; c < kAccs; ++c) w[c] = c >= c0 && c < c1 ? v[i * kAccs + c][q] : 0.f;
#pragma unroll
                            for (int o = kAccs / 2; o; o >>= 1)
#pragma unroll
                                for (int c = 0; c < o; ++c) w[c] += w[c + o];
                            x[i][q] += w[0];
                        }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&s_acc_empty[set]);
            }
            if (ok) {
#ifdef VT_STAMPS
                if (e == 0 && lane == 0) VT_STAMP(4);
#endif
                if (COMB ? quad * 32 < comb * geo.pitch : quad * qrows < nrow && lane < qrows) {
#pragma unroll
                    for (int i = 0; i < kUnits; ++i)
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const int b = (part + i * kParts) * 4 + q;
                            if (b < B) zt[(size_t)b * kBM + quad * qrows + lane] = x[i][q];
                        }
                }
            }
            {   // every epilogue warp has written its part, and all of them agree whether to go on
                int all_ok;
                asm volatile("{ .reg .pred p, q; setp.ne.s32 p, %1, 0; bar.red.and.pred q, 1, %2, p; selp.s32 %0, 1, 0, q; }"
                             : "=r"(all_ok) : "r"(ok ? 1 : 0), "n"(EW * 32) : "memory");
                if (!all_ok) break;
            }
            // ---- the warp's hidden rows over this tile.  (A rolled loop, with the per-lane state in shared memory:
            // unrolled over the rows its code would be fetched anew for every row.)
#pragma unroll 1
            for (int b = e; b < B; b += EW) {
                const float u[4] = {un[0], un[1], un[2], un[3]};
                load_u(b + EW);
                RowState* rs = &states[b * 32 + lane];
                RowState st = *rs;
                const float invT = s_invT[b];
                unsigned long long* list = lists + (size_t)b * topk;
                const int cnt = s_cnt[b];
                const float last = key_val(list[topk - 1]);
                const float thr = cnt == topk ? last : -CUDART_INF_F;
                const int ni = (nrow + 31) >> 5;                    // the tile's rows per lane
                float z[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const bool valid = lane + 32 * i < nrow;
                    float x1 = valid ? zt[(size_t)b * kBM + lane + 32 * i] : 0.f;
                    if (COMB && i < 2) {                            // the logit's parts of the steps that lay side by side (tiles of up to 64 rows)
                        const float* zc = zt + (size_t)b * kBM + lane + 32 * i;
                        const float p1 = valid ? zc[geo.pitch] : 0.f;
                        const float p2 = valid && comb > 2 ? zc[2 * geo.pitch] : 0.f;
                        const float p3 = valid && comb > 3 ? zc[3 * geo.pitch] : 0.f;
                        x1 = (x1 + p1) + (p2 + p3);
                    }
                    if (a.dbg_logits && valid) a.dbg_logits[(size_t)b * K + j0 + lane + 32 * i] = x1;
                    z[i] = valid ? x1 * invT : -CUDART_INF_F;
                }
                {   // running max / sum-exp: one rescale per tile, independent exponentials (a NaN logit is left out of
                    // the maximum and poisons the sum)
                    const float m_new = fmaxf(st.m, fmaxf(fmaxf(z[0], z[1]), fmaxf(z[2], z[3])));
                    const float m_ref = (m_new == -CUDART_INF_F) ? 0.f : m_new;
                    st.s = st.s * exp_fast(st.m - m_ref) + ((exp_fast(z[0] - m_ref) + exp_fast(z[1] - m_ref)) +
                                                            (exp_fast(z[2] - m_ref) + exp_fast(z[3] - m_ref)));
                    st.m = m_new;
                }
                if (a.uniforms) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        if (i < ni) {
                            // g = -log(-log u): -log u from a short series in 1-u near 1 (where a fast logarithm's absolute
                            // error would dominate the tiny result), fast logarithms elsewhere
                            const float uc = fminf(fmaxf(u[i], 0x1p-24f), 1.f - 0x1p-24f);
                            const float t1 = 1.f - uc;
                            const float lp = t1 * (1.f + t1 * (0.5f + t1 * (0.33333334f + t1 * (0.25f + t1 * 0.2f))));
                            const float L = uc > 0.95f ? lp : -log_fast(uc);
                            const float sc = z[i] - log_fast(L);
                            const bool win = sc > st.gs;            // (rows that do not exist carry -inf)
                            st.gs = win ? sc : st.gs;
                            st.gj = win ? j0 + lane + 32 * i : st.gj;
                            st.gz = win ? z[i] : st.gz;
                        }
                    }
                }
                // top-k: the rows that beat the list's last entry join the list.  While the list is not full that is
                // nearly every row of the tile; the topk-th largest of the lanes' best values is then a lower bound of
                // the answer and leaves a few more than topk of them.
                unsigned cm[4];
                int n_c = 0;
#pragma unroll
                for (int i = 0; i < 4; ++i) { cm[i] = __ballot_sync(0xffffffffu, z[i] > thr); n_c += __popc(cm[i]); }
                if (n_c > 32 && topk <= 32) {
                    unsigned lb = 0u;                               // the lane's best candidate (no NaN is a candidate)
#pragma unroll
                    for (int i = 0; i < 4; ++i) lb = (z[i] > thr) ? max(lb, f2ord(z[i])) : lb;
                    const unsigned tau = kth_of_lanes(lb, topk, reinterpret_cast<unsigned*>(buf));
                    n_c = 0;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        cm[i] = __ballot_sync(0xffffffffu, z[i] > thr && f2ord(z[i]) >= tau);
                        n_c += __popc(cm[i]);
                    }
                }
                int now = cnt;                                      // entries of the list from here on
                if (n_c) {
                    for (int i = lane; i < cnt; i += 32) buf[i] = list[i];
                    int pos = cnt;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        if ((cm[i] >> lane) & 1u) buf[pos + __popc(cm[i] & lanemask_lt())] = key64(z[i], j0 + lane + 32 * i);
                        pos += __popc(cm[i]);
                    }
                    if (lane < 4) buf[pos + lane] = 0ull;           // (read in groups of four)
                    __syncwarp();                                   // (every read of the old list is done, too)
                    if (pos <= 32) rank_scatter<1>(list, buf, pos, topk);
                    else if (pos <= 64) rank_scatter<2>(list, buf, pos, topk);
                    else rank_scatter<(VT_MAX_TOPK + kBM) / 32>(list, buf, pos, topk);
                    now = min(topk, pos);
                    __syncwarp();
                }
                if (t + 1 < geo.n_tiles) {
                    *rs = st;
                    if (lane == 0) s_cnt[b] = now;
                    continue;
                }
                // ---- last tile: this CTA's record of the hidden row, the lanes folded -- the maximum by one warp reduction,
                // every lane's sum rescaled to it once, a butterfly of additions; the Gumbel candidate by two reductions
                // over its 64-bit key.  (The merge kernel starts when this grid has ended.)
                unsigned long long* kp = rec_keys(recs, b, topk);
                float* fp = rec_f32(recs, b, topk);
                const int c = blockIdx.x;
                for (int k = lane; k < topk; k += 32) kp[(size_t)(1 + k) * kMaxGrid + c] = k < now ? list[k] : 0ull;
                const float Mall = ord2f(__reduce_max_sync(0xffffffffu, f2ord(st.m)));
                float sc = (st.m != -CUDART_INF_F) ? st.s * exp_fast(st.m - Mall) : st.s;
#pragma unroll
                for (int o = 16; o; o >>= 1) sc += __shfl_xor_sync(0xffffffffu, sc, o);
                if (lane == 0) {
                    fp[c] = Mall;
                    fp[kMaxGrid + c] = sc;
                }
                if (a.uniforms) {
                    const unsigned long long gk = st.gj >= 0 ? key64(st.gs, st.gj) : 0ull;
                    const unsigned ghi = (unsigned)(gk >> 32);
                    const unsigned gmax = __reduce_max_sync(0xffffffffu, ghi);
                    const unsigned glo = __reduce_max_sync(0xffffffffu, ghi == gmax ? (unsigned)gk : 0u);
                    if (gk == (((unsigned long long)gmax << 32) | glo)) {     // (one lane, or all of them when no row has a candidate)
                        fp[2 * kMaxGrid + c] = st.gz;
                        kp[c] = gk;
                    }
                }
            }
            if (t + 1 < geo.n_tiles) {
                asm volatile("bar.sync 1, %0;" ::"n"(EW * 32) : "memory");           // the tile buffer is free
            }
        }
#ifdef VT_STAMPS
        if (e == 0 && lane == 0) VT_STAMP(5);
#endif
    }
    tc_fence_before();
    __syncwarp();                                                   // lanes of the single-thread roles rejoin their warps
    __syncthreads();                                                // no copy, no MMA and no read of tensor memory is left
    if (warp == 1) {
        if (s_abort && lane == 0) {
            // a wait expired somewhere: the last release of every stage that was released has arrived, whoever issued it
            const int S = geo.n_stages, ni = geo.issuers;
            int top = -1;
            for (int i = 0; i < ni; ++i) top = max(top, i + ni * (s_issued[i] - 1));
            for (int g = top; g > top - S && g >= 0; --g) {
                int r = g;
                while (r >= 0 && r / ni >= s_issued[r % ni]) r -= S;
                if (r >= 0) drain_wait(&s_empty[r % S], (uint32_t)((r / S) & 1));
            }
        }
        __syncwarp();
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols) : "memory");
    }
    if (threadIdx.x == 0) {
        if (s_abort) {
            atomicOr(&ctrl->flags, (uint32_t)VT_FLAG_TIMEOUT);
            atomicOr(&ctrl->head_aborted, 1u);                      // the merge reports every row as missing
        }
        VT_STAMP(6);
    }
}

// ---- host side ---------------------------------------------------------------------------------------
// Shapes of the few-row contract: what vt_workspace_bytes and the entry points take with topk up to VT_MAX_TOPK.
bool shape_ok(int B, int d) {
    if (B < 1 || B > 16 || d < 8 || (d & 7)) return false;
    return d <= (B <= 8 ? 8192 : 4096);
}

Geo make_geo(int B, int K, int d, int topk, int sms, size_t* smem_bytes) {
    Geo g{};
    g.grid = sms;
    if (g.grid > (K + 7) / 8) g.grid = (K + 7) / 8;
    const int slab = (K + g.grid - 1) / g.grid;
    g.n_tiles = (slab + kBM - 1) / kBM;
    g.rows = (slab + g.n_tiles - 1) / g.n_tiles;
    g.n_kc = (d + kBK - 1) / kBK;
    g.h_bytes = (int)align_up((size_t)B * kBK * 2, 1024);
    const int ew = B <= 8 ? 8 : 16;
    // Tiles of up to 64 rows and up to 16 hidden rows: an MMA takes about 40 cycles whatever its size, so two to four steps
    // of d go into one, side by side: vocabulary rows [c * pitch, (c + 1) * pitch) are those of step c, columns [c * 8 or 16,
    // ...) its hidden rows, and the blocks of the product where both are of the same step are its result.  The rest is
    // computed for nothing; steps beyond d are copies of zeros.  (One row, L2, two issuers
    // without / with: 3000 x 2048 9.8 / 8.3 us, 3000 x 4096 12.6 / 9.9, 5000 x 3072 11.7 / 10.2, 8000 x 4096 13.5 / 12.6; 9 rows of
    // 5000 x 3072 17.1 / 15.2, 16 rows 15.9 / 15.8; the warp-level kernel before took 8.4, 11.0, 12.6, 15.4; 16.8, 21.1.)
    g.comb = 1;
    g.pitch = (int)align_up((size_t)g.rows, 8);
    if (B <= 16 && g.rows <= 64 && g.n_kc > 1) {
        if (g.pitch < 16) g.pitch = 16;                                    // (a TMEM quadrant then holds rows of two steps at most)
        g.comb = kBM / g.pitch < 4 ? kBM / g.pitch : 4;
        if (g.comb > g.n_kc) g.comb = g.n_kc;
        g.n_kc = (g.n_kc + g.comb - 1) / g.comb * g.comb;
    }
    g.mma_rows = g.comb == 1 && g.rows <= 64 ? 64 : kBM;
    const int w_bytes = g.pitch * kBK * 2;
    g.step_bytes = g.h_bytes + w_bytes;
    g.buf_bytes = (B < ew ? B : ew) * kBufKeys * 8;
    const size_t fixed = (size_t)B * kBM * 4 + align_up((size_t)B * topk * 8, 16) + (size_t)g.buf_bytes + (size_t)B * (32 * sizeof(RowState) + 8);
    // the MMA reads mma_rows rows from the start of a W part: what may lie beyond the ring's end
    const long over = (long)g.mma_rows * kBK * 2 - (long)g.comb * g.step_bytes;
    const size_t tail = (long)fixed > over ? fixed : (size_t)over;
    const size_t room = kSmemLimit - 1024 - tail;
    // Four steps to a stage where three such stages fit: the two threads that drive the ring wait and release once
    // per stage (201 MB cold through the bare ring: 34.9 us with one step, 33.3 with two, 32.8 with four).
    g.sub = kMaxSub / g.comb * g.comb;
    while (g.sub > g.comb && (g.sub > g.n_kc || (size_t)3 * g.sub * g.step_bytes > room)) g.sub >>= 1;
    // h of a stage in one copy where its rows end on a step: the producer spends 50 ns on every copy it asks for
    g.h_steps = B <= 16 && d % kBK == 0 ? g.sub : 1;
    const size_t stage = (size_t)g.sub * g.step_bytes;
    const long total = (long)g.n_tiles * ((g.n_kc + g.sub - 1) / g.sub);
    g.n_stages = (int)(room / stage);
    if (g.n_stages > kMaxStages) g.n_stages = kMaxStages;
    if (g.n_stages > total) g.n_stages = (int)total;
    // A phase: eight steps, up to four MMAs in a row per accumulator.  Steps side by side need half the accumulations where
    // there are three or four of them and two issuers; there a phase may be twice as long, and it pays: reading a set takes the
    // epilogue as long as the MMAs of four stages.
    g.spp = kPhase / g.sub;
    if (g.comb >= 3 && ew == 8 && (g.n_stages >= total || g.n_stages >= 4 * g.spp)) g.spp *= 2;
    // A single thread needs 250-300 cycles per 64-column step for its waits, releases and four MMAs, which a small head waits
    // for from the moment h has landed; two threads take every other stage each (one row, L2, one / two issuers: 3000 x
    // 1024 8.8 / 7.9 us, 5000 x 3072 15.0 / 12.9, 8000 x 4096 16.4 / 13.1, 20001 x 3072 22.4 / 20.3).  An issuer that is ahead must not take
    // a stage's former fill, which the other one has yet to wait for, for the one it expects: it is at most two phases less
    // a stage ahead (an accumulator set is read before its next use), so the ring has to be longer than that, or never
    // reused, or even (a stage then always has the same issuer).  A large head's ring of three stages is none of these; there
    // the copies are what is waited for (three stages of four steps, one issuer / six of two, two issuers: 788 MB 114.4 / 116.5).
    g.issuers = max_issuers(ew) == 2 && (g.n_stages >= total || (g.n_stages & 1) == 0 || g.n_stages >= 2 * g.spp) ? 2 : 1;
    g.ring_bytes = (int)(g.n_stages * stage);
    // A drafting loop reads the same head again a few tens of microseconds later.  A head that is larger than L2
    // leaves nothing behind when all of it streams through under one policy; so 56 MB of it, spread evenly over
    // every CTA's fills, keep the ordinary priority and the rest is evicted first.  (56 MB: of the 126 MB about
    // half serves a line that one die's SMs ask for; 201 MB per step 36.0 -> 31.5 us, 24 / 40 / 72 MB 34.3 / 33.1 /
    // 32.1; 268 MB with 10 rows 54.3 -> 53.5.)  A head under 96 MB stays resident anyway, and there the ordinary
    // priority would only push out the records and the uniforms (61 MB: 69.5 -> 73 us per three steps).
    const double mb = (double)K * d * 2.0 / 1e6;
    const int share = mb > 96.0 ? (int)(56.0 / mb * 32.0) : 0;
    for (int i = 0; i < 32; ++i)
        if ((i + 1) * share / 32 != i * share / 32) g.keep |= 1u << i;
    *smem_bytes = (size_t)g.ring_bytes + tail + 1024;              // + slack to align the ring to 1024 bytes
    return g;
}

template <int EW, int RPW, bool COMB>
cudaError_t launch_variant(const HeadArgs& a, Ctrl* ctrl, float* recs, const Geo& geo, const CUtensorMap& tm_h,
                           const CUtensorMap& tm_w, size_t smem, cudaStream_t s) {
    static int attr_done[64] = {0};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64 || !attr_done[dev]) {
        cudaError_t e = cudaFuncSetAttribute(k_head_stream<EW, RPW, COMB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemLimit);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) attr_done[dev] = 1;
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)geo.grid);
    cfg.blockDim = dim3((unsigned)(EW + 1 + geo.issuers) * 32);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = a.overlap ? 1 : 0;
    count_launch();
    return cudaLaunchKernelEx(&cfg, k_head_stream<EW, RPW, COMB>, a, ctrl, recs, geo, tm_h, tm_w);
}

}  // namespace

bool head_skinny_supported(int32_t B, int32_t d) { return shape_ok(B, d); }

// Up to 32 rows the two kernels are within 11 % of one another (us per call, this / batched kernel, greedy: 24 rows of 5000 x 2048
// 15.9 / 14.9, of 20001 x 3072 32.7 / 30.8, of 80000 x 3072 85.2 / 87.0; 32 rows of 32768 x 3072 41.6 / 43.4), and the smaller sums are this
// one's advantage: it adds up phases of eight steps, and its logits' rms error is a tenth of the batched kernel's (2.6e-7 against
// 3.6e-6 at 40 rows).  From 33 to 64 rows its second pass over h for slabs of more than 128 rows and four hidden rows per
// epilogue warp make it the slower one throughout: 40 rows of 123 MB 39.9 / 33.1, of 201 MB 47.1 / 44.1, of 268 MB 58.8 / 53.9, of 491
// MB 95.1 / 88.5.  It keeps the heads of 192 MB and more there for the sake of those logits.
bool head_stream_takes(int32_t B, int32_t K, int32_t d) {
    return B >= 1 && (B <= 32 || (B <= kMaxB && (size_t)K * d * 2 >= ((size_t)192 << 20)));
}

size_t head_skinny_scratch_bytes(int32_t B, int32_t K, int32_t topk) {
    (void)K;
    return align_up((size_t)kMaxGrid * B * rec_fields(topk) * 4, 256) + kStampBytes;
}

cudaError_t launch_head_skinny(const HeadArgs& a, Ctrl* ctrl, uint8_t* scratch, cudaStream_t s) {
    if (!head_stream_takes(a.B, a.K, a.d) || a.d < 8 || (a.d & 7)) return cudaErrorInvalidValue;
    int sms = num_sms();
    if (sms > kMaxGrid) sms = kMaxGrid;
    size_t smem = 0;
    const Geo geo = make_geo(a.B, a.K, a.d, a.topk, sms, &smem);
    if (geo.n_stages < 1 || smem > kSmemLimit) return cudaErrorInvalidValue;
    CUtensorMap tm_h, tm_w;
    const int box_h = geo.h_steps > 1 ? geo.h_bytes / (kBK * 2) : a.B;
    if (!encode_map(&tm_h, a.h, a.B, a.d, box_h, geo.h_steps > 1 ? geo.h_steps : 0) || !encode_map(&tm_w, a.W, a.K, a.d, geo.rows)) return cudaErrorInvalidValue;
    float* recs = reinterpret_cast<float*>(scratch);
    const bool comb = geo.comb > 1;
    const cudaError_t e = a.B <= 8 ? (comb ? launch_variant<8, 1, true>(a, ctrl, recs, geo, tm_h, tm_w, smem, s)
                                           : launch_variant<8, 1, false>(a, ctrl, recs, geo, tm_h, tm_w, smem, s))
                        : a.B <= 16 ? (comb ? launch_variant<16, 1, true>(a, ctrl, recs, geo, tm_h, tm_w, smem, s)
                                            : launch_variant<16, 1, false>(a, ctrl, recs, geo, tm_h, tm_w, smem, s))
                        : a.B <= 32 ? launch_variant<16, 2, false>(a, ctrl, recs, geo, tm_h, tm_w, smem, s)
                                    : launch_variant<16, 4, false>(a, ctrl, recs, geo, tm_h, tm_w, smem, s);
    if (e != cudaSuccess) return e;
    return launch_head_merge(a, ctrl, recs, geo.grid, a.B > 8, s);
}

}  // namespace vt
