// Shared device/host helpers of the uncomp CUDA library (sm_100a only).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <utility>

#include "../../include/uncomp.h"

namespace uncomp {

constexpr int kD = 128;          // head dimension supported by every kernel
constexpr int kMaxRows = 512;    // G * w upper bound (window rows of all grouped query heads)
constexpr int kTargetSms = 148;  // SM count of the part the grids are sized for (B200)

// Carve-up of the caller's workspace, decided by the shape alone (see api.cu).
struct Plan {
    uncomp_shape shape;
    int units;          // B * L * H
    int G;              // query heads per KV head
    int rows;           // G * w
    int prefix;         // N - w
    int gram_splits;    // token chunks per unit in the Gram stage (P)
    int gram_chunk;     // tokens per chunk
    int score_splits;   // token chunks per unit in the scorer's statistics pass
    int score_chunk;    // tokens per chunk
    size_t off_status, off_gram, off_stats_part, off_stats, off_raw, off_pooled, off_rank, off_rem;
    size_t off_ev_logits, off_ev_stats, off_ev_raw, off_ev_pooled, off_ev_budgets, off_ev_offsets;   // hidden-state eviction
    size_t off_dec_stats, off_dec_part, off_dec_new;   // decode-time update (its logits reuse off_raw .. off_rank)
    size_t bytes;
};

Plan make_plan(const uncomp_shape &s);

// Place of the 16-byte vector (row r, columns 4 c4 .. 4 c4 + 3) in a Gram partial of the scorer: the vectors of four rows lie
// side by side, so that a warp that holds a row per lane (as TMEM hands it out) stores 64-byte pieces, eight cache lines an
// instruction, and a warp of the eigenvalue kernel reads four rows x 128 bytes as one run.  Row by row a store touched 32
// lines, and the 128 x 128 block took 4,000 cycles of an item whose tiles take 25,000.
__host__ __device__ __forceinline__ int gram_vec4(int r, int c4) { return ((r >> 2) * (kD / 4) + c4) * 4 + (r & 3); }

struct UnitAddr {
    int L, H;
    int64_t sB, sL, sH, sN;
    __host__ __device__ inline int64_t base(int u) const {
        const int h = u % H;
        const int l = (u / H) % L;
        const int b = u / (H * L);
        return (int64_t)b * sB + (int64_t)l * sL + (int64_t)h * sH;
    }
};

inline UnitAddr make_addr(const uncomp_shape &s, const uncomp_strides &st) {
    UnitAddr a;
    a.L = s.L; a.H = s.H; a.sB = st.sB; a.sL = st.sL; a.sH = st.sH; a.sN = st.sN;
    return a;
}

// Debug library (-DUNCOMP_DEBUG, built as libuncomp_debug.so): the kernels that place data at computed positions
// (selection, compaction, decode-time commit, hidden-state gather) check every such
// index against the extent it must stay in.  A violation raises UNCOMP_STATUS_BOUNDS and the access is skipped:
// no trap, no assert.  In the release library the check is the constant `true`.
#ifdef UNCOMP_DEBUG
__device__ __forceinline__ bool debug_index_ok(int64_t i, int64_t extent, uint32_t *status) {
    if (i >= 0 && i < extent) return true;
    atomicOr(status, (uint32_t)UNCOMP_STATUS_BOUNDS);
    return false;
}
#define UNCOMP_INDEX_OK(i, extent, status) (::uncomp::debug_index_ok((int64_t)(i), (int64_t)(extent), (status)))
#else
#define UNCOMP_INDEX_OK(i, extent, status) (true)
#endif

__device__ __forceinline__ float to_float(float x) { return x; }
__device__ __forceinline__ float to_float(__nv_bfloat16 x) { return __bfloat162float(x); }

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ int64_t warp_sum_i64(int64_t v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// ---- packed fp32 pairs (one instruction works on two values; each half rounds as the scalar form) ---
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float &lo, float &hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ float sum2(f32x2 v) {
    float lo, hi;
    unpack2(v, lo, hi);
    return lo + hi;
}

// cudaFuncSetAttribute is sticky per function and device: once per device.  `done` belongs to the one function.
inline cudaError_t allow_dynamic_smem(const void *fn, size_t bytes, bool (&done)[64]) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < 64 && done[dev]) return cudaSuccess;
    e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess && dev >= 0 && dev < 64) done[dev] = true;
    return e;
}

// Kernels that follow one another on a stream are launched with programmatic serialization: the next kernel is set up while
// the one before ends, not after.  Every kernel of such a chain calls chain_wait() before it touches global memory: it
// returns when the kernel before has completed and its writes are visible (at once where there is none), and because each
// kernel waits, so have all before it.  Nobody signals before its end: a signal at the start lets the next kernel's CTAs
// take places early, and the kernels that fill the registers of an SM lost by it more than the launches cost.  Launches
// with full serialization / signal at the start / at the end, back to back: fp32 pass of 512 tokens 251 / 248 / 232 us, one
// layer of 7001 tokens 146 / 160 / 129, 256 units of 8192 tokens 427 / 453 / 414, 1024 of 3712 836 / 862 / 819, a decode
// step on 256 caches of 410 rows 11.1 / 9.4 / 9.4.  The exception are the kernels that end the eigenvalues of up to 296
// units: next are the budgets, one CTA with work that depends on nothing (the table of the groups); a signal is no promise
// about memory, chain_wait() still waits for the end.  All of this loosens the order behind the stream's previous kernel and
// nothing else: copies, event waits and, in a captured graph, kernels of other branches are waited for as by any launch, so it
// holds for the first kernel of a call, whatever the caller has put on the stream, and behind the library's own joins.
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void chain_signal() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

struct LaunchShape {
    dim3 grid;
    unsigned block;
    size_t smem;
    unsigned cluster;    // CTAs per cluster
};
template <typename... P, typename... A>
inline cudaError_t launch_kernel(void (*kernel)(P...), const LaunchShape &s, cudaStream_t st, A &&...args) {
    cudaLaunchAttribute attr[2];
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = s.grid;
    cfg.blockDim = dim3(s.block);
    cfg.dynamicSmemBytes = s.smem;
    cfg.stream = st;
    cfg.attrs = attr;
    attr[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[cfg.numAttrs++].val.programmaticStreamSerializationAllowed = 1;
    if (s.cluster > 1) {
        attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
        attr[cfg.numAttrs].val.clusterDim.x = s.cluster;
        attr[cfg.numAttrs].val.clusterDim.y = attr[cfg.numAttrs].val.clusterDim.z = 1;
        ++cfg.numAttrs;
    }
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
    // a refused launch is this call's error; the runtime also keeps it as its last one, where the caller's next check would find it
    if (e != cudaSuccess) cudaGetLastError();
    return e;
}

// Optional per-kernel timing with CUDA events on the launching stream (host objects only).
enum Slot { kSlotGram = 0, kSlotEigen, kSlotBudgets, kSlotScoreStats, kSlotStatsMerge, kSlotScoreColsum,
            kSlotPoolSelect, kSlotCompact, kSlotGramStats, kSlotEvictLogits, kSlotEvictScores, kSlotEvictGather,
            kSlotDecodeLogits, kSlotDecodeAccumulate, kSlotDecodeCommit, kSlotPrepareVote,
            kSlotPrepareFinish, kSlotWideGram, kSlotWideAssemble, kSlotWideTridiag, kSlotWideSturm, kSlotGramColsum, kSlotDecodeStep, kSlotWideKrylov, kSlotCount };
enum { kScorePhaseStats = 1, kScorePhaseColsum = 2 };
struct Profiler;
void prof_begin(Profiler *p, int slot, cudaStream_t st);
void prof_end(Profiler *p, cudaStream_t st);
struct ProfScope {
    Profiler *p; cudaStream_t st;
    ProfScope(Profiler *p_, int slot, cudaStream_t st_) : p(p_), st(st_) { if (p) prof_begin(p, slot, st); }
    ~ProfScope() { if (p) prof_end(p, st); }
};

// ---- kernel launchers (each returns the cudaError_t of its launches) -------------------------------
cudaError_t launch_gram_simt(const Plan &p, const void *dK, const UnitAddr &addr, void *d_partials, cudaStream_t st);
cudaError_t launch_gram_tc(const Plan &p, const void *dK, const UnitAddr &addr, void *d_partials, uint32_t *d_status,
                           cudaStream_t st);
cudaError_t launch_eigen_entropy(const Plan &p, void *d_partials, const uncomp_entropy_params &ep,
                                 float *d_entropy, float *d_erank, double *d_spectrum, uint32_t *d_status,
                                 cudaStream_t st);
// The partials are scratch of the eigenvalue stage: overwritten.
cudaError_t launch_eigen_tail(int units, float *d_partials, int partials_per_unit, const uncomp_entropy_params &ep,
                              float *d_entropy, float *d_erank, double *d_spectrum, uint32_t *d_status, cudaStream_t st);
// tiled: the partials' matrices are laid out by gram_vec4 (the scorer's), else row by row
cudaError_t launch_eigen_f32(const Plan &p, void *d_partials, int partials_per_unit, bool tiled, const uncomp_entropy_params &ep,
                             float *d_entropy, float *d_erank, double *d_spectrum, uint32_t *d_status, cudaStream_t st);
cudaError_t launch_gram_reduce(const Plan &p, const void *d_partials, double *d_out, cudaStream_t st);
int check_budget_params(const uncomp_shape &s, const uncomp_budget_params &bp);
cudaError_t launch_budgets(const Plan &p, const float *d_erank, const uncomp_budget_params &bp, int32_t *d_budgets,
                           int64_t *d_offsets, int32_t *d_layer_group, int32_t *d_layer_ctx, int32_t *d_rank,
                           int64_t *d_rem, cudaStream_t st);
// d_lse != NULL: the caller's log-sum-exp per window row replaces the statistics pass and the merge
cudaError_t launch_scores_simt(const Plan &p, const void *dQw, const void *dK, const UnitAddr &addr, float scale,
                               const float *d_lse, float *d_stats_part, float *d_stats, float *d_raw,
                               uint32_t *d_status, Profiler *prof, cudaStream_t st);
struct TmapCache;
// phases: kScorePhaseStats (pass A; with d_gram_part != NULL the Gram partials of every (unit, scorer chunk) are
// produced in the same sweep) and / or kScorePhaseColsum (pass B, which merges the chunk statistics or takes d_lse).
// kScorePhaseColsum alone with d_gram_part != NULL: pass B and the Gram partials from one sweep (needs d_lse).
cudaError_t launch_scores_tc(const Plan &p, const void *dQw, const void *dK, const UnitAddr &addr, float scale,
                             const float *d_lse, float *d_stats_part, float *d_raw, float *d_gram_part,
                             int phases, uint32_t *d_status, TmapCache *cache, Profiler *prof, cudaStream_t st);
cudaError_t launch_pool_select(const Plan &p, const float *d_raw, float *d_pooled, int pool_kernel, int pool_mode,
                               const int32_t *d_budgets, const int64_t *d_offsets, int32_t *d_indices,
                               uint32_t *d_status, cudaStream_t st);
int evict_chunks(const uncomp_shape &s);
cudaError_t launch_evict_hidden(const Plan &p, const void *d_qlast, const void *d_K, int64_t sB, int64_t sH, int64_t sN,
                                const void *d_X, int64_t row_bytes, int n_keep, float scale, float *d_logits,
                                float *d_stats, float *d_raw, int32_t *d_budgets, int64_t *d_offsets, float *d_scores,
                                int32_t *d_indices, void *d_Xout, uint32_t *d_status, Profiler *prof, cudaStream_t st);
cudaError_t launch_decode_seed(const Plan &p, const float *d_scores, const int32_t *d_indices, const int64_t *d_offsets,
                               float *d_cum, cudaStream_t st);
int decode_chunks(int max_cap);
size_t decode_partial_bytes();
cudaError_t launch_decode_update(const Plan &p, const void *d_q, const void *d_knew, const void *d_vnew,
                                 const int32_t *d_new_pos, const int64_t *d_offsets, int32_t *d_lens, int max_cap,
                                 int protect, float scale, void *d_Kc, void *d_Vc, int32_t *d_pos, float *d_cum,
                                 float *d_p, int32_t *d_evicted, float *d_logits, float *d_stats, void *d_partial,
                                 float *d_new_cum, uint32_t *d_status, Profiler *prof, cudaStream_t st);
cudaError_t launch_retrieval_layer(const float *d_values, int L, int H, int32_t *d_layer, float *d_increase,
                                   cudaStream_t st);
cudaError_t launch_prepare_groups(const float *d_erank, int S, int L, int H, int M, int scope, float *d_mean,
                                  int32_t *d_group_mean, int32_t *d_votes, int32_t *d_group_vote, Profiler *prof,
                                  cudaStream_t st);
size_t entropy_wide_scratch_bytes(int N, int D);
cudaError_t launch_entropy_wide(const void *d_X, int64_t sN, int N, int D, const uncomp_entropy_params &ep,
                                unsigned char *scratch, float *d_entropy, float *d_erank, double *d_spectrum,
                                uint32_t *d_status, Profiler *prof, cudaStream_t st);
cudaError_t launch_l2_sweep(float *d_A, int rows, int cols, int passes, cudaStream_t st);
cudaError_t launch_compact(const Plan &p, const void *dK, const void *dV, const UnitAddr &aK, const UnitAddr &aV,
                           const int32_t *d_indices, const int64_t *d_offsets, void *dKc, void *dVc,
                           uint32_t *d_status, cudaStream_t st);

}  // namespace uncomp
