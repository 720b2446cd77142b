// Pooling of the raw window scores and variable-k top-k selection per unit (paper Section 3.3.3:
// the tokens with the highest cumulative window attention are kept within the head's budget; the w
// window tokens are part of the budget).
//
//   1. pooled[j] = max / mean of raw over the pool window clipped to the prefix (written out: it is the
//      `d_scores` output of the pass).
//   2. the k-th largest pooled score, k = budget - w, on the order-preserving 32-bit image of the float: the exact
//      threshold T, the number of scores above it and how many scores equal to T are still needed.
//   3. Ordered compaction: each warp owns a contiguous segment; ballots and population counts give every
//      kept position its output slot, so the kept positions come out ascending, and among scores equal to
//      T the lowest positions win.  The window positions follow.
// Counting is integer work: the result does not depend on the order in which threads run.
#include <cooperative_groups.h>

#include "common.cuh"

namespace uncomp {

constexpr int kSelThreads = 1024;
constexpr int kSelWarps = kSelThreads / 32;

__device__ __forceinline__ uint32_t ordered_bits(float f) {
    const uint32_t b = __float_as_uint(f);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

struct SelSmem {
    int hist[2048];
    int scan[kSelThreads];
    int warp_gt[kSelWarps], warp_eq[kSelWarps];
    int bin, above;
};

// What a unit may write: its slab of d_indices is offsets[u] .. offsets[u+1].  The budget should equal the slab
// length and lie in [w, P + w]; whatever disagrees raises UNCOMP_STATUS_BOUNDS and the unit is cut to what the
// slab and the budget both allow, so that every slot of the slab holds a valid position and nothing outside it
// is touched: k top positions, then wn window positions, then `fill` copies of the last position.
struct Slab {
    int64_t begin, seg;
    int k, wn;
    int64_t fill;
};

__device__ __forceinline__ Slab slab_of(const int32_t *__restrict__ budgets, const int64_t *__restrict__ offsets,
                                        int units, int u, int P, int w, bool reporter, uint32_t *status) {
    const int64_t o0 = offsets[u], o1 = offsets[u + 1], oend = offsets[units];
    const int budget = budgets[u];
    const bool off_ok = o0 >= 0 && o1 >= o0 && o1 <= oend;
    const int64_t seg = off_ok ? o1 - o0 : 0;
    if (!(off_ok && (int64_t)budget == seg && budget >= w && budget <= P + w) && reporter)
        atomicOr(status, (uint32_t)UNCOMP_STATUS_BOUNDS);
    int64_t b = min(max(budget, 0), P + w);
    b = min(b, seg);
    Slab s;
    s.begin = off_ok ? o0 : 0;
    s.seg = seg;
    s.k = (int)max((int64_t)0, min(b - w, (int64_t)P));
    s.wn = (int)min((int64_t)w, b - s.k);
    s.fill = seg - s.k - s.wn;
    return s;
}

// Finds the bin (counting down from the top) that holds the kr-th largest element.  All threads call it.
__device__ void find_bin(SelSmem &S, int nbins, int kr, int tid) {
    // thread t covers bins nbins-1-2t and nbins-2-2t
    const int b0 = nbins - 1 - 2 * tid;
    const int h0 = b0 >= 0 ? S.hist[b0] : 0;
    const int h1 = b0 - 1 >= 0 ? S.hist[b0 - 1] : 0;
    S.scan[tid] = h0 + h1;
    __syncthreads();
    for (int o = 1; o < kSelThreads; o <<= 1) {
        const int add = tid >= o ? S.scan[tid - o] : 0;
        __syncthreads();
        S.scan[tid] += add;
        __syncthreads();
    }
    const int excl = S.scan[tid] - (h0 + h1);
    if (b0 >= 0 && excl < kr && kr <= excl + h0) { S.bin = b0; S.above = excl; }
    else if (b0 - 1 >= 0 && excl + h0 < kr && kr <= excl + h0 + h1) { S.bin = b0 - 1; S.above = excl + h0; }
    __syncthreads();
}

// ---- prefixes beyond 262144: radix select of the pooled scores in global memory -----------------------------------
// A cluster of 8 CTAs per unit.  CTA r owns the r-th eighth of the positions; histograms and counts are combined through
// distributed shared memory by CTA 0 and read back by the others.
constexpr int kSelCluster = 8;

__global__ void __cluster_dims__(kSelCluster, 1, 1) __launch_bounds__(kSelThreads)
pool_select_cluster_kernel(const float *__restrict__ raw, float *__restrict__ pooled, int P, int w, int pool_kernel,
                           int pool_mode, const int32_t *__restrict__ budgets, const int64_t *__restrict__ offsets,
                           int units, int32_t *__restrict__ indices, uint32_t *__restrict__ status) {
    namespace cg = cooperative_groups;
    __shared__ SelSmem S;
    __shared__ int slice_gt, slice_eq;
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const int u = blockIdx.x / kSelCluster, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const float *r = raw + (size_t)u * P;
    float *s = pooled + (size_t)u * P;
    chain_wait();
    // this CTA's positions: a multiple of 1024 per CTA, so that warps own aligned segments of 32
    const int per = ((P + kSelCluster - 1) / kSelCluster + kSelThreads - 1) / kSelThreads * kSelThreads;
    const int p0 = min(P, rank * per), p1 = min(P, p0 + per);

    const int half = pool_kernel >> 1;
    for (int j = p0 + tid; j < p1; j += kSelThreads) {
        const int lo = max(0, j - half), hi = min(P - 1, j + half);
        float acc = pool_mode ? 0.f : r[lo];
        for (int t = lo; t <= hi; ++t) acc = pool_mode ? acc + r[t] : fmaxf(acc, r[t]);
        s[j] = pool_mode ? acc / (float)(hi - lo + 1) : acc;
    }
    const Slab slab = slab_of(budgets, offsets, units, u, P, w, tid == 0 && rank == 0, status);
    const int k = slab.k;
    int32_t *out = indices + slab.begin;
    if (rank == 0) {
        for (int i = tid; i < slab.wn; i += kSelThreads)
            if (UNCOMP_INDEX_OK(k + i, slab.seg, status)) out[k + i] = P + i;
        for (int64_t i = tid; i < slab.fill; i += kSelThreads)
            if (UNCOMP_INDEX_OK(k + slab.wn + i, slab.seg, status)) out[k + slab.wn + i] = P + w - 1;
    }
    if (k == 0) return;   // uniform over the cluster
    __syncthreads();      // this CTA reads only the pooled scores it wrote itself

    SelSmem *S0 = cluster.map_shared_rank(&S, 0);
    uint32_t prefix = 0;
    int kr = k;
    if (k < P) {
#pragma unroll 1
        for (int pass = 0; pass < 3; ++pass) {
            const int shift = pass == 0 ? 21 : (pass == 1 ? 10 : 0);
            const int nbits = pass == 2 ? 10 : 11;
            const int nbins = 1 << nbits;
            const uint32_t himask = pass == 0 ? 0u : (0xffffffffu << (shift + nbits));
            for (int b = tid; b < 2048; b += kSelThreads) S.hist[b] = 0;
            __syncthreads();
            for (int j = p0 + tid; j < p1; j += kSelThreads) {
                const uint32_t v = ordered_bits(s[j]);
                if ((v & himask) == prefix && UNCOMP_INDEX_OK((v >> shift) & (nbins - 1), 2048, status))
                    atomicAdd(&S.hist[(v >> shift) & (nbins - 1)], 1);
            }
            cluster.sync();                       // every CTA's histogram is complete
            if (rank == 0) {
                for (int b = tid; b < nbins; b += kSelThreads) {
                    int sum = S.hist[b];
                    for (int c = 1; c < kSelCluster; ++c) sum += cluster.map_shared_rank(&S, c)->hist[b];
                    S.hist[b] = sum;              // only this thread reads or writes bin b of CTA 0 here
                }
                __syncthreads();
                find_bin(S, nbins, kr, tid);
            }
            cluster.sync();                       // bin and count above it are published by CTA 0
            prefix |= (uint32_t)S0->bin << shift;
            kr -= S0->above;
            cluster.sync();                       // all have read them before the next pass clears the histograms
        }
    }
    const uint32_t T = k < P ? prefix : 0u;
    const int need_eq = k < P ? kr : P;

    // ordered compaction: counts of the lower CTAs first, then of the lower warps of this CTA
    const int seg = per / kSelWarps;              // a multiple of 32
    const int j0 = min(p1, p0 + wid * seg), j1 = min(p1, j0 + seg);
    int cg_ = 0, ce = 0;
    for (int j = j0 + lane; j < j1; j += 32) {
        const uint32_t v = ordered_bits(s[j]);
        cg_ += v > T;
        ce += v == T;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        cg_ += __shfl_xor_sync(0xffffffffu, cg_, o);
        ce += __shfl_xor_sync(0xffffffffu, ce, o);
    }
    if (lane == 0) { S.warp_gt[wid] = cg_; S.warp_eq[wid] = ce; }
    __syncthreads();
    if (tid == 0) {
        int a = 0, b = 0;
        for (int x = 0; x < kSelWarps; ++x) { a += S.warp_gt[x]; b += S.warp_eq[x]; }
        slice_gt = a;
        slice_eq = b;
    }
    cluster.sync();
    int gt_run = 0, eq_run = 0;
    for (int c = 0; c < rank; ++c) {
        gt_run += *cluster.map_shared_rank(&slice_gt, c);
        eq_run += *cluster.map_shared_rank(&slice_eq, c);
    }
    for (int x = 0; x < wid; ++x) { gt_run += S.warp_gt[x]; eq_run += S.warp_eq[x]; }
    const unsigned lt = (1u << lane) - 1u;
    for (int jb = j0; jb < j1; jb += 32) {
        const int j = jb + lane;
        const uint32_t v = j < j1 ? ordered_bits(s[j]) : 0u;
        const bool gt = j < j1 && v > T;
        const bool eq = j < j1 && v == T;
        const unsigned mg = __ballot_sync(0xffffffffu, gt), me = __ballot_sync(0xffffffffu, eq);
        const int gtb = gt_run + __popc(mg & lt);
        const int eqb = eq_run + __popc(me & lt);
        if ((gt || (eq && eqb < need_eq)) && UNCOMP_INDEX_OK(gtb + min(eqb, need_eq), k, status))
            out[gtb + min(eqb, need_eq)] = j;
        gt_run += __popc(mg);
        eq_run += __popc(me);
    }
    cluster.sync();       // no CTA leaves while another may still read its shared memory
}

// ---- prefixes up to 262144 positions: keys in shared memory --------------------------------------------------------
// A unit is a CTA of 1024 threads (up to 32768 positions) or a cluster of 2, 4 or 8; a warp owns NBK x 128 consecutive
// positions, a lane 4 consecutive ones of every 128.  The pooled scores replace the raw ones in shared memory as
// order-preserving integers.  The threshold comes from
// histograms of 2048 bins over the range the keys really span (not over their leading bits: scores share most of those,
// and the shared-memory atomics of a warp would meet in a few bins), then over the chosen bin, at most three times.  One
// cluster barrier per histogram: every CTA adds up all of them, the next pass uses another array.
// Bound by shared-memory atomics, barriers and, with many units, issue.  256 units of 32704 positions / 1024 of 3704 / 8
// of 6969: radix select that read the pooled scores from global memory three times with 20 barriers a pass 75 / 61 / 23 us,
// keys in registers and a search bit by bit with counts (no atomics, 20 to 30 rounds) 163 / 74 / 25 us, this 39 / 36 / 14 us
// (128 of 131008: 101 us, was 201).
constexpr int kKeyThreads = 1024;
constexpr int kKeyWarps = kKeyThreads / 32;
constexpr int kKeyMaxCluster = 8;
constexpr int kKeyHalo = 32;                             // pool windows reach at most 31 positions beyond a CTA's share
constexpr int kKeyBins = 2 * kKeyThreads;
constexpr int kCandidates = 256;                         // keys ranked against one another instead of by another histogram
// How the scores are pooled: width 1 takes them as they are; the 7-wide maximum, what the pass defaults to, from the four
// scores of a lane and shuffles; any other width by a loop per position.  256 units of 32704 positions / 1024 of 3704 / 8 of
// 6969: 33 / 31 / 13 us, 39 / 36 / 14 us, and by the loop 55 / 45 / 17 us for a maximum over 5, 54 / 44 / 17 over 9, 119 /
// 72 / 25 over 63.
enum { kPoolAny, kPoolNone, kPoolMax7 };

template <int NBK> struct KeySmem {
    float raw[2 * kKeyHalo + kKeyWarps * NBK * 128];     // this CTA's raw scores with their neighbours, later its keys
    int hist[3][kKeyBins];
    unsigned slot[2][2][kKeyMaxCluster];                 // [exchange][value][CTA of the cluster]
    unsigned warp_a[kKeyWarps], warp_b[kKeyWarps];
    int warp_sum[kKeyWarps];
    uint4 above_bits[kKeyWarps * NBK], equal_bits[kKeyWarps * NBK];      // of 128 positions: bit l of word c is position 4 l + c
    uint32_t threshold;
    int bin, above, in_bin, candidates, all_equal;
};

// bit i of a byte to bit 4 i
__device__ __forceinline__ uint32_t spread4(uint32_t x) {
    x = (x | (x << 12)) & 0x000f000fu;
    x = (x | (x << 6)) & 0x03030303u;
    return (x | (x << 3)) & 0x11111111u;
}
// the 32 positions 32 g .. 32 g + 31 of 128, in their order
__device__ __forceinline__ uint32_t in_order(const uint4 &w, int g) {
    const int s = 8 * g;
    return spread4((w.x >> s) & 255u) | spread4((w.y >> s) & 255u) << 1 | spread4((w.z >> s) & 255u) << 2 | spread4((w.w >> s) & 255u) << 3;
}

// Two CTAs per SM up to four blocks of keys: with many units one CTA's barriers hide behind the other.  That bound leaves
// 32 registers and spills 36 to 64 bytes of a thread, also in calls whose few units leave the second place empty.
template <int NBK, int POOL>
__global__ void __launch_bounds__(kKeyThreads, NBK <= 4 ? 2 : 1)
pool_select_keys_kernel(const float *__restrict__ raw, float *__restrict__ pooled, int P, int w, int pool_kernel, int pool_mode,
                        const int32_t *__restrict__ budgets, const int64_t *__restrict__ offsets, int units,
                        int32_t *__restrict__ indices, uint32_t *__restrict__ status) {
    namespace cg = cooperative_groups;
    constexpr int kShare = kKeyWarps * NBK * 128, kWarpShare = NBK * 128;
    extern __shared__ __align__(16) unsigned char key_smem[];
    KeySmem<NBK> &S = *reinterpret_cast<KeySmem<NBK> *>(key_smem);
    cg::cluster_group cluster = cg::this_cluster();
    const int ctas = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const int u = blockIdx.x / ctas, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const float *r = raw + (size_t)u * P;
    float *s = pooled + (size_t)u * P;
    const int p0 = rank * kShare;                        // S.raw[i] is position p0 - kKeyHalo + i
    const int half = pool_kernel >> 1;
    if (ctas > 1) cluster.barrier_arrive();              // waited for before anybody's shared memory is touched
    chain_wait();

    // ---- 1. raw scores to shared memory, pooled scores out and, as keys, in their place ---------------------
    const float outside = pool_mode ? 0.f : -INFINITY;
    constexpr int kVec = (kShare + 2 * kKeyHalo) / 4;
    if ((reinterpret_cast<uintptr_t>(r) & 15u) == 0) {               // asynchronous copies: all on their way at once
#pragma unroll 4
        for (int i = tid; i < kVec; i += kKeyThreads) {
            const int j = p0 - kKeyHalo + 4 * i;
            if (j >= 0 && j + 3 < P) {
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(S.raw + 4 * i)), "l"(r + j) : "memory");
            } else {
                float4 x = make_float4(outside, outside, outside, outside);
                if (j >= 0 && j < P) {
                    x.x = r[j];
                    if (j + 1 < P) x.y = r[j + 1];
                    if (j + 2 < P) x.z = r[j + 2];
                }
                reinterpret_cast<float4 *>(S.raw)[i] = x;
            }
        }
    } else {
#pragma unroll 8
        for (int i = tid; i < kShare + 2 * kKeyHalo; i += kKeyThreads) {
            const int j = p0 - kKeyHalo + i;
            S.raw[i] = j >= 0 && j < P ? __ldg(r + j) : outside;
        }
    }
#pragma unroll
    for (int i = 0; i < 3 * kKeyBins / kKeyThreads; ++i) (&S.hist[0][0])[tid + i * kKeyThreads] = 0;
    const Slab slab = slab_of(budgets, offsets, units, u, P, w, tid == 0 && rank == 0, status);
    const int k = slab.k;
    int32_t *out = indices + slab.begin;
    if (rank == 0) {
        for (int i = tid; i < slab.wn; i += kKeyThreads)
            if (UNCOMP_INDEX_OK(k + i, slab.seg, status)) out[k + i] = P + i;
        for (int64_t i = tid; i < slab.fill; i += kKeyThreads)
            if (UNCOMP_INDEX_OK(k + slab.wn + i, slab.seg, status)) out[k + slab.wn + i] = P + w - 1;
    }
    if (tid == 0) S.candidates = 0;
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    const int at0 = wid * kWarpShare + lane * 4, j0 = p0 + at0;        // block b: 128 b further
    float *mine = S.raw + kKeyHalo + at0;
    const bool vec = (reinterpret_cast<uintptr_t>(s) & 15u) == 0;
    uint32_t hi = 0u, lo = 0xffffffffu;
    auto finish = [&](int b, const float4 &o) {          // pooled scores out, keys in place; 0 beyond the prefix
        const int j = j0 + 128 * b;
        if (vec && j + 3 < P) {
            *reinterpret_cast<float4 *>(s + j) = o;
        } else {
            if (j < P) s[j] = o.x;
            if (j + 1 < P) s[j + 1] = o.y;
            if (j + 2 < P) s[j + 2] = o.z;
            if (j + 3 < P) s[j + 3] = o.w;
        }
        uint4 key = make_uint4(ordered_bits(o.x), ordered_bits(o.y), ordered_bits(o.z), ordered_bits(o.w));
        if (j + 3 < P) {
            hi = max(max(hi, max(key.x, key.y)), max(key.z, key.w));
            lo = min(min(lo, min(key.x, key.y)), min(key.z, key.w));
        } else {
            if (j < P) { hi = max(hi, key.x); lo = min(lo, key.x); } else key.x = 0u;
            if (j + 1 < P) { hi = max(hi, key.y); lo = min(lo, key.y); } else key.y = 0u;
            if (j + 2 < P) { hi = max(hi, key.z); lo = min(lo, key.z); } else key.z = 0u;
            key.w = 0u;
        }
        *reinterpret_cast<uint4 *>(mine + 128 * b) = key;
    };
    if (POOL == kPoolMax7) {
        // the neighbours that other warps overwrite are taken before anybody writes
        const float4 left = *reinterpret_cast<const float4 *>(mine - 4);                       // lane 0 uses it
        const float4 right = *reinterpret_cast<const float4 *>(mine + 128 * (NBK - 1) + 4);    // lane 31 uses it
        __syncthreads();
        float4 m = *reinterpret_cast<const float4 *>(mine);
        float py = left.y, pz = left.z, pw = left.w;     // raw scores left of the lane's first position
#pragma unroll
        for (int b = 0; b < NBK; ++b) {
            const float4 next = b + 1 < NBK ? *reinterpret_cast<const float4 *>(mine + 128 * (b + 1)) : right;
            // right of the lane: the next lane's, for lane 31 the first of the next 128
            float ax = __shfl_up_sync(0xffffffffu, m.y, 1), ay = __shfl_up_sync(0xffffffffu, m.z, 1), az = __shfl_up_sync(0xffffffffu, m.w, 1);
            const float nx = b + 1 < NBK ? __shfl_sync(0xffffffffu, next.x, 0) : right.x;
            const float ny = b + 1 < NBK ? __shfl_sync(0xffffffffu, next.y, 0) : right.y;
            const float nz = b + 1 < NBK ? __shfl_sync(0xffffffffu, next.z, 0) : right.z;
            float zx = __shfl_down_sync(0xffffffffu, m.x, 1), zy = __shfl_down_sync(0xffffffffu, m.y, 1), zz = __shfl_down_sync(0xffffffffu, m.z, 1);
            if (lane == 0) { ax = py; ay = pz; az = pw; }
            if (lane == 31) { zx = nx; zy = ny; zz = nz; }
            py = __shfl_sync(0xffffffffu, m.y, 31);
            pz = __shfl_sync(0xffffffffu, m.z, 31);
            pw = __shfl_sync(0xffffffffu, m.w, 31);
            const float mid = fmaxf(fmaxf(m.x, m.y), fmaxf(m.z, m.w));
            const float4 o = make_float4(fmaxf(mid, fmaxf(ax, fmaxf(ay, az))), fmaxf(mid, fmaxf(fmaxf(ay, az), zx)),
                                         fmaxf(mid, fmaxf(az, fmaxf(zx, zy))), fmaxf(mid, fmaxf(zx, fmaxf(zy, zz))));
            finish(b, o);
            m = next;
        }
    } else if (POOL == kPoolNone) {
#pragma unroll
        for (int b = 0; b < NBK; ++b) finish(b, *reinterpret_cast<const float4 *>(mine + 128 * b));
    } else {
        auto pooled_at = [&](int at, int j) {
            const float *x = S.raw + kKeyHalo + at;
            float acc;
            if (pool_mode) {
                const int lo_j = max(0, j - half), hi_j = min(P - 1, j + half);
                acc = 0.f;
                for (int t = lo_j; t <= hi_j; ++t) acc += x[t - j];
                return acc / (float)(hi_j - lo_j + 1);
            }
            acc = x[-half];
            for (int t = 1 - half; t <= half; ++t) acc = fmaxf(acc, x[t]);
            return acc;
        };
        for (int i = tid; i < kShare; i += kKeyThreads)
            if (p0 + i < P) s[p0 + i] = pooled_at(i, p0 + i);
        __syncthreads();                                 // nobody reads raw scores any more; s is visible to the CTA
#pragma unroll 1
        for (int b = 0; b < NBK; ++b) {
            const int j = j0 + 128 * b;
            finish(b, make_float4(j < P ? s[j] : 0.f, j + 1 < P ? s[j + 1] : 0.f, j + 2 < P ? s[j + 2] : 0.f, j + 3 < P ? s[j + 3] : 0.f));
        }
    }
    if (ctas > 1) cluster.barrier_wait();
    if (k == 0) return;                                  // uniform over the cluster, nobody has touched a peer's memory

    // From here on a thread reads only the keys it has written.
    auto keys = [&](int b) { return *reinterpret_cast<const uint4 *>(mine + 128 * b); };

    // ---- 2. threshold ------------------------------------------------------------------------------
    uint32_t T = 0;
    bool all_equal_kept = k >= P;                        // every key that equals T is kept
    if (k < P) {
        hi = __reduce_max_sync(0xffffffffu, hi);
        lo = __reduce_min_sync(0xffffffffu, lo);
        if (lane == 0) { S.warp_a[wid] = hi; S.warp_b[wid] = lo; }
        __syncthreads();
        hi = __reduce_max_sync(0xffffffffu, S.warp_a[lane]);
        lo = __reduce_min_sync(0xffffffffu, S.warp_b[lane]);
        if (ctas > 1) {
            if (tid < ctas) {
                KeySmem<NBK> *R = cluster.map_shared_rank(&S, tid);
                R->slot[0][0][rank] = hi;
                R->slot[0][1][rank] = lo;
            }
            cluster.sync();
            for (int c = 0; c < ctas; ++c) { hi = max(hi, S.slot[0][0][c]); lo = min(lo, S.slot[0][1][c]); }
        }
        int kr = k;                                      // rank to resolve inside [lo, lo + width)
        uint32_t width = hi - lo;                        // first as the largest distance
        int shift = max(0, 21 - __clz((int)width));      // 11 bits of it
        if (width == 0u) { T = lo; __syncthreads(); }    // all keys equal; warp_a is written again below
#pragma unroll 1
        for (int pass = 0; width != 0u; ++pass) {
            int *hist = S.hist[pass];
            const uint32_t last = pass == 0 ? width : width - 1;      // largest distance from lo that counts
#pragma unroll
            for (int b = 0; b < NBK; ++b) {
                const uint4 key = keys(b);
                const uint32_t d[4] = {key.x - lo, key.y - lo, key.z - lo, key.w - lo};
                const int left = P - (j0 + 128 * b);     // of the four, those before the prefix' end
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    if (d[c] <= last && c < left && UNCOMP_INDEX_OK(d[c] >> shift, kKeyBins, status)) atomicAdd(&hist[d[c] >> shift], 1);
            }
            if (ctas > 1) cluster.sync();                // every histogram of the cluster is complete
            else __syncthreads();
            // bins from the top: this thread has bins b0 and b0 - 1
            const int b0 = kKeyBins - 1 - 2 * tid;
            int h0 = 0, h1 = 0;
            for (int c = 0; c < ctas; ++c) {
                const int2 h = *reinterpret_cast<const int2 *>(&(ctas > 1 ? cluster.map_shared_rank(&S, c) : &S)->hist[pass][b0 - 1]);
                h0 += h.y;
                h1 += h.x;
            }
            int incl = h0 + h1;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int below = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += below;
            }
            if (lane == 31) S.warp_sum[wid] = incl;
            __syncthreads();
            const int excl = incl - h0 - h1 + __reduce_add_sync(0xffffffffu, lane < wid ? S.warp_sum[lane] : 0);
            if (excl < kr && kr <= excl + h0) { S.bin = b0; S.above = excl; S.in_bin = h0; }
            else if (excl + h0 < kr && kr <= excl + h0 + h1) { S.bin = b0 - 1; S.above = excl + h0; S.in_bin = h1; }
            __syncthreads();
            lo += (uint32_t)S.bin << shift;
            kr -= S.above;
            T = lo;
            all_equal_kept = S.in_bin == kr;             // the whole bin is kept: T is its lower end
            if (all_equal_kept || shift == 0) break;
            if (ctas == 1 && S.in_bin <= kCandidates) {
                // few keys are left in the bin: they are collected, and each is ranked against all of them
                uint32_t *list = reinterpret_cast<uint32_t *>(S.hist[2]);
                const int m = S.in_bin;
#pragma unroll 1
                for (int b = 0; b < NBK; ++b) {
                    const uint4 kv = keys(b);
                    const uint32_t key[4] = {kv.x, kv.y, kv.z, kv.w};
                    const int left = P - (j0 + 128 * b);
#pragma unroll
                    for (int c = 0; c < 4; ++c)
                        if ((key[c] - lo) >> shift == 0u && c < left) {
                            const int at = atomicAdd(&S.candidates, 1);
                            if (UNCOMP_INDEX_OK(at, kCandidates, status)) list[at] = key[c];
                        }
                }
                __syncthreads();
                if (tid < m) {
                    const uint32_t own = list[tid];
                    int above = 0, equal = 0;
#pragma unroll 4
                    for (int i = 0; i < m; ++i) {
                        const uint32_t x = list[i];
                        above += x > own;
                        equal += x == own;
                    }
                    if (above < kr && kr <= above + equal) {      // the same for all keys equal to it
                        S.threshold = own;
                        S.all_equal = kr == above + equal;
                    }
                }
                __syncthreads();
                T = S.threshold;
                all_equal_kept = S.all_equal != 0;
                break;
            }
            width = 1u << shift;
            shift = max(0, shift - 11);
            __syncthreads();                             // bin, above and in_bin are read before the next pass writes them
        }
    }

    // ---- 3. ordered compaction ---------------------------------------------------------------------------
    // kept: above T, and of those equal to T the first; when all equal ones are kept they count as above.  The warps leave a bit
    // per position; then a thread has 32 consecutive positions, so one scan of the block gives every thread its first
    // slot.  (A scan per 128 positions took 15,000 cycles of a unit of 32768.)
    auto is_above = [&](uint32_t x) { return all_equal_kept ? x >= T : x > T; };
#pragma unroll
    for (int b = 0; b < NBK; ++b) {
        const uint4 key = keys(b);
        const int left = P - (j0 + 128 * b);
        const uint4 above = make_uint4(__ballot_sync(0xffffffffu, is_above(key.x) && 0 < left), __ballot_sync(0xffffffffu, is_above(key.y) && 1 < left),
                                       __ballot_sync(0xffffffffu, is_above(key.z) && 2 < left), __ballot_sync(0xffffffffu, is_above(key.w) && 3 < left));
        if (lane == 0) S.above_bits[wid * NBK + b] = above;
        if (!all_equal_kept) {
            const uint4 equal = make_uint4(__ballot_sync(0xffffffffu, key.x == T && 0 < left), __ballot_sync(0xffffffffu, key.y == T && 1 < left),
                                           __ballot_sync(0xffffffffu, key.z == T && 2 < left), __ballot_sync(0xffffffffu, key.w == T && 3 < left));
            if (lane == 0) S.equal_bits[wid * NBK + b] = equal;
        }
    }
    __syncthreads();
    constexpr int kGroups = 4 * kKeyWarps * NBK;         // of 32 positions, at most one per thread
    uint32_t above = 0u, equal = 0u;
    if (tid < kGroups) {
        above = in_order(S.above_bits[tid >> 2], tid & 3);
        if (!all_equal_kept) equal = in_order(S.equal_bits[tid >> 2], tid & 3);
    }
    const unsigned own = __popc(above) | (unsigned)__popc(equal) << 16;         // 32768 of each at most
    unsigned incl = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned below = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += below;
    }
    if (lane == 31) S.warp_a[wid] = incl;
    __syncthreads();
    const unsigned warp_all = S.warp_a[lane];
    const unsigned before = __reduce_add_sync(0xffffffffu, lane < wid ? warp_all : 0u) + incl - own;
    const unsigned all = __reduce_add_sync(0xffffffffu, warp_all);
    unsigned g = before & 0xffffu, e = before >> 16, gt_all = all & 0xffffu;
    if (ctas > 1) {
        if (tid < ctas) {
            KeySmem<NBK> *R = cluster.map_shared_rank(&S, tid);
            R->slot[1][0][rank] = gt_all;
            R->slot[1][1][rank] = all >> 16;
        }
        cluster.sync();                                  // also the last access to a peer's memory
        gt_all = 0;
        for (int c = 0; c < ctas; ++c) {
            gt_all += S.slot[1][0][c];
            if (c < rank) { g += S.slot[1][0][c]; e += S.slot[1][1][c]; }
        }
    }
    const unsigned need_eq = all_equal_kept ? 0u : (unsigned)k - gt_all;
    const int j = p0 + 32 * tid;
    for (uint32_t rest = above | equal; rest != 0u; rest &= rest - 1u) {
        const int bit = __ffs(rest) - 1;
        const bool is_gt = (above >> bit) & 1u;
        const unsigned at = g + min(e, need_eq);
        if ((is_gt || e < need_eq) && UNCOMP_INDEX_OK(at, k, status)) out[at] = j + bit;
        g += is_gt;
        e += !is_gt;
    }
}

template <int NBK, int POOL>
cudaError_t launch_keys(const Plan &p, int ctas, const float *d_raw, float *d_pooled, int pool_kernel, int pool_mode,
                        const int32_t *d_budgets, const int64_t *d_offsets, int32_t *d_indices, uint32_t *d_status, cudaStream_t st) {
    static bool done[64] = {};
    cudaError_t e = allow_dynamic_smem((const void *)pool_select_keys_kernel<NBK, POOL>, sizeof(KeySmem<NBK>), done);
    if (e != cudaSuccess) return e;
    return launch_kernel(pool_select_keys_kernel<NBK, POOL>,
                         LaunchShape{dim3(p.units * ctas), kKeyThreads, sizeof(KeySmem<NBK>), (unsigned)ctas}, st, d_raw, d_pooled,
                         p.prefix, p.shape.w, pool_kernel, pool_mode, d_budgets, d_offsets, p.units, d_indices, d_status);
}

template <int POOL>
cudaError_t launch_keys_nbk(const Plan &p, int n, int ctas, const float *d_raw, float *d_pooled, int pool_kernel, int pool_mode,
                            const int32_t *d_budgets, const int64_t *d_offsets, int32_t *d_indices, uint32_t *d_status, cudaStream_t st) {
    const auto f = n > 4 * ctas ? launch_keys<8, POOL> : n > 2 * ctas ? launch_keys<4, POOL> : n > ctas ? launch_keys<2, POOL> : launch_keys<1, POOL>;
    return f(p, ctas, d_raw, d_pooled, pool_kernel, pool_mode, d_budgets, d_offsets, d_indices, d_status, st);
}

cudaError_t launch_pool_select(const Plan &p, const float *d_raw, float *d_pooled, int pool_kernel, int pool_mode,
                               const int32_t *d_budgets, const int64_t *d_offsets, int32_t *d_indices,
                               uint32_t *d_status, cudaStream_t st) {
    // 4096 positions per CTA and block of keys.  One CTA per unit up to 16384 positions (a cluster barrier costs a microsecond:
    // 16 units of 16000 positions 17 us on one CTA, 20 on two), and up to 32768 unless most of the GPU would idle (8 units of
    // 32768: 23 us on one or two, 21 on four); clusters beyond.
    const int n = (p.prefix + 4095) / 4096;
    if (n > 64) {
        return launch_kernel(pool_select_cluster_kernel, LaunchShape{dim3(p.units * kSelCluster), kSelThreads, 0, 1}, st,
                             d_raw, d_pooled, p.prefix, p.shape.w, pool_kernel, pool_mode, d_budgets, d_offsets, p.units,
                             d_indices, d_status);
    }
    int ctas = 1;
    while (ctas < kKeyMaxCluster && (n > 8 * ctas || (n > 4 && n > 2 * ctas && (int64_t)p.units * ctas * 2 <= kTargetSms))) ctas *= 2;
    const auto f = pool_kernel == 1 ? launch_keys_nbk<kPoolNone>
                                    : pool_kernel == 7 && pool_mode == 0 ? launch_keys_nbk<kPoolMax7> : launch_keys_nbk<kPoolAny>;
    return f(p, n, ctas, d_raw, d_pooled, pool_kernel, pool_mode, d_budgets, d_offsets, d_indices, d_status, st);
}

}  // namespace uncomp
