// Decode-time update of the ragged per-head cache (paper Section 3.3.3, "Dynamic KV Cache Eviction", last
// sentence: as new tokens are generated, the token with the lowest cumulative attention score leaves;
// Algorithm 2, decoding loop: the new token is concatenated with the head's cache and attends over it).
//
// Per unit (batch, layer, KV head) with a cache of len entries inside a slab of cap rows:
//   p[j]   = sum over the G query heads of softmax_j(scale * q_g . k_j), j over the len cached keys and the
//            new token's own key (entry len);
//   cum[j] += p[j] for the cached entries; the new token starts with p[len];
//   len < cap : the new token is appended;
//   len == cap: the entry with the lowest cum among those with pos <= new_pos - protect leaves (equal
//               scores: the lower position; no such entry: every cached entry is a candidate) and the new
//               token takes its row, so the slab is not kept in position order: `pos` names each row.
//
// The step is bound by reading the cached keys once.  One launch while the logits of a unit fit into the shared memory
// of a cluster (decode_step_kernel below); otherwise three:
//   1. logits      grid (chunks of 1024 entries, units): the G logits of every entry (log2 domain) to scratch,
//                  per chunk the softmax statistics (max, sum of 2^(x - max)) per query head;
//   2. accumulate  same grid: merges the chunk statistics, forms p, updates cum, and leaves per chunk the
//                  lexicographic minimum of (cum, pos) over the candidates and over all entries;
//   3. commit      one small CTA per unit: picks the row, copies the new key / value rows, updates pos, cum, len.
// Positions are unique inside a unit, so every minimum is unique and no result depends on thread order.
#include <cooperative_groups.h>

#include "common.cuh"

namespace uncomp {

namespace {
constexpr int kDecThreads = 256;
constexpr int kDecWarps = kDecThreads / 32;
constexpr int kDecChunk = 1024;

__device__ __forceinline__ float ex2f(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

struct MinRec {          // candidate for eviction: (cum, pos) ordered lexicographically; pos < 0 means none
    float c;
    int32_t pos, j;
};
struct MinPair {
    MinRec el, any;      // among the entries old enough / among all cached entries
};

__device__ __forceinline__ bool rec_less(float c, int32_t pos, const MinRec &b) {
    return b.pos < 0 || c < b.c || (c == b.c && pos < b.pos);
}
__device__ __forceinline__ void rec_take(MinRec &a, const MinRec &b) {
    if (b.pos >= 0 && rec_less(b.c, b.pos, a)) a = b;
}

__device__ __forceinline__ void mma_bf16_16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                               uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

struct DecArgs {
    const void *q, *knew;            // [units * G, d], [units, d]
    const void *Kc;                  // [total_cap, d]
    const int64_t *offsets;          // [units + 1]
    const int32_t *lens;             // [units]
    int units, G, max_cap, chunks_max;
    float c_log2;
    float *logits;                   // [(total_cap + units) * G]
    float *stats;                    // [units, chunks_max, G, 2]
};

// Entry e of unit u sits at row offsets[u] + u + e of the scratch (and of the optional p output): every unit
// has one more entry than its slab has rows.
__device__ __forceinline__ bool unit_ok(const DecArgs &a, int u, int64_t &off, int &len) {
    off = a.offsets[u];
    const int64_t cap = a.offsets[u + 1] - off;
    len = a.lens[u];
    return cap >= 1 && cap <= a.max_cap && len >= 0 && len <= cap;
}

// bf16: the warp-level tensor-core instruction on 16 entries x 16 features times 16 features x 8 heads.  Both
// operands are loaded in the order that makes the loads contiguous (lane (gid, tig) reads bytes
// [64 j + 16 tig, +16) of key rows gid and gid + 8 and of query head gid); a dot product does not depend on the
// order in which the features are visited.  fp32 accumulation, scaled afterwards.
template <int G>
__global__ void __launch_bounds__(kDecThreads) decode_logits_mma_kernel(DecArgs a) {
    constexpr int NB = (G + 7) / 8;
    __shared__ float red_m[kDecWarps][32][NB * 2], red_l[kDecWarps][32][NB * 2];
    const int c = blockIdx.x, u = blockIdx.y;
    int64_t off;
    int len;
    if (!unit_ok(a, u, off, len)) return;
    const int n = len + 1;
    const int t0 = c * kDecChunk, t1 = min(n, t0 + kDecChunk);
    if (t0 >= n) return;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, gid = lane >> 2, tig = lane & 3;
    const __nv_bfloat16 *qb = (const __nv_bfloat16 *)a.q + (size_t)u * G * kD;
    const __nv_bfloat16 *Kb = (const __nv_bfloat16 *)a.Kc + off * kD;
    const __nv_bfloat16 *kn = (const __nv_bfloat16 *)a.knew + (size_t)u * kD;
    uint32_t bq[NB][16];
#pragma unroll
    for (int nb = 0; nb < NB; ++nb) {
        const int h = nb * 8 + gid;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            uint4 x = make_uint4(0u, 0u, 0u, 0u);
            if (h < G) x = reinterpret_cast<const uint4 *>(qb + (size_t)h * kD)[4 * j + tig];
            bq[nb][4 * j] = x.x; bq[nb][4 * j + 1] = x.y; bq[nb][4 * j + 2] = x.z; bq[nb][4 * j + 3] = x.w;
        }
    }
    float m_run[NB][2], l_run[NB][2];
#pragma unroll
    for (int nb = 0; nb < NB; ++nb)
#pragma unroll
        for (int i = 0; i < 2; ++i) { m_run[nb][i] = -1e30f; l_run[nb][i] = 0.f; }
    float *lg = a.logits + (off + u) * G;
    for (int base = t0 + wid * 32; base < t1; base += kDecWarps * 32) {
        uint4 ka[2][2][4];
#pragma unroll
        for (int tile = 0; tile < 2; ++tile)
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                const int row = base + tile * 16 + half * 8 + gid;
                const uint4 *src = reinterpret_cast<const uint4 *>(row < len ? Kb + (int64_t)row * kD : kn);
#pragma unroll
                for (int j = 0; j < 4; ++j) ka[tile][half][j] = row < t1 ? src[4 * j + tig] : make_uint4(0u, 0u, 0u, 0u);
            }
#pragma unroll
        for (int tile = 0; tile < 2; ++tile)
#pragma unroll
            for (int nb = 0; nb < NB; ++nb) {
                float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const uint4 lo = ka[tile][0][j], hi = ka[tile][1][j];
                    mma_bf16_16816(acc, lo.x, hi.x, lo.y, hi.y, bq[nb][4 * j], bq[nb][4 * j + 1]);
                    mma_bf16_16816(acc, lo.z, hi.z, lo.w, hi.w, bq[nb][4 * j + 2], bq[nb][4 * j + 3]);
                }
                // acc[0], acc[1]: entry gid, heads 2 tig and 2 tig + 1;  acc[2], acc[3]: entry gid + 8
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const int h = nb * 8 + 2 * tig + i;
                    if (h < G) {
#pragma unroll
                        for (int half = 0; half < 2; ++half) {
                            const int t = base + tile * 16 + half * 8 + gid;
                            if (t < t1) {
                                const float v = acc[2 * half + i] * a.c_log2;
                                lg[(int64_t)t * G + h] = v;
                                const float m_new = fmaxf(m_run[nb][i], v);
                                l_run[nb][i] = fmaf(l_run[nb][i], ex2f(m_run[nb][i] - m_new), ex2f(v - m_new));
                                m_run[nb][i] = m_new;
                            }
                        }
                    }
                }
            }
    }
#pragma unroll
    for (int nb = 0; nb < NB; ++nb)
#pragma unroll
        for (int i = 0; i < 2; ++i) { red_m[wid][lane][nb * 2 + i] = m_run[nb][i]; red_l[wid][lane][nb * 2 + i] = l_run[nb][i]; }
    __syncthreads();
    if (tid < G) {   // fixed order: warps 0.., then the 8 row lanes that hold this head
        const int nb = tid >> 3, tg = (tid & 7) >> 1, i = tid & 1;
        float m = -1e30f;
        for (int x = 0; x < kDecWarps; ++x)
            for (int g8 = 0; g8 < 8; ++g8) m = fmaxf(m, red_m[x][g8 * 4 + tg][nb * 2 + i]);
        float l_sum = 0.f;
        for (int x = 0; x < kDecWarps; ++x)
            for (int g8 = 0; g8 < 8; ++g8)
                l_sum += red_l[x][g8 * 4 + tg][nb * 2 + i] * ex2f(red_m[x][g8 * 4 + tg][nb * 2 + i] - m);
        float *o = a.stats + (((size_t)u * a.chunks_max + c) * G + tid) * 2;
        o[0] = m;
        o[1] = l_sum;
    }
}

// fp32 keys: a warp per entry, a lane holds 4 features, the G dot products are reduced by shuffles.
__global__ void __launch_bounds__(kDecThreads) decode_logits_f32_kernel(DecArgs a) {
    __shared__ __align__(16) float qs[16][kD];
    __shared__ float red_m[kDecWarps][16], red_l[kDecWarps][16];
    const int c = blockIdx.x, u = blockIdx.y, G = a.G;
    int64_t off;
    int len;
    if (!unit_ok(a, u, off, len)) return;
    const int n = len + 1;
    const int t0 = c * kDecChunk, t1 = min(n, t0 + kDecChunk);
    if (t0 >= n) return;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const float *qb = (const float *)a.q + (size_t)u * G * kD;
    for (int e = tid; e < G * kD; e += kDecThreads) qs[e / kD][e % kD] = qb[e];
    __syncthreads();
    const float *Kb = (const float *)a.Kc + off * kD;
    const float *kn = (const float *)a.knew + (size_t)u * kD;
    float *lg = a.logits + (off + u) * G;
    float m_run = -1e30f, l_run = 0.f;   // lane g < G keeps the statistics of head g
    for (int t = t0 + wid; t < t1; t += kDecWarps) {
        const float4 k4 = *reinterpret_cast<const float4 *>((t < len ? Kb + (int64_t)t * kD : kn) + lane * 4);
        float mine = 0.f;
        for (int g = 0; g < G; ++g) {
            const float4 q4 = *reinterpret_cast<const float4 *>(&qs[g][lane * 4]);
            float v = fmaf(k4.x, q4.x, fmaf(k4.y, q4.y, fmaf(k4.z, q4.z, k4.w * q4.w)));
            v = warp_sum(v) * a.c_log2;
            if (lane == g) mine = v;
        }
        if (lane < G) {
            lg[(int64_t)t * G + lane] = mine;
            const float m_new = fmaxf(m_run, mine);
            l_run = fmaf(l_run, ex2f(m_run - m_new), ex2f(mine - m_new));
            m_run = m_new;
        }
    }
    if (lane < G) { red_m[wid][lane] = m_run; red_l[wid][lane] = l_run; }
    __syncthreads();
    if (tid < G) {
        float m = -1e30f;
        for (int x = 0; x < kDecWarps; ++x) m = fmaxf(m, red_m[x][tid]);
        float l_sum = 0.f;
        for (int x = 0; x < kDecWarps; ++x) l_sum += red_l[x][tid] * ex2f(red_m[x][tid] - m);
        float *o = a.stats + (((size_t)u * a.chunks_max + c) * G + tid) * 2;
        o[0] = m;
        o[1] = l_sum;
    }
}

__global__ void __launch_bounds__(kDecThreads) decode_accumulate_kernel(DecArgs a, int H_per_seq, const int32_t *new_pos,
                                                                       int protect, const int32_t *pos, float *cum,
                                                                       float *p_out, MinPair *partial, float *new_cum) {
    __shared__ float mprime[16];
    __shared__ MinPair red[kDecWarps];
    const int c = blockIdx.x, u = blockIdx.y, G = a.G, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    int64_t off;
    int len;
    if (!unit_ok(a, u, off, len)) return;
    const int n = len + 1, chunks = (n + kDecChunk - 1) / kDecChunk;
    if (c >= chunks) return;
    if (tid < G) {
        const float *s = a.stats + ((size_t)u * a.chunks_max * G + tid) * 2;
        float m = -1e30f;
        for (int x = 0; x < chunks; ++x) m = fmaxf(m, s[(size_t)x * G * 2]);
        float l = 0.f;
        for (int x = 0; x < chunks; ++x) l += s[(size_t)x * G * 2 + 1] * exp2f(s[(size_t)x * G * 2] - m);
        mprime[tid] = m + log2f(l);
    }
    __syncthreads();
    const int limit = new_pos[u / H_per_seq] - protect;   // candidates have pos <= limit
    const float *lg = a.logits + (off + u) * G;
    MinPair best;
    best.el.c = best.any.c = 0.f;
    best.el.pos = best.any.pos = -1;
    best.el.j = best.any.j = -1;
    const int t1 = min(n, (c + 1) * kDecChunk);
    for (int j = c * kDecChunk + tid; j < t1; j += kDecThreads) {
        float p = 0.f;   // heads in ascending order, whichever load width is used
        if ((G & 3) == 0) {
            const float4 *l4 = reinterpret_cast<const float4 *>(lg + (int64_t)j * G);
            for (int g = 0; g < G; g += 4) {
                const float4 x = l4[g >> 2];
                p += ex2f(x.x - mprime[g]);
                p += ex2f(x.y - mprime[g + 1]);
                p += ex2f(x.z - mprime[g + 2]);
                p += ex2f(x.w - mprime[g + 3]);
            }
        } else {
            for (int g = 0; g < G; ++g) p += ex2f(lg[(int64_t)j * G + g] - mprime[g]);
        }
        if (p_out) p_out[off + u + j] = p;
        if (j < len) {
            const float cn = cum[off + j] + p;
            cum[off + j] = cn;
            const int32_t ps = pos[off + j];
            if (rec_less(cn, ps, best.any)) { best.any.c = cn; best.any.pos = ps; best.any.j = j; }
            if (ps <= limit && rec_less(cn, ps, best.el)) { best.el.c = cn; best.el.pos = ps; best.el.j = j; }
        } else {
            new_cum[u] = p;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        MinPair other;
        other.el.c = __shfl_xor_sync(0xffffffffu, best.el.c, o);
        other.el.pos = __shfl_xor_sync(0xffffffffu, best.el.pos, o);
        other.el.j = __shfl_xor_sync(0xffffffffu, best.el.j, o);
        other.any.c = __shfl_xor_sync(0xffffffffu, best.any.c, o);
        other.any.pos = __shfl_xor_sync(0xffffffffu, best.any.pos, o);
        other.any.j = __shfl_xor_sync(0xffffffffu, best.any.j, o);
        rec_take(best.el, other.el);
        rec_take(best.any, other.any);
    }
    if (lane == 0) red[wid] = best;
    __syncthreads();
    if (tid == 0) {
        for (int x = 1; x < kDecWarps; ++x) { rec_take(best.el, red[x].el); rec_take(best.any, red[x].any); }
        partial[(size_t)u * a.chunks_max + c] = best;
    }
}

__global__ void __launch_bounds__(64) decode_commit_kernel(DecArgs a, int H_per_seq, const int32_t *new_pos,
                                                          const void *vnew, int row_bytes, void *Kc, void *Vc,
                                                          int32_t *pos, float *cum, int32_t *lens, int32_t *evicted,
                                                          const MinPair *partial, const float *new_cum,
                                                          uint32_t *status) {
    __shared__ int slot_s;
    const int u = blockIdx.x, tid = threadIdx.x;
    int64_t off;
    int len;
    if (!unit_ok(a, u, off, len)) {
        if (tid == 0) {
            atomicOr(status, (uint32_t)UNCOMP_STATUS_BOUNDS);
            if (evicted) evicted[u] = -1;
        }
        return;
    }
    const int64_t cap = a.offsets[u + 1] - off;
    if (tid == 0) {
        int slot = len, gone = -1;
        if (len >= cap) {
            const int chunks = (len + 1 + kDecChunk - 1) / kDecChunk;
            MinPair best = partial[(size_t)u * a.chunks_max];
            for (int x = 1; x < chunks; ++x) {
                const MinPair o = partial[(size_t)u * a.chunks_max + x];
                rec_take(best.el, o.el);
                rec_take(best.any, o.any);
            }
            const MinRec &r = best.el.pos >= 0 ? best.el : best.any;
            slot = r.j;
            gone = r.pos;
        } else {
            lens[u] = len + 1;
        }
        if (!UNCOMP_INDEX_OK(slot, cap, status)) slot = -1;       // debug library: the row must lie in the unit's slab
        if (slot >= 0) {
            pos[off + slot] = new_pos[u / H_per_seq];
            cum[off + slot] = new_cum[u];
        }
        if (evicted) evicted[u] = gone;
        slot_s = slot;
    }
    __syncthreads();
    const int slot = slot_s, vecs = row_bytes >> 4;      // 16-byte vectors per row: 16 (bf16) or 32 (fp32)
    if (slot < 0) return;                                // only the debug library can get here
    const int4 *srcK = reinterpret_cast<const int4 *>((const char *)a.knew + (size_t)u * row_bytes);
    const int4 *srcV = reinterpret_cast<const int4 *>((const char *)vnew + (size_t)u * row_bytes);
    int4 *dstK = reinterpret_cast<int4 *>((char *)Kc + (off + slot) * row_bytes);
    int4 *dstV = reinterpret_cast<int4 *>((char *)Vc + (off + slot) * row_bytes);
    if (tid < 32) { if (tid < vecs) dstK[tid] = srcK[tid]; }
    else if (tid - 32 < vecs) dstV[tid - 32] = srcV[tid - 32];
}
// ---- the whole step in one launch: a cluster of CTAs per unit ---------------------------------------------------
// Bound by reading the cached keys once.  A unit is one CTA, or a cluster of 2, 4 or 8 when its cache is large or the
// units are few.  The logits stay in shared memory between the statistics and the probabilities; softmax statistics and
// eviction minima of a cluster meet in distributed shared memory, and CTA 0 writes the new token.  Three CTAs per SM are
// in different phases, so the latency of the barriers hides behind other units' loads; scores, positions and the new
// token's row are prefetched past the barriers.  Against three launches over a logits array in global memory (device
// time, back to back): 1024 caches of 3080 rows 194 -> 145 us = 5.9 TB/s of keys, scores and positions, 256 caches of
// 410 rows 16.0 -> 8.2 us.
constexpr int kStepMaxCluster = 8;
constexpr int kPre = 3;                                  // entries per thread whose score and position are prefetched
constexpr size_t kStepSmem = 200 * 1024;                 // logits of one CTA's share at most

struct StepSmem {
    unsigned long long wkey[kDecWarps][2];
    float red_m[kDecWarps][16], red_l[kDecWarps][16];
    float stat_m[16], stat_l[16];                        // this CTA's softmax statistics per head
    float mprime[16];
    unsigned long long key[kStepMaxCluster][2];          // CTA 0: smallest (cum, pos) of every CTA, old enough / any
    int32_t slot[kStepMaxCluster][2];
    float new_cum;                                       // CTA 0
    int row;
};

// order-preserving image of (cum, pos): the lexicographic minimum is the smallest key
__device__ __forceinline__ unsigned long long min_key(float c, int32_t pos) {
    const uint32_t b = __float_as_uint(c + 0.f);         // -0 and +0 are equal scores
    const uint32_t o = (b & 0x80000000u) ? ~b : (b | 0x80000000u);
    return ((unsigned long long)o << 32) | (uint32_t)pos;
}
__device__ __forceinline__ unsigned long long warp_min(unsigned long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = min(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// logits of the entries t0 .. t1 - 1 to lg[head * pitch + t - t0]; running (max, sum) of this thread's heads
template <int G>
__device__ __forceinline__ void step_logits(const DecArgs &a, int u, int64_t off, int len, int t0, int t1, float *lg, int pitch,
                                            StepSmem &S, __nv_bfloat16) {
    constexpr int NB = (G + 7) / 8;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, gid = lane >> 2, tig = lane & 3;
    const __nv_bfloat16 *qb = (const __nv_bfloat16 *)a.q + (size_t)u * G * kD;
    const __nv_bfloat16 *Kb = (const __nv_bfloat16 *)a.Kc + off * kD;
    const __nv_bfloat16 *kn = (const __nv_bfloat16 *)a.knew + (size_t)u * kD;
    uint32_t bq[NB][16];
#pragma unroll
    for (int nb = 0; nb < NB; ++nb) {
        const int h = nb * 8 + gid;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            uint4 x = make_uint4(0u, 0u, 0u, 0u);
            if (h < G) x = reinterpret_cast<const uint4 *>(qb + (size_t)h * kD)[4 * j + tig];
            bq[nb][4 * j] = x.x; bq[nb][4 * j + 1] = x.y; bq[nb][4 * j + 2] = x.z; bq[nb][4 * j + 3] = x.w;
        }
    }
    float m_run[NB][2], l_run[NB][2];
#pragma unroll
    for (int nb = 0; nb < NB; ++nb)
#pragma unroll
        for (int i = 0; i < 2; ++i) { m_run[nb][i] = -1e30f; l_run[nb][i] = 0.f; }
    for (int base = t0 + wid * 32; base < t1; base += kDecWarps * 32) {
        uint4 ka[2][2][4];
#pragma unroll
        for (int tile = 0; tile < 2; ++tile)
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                const int row = base + tile * 16 + half * 8 + gid;
                const uint4 *src = reinterpret_cast<const uint4 *>(row < len ? Kb + (int64_t)row * kD : kn);
#pragma unroll
                for (int j = 0; j < 4; ++j) ka[tile][half][j] = row < t1 ? src[4 * j + tig] : make_uint4(0u, 0u, 0u, 0u);
            }
#pragma unroll
        for (int tile = 0; tile < 2; ++tile)
#pragma unroll
            for (int nb = 0; nb < NB; ++nb) {
                float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const uint4 lo = ka[tile][0][j], hi = ka[tile][1][j];
                    mma_bf16_16816(acc, lo.x, hi.x, lo.y, hi.y, bq[nb][4 * j], bq[nb][4 * j + 1]);
                    mma_bf16_16816(acc, lo.z, hi.z, lo.w, hi.w, bq[nb][4 * j + 2], bq[nb][4 * j + 3]);
                }
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const int h = nb * 8 + 2 * tig + i;
                    if (h < G) {
#pragma unroll
                        for (int half = 0; half < 2; ++half) {
                            const int t = base + tile * 16 + half * 8 + gid;
                            if (t < t1) {
                                const float v = acc[2 * half + i] * a.c_log2;
                                lg[h * pitch + t - t0] = v;
                                const float m_new = fmaxf(m_run[nb][i], v);
                                l_run[nb][i] = fmaf(l_run[nb][i], ex2f(m_run[nb][i] - m_new), ex2f(v - m_new));
                                m_run[nb][i] = m_new;
                            }
                        }
                    }
                }
            }
    }
    // over the 8 row lanes, then one value per warp and head
#pragma unroll
    for (int nb = 0; nb < NB; ++nb)
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            float m = m_run[nb][i], l = l_run[nb][i];
#pragma unroll
            for (int o = 4; o < 32; o <<= 1) {
                const float mo = __shfl_xor_sync(0xffffffffu, m, o), lo = __shfl_xor_sync(0xffffffffu, l, o);
                const float mn = fmaxf(m, mo);
                l = l * ex2f(m - mn) + lo * ex2f(mo - mn);
                m = mn;
            }
            const int h = nb * 8 + 2 * tig + i;
            if (gid == 0 && h < G) { S.red_m[wid][h] = m; S.red_l[wid][h] = l; }
        }
}

template <int G>
__device__ __forceinline__ void step_logits(const DecArgs &a, int u, int64_t off, int len, int t0, int t1, float *lg, int pitch,
                                            StepSmem &S, float) {
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const float4 *q4 = reinterpret_cast<const float4 *>((const float *)a.q + (size_t)u * G * kD) + lane;
    float4 q[G];
#pragma unroll
    for (int g = 0; g < G; ++g) q[g] = q4[g * (kD / 4)];
    const float *Kb = (const float *)a.Kc + off * kD;
    const float *kn = (const float *)a.knew + (size_t)u * kD;
    float m_run = -1e30f, l_run = 0.f;                   // lane g < G keeps the statistics of head g
    for (int t = t0 + wid; t < t1; t += kDecWarps) {
        const float4 k4 = *reinterpret_cast<const float4 *>((t < len ? Kb + (int64_t)t * kD : kn) + lane * 4);
        float mine = 0.f;
#pragma unroll
        for (int g = 0; g < G; ++g) {
            float v = fmaf(k4.x, q[g].x, fmaf(k4.y, q[g].y, fmaf(k4.z, q[g].z, k4.w * q[g].w)));
            v = warp_sum(v) * a.c_log2;
            if (lane == g) mine = v;
        }
        if (lane < G) {
            lg[lane * pitch + t - t0] = mine;
            const float m_new = fmaxf(m_run, mine);
            l_run = fmaf(l_run, ex2f(m_run - m_new), ex2f(mine - m_new));
            m_run = m_new;
        }
    }
    if (lane < G) { S.red_m[wid][lane] = m_run; S.red_l[wid][lane] = l_run; }
}

struct StepArgs {
    const int32_t *new_pos;
    const void *vnew;
    void *Kc, *Vc;
    int32_t *pos, *lens, *evicted;
    float *cum, *p_out;
    uint32_t *status;
    int H_per_seq, protect, pitch;
};

// The bound of three CTAs leaves 80 registers: enough up to 8 heads per key (16 bytes spilled at most); 16 heads spill 432
// bytes in bf16 and 64 in fp32.
template <int G, typename T>
__global__ void __launch_bounds__(kDecThreads, 3) decode_step_kernel(DecArgs a, StepArgs b) {
    namespace cg = cooperative_groups;
    __shared__ StepSmem S;
    extern __shared__ float lg[];                        // [G][pitch]
    cg::cluster_group cluster = cg::this_cluster();
    const int ctas = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const int u = blockIdx.x / ctas, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    chain_wait();
    // the new token's row and position are not needed before the end: on their way from the start
    constexpr int kVecs = kD * (int)sizeof(T) / 16;      // 16-byte vectors per row
    int4 fresh = make_int4(0, 0, 0, 0);
    if (rank == 0 && tid < 2 * kVecs)
        fresh = (reinterpret_cast<const int4 *>(tid < kVecs ? a.knew : b.vnew) + (size_t)u * kVecs)[tid % kVecs];
    const int32_t newest = b.new_pos[u / b.H_per_seq], limit = newest - b.protect;     // candidates have pos <= limit
    int64_t off;
    int len;
    if (!unit_ok(a, u, off, len)) {                      // uniform over the cluster
        if (tid == 0 && rank == 0) {
            atomicOr(b.status, (uint32_t)UNCOMP_STATUS_BOUNDS);
            if (b.evicted) b.evicted[u] = -1;
        }
        return;
    }
    const int64_t cap = a.offsets[u + 1] - off;
    const bool full = len >= cap;
    const int n = len + 1, share = (n + ctas - 1) / ctas;
    const int t0 = min(n, rank * share), t1 = min(n, t0 + share);
    StepSmem *S0 = cluster.map_shared_rank(&S, 0);

    // ---- logits, softmax statistics over the cluster -------------------------------------------------
    step_logits<G>(a, u, off, len, t0, t1, lg, b.pitch, S, T());
    // cumulative scores and positions of this thread's first entries are on their way during the barriers
    float c_pre[kPre];
    int32_t p_pre[kPre];
#pragma unroll
    for (int i = 0; i < kPre; ++i) {
        const int j = t0 + tid + i * kDecThreads;
        c_pre[i] = j < t1 && j < len ? b.cum[off + j] : 0.f;
        p_pre[i] = j < t1 && j < len ? b.pos[off + j] : 0;
    }
    __syncthreads();
    if (tid < G) {
        float m = -1e30f, l = 0.f;
#pragma unroll
        for (int x = 0; x < kDecWarps; ++x) m = fmaxf(m, S.red_m[x][tid]);
#pragma unroll
        for (int x = 0; x < kDecWarps; ++x) l += S.red_l[x][tid] * ex2f(S.red_m[x][tid] - m);
        S.stat_m[tid] = m;
        S.stat_l[tid] = l;
        if (ctas == 1) S.mprime[tid] = m + log2f(l);
    }
    if (ctas > 1) {
        cluster.sync();
        if (tid < G) {
            float m[kStepMaxCluster], l[kStepMaxCluster], top = -1e30f, sum = 0.f;
#pragma unroll
            for (int c = 0; c < kStepMaxCluster; ++c) {
                const StepSmem *Sc = cluster.map_shared_rank(&S, c < ctas ? c : 0);
                m[c] = c < ctas ? Sc->stat_m[tid] : -1e30f;
                l[c] = c < ctas ? Sc->stat_l[tid] : 0.f;
            }
#pragma unroll
            for (int c = 0; c < kStepMaxCluster; ++c) top = fmaxf(top, m[c]);
#pragma unroll
            for (int c = 0; c < kStepMaxCluster; ++c) sum += l[c] * exp2f(m[c] - top);
            S.mprime[tid] = top + log2f(sum);
        }
    }
    __syncthreads();

    // ---- probabilities, cumulative scores, the lowest of this CTA -------------------------------------
    float mp[G];
#pragma unroll
    for (int g = 0; g < G; ++g) mp[g] = S.mprime[g];
    unsigned long long best_el = ~0ull, best_any = ~0ull;
    int j_el = -1, j_any = -1;
    auto entry = [&](int j, float c_old, int32_t ps) {
        float p = 0.f;                                   // heads in ascending order
#pragma unroll
        for (int g = 0; g < G; ++g) p += ex2f(lg[g * b.pitch + j - t0] - mp[g]);
        if (b.p_out) b.p_out[off + u + j] = p;
        if (j < len) {
            const float cn = c_old + p;
            b.cum[off + j] = cn;
            if (full) {
                const unsigned long long k = min_key(cn, ps);
                if (k < best_any) { best_any = k; j_any = j; }
                if (ps <= limit && k < best_el) { best_el = k; j_el = j; }
            }
        } else {
            S0->new_cum = p;
        }
    };
#pragma unroll
    for (int i = 0; i < kPre; ++i) {
        const int j = t0 + tid + i * kDecThreads;
        if (j < t1) entry(j, c_pre[i], p_pre[i]);
    }
#pragma unroll 4
    for (int j = t0 + tid + kPre * kDecThreads; j < t1; j += kDecThreads)
        entry(j, j < len ? b.cum[off + j] : 0.f, j < len ? b.pos[off + j] : 0);
    if (full) {
        const unsigned long long we = warp_min(best_el), wa = warp_min(best_any);
        if (lane == 0) { S.wkey[wid][0] = we; S.wkey[wid][1] = wa; }
        __syncthreads();
        unsigned long long be = ~0ull, ba = ~0ull;
#pragma unroll
        for (int x = 0; x < kDecWarps; ++x) { be = min(be, S.wkey[x][0]); ba = min(ba, S.wkey[x][1]); }
        // keys are unique inside a unit: the one thread that holds the minimum names its row
        if (be != ~0ull ? best_el == be : tid == 0) { S0->key[rank][0] = be; S0->slot[rank][0] = j_el; }
        if (ba != ~0ull ? best_any == ba : tid == 0) { S0->key[rank][1] = ba; S0->slot[rank][1] = j_any; }
    }
    if (ctas > 1) cluster.sync();
    else __syncthreads();
    if (rank != 0) return;

    // ---- the new token takes its row -----------------------------------------------------------------
    if (tid == 0) {
        int slot = len, gone = -1;
        if (full) {
            unsigned long long k[2] = {~0ull, ~0ull};
            int s[2] = {-1, -1};
            for (int c = 0; c < ctas; ++c)
                for (int w = 0; w < 2; ++w)
                    if (S.key[c][w] < k[w]) { k[w] = S.key[c][w]; s[w] = S.slot[c][w]; }
            const int w = s[0] >= 0 ? 0 : 1;
            slot = s[w];
            gone = (int32_t)(uint32_t)k[w];
        } else {
            b.lens[u] = len + 1;
        }
        if (!UNCOMP_INDEX_OK(slot, cap, b.status)) slot = -1;     // debug library: the row must lie in the unit's slab
        if (slot >= 0) {
            b.pos[off + slot] = newest;
            b.cum[off + slot] = S.new_cum;
        }
        if (b.evicted) b.evicted[u] = gone;
        S.row = slot;
    }
    __syncthreads();
    if (S.row < 0) return;                               // only the debug library can get here
    if (tid < 2 * kVecs)
        (reinterpret_cast<int4 *>(tid < kVecs ? b.Kc : b.Vc) + (off + S.row) * kVecs)[tid % kVecs] = fresh;
}

template <int G, typename T>
cudaError_t launch_step(const DecArgs &a, const StepArgs &b, int units, int ctas, size_t smem, cudaStream_t st) {
    static bool done[64] = {};
    cudaError_t e = allow_dynamic_smem((const void *)decode_step_kernel<G, T>, kStepSmem, done);
    if (e != cudaSuccess) return e;
    return launch_kernel(decode_step_kernel<G, T>, LaunchShape{dim3(units * ctas), kDecThreads, smem, (unsigned)ctas}, st, a, b);
}
template <typename T>
cudaError_t launch_step_g(const DecArgs &a, const StepArgs &b, int units, int ctas, size_t smem, cudaStream_t st) {
    switch (a.G) {
        case 1: return launch_step<1, T>(a, b, units, ctas, smem, st);
        case 2: return launch_step<2, T>(a, b, units, ctas, smem, st);
        case 4: return launch_step<4, T>(a, b, units, ctas, smem, st);
        case 8: return launch_step<8, T>(a, b, units, ctas, smem, st);
        case 16: return launch_step<16, T>(a, b, units, ctas, smem, st);
        default: return cudaErrorInvalidValue;
    }
}

// Cumulative scores right after prefill: a kept prefix position takes its prefill score, a window position the
// largest score among the kept prefix positions of its head (0 if there is none).  One CTA per unit.
__global__ void __launch_bounds__(256) decode_seed_kernel(const float *__restrict__ scores, int P,
                                                         const int32_t *__restrict__ indices,
                                                         const int64_t *__restrict__ offsets, float *__restrict__ cum) {
    __shared__ float red[8];
    const int u = blockIdx.x, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int64_t off = offsets[u];
    const int n = (int)(offsets[u + 1] - off);
    const float *s = scores + (size_t)u * P;
    float top = -INFINITY;
    for (int t = tid; t < n; t += 256) {
        const int j = indices[off + t];
        if (j < P) top = fmaxf(top, s[j]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, o));
    if (lane == 0) red[wid] = top;
    __syncthreads();
    top = red[0];
#pragma unroll
    for (int i = 1; i < 8; ++i) top = fmaxf(top, red[i]);
    if (top == -INFINITY) top = 0.f;
    for (int t = tid; t < n; t += 256) {
        const int j = indices[off + t];
        cum[off + t] = j < P ? s[j] : top;
    }
}
}  // namespace

cudaError_t launch_decode_seed(const Plan &p, const float *d_scores, const int32_t *d_indices, const int64_t *d_offsets,
                               float *d_cum, cudaStream_t st) {
    decode_seed_kernel<<<p.units, 256, 0, st>>>(d_scores, p.prefix, d_indices, d_offsets, d_cum);
    return cudaGetLastError();
}

int decode_chunks(int max_cap) { return (max_cap + 1 + kDecChunk - 1) / kDecChunk; }
size_t decode_partial_bytes() { return sizeof(MinPair); }

cudaError_t launch_decode_update(const Plan &p, const void *d_q, const void *d_knew, const void *d_vnew,
                                 const int32_t *d_new_pos, const int64_t *d_offsets, int32_t *d_lens, int max_cap,
                                 int protect, float scale, void *d_Kc, void *d_Vc, int32_t *d_pos, float *d_cum,
                                 float *d_p, int32_t *d_evicted, float *d_logits, float *d_stats, void *d_partial,
                                 float *d_new_cum, uint32_t *d_status, Profiler *prof, cudaStream_t st) {
    const uncomp_shape &s = p.shape;
    DecArgs a;
    a.q = d_q; a.knew = d_knew; a.Kc = d_Kc; a.offsets = d_offsets; a.lens = d_lens;
    a.units = p.units; a.G = p.G; a.max_cap = max_cap; a.chunks_max = decode_chunks(max_cap);
    a.c_log2 = scale * 1.4426950408889634f;
    a.logits = d_logits; a.stats = d_stats;
    {
        // One launch with the logits in shared memory.  A cluster barrier costs a microsecond of a CTA's time, so a unit
        // stays on one CTA up to 4096 entries (64 KB of logits at 4 heads, three CTAs per SM); beyond, the cluster grows
        // to 8 CTAs, then the share.  Only where the units leave half the SMs idle smaller shares pay.
        int ctas = 1;
        while (ctas < kStepMaxCluster && (max_cap + 1 > 4096 * ctas ||
                                          ((int64_t)p.units * ctas * 2 <= kTargetSms && max_cap + 1 > 512 * ctas)))
            ctas *= 2;
        const int share = (max_cap + 1 + ctas - 1) / ctas;
        StepArgs b;
        b.pitch = (share + 31) / 32 * 32 + 8;            // heads 8 banks apart
        const size_t smem = (size_t)b.pitch * p.G * sizeof(float);
        if (smem <= kStepSmem) {
            b.new_pos = d_new_pos; b.vnew = d_vnew; b.Kc = d_Kc; b.Vc = d_Vc; b.pos = d_pos; b.lens = d_lens;
            b.evicted = d_evicted; b.cum = d_cum; b.p_out = d_p; b.status = d_status;
            b.H_per_seq = s.L * s.H; b.protect = protect;
            ProfScope ps(prof, kSlotDecodeStep, st);
            return s.dtype == UNCOMP_FP32 ? launch_step_g<float>(a, b, p.units, ctas, smem, st)
                                          : launch_step_g<__nv_bfloat16>(a, b, p.units, ctas, smem, st);
        }
    }
    // caches whose logits do not fit into the shared memory of a cluster: three launches over a global logits array
    const dim3 grid(a.chunks_max, p.units);
    const int row_bytes = kD * (s.dtype == UNCOMP_FP32 ? 4 : 2);
    {
        ProfScope ps(prof, kSlotDecodeLogits, st);
        if (s.dtype == UNCOMP_FP32) decode_logits_f32_kernel<<<grid, kDecThreads, 0, st>>>(a);
        else switch (p.G) {
            case 1: decode_logits_mma_kernel<1><<<grid, kDecThreads, 0, st>>>(a); break;
            case 2: decode_logits_mma_kernel<2><<<grid, kDecThreads, 0, st>>>(a); break;
            case 4: decode_logits_mma_kernel<4><<<grid, kDecThreads, 0, st>>>(a); break;
            case 8: decode_logits_mma_kernel<8><<<grid, kDecThreads, 0, st>>>(a); break;
            case 16: decode_logits_mma_kernel<16><<<grid, kDecThreads, 0, st>>>(a); break;
            default: return cudaErrorInvalidValue;
        }
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    {
        ProfScope ps(prof, kSlotDecodeAccumulate, st);
        decode_accumulate_kernel<<<grid, kDecThreads, 0, st>>>(a, s.L * s.H, d_new_pos, protect, d_pos, d_cum, d_p,
                                                               (MinPair *)d_partial, d_new_cum);
    }
    {
        ProfScope ps(prof, kSlotDecodeCommit, st);
        decode_commit_kernel<<<p.units, 64, 0, st>>>(a, s.L * s.H, d_new_pos, d_vnew, row_bytes, d_Kc, d_Vc, d_pos, d_cum,
                                                     d_lens, d_evicted, (const MinPair *)d_partial, d_new_cum, d_status);
    }
    return cudaGetLastError();
}

}  // namespace uncomp
