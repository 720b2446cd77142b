// Observation-window scores for bf16 keys on the tcgen05 tensor cores (paper Section 3.3.3, "Dynamic KV
// Cache Eviction": the attention of the last w query positions, summed per key position).
//
// Two kernels with one pipeline skeleton; softmax needs the row statistics before the column sums:
//   pass A  S = Qw K^T with the window rows on the TMEM lanes (M = 128 rows, N = 128 tokens per MMA tile):
//           a thread owns a row, so its running maximum and sum of exponentials are thread-local;
//           every (unit, chunk) writes partial statistics (m, l) in the log2 domain;
//           pass B combines them in index order into m'_r = m_r + log2 l_r when it comes to a unit;
//   pass B  operands swapped (M = 128 tokens on the lanes, N = 128 rows): a thread owns a token and adds
//           2^(s c - m'_r) along its TMEM row; tokens of a warp are consecutive, the store is coalesced.
// K tiles (128 tokens x 128 features, two 128B-swizzled boxes of 64 features) stream through a TMA ring;
// the unit's window queries stay in shared memory for the whole CTA.  Both operands are K-major.
//
// One CTA per SM works through its share of the (unit, token chunk) items.  The TMA producer runs ahead into the next item,
// so a CTA's pipeline fills once and not once per item (a CTA per item spent 8,000 of 38,000 cycles on a 3712-token unit
// before its first tile arrived and 6,000 after its last).
// Warps 0-15 softmax in two groups of eight that take alternate 128-row blocks or token tiles (so the four
// warps of an SM sub-partition are in different phases: while one group waits for its accumulator, the
// other keeps the exponential unit busy); inside a group warp % 4 selects the TMEM lane quarter and bit 2
// of the warp index the 64-column half of an accumulator.  Warp 16 is the TMA producer, warp 17 allocates
// TMEM and issues the MMAs: one ELECTED lane (elect.sync lets the compiler keep descriptors in uniform registers; with
// `lane == 0` an MMA took 130 cycles to issue, twice what the tensor pipe needs for it, and paced the kernel).  The
// 128-column accumulators are four buffers in modes 0 and 1, two in modes 2 and 3.
// Mode 2 of the kernel is pass A with the Gram stage folded in: the K tile that is in shared memory for
// Qw K^T is also the MN-major operand of G += K_tile^T K_tile, so the entropy stage costs no second sweep
// over K.  The column sums s = K^T 1 come out of the same MMAs, as 16 more columns whose operand is ones.  (Two warps that
// read the tile from shared memory once more took a sixth of what the MMAs and TMA leave of its bandwidth: 256 units of 8192
// tokens 128.5 us, now 123; 1024 of 3712 205, now 190; of 32768 2052, now 1995; 256 of 32768 with two row blocks 833, now
// 803.  From global memory, 3,000 cycles of latency per tile paced the kernel.)  The errors are those of the warps' fp32 sums:
// entropies of keys with means of 0, 1, 10 and 100 times their spread are as far from 64 bits as before.
// Mode 3 is pass B with the Gram stage folded in the same way, for callers who bring the row normalisers (their
// prefill attention kernel's log-sum-exp): entropy stage and scores from ONE sweep over K.
// What bounds it.  The clock that power allows, 1.6 to 1.7 GHz from the first pass on (four row blocks 1.83), repeated for more
// than half a second 1.75 (8192 and 131072 tokens), 1.57 (32768) or 1.40 GHz (4 x 32768) at 985 W; and at that clock, with two
// row blocks or more, the exponential unit, 75 % (mode 2) and 80 % (mode 1) busy: 2,700 and 2,540 cycles per tile of two row
// blocks, which need 2,048 of it.  The exponential loops alone keep it 97 % busy with two warps per scheduler.  Letting the
// groups take turns on it (named barriers) was slower (1,600 cycles per block against 1,300), three accumulators beside the
// Gram block and blocks by tile in pass A were the same.  One row block: shared memory (the MMAs read 128 bytes per cycle, which
// is all it has) and, in mode 1, HBM (5.4 TB/s).
// Every wait is bounded; a timeout raises UNCOMP_STATUS_TIMEOUT and the CTA drains and exits.
#include "tc_common.cuh"

namespace uncomp {

namespace {
constexpr int kTile = 128;
constexpr int kHalfBytes = 128 * 128;            // 64 features x 128 rows/tokens, bf16
constexpr int kBlockBytes = 2 * kHalfBytes;      // one K tile or one block of 128 query rows
constexpr int kNB = 4;                           // accumulator buffers (x 128 TMEM columns = all 512)
constexpr int kSoftThreads = 512;
constexpr int kScoreThreads = kSoftThreads + 64;
// The compiler may use 96 registers, as if there were two more warps.  With the 112 that 576 threads leave it puts the
// loads of the normalisers elsewhere: column sums of 1024 units of 32768 tokens 1865 us against 1600 (88 registers 1763, 80
// 1823).
constexpr int kBoundThreads = kScoreThreads + 64;
constexpr int kMaxStages = 4;

struct ScoreTail {
    uint64_t full[kMaxStages], empty[kMaxStages], qfull[2], qempty[2], tfull[2 * kNB], tempty[kNB], gfull, gdrained;
    uint32_t tmem_base;
};

__host__ __device__ constexpr int score_stages(int MB) { return MB <= 2 ? 4 : (MB == 3 ? 3 : 2); }
__host__ __device__ constexpr int query_buffers(int MB) { return MB == 1 ? 2 : 1; }

// Places in shared memory, in halves (16 KB: 64 features of a K tile or of 128 query rows).  Without the Gram stage: queries, then
// stages.  With it (modes 2 and 3) half kOnesHalf is filled with ones, and the halves of stage s lie at kOnesHalf - 2 x and
// kOnesHalf - x, so that to the tensor core, which finds the 64-feature regions of an MN-major operand at equal distances, the
// ones are features 128 .. of every tile: N = 144 instead of 128 columns give the Gram block and, in the last 16, the column
// sums.  x = 1, 3, 4, 5 keeps all of them apart; the queries take what is left.
constexpr int kOnesHalf = 12;
__host__ __device__ constexpr int stage_x(int s) { return s + 1 + (s != 0); }
template <bool GRAM> __host__ __device__ constexpr int stage_half(int MB, int s, int h) {
    return GRAM ? kOnesHalf - (2 - h) * stage_x(s) : 2 * (query_buffers(MB) * MB + s) + h;
}
// the i-th half that no stage takes
__host__ __device__ constexpr int free_half(int MB, int i) {
    return MB <= 2 ? i + (i > 1) + (i > 2) : (MB == 3 ? i + (i > 3) + (i > 4) : i + (i > 5));
}
constexpr bool halves_apart(int MB) {
    bool taken[kOnesHalf + 1] = {}, ok = true;
    for (int s = 0; s < score_stages(MB); ++s)
        for (int h = 0; h < 2; ++h) {
            const int at = stage_half<true>(MB, s, h);
            ok = ok && at >= 0 && at < kOnesHalf && !taken[at];
            taken[at] = true;
        }
    for (int i = 0; i < 2 * query_buffers(MB) * MB; ++i) {
        const int at = free_half(MB, i);
        ok = ok && at >= 0 && at < kOnesHalf && !taken[at];
        taken[at] = true;
    }
    return ok;
}
static_assert(halves_apart(1) && halves_apart(2) && halves_apart(3) && halves_apart(4), "every half has one owner");
template <bool GRAM> __host__ __device__ constexpr int query_half(int MB, int buf, int mb, int h) {
    return GRAM ? free_half(MB, 2 * (buf * MB + mb) + h) : 2 * (buf * MB + mb) + h;
}
__host__ __device__ constexpr int score_halves(int MB, bool gram) {
    return gram ? kOnesHalf + 1 : 2 * (query_buffers(MB) * MB + score_stages(MB));
}
// pass B: normalisers of two units and column sums; pass A: statistics to be merged
__host__ __device__ constexpr int score_smem(int MB, int mode) {
    return 1024 + score_halves(MB, mode >= 2) * kHalfBytes + (mode == 1 || mode == 3 ? 2 * MB * 128 * 4 + 2 * 4 * 128 * 4 : 4 * MB * 128 * 8) +
           (int)sizeof(ScoreTail);
}
static_assert(score_smem(4, 2) <= 227 * 1024 && score_smem(4, 0) <= 227 * 1024, "shared memory of one CTA");

__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ void all_soft_barrier() { asm volatile("bar.sync 3, 512;" ::: "memory"); }
__device__ __forceinline__ void group_barrier(int g) { asm volatile("bar.sync %0, 256;" ::"r"(1 + g) : "memory"); }
__device__ __forceinline__ float max3(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// Pass A: fold NC logits of one row into its running (m, l), log2 domain.  m only has to stay at or above
// every logit seen so far (it is the exact running maximum here, raised lazily), l = sum 2^(x c - m).  Multiply-adds and
// sums work on pairs.
template <bool MASKED, int NC>
__device__ __forceinline__ void stats_update(uint32_t (&v)[NC], float c_log2, int pos0, int last, float &m_run,
                                             float &l_run) {
    if (MASKED) {
#pragma unroll
        for (int j = 0; j < NC; ++j)
            if (pos0 + j > last) v[j] = 0xff800000u;            // -inf: not visible to this row
    }
    float pm[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
    for (int j = 0; j < NC; j += 8) {
        pm[0] = max3(pm[0], __uint_as_float(v[j]), __uint_as_float(v[j + 1]));
        pm[1] = max3(pm[1], __uint_as_float(v[j + 2]), __uint_as_float(v[j + 3]));
        pm[2] = max3(pm[2], __uint_as_float(v[j + 4]), __uint_as_float(v[j + 5]));
        pm[3] = max3(pm[3], __uint_as_float(v[j + 6]), __uint_as_float(v[j + 7]));
    }
    const float mx = fmaxf(fmaxf(pm[0], pm[1]), fmaxf(pm[2], pm[3])) * c_log2;
    if (mx > m_run) {                                           // rare after the first tiles
        l_run *= ex2(m_run - mx);
        m_run = mx;
    }
    if (m_run > -INFINITY) {
        const f32x2 c2 = pack2(c_log2, c_log2), m2 = pack2(-m_run, -m_run);
        f32x2 sum[2] = {0ull, 0ull};
#pragma unroll
        for (int j = 0; j < NC; j += 2) {
            float a, b;
            unpack2(fma2(pack2(__uint_as_float(v[j]), __uint_as_float(v[j + 1])), c2, m2), a, b);
            sum[(j >> 1) & 1] = add2(sum[(j >> 1) & 1], pack2(ex2(a), ex2(b)));
        }
        l_run += sum2(sum[0]) + sum2(sum[1]);
    }
}

// Pass B: sum over NC window rows of 2^(s c - m'_r) for one token; `mneg` holds -m'_r.
template <int NC>
__device__ __forceinline__ float colsum_partial(const uint32_t (&v)[NC], float c_log2, const float *mneg) {
    const f32x2 c2 = pack2(c_log2, c_log2);
    f32x2 acc[2] = {0ull, 0ull};
#pragma unroll
    for (int j = 0; j < NC; j += 4) {
        const ulonglong2 m4 = *reinterpret_cast<const ulonglong2 *>(mneg + j);
        float a, b;
        unpack2(fma2(pack2(__uint_as_float(v[j]), __uint_as_float(v[j + 1])), c2, m4.x), a, b);
        acc[0] = add2(acc[0], pack2(ex2(a), ex2(b)));
        unpack2(fma2(pack2(__uint_as_float(v[j + 2]), __uint_as_float(v[j + 3])), c2, m4.y), a, b);
        acc[1] = add2(acc[1], pack2(ex2(a), ex2(b)));
    }
    return sum2(acc[0]) + sum2(acc[1]);
}

// NC columns of this warp's 32 TMEM lanes
template <int NC>
__device__ __forceinline__ void load_columns(uint32_t taddr, uint32_t (&v)[NC]) {
    if constexpr (NC == 16) {
        tc::tmem_ld16(taddr, v);
        tc::tmem_ld_wait();
    } else if constexpr (NC == 32) {
        tc::tmem_ld32(taddr, v);
        tc::tmem_ld_wait();
    } else {
        uint32_t va[32], vb[32];
        tc::tmem_ld32(taddr, va);
        tc::tmem_ld32(taddr + 32, vb);
        tc::tmem_ld_wait();
#pragma unroll
        for (int j = 0; j < 32; ++j) { v[j] = va[j]; v[32 + j] = vb[j]; }
    }
}
}  // namespace

// m'_r of row r of unit u in the log2 domain, for pass B: from the caller's log-sum-exp, or from the partial (m, l) of pass A,
// combined in chunk order.  A non-finite log-sum-exp raises UNCOMP_STATUS_NONFINITE and its row adds nothing.
__device__ __forceinline__ float row_norm(const float *__restrict__ stats, int parts, const float *__restrict__ lse, size_t u, int r,
                                          int rows, uint32_t *status) {
    if (lse) {
        const float v = lse[u * rows + r];
        if (isfinite(v)) return v * 1.4426950408889634f;
        atomicOr(status, (uint32_t)UNCOMP_STATUS_NONFINITE);
        return INFINITY;
    }
    const float2 *s = reinterpret_cast<const float2 *>(stats) + u * parts * kMaxRows + r;
    float m = -INFINITY, l = 0.f;
#pragma unroll 4
    for (int p = 0; p < parts; ++p) m = fmaxf(m, s[(size_t)p * kMaxRows].x);
#pragma unroll 4
    for (int p = 0; p < parts; ++p) {
        const float2 x = s[(size_t)p * kMaxRows];
        if (x.x > -INFINITY) l += x.y * exp2f(x.x - m);
    }
    return m + log2f(l);
}

// MODE 0: pass A, 1: pass B, 2: pass A fused with the Gram stage, 3: pass B fused with it.
// SPLIT 2 and 4 (MB = 1 only): at most 64 or 32 window rows.  A block of 128 rows would be mostly padding, and every
// padded row costs as many exponentials as a real one.  Pass A keeps M = 128 but fills it with SPLIT copies of the rows;
// the lanes of a copy take their own part of the tile's tokens.  Pass B takes N = 128 / SPLIT instead of 128.  (Copies of
// 16 rows were no faster: the keys' bandwidth and the Gram MMAs bound it then.)
template <int MB, int MODE, int SPLIT>
__global__ void __launch_bounds__(kBoundThreads, 1)
score_tc_kernel(const __grid_constant__ CUtensorMap tmapQ, const __grid_constant__ CUtensorMap tmapK, int L, int H,
                int N, int w, int rows, int units, int chunk, int splits, float c_log2, float *__restrict__ stats_part,
                const float *__restrict__ stats_in, int stats_splits, const float *__restrict__ lse, float *__restrict__ raw,
                float *__restrict__ gram_part,
                uint32_t *__restrict__ status) {
    constexpr bool PASS_B = MODE == 1 || MODE == 3, GRAM = MODE >= 2, RING = MODE != 1;
    // Accumulator buffers (128 TMEM columns each).  An accumulator holds one 128-row block of one tile; blocks are counted over
    // everything the CTA does, block (tile n, mb) is number n MB + mb.
    // RING: the buffers are used in the order of the blocks.  Pass A: blocks go to the two softmax groups in turn, whichever
    // tile they belong to, so both groups always have one (four buffers without the Gram stage, two beside it: an accumulator is
    // free again as soon as its values are in registers, a third made no difference).
    // Pass B: a token's sum takes all blocks of its tile, so tile n belongs to group n & 1.  Mode 1: four buffers, two owned
    // by each group, which it fills alternately (so each group runs up to two blocks ahead, independent of the other).
    constexpr int NB = GRAM ? 2 : kNB;
    // RING: "block q is ready" is signalled on barrier q % NF.  A softmax group that waits for its next block may get
    // there before the blocks in between have completed, and the parity of an unfinished phase could not be told from the one
    // waited for: the user of the barrier before, block q - NF, must not lie behind the last block this group has consumed,
    // which is q - MB - 1 at the earliest.
    constexpr int NF = RING ? 2 * kNB : kNB;
    static_assert(!RING || NF > MB, "see above");
    // block -> buffer, ready barrier and its parity, and the drain phase the MMA thread waits for
    // (-1: the buffer has not been used yet)
    auto item_buf = [](int n, int mb) { return RING ? (n * MB + mb) % NB : 2 * (n & 1) + (((n >> 1) * MB + mb) & 1); };
    auto item_ready_bar = [](int n, int mb) { return RING ? (n * MB + mb) % NF : 2 * (n & 1) + (((n >> 1) * MB + mb) & 1); };
    auto item_ready_parity = [](int n, int mb) { return RING ? ((n * MB + mb) / NF) & 1 : ((((n >> 1) * MB + mb) >> 1) & 1); };
    auto item_drain_phase = [](int n, int mb) { return RING ? (n * MB + mb) / NB - 1 : ((((n >> 1) * MB + mb) >> 1) - 1); };
    constexpr uint32_t kGramCol = NB * 128;          // TMEM columns of the Gram block (modes 2 and 3): 128 and 16 of column sums
    constexpr int kRows = 128 / SPLIT;               // rows of a copy (pass A), columns of an accumulator (pass B)
    constexpr int NC = 64 / SPLIT;                   // logits a thread takes from an accumulator
    static_assert(kRows >= 32, "a TMEM load has one address per warp: a warp belongs to one copy");
    static_assert(SPLIT == 1 || MB == 1, "more than 128 rows are never split");
    constexpr int S = score_stages(MB), QB = query_buffers(MB);
    extern __shared__ unsigned char smem_raw[];
    const uint32_t raw_addr = tc::smem_u32(smem_raw);
    const uint32_t pad = (1024u - (raw_addr & 1023u)) & 1023u;
    unsigned char *smem = smem_raw + pad;
    const uint32_t base = raw_addr + pad;
    auto stage_addr = [&](int st, int h) { return base + (uint32_t)(stage_half<GRAM>(MB, st, h) * kHalfBytes); };
    auto query_addr = [&](int buf, int mb, int h) {
        const int at = QB == 2 && buf ? query_half<GRAM>(MB, 1, mb, h) : query_half<GRAM>(MB, 0, mb, h);
        return base + (uint32_t)(at * kHalfBytes);
    };
    unsigned char *behind = smem + score_halves(MB, GRAM) * kHalfBytes;
    float *mp = reinterpret_cast<float *>(behind);                                 // pass B: [2][MB * 128], by unit
    float *colsum = mp + 2 * MB * 128;                                             // pass B: [2][4][128]
    float2 *merge = reinterpret_cast<float2 *>(behind);                            // pass A: [4][MB * 128]
    ScoreTail &T = *reinterpret_cast<ScoreTail *>(behind + (PASS_B ? 2 * MB * 128 * 4 + 2 * 4 * 128 * 4 : 4 * MB * 128 * 8));

    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const int P = N - w;
    const int limit = (PASS_B && !GRAM) ? P : N;   // pass B only scores the prefix; the Gram stage needs every token
    // this CTA's share of the work items; item j is chunk j % splits of unit j / splits
    const int64_t total = (int64_t)units * splits;
    const int first = (int)(total * blockIdx.x / gridDim.x), last_item = (int)(total * (blockIdx.x + 1) / gridDim.x);
    auto tiles_of = [&](int j) {
        const int t0 = (j % splits) * chunk;
        return (min(limit, t0 + chunk) - t0 + kTile - 1) / kTile;
    };

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            tc::mbar_init(tc::smem_u32(&T.full[s]), 1);
            tc::mbar_init(tc::smem_u32(&T.empty[s]), 1);
        }
        for (int q = 0; q < QB; ++q) {
            tc::mbar_init(tc::smem_u32(&T.qfull[q]), 1);
            tc::mbar_init(tc::smem_u32(&T.qempty[q]), 1);
        }
        tc::mbar_init(tc::smem_u32(&T.gfull), 1);
        tc::mbar_init(tc::smem_u32(&T.gdrained), kSoftThreads / 32);
        for (int i = 0; i < 2 * kNB; ++i) tc::mbar_init(tc::smem_u32(&T.tfull[i]), 1);
        for (int i = 0; i < kNB; ++i) tc::mbar_init(tc::smem_u32(&T.tempty[i]), kSoftThreads / 64);   // the 8 warps of one group
        tc::fence_mbar_init();
    }
    if (GRAM) {                                        // ones; what the tensor core reads goes through the asynchronous proxy
        uint4 *ones = reinterpret_cast<uint4 *>(smem + kOnesHalf * kHalfBytes);
        for (int i = threadIdx.x; i < kHalfBytes / 16; i += kScoreThreads) ones[i] = make_uint4(0x3f803f80u, 0x3f803f80u, 0x3f803f80u, 0x3f803f80u);
        tc::fence_proxy_async();
    }
    if (warp == 17) {
        tc::tmem_alloc(tc::smem_u32(&T.tmem_base), 512);
        tc::tmem_relinquish();
    }
    if (warp == 16 && lane == 0) {
        tc::prefetch_tmap(&tmapQ);
        tc::prefetch_tmap(&tmapK);
    }
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = T.tmem_base;
    chain_wait();               // barriers, TMEM and descriptors are ready by then

    if (warp == 16) {
        // ---------------- TMA producer: runs ahead into the next items ----------------
        if (lane == 0) {
            int n = 0, useq = -1, cur_u = -1, q_sent = 0;      // tiles sent, units seen, query blocks sent
            bool ok = true, q_pending = false;
            auto q_free = [&]() {
                return useq < QB || tc::mbar_test_wait(tc::smem_u32(&T.qempty[useq % QB]), ((useq / QB) - 1) & 1);
            };
            auto send_q = [&]() {
                constexpr int kCopies = PASS_B ? 1 : SPLIT;
                const uint32_t bar = tc::smem_u32(&T.qfull[useq % QB]);
                tc::mbar_expect_tx(bar, MB * kCopies * (kBlockBytes / SPLIT));
                for (int mb = 0; mb < MB; ++mb)
                    for (int cp = 0; cp < kCopies; ++cp) {
                        const uint32_t at = cp * (kHalfBytes / SPLIT);
                        tc::tma_load_3d(query_addr(useq % QB, mb, 0) + at, &tmapQ, bar, 0, mb * 128, cur_u);
                        tc::tma_load_3d(query_addr(useq % QB, mb, 1) + at, &tmapQ, bar, 64, mb * 128, cur_u);
                    }
                q_pending = false;
                ++q_sent;
            };
            // the queries' buffer may still be in use by the unit before: key tiles go ahead, the queries as soon as it is free
            auto wait_q = [&]() {
                if (useq >= QB) ok = tc::mbar_wait(tc::smem_u32(&T.qempty[useq % QB]), ((useq / QB) - 1) & 1, status);
                if (ok) send_q();
            };
            for (int j = first; j < last_item && ok; ++j) {
                const int u = j / splits, t0 = (j % splits) * chunk, ntiles = tiles_of(j);
                const int h = u % H, l = (u / H) % L, b = u / (H * L);
                if (u != cur_u) {
                    if (q_pending) wait_q();
                    if (!ok) break;
                    cur_u = u;
                    ++useq;
                    q_pending = true;
                    if (q_free()) send_q();
                }
                for (int i = 0; i < ntiles; ++i, ++n) {
                    const int s = n % S;
                    if (n >= S) {
                        const uint32_t bar = tc::smem_u32(&T.empty[s]), parity = ((n / S) - 1) & 1;
                        uint32_t spins = 0;
                        while (q_pending && !tc::mbar_test_wait(bar, parity) && ++spins < tc::kSpinLimit)
                            if (q_free()) send_q();
                        ok = tc::mbar_wait(bar, parity, status);
                        if (!ok) break;
                    }
                    const uint32_t bar = tc::smem_u32(&T.full[s]);
                    tc::mbar_expect_tx(bar, kBlockBytes);
                    tc::tma_load_5d(stage_addr(s, 0), &tmapK, bar, 0, t0 + i * kTile, h, l, b);
                    tc::tma_load_5d(stage_addr(s, 1), &tmapK, bar, 64, t0 + i * kTile, h, l, b);
                    if (q_pending && q_free()) send_q();
                }
            }
            if (ok && q_pending) wait_q();
            if (!ok) {   // let the copies in flight land before the CTA may exit (bounded)
                for (int q = max(0, q_sent - QB); q < q_sent; ++q)
                    tc::mbar_wait(tc::smem_u32(&T.qfull[q % QB]), (q / QB) & 1, status);
                for (int i = max(0, n - S); i < n; ++i)
                    tc::mbar_wait(tc::smem_u32(&T.full[i % S]), (i / S) & 1, status);
            }
        }
    } else if (warp == 17) {
        // ---------------- MMA issue ----------------
        if (tc::elect_one()) {
            constexpr uint32_t idesc = tc::idesc_bf16_f32(128, PASS_B ? kRows : 128, 0, 0);
            // descriptors: K-major, 128-byte swizzle, 8-row groups 1024 B apart.  Only the address field
            // (16-byte units) of the lower half changes: +2 per 16 features inside a 128-byte row.
            auto half_desc = [](uint32_t addr) { return tc::desc_lo(tc::smem_desc_sw128(addr, 16, 1024)); };
            const uint32_t dhi = tc::desc_hi(tc::smem_desc_sw128(base, 16, 1024));
            int n = 0, useq = -1, cur_u = -1, iseq = 0, item_start = 0;
            bool ok = true;
            bool have_tile = false, have_buf = false;   // known of the next tile before this one's Gram MMAs are issued
            // Modes 2 and 3: the Gram MMAs of a tile only have to be issued before its stage is handed back, so they
            // are deferred by up to one tile: the latency-critical QK^T MMAs never queue behind them, and while the
            // tensor pipe works on them this thread finds out about the next tile and accumulator.
            // One 128-row block per tile: little waits behind the Gram MMAs, and issuing them at once frees the stage earlier
            // (1024 units of 3712 tokens 188 us, 196 with the lag; 256 of 8192 124 and 127).  With more blocks the lag pays: two
            // in mode 3 751 us with it, 758 without (256 units of 32768), four in mode 2 725 and 730 (32 units of 131072), two in
            // mode 2 756 both.
            constexpr int kLag = MB == 1 ? 0 : 1;
            int g_done = 0;                    // tiles whose Gram MMAs are issued (and whose stage is released)
            auto issue_gram = [&]() {
                constexpr uint32_t idesc_g = tc::idesc_bf16_f32(128, 144, 1, 1);
                const int t = g_done, sg = t % S;
                if (t == item_start && iseq > 0) {      // the softmax warps have read the item before
                    ok = tc::mbar_wait(tc::smem_u32(&T.gdrained), (iseq - 1) & 1, status);
                    tc::tc_fence_after();
                    if (!ok) return;
                }
                const uint32_t g_lo = tc::desc_lo(tc::smem_desc_sw128(stage_addr(sg, 0), (uint32_t)(stage_x(sg) * kHalfBytes), 1024));
#pragma unroll
                for (int k = 0; k < kTile / 16; ++k) {
                    // the same stage read MN-major (feature halves and the ones equally far apart, 8-token groups 1024 B
                    // apart); 16 tokens further = +128 address units
                    const uint32_t acc = (t > item_start || k > 0) ? 1u : 0u;
                    tc::mma_f16_ss_lohi(tmem + kGramCol, g_lo + k * 128, g_lo + k * 128, dhi, idesc_g, acc);
                }
                tc::mma_commit(tc::smem_u32(&T.empty[sg]));
                ++g_done;
            };
            for (int j = first; j < last_item && ok; ++j) {
                const int u = j / splits, ntiles = tiles_of(j);
                const bool more = j + 1 < last_item;
                if (u != cur_u) {
                    cur_u = u;
                    ++useq;
                    ok = tc::mbar_wait(tc::smem_u32(&T.qfull[useq % QB]), (useq / QB) & 1, status);
                }
                const bool leaves_q = !more || (j + 1) / splits != u;      // the unit's last item of this CTA
                item_start = n;
                for (int i = 0; i < ntiles && ok; ++i, ++n) {
                    const int s = n % S;
                    if (!have_tile) ok = tc::mbar_wait(tc::smem_u32(&T.full[s]), (n / S) & 1, status);
                    if (!ok) break;
                    const uint32_t k_lo[2] = {half_desc(stage_addr(s, 0)), half_desc(stage_addr(s, 1))};
#pragma unroll
                    for (int mb = 0; mb < MB; ++mb) {
                        // the block's buffer must have been drained of its previous block
                        const int buf = item_buf(n, mb), drain = item_drain_phase(n, mb);
                        if (ok && drain >= 0 && !(mb == 0 && have_buf)) {
                            const uint32_t bar = tc::smem_u32(&T.tempty[buf]);
                            const uint32_t parity = drain & 1;
                            if (GRAM) {
                                while (ok && g_done < n && !tc::mbar_test_wait(bar, parity)) issue_gram();
                            }
                            if (ok) ok = tc::mbar_wait(bar, parity, status);
                        }
                        if (!ok) break;
                        tc::tc_fence_after();
                        const uint32_t d_tmem = tmem + buf * 128;
                        const uint32_t q_lo[2] = {half_desc(query_addr(useq % QB, mb, 0)), half_desc(query_addr(useq % QB, mb, 1))};
#pragma unroll
                        for (int k = 0; k < 8; ++k) {
                            const uint32_t kd = k_lo[k >> 2] + (k & 3) * 2, qd = q_lo[k >> 2] + (k & 3) * 2;
                            if (PASS_B) tc::mma_f16_ss_lohi(d_tmem, kd, qd, dhi, idesc, k > 0);
                            else tc::mma_f16_ss_lohi(d_tmem, qd, kd, dhi, idesc, k > 0);
                        }
                        tc::mma_commit(tc::smem_u32(&T.tfull[item_ready_bar(n, mb)]));
                    }
                    if (!ok) break;
                    if (leaves_q && i == ntiles - 1) tc::mma_commit(tc::smem_u32(&T.qempty[useq % QB]));
                    if (!GRAM) tc::mma_commit(tc::smem_u32(&T.empty[s]));
                    const int m = n + 1, nd = item_drain_phase(m, 0);
                    const bool next = i + 1 < ntiles || more;
                    have_tile = next && tc::mbar_test_wait(tc::smem_u32(&T.full[m % S]), (m / S) & 1);
                    have_buf = next && nd >= 0 && tc::mbar_test_wait(tc::smem_u32(&T.tempty[item_buf(m, 0)]), nd & 1);
                    if (GRAM) {
                        while (ok && g_done < n + 1 - kLag) issue_gram();  // at most kLag tiles may stay pending
                    }
                }
                if (GRAM && ok) {
                    while (ok && g_done < n) issue_gram();
                    if (ok) tc::mma_commit(tc::smem_u32(&T.gfull));
                    ++iseq;
                }
            }
        }
    } else {
        // ---------------- softmax warps ----------------
        const int quarter = warp & 3, half = (warp >> 2) & 1, group = warp >> 3;
        const int lane_row = quarter * 32 + lane;          // TMEM lane: a window row (A) or a token (B)
        const int copy = PASS_B ? 0 : lane_row / kRows;    // pass A: the copy of the rows this lane belongs to
        const int col0 = PASS_B ? half * NC : half * 64 + copy * NC;
        const uint32_t tbase = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)col0;
        bool dead = false;
        int n0 = 0, useq = -1, cur_u = -1;                 // tiles before this item, units seen
        for (int j = first; j < last_item; ++j) {
            const int u = j / splits, t0 = (j % splits) * chunk, t1 = min(limit, t0 + chunk), ntiles = tiles_of(j);
            if (PASS_B && u != cur_u) {
                // two arrays in turn: the one written here belonged to the unit before the last, which everyone has left
                // since the barrier of the last
                cur_u = u;
                ++useq;
                for (int r = threadIdx.x; r < MB * 128; r += kSoftThreads)
                    mp[(useq & 1) * (MB * 128) + r] =
                        r < rows ? -row_norm(stats_in, stats_splits, lse, (size_t)u, r, rows, status) : -INFINITY;
                all_soft_barrier();
            }
            const float *mpu = mp + (useq & 1) * (MB * 128);
            float m_run[MB], l_run[MB];
#pragma unroll
            for (int mb = 0; mb < MB; ++mb) { m_run[mb] = -INFINITY; l_run[mb] = 0.f; }

            for (int i = PASS_B ? group ^ (n0 & 1) : 0; i < ntiles; i += PASS_B ? 2 : 1) {    // pass B: this group's tiles
                const int n = n0 + i, tile_t0 = t0 + i * kTile;
                const bool masked = tile_t0 + kTile > P;            // uniform over the CTA
                float acc = 0.f;
#pragma unroll
                for (int mb = 0; mb < MB; ++mb) {
                    if (!PASS_B && ((n * MB + mb) & 1) != group) continue;            // pass A: this group's blocks
                    const int buf = item_buf(n, mb);
                    uint32_t v[NC];
                    if (!dead) {
                        const bool ok = tc::mbar_wait(tc::smem_u32(&T.tfull[item_ready_bar(n, mb)]), item_ready_parity(n, mb),
                                                      status);
                        dead = !__all_sync(0xffffffffu, ok);
                    }
                    if (!dead) {
                        tc::tc_fence_after();
                        load_columns<NC>(tbase + buf * 128, v);
                        tc::tc_fence_before();
                        __syncwarp();
                        if (lane == 0) tc::mbar_arrive(tc::smem_u32(&T.tempty[buf]));
                    } else {
#pragma unroll
                        for (int e = 0; e < NC; ++e) v[e] = 0u;
                    }
                    if (PASS_B) {
                        acc += colsum_partial<NC>(v, c_log2, mpu + mb * 128 + half * NC);
                    } else {
                        const int r = mb * 128 + lane_row % kRows;
                        const int last = P + (r % w);                       // last visible position of this row
                        const int pos0 = tile_t0 + col0;
                        if (masked) stats_update<true, NC>(v, c_log2, pos0, last, m_run[mb], l_run[mb]);
                        else stats_update<false, NC>(v, c_log2, pos0, last, m_run[mb], l_run[mb]);
                    }
                }
                if (PASS_B) {
                    // the two column halves of this group meet in shared memory (slot = tile parity within the group)
                    float *cs = colsum + ((n >> 1) & 1) * 512 + group * 256;
                    cs[half * 128 + lane_row] = acc;
                    group_barrier(group);
                    const int pos = tile_t0 + lane_row;
                    if (half == 0 && pos < min(t1, P) && !dead) raw[(size_t)u * P + pos] = cs[lane_row] + cs[128 + lane_row];
                }
            }
            n0 += ntiles;
            if (GRAM) {
                // drain the Gram block: warp (quarter, cb) stores rows 32 quarter .. +31, columns 32 cb .. +31
                if (!dead) {
                    const bool ok = tc::mbar_wait(tc::smem_u32(&T.gfull), (j - first) & 1, status);
                    dead = !__all_sync(0xffffffffu, ok);
                }
                if (!dead) {
                    tc::tc_fence_after();
                    const int cb = warp >> 2;
                    float *out = gram_part + (size_t)j * (kD * kD + kD);
                    const uint32_t rows_at = tmem + ((uint32_t)(quarter * 32) << 16) + kGramCol;
                    uint32_t r[32], sum = 0u;
                    tc::tmem_ld32(rows_at + cb * 32, r);
                    if (cb == 0) sum = tc::tmem_ld1(rows_at + 128);
                    tc::tmem_ld_wait();
                    tc::tc_fence_before();
                    __syncwarp();
                    if (lane == 0) tc::mbar_arrive(tc::smem_u32(&T.gdrained));
                    if (cb == 0) out[kD * kD + lane_row] = __uint_as_float(sum);
                    float4 *dst = reinterpret_cast<float4 *>(out) + gram_vec4(lane_row, cb * 8);
#pragma unroll
                    for (int q4 = 0; q4 < 8; ++q4)
                        dst[4 * q4] = make_float4(__uint_as_float(r[4 * q4]), __uint_as_float(r[4 * q4 + 1]),
                                              __uint_as_float(r[4 * q4 + 2]), __uint_as_float(r[4 * q4 + 3]));
                }
            }
            if (!PASS_B) {
                // merge the four (group, half) partials of every row, and of its copies, in a fixed order
                all_soft_barrier();            // the item before has been read
                const int slot = group * 2 + half;
#pragma unroll
                for (int mb = 0; mb < MB; ++mb) merge[slot * (MB * 128) + mb * 128 + lane_row] = make_float2(m_run[mb], l_run[mb]);
                all_soft_barrier();
                if (slot == 0 && !dead) {
#pragma unroll
                    for (int mb = 0; mb < MB; ++mb) {
                        const int r = mb * 128 + lane_row;
                        if (r < rows) {                                 // SPLIT > 1: rows <= kRows, the lanes of copy 0
                            float m = -INFINITY;
#pragma unroll
                            for (int sl = 0; sl < 4 * SPLIT; ++sl)
                                m = fmaxf(m, merge[(sl / SPLIT) * (MB * 128) + r + (sl % SPLIT) * kRows].x);
                            float lsum = 0.f;
#pragma unroll
                            for (int sl = 0; sl < 4 * SPLIT; ++sl) {
                                const float2 ml = merge[(sl / SPLIT) * (MB * 128) + r + (sl % SPLIT) * kRows];
                                if (ml.x > -INFINITY) lsum += ml.y * ex2(ml.x - m);
                            }
                            float *o = stats_part + ((size_t)j * kMaxRows + r) * 2;
                            o[0] = m;
                            o[1] = lsum;
                        }
                    }
                }
            }
        }
    }
    tc::tc_fence_before();
    __syncthreads();
    if (warp == 17) tc::tmem_dealloc(tmem, 512);
}

template <int MB, int MODE, int SPLIT>
static cudaError_t raise_smem_limit() {
    static bool done[64] = {};
    return allow_dynamic_smem((const void *)score_tc_kernel<MB, MODE, SPLIT>, score_smem(MB, MODE), done);
}

template <int MB, int SPLIT>
static cudaError_t launch_scores_tc_mb(const Plan &p, const CUtensorMap &tq, const CUtensorMap &tk, float c_log2,
                                       const float *d_lse, float *d_stats_part, float *d_raw,
                                       float *d_gram_part, int phases, uint32_t *d_status, Profiler *prof,
                                       cudaStream_t st) {
    const uncomp_shape &s = p.shape;
    cudaError_t e = cudaSuccess;
    int dev = 0, sms = kTargetSms;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // one CTA per SM, each with an equal share of the (unit, chunk) items
    auto ctas = [&](int splits) { return (unsigned)min((int64_t)sms, (int64_t)p.units * splits); };
    auto launch = [&](auto kernel, int mode, int splits, float *stats_out, const float *stats_in, int stats_splits, const float *lse,
                      float *raw, float *gram) {
        return launch_kernel(kernel, LaunchShape{dim3(ctas(splits)), kScoreThreads, (size_t)score_smem(MB, mode), 1}, st, tq, tk, s.L, s.H,
                             s.N, s.w, p.rows, p.units, p.score_chunk, splits, c_log2, stats_out, stats_in, stats_splits, lse, raw,
                             gram, d_status);
    };
    if (phases & kScorePhaseStats) {
        e = d_gram_part ? raise_smem_limit<MB, 2, SPLIT>() : raise_smem_limit<MB, 0, SPLIT>();
        if (e != cudaSuccess) return e;
        ProfScope ps(prof, d_gram_part ? kSlotGramStats : kSlotScoreStats, st);
        e = launch(d_gram_part ? score_tc_kernel<MB, 2, SPLIT> : score_tc_kernel<MB, 0, SPLIT>, d_gram_part ? 2 : 0, p.score_splits, d_stats_part, nullptr, 0, nullptr, nullptr, d_gram_part);
        if (e != cudaSuccess) return e;
    }
    if (phases & kScorePhaseColsum) {
        const bool with_gram = (phases & kScorePhaseStats) == 0 && d_gram_part != nullptr;   // mode 3
        ProfScope ps(prof, with_gram ? kSlotGramColsum : kSlotScoreColsum, st);
        const int splitsB = (p.prefix + p.score_chunk - 1) / p.score_chunk;
        e = with_gram ? raise_smem_limit<MB, 3, SPLIT>() : raise_smem_limit<MB, 1, SPLIT>();
        if (e != cudaSuccess) return e;
        e = launch(with_gram ? score_tc_kernel<MB, 3, SPLIT> : score_tc_kernel<MB, 1, SPLIT>, with_gram ? 3 : 1,
                   with_gram ? p.score_splits : splitsB, nullptr, d_stats_part, p.score_splits, d_lse, d_raw,
                   with_gram ? d_gram_part : nullptr);
    }
    return e;
}

cudaError_t launch_scores_tc(const Plan &p, const void *dQw, const void *dK, const UnitAddr &addr, float scale,
                             const float *d_lse, float *d_stats_part, float *d_raw, float *d_gram_part,
                             int phases, uint32_t *d_status, TmapCache *cache, Profiler *prof, cudaStream_t st) {
    CUtensorMap tq, tk;
    cudaError_t e = cached_scorer_maps(cache, p, addr, dQw, dK, kTile, &tq, &tk);
    if (e != cudaSuccess) return e;
    const float c_log2 = scale * 1.4426950408889634f;
    const int MB = (p.rows + 127) / 128;
    if (p.rows <= 32) return launch_scores_tc_mb<1, 4>(p, tq, tk, c_log2, d_lse, d_stats_part, d_raw, d_gram_part, phases, d_status, prof, st);
    if (p.rows <= 64) return launch_scores_tc_mb<1, 2>(p, tq, tk, c_log2, d_lse, d_stats_part, d_raw, d_gram_part, phases, d_status, prof, st);
    switch (MB) {
        case 1: return launch_scores_tc_mb<1, 1>(p, tq, tk, c_log2, d_lse, d_stats_part, d_raw, d_gram_part, phases, d_status, prof, st);
        case 2: return launch_scores_tc_mb<2, 1>(p, tq, tk, c_log2, d_lse, d_stats_part, d_raw, d_gram_part, phases, d_status, prof, st);
        case 3: return launch_scores_tc_mb<3, 1>(p, tq, tk, c_log2, d_lse, d_stats_part, d_raw, d_gram_part, phases, d_status, prof, st);
        default: return launch_scores_tc_mb<4, 1>(p, tq, tk, c_log2, d_lse, d_stats_part, d_raw, d_gram_part, phases, d_status, prof, st);
    }
}

}  // namespace uncomp
