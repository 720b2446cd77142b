// Head-group token budgets and the layer-group partition (paper Section 3.3.3 and 3.3.2).
//
// A single CTA: the input is at most a few thousand effective ranks, and the kernel exists so that the
// pass needs no host synchronisation between the entropy stage and the selection stage.
//
// Ranking is by counting (rank = number of heads of the ranking set that come first), the group target
// t_g = n_max - g * n (n_max - avg) / S, S = sum_g n_g g, is kept as the exact fraction num_g / S, heads
// get floor(t_g) and the tokens still missing go to the largest remainders (ties: better rank).  Every
// step is integer arithmetic, so the budgets are reproducible bit for bit.
//
// What bounds it is latency.  A remainder belongs to a group, so who gets a missing token follows from a table of the M
// groups (remainder, heads ahead of the group) and a head's rank inside its group; S and the number of missing tokens
// come from the host; ranks are counted in shared memory; the prefix sum is one of warps.  With 64-bit divisions in every
// thread, remainders compared head by head in global memory and a scan with 20 barriers 256 units took 15 us
// (of which 9 are the launch and its event records), now 11.  The table of the groups is made before the effective ranks are
// there: the kernels of the eigenvalues let this one start when all of theirs run (passes of few units 2.4 us shorter).
#include "common.cuh"

namespace uncomp {

constexpr int kBudThreads = 1024;
constexpr int kBudShared = 4096;      // effective ranks and groups held in shared memory

// first rank of group g: floor(g n / M)
__host__ __device__ __forceinline__ int group_lo(int g, int n, int M) {
    const uint64_t p = (uint64_t)g * (uint64_t)n;
    return p >> 32 ? (int)(p / (uint64_t)M) : (int)((uint32_t)p / (uint32_t)M);
}

struct BudSched {
    int64_t S;            // sum_g n_g g
    int missing;          // tokens of a ranking set that the floors leave undistributed
};

// grid (1).  table_ahead [M] and table_rem [M]: scratch for the group table when M > kBudShared.
__global__ void __launch_bounds__(kBudThreads) budgets_kernel(const float *__restrict__ erank, int B, int L, int H,
                                                             int N, int w, uncomp_budget_params bp, BudSched sched,
                                                             int32_t *__restrict__ budgets,
                                                             int64_t *__restrict__ offsets,
                                                             int32_t *__restrict__ layer_group,
                                                             int32_t *__restrict__ layer_ctx,
                                                             int32_t *__restrict__ table_ahead,
                                                             int64_t *__restrict__ table_rem) {
    extern __shared__ int64_t bud_smem[];
    __shared__ int64_t warp_total[kBudThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int units = B * L * H;
    const int n = bp.scope ? L * H : H;          // ranking-set size
    const int M = bp.M;
    const int64_t avg = bp.avg_budget, n_max = bp.n_max, S = sched.S;
    const bool shared_tab = M <= kBudShared, shared_er = units <= kBudShared;
    int64_t *rem_t = shared_tab ? bud_smem : table_rem;                              // [M]
    int32_t *ahead_t = shared_tab ? reinterpret_cast<int32_t *>(bud_smem + M) : table_ahead;   // [M]
    float *er_s = reinterpret_cast<float *>(shared_tab ? reinterpret_cast<int32_t *>(bud_smem + M) + M
                                                       : reinterpret_cast<int32_t *>(bud_smem));
    const float *er = shared_er ? er_s : erank;
    if (!shared_tab) chain_wait();                     // the scratch may still be read
    auto target = [&](int g) { return n_max * S - (int64_t)g * n * (n_max - avg); };   // t_g S
    for (int g = tid; g < M; g += kBudThreads) rem_t[g] = M == 1 ? 0 : target(g) % S;
    __syncthreads();
    // heads ahead of group g when the missing tokens are handed out: larger remainder, or the same and a better rank
    for (int g = tid; g < M; g += kBudThreads) {
        const int64_t rem = rem_t[g];
        int ahead = 0;
        for (int o = 0; o < M; ++o) {
            const int64_t ro = rem_t[o];
            if (ro > rem || (ro == rem && o < g)) ahead += group_lo(o + 1, n, M) - group_lo(o, n, M);
        }
        ahead_t[g] = ahead;
    }
    __syncthreads();
    chain_wait();                                      // what came before depends on the parameters alone
    if (shared_er) {
        for (int u = tid; u < units; u += kBudThreads) er_s[u] = erank[u];
        __syncthreads();
    }
    // budgets and their exclusive prefix sum over the units, 1024 units at a time
    int64_t carry = 0;
    if (tid == 0) offsets[0] = 0;
    for (int base = 0; base < units; base += kBudThreads) {
        const int u = base + tid;
        int64_t budget = 0;
        if (u < units) {
            const int set_base = (u / n) * n;
            const float e = er[u];
            int r = 0;
            for (int j = set_base; j < u; ++j) r += er[j] >= e;            // equal values: the lower index first
            for (int j = u + 1; j < set_base + n; ++j) r += er[j] > e;
            const uint64_t rm = (uint64_t)r * (uint64_t)M;
            int g = rm >> 32 ? (int)(rm / (uint64_t)n) : (int)((uint32_t)rm / (uint32_t)n);
            while (g + 1 < M && group_lo(g + 1, n, M) <= r) ++g;
            while (g > 0 && group_lo(g, n, M) > r) --g;
            budget = M == 1 ? avg : target(g) / S;
            if (ahead_t[g] + r - group_lo(g, n, M) < sched.missing) budget += 1;
            budgets[u] = (int32_t)budget;
        }
        int64_t incl = budget;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t below = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += below;
        }
        if (lane == 31) warp_total[wid] = incl;
        __syncthreads();
        int64_t before = 0, all = warp_total[lane];
        if (lane < wid) before = all;
        before = warp_sum_i64(before);
        all = warp_sum_i64(all);
        if (u < units) offsets[u + 1] = carry + before + incl;
        carry += all;
        __syncthreads();
    }
    // layer groups
    if (layer_group && layer_ctx && bp.dn <= 0) {
        for (int i = tid; i < B * L; i += kBudThreads) { layer_group[i] = 0; layer_ctx[i] = N; }
    } else if (layer_group && layer_ctx) {
        for (int b = tid; b < B; b += kBudThreads) {
            int32_t *lg = layer_group + (size_t)b * L, *lc = layer_ctx + (size_t)b * L;
            int boundaries = 0;
            lg[0] = 0;
            double prev = 0.0;
            for (int h = 0; h < H; ++h) prev += (double)erank[((size_t)b * L) * H + h];
            prev /= (double)H;
            for (int l = 0; l + 1 < L; ++l) {
                double next = 0.0;
                for (int h = 0; h < H; ++h) next += (double)erank[((size_t)b * L + l + 1) * H + h];
                next /= (double)H;
                if (prev - next > (double)bp.eps) ++boundaries;
                lg[l + 1] = boundaries;
                prev = next;
            }
            for (int l = 0; l < L; ++l) {
                if (lg[l] == 0) lc[l] = N;
                else {
                    const int64_t c = (int64_t)bp.n_last + (int64_t)(boundaries - lg[l]) * bp.dn;
                    lc[l] = (int32_t)(c < N ? c : N);
                }
            }
        }
    }
}

// Host-side check of the schedule's preconditions; mirrors the arithmetic of the kernel.
int check_budget_params(const uncomp_shape &s, const uncomp_budget_params &bp) {
    const int n = bp.scope ? s.L * s.H : s.H;
    if (bp.M < 1 || bp.M > n) return UNCOMP_E_PARAM;
    if (bp.avg_budget < s.w || bp.n_max < bp.avg_budget || bp.n_max > s.N) return UNCOMP_E_PARAM;
    if (bp.dn < 0 || (bp.dn > 0 && bp.n_last < 1)) return UNCOMP_E_PARAM;
    if (bp.M > 1) {
        int64_t S = 0;
        for (int g = 0; g < bp.M; ++g) S += (int64_t)(group_lo(g + 1, n, bp.M) - group_lo(g, n, bp.M)) * g;
        const int64_t num_last = (int64_t)bp.n_max * S - (int64_t)(bp.M - 1) * n * (bp.n_max - bp.avg_budget);
        if (num_last < (int64_t)s.w * S) return UNCOMP_E_PARAM;
    }
    return UNCOMP_OK;
}

cudaError_t launch_budgets(const Plan &p, const float *d_erank, const uncomp_budget_params &bp, int32_t *d_budgets,
                           int64_t *d_offsets, int32_t *d_layer_group, int32_t *d_layer_ctx, int32_t *d_rank,
                           int64_t *d_rem, cudaStream_t st) {
    const int n = bp.scope ? p.shape.L * p.shape.H : p.shape.H, M = bp.M;
    BudSched sched{0, 0};
    int64_t floor_total = 0;
    for (int g = 0; g < M; ++g) sched.S += (int64_t)(group_lo(g + 1, n, M) - group_lo(g, n, M)) * g;
    for (int g = 0; g < M; ++g) {
        const int64_t ng = group_lo(g + 1, n, M) - group_lo(g, n, M);
        const int64_t fl = M == 1 ? bp.avg_budget
                                  : (bp.n_max * sched.S - (int64_t)g * n * (bp.n_max - bp.avg_budget)) / sched.S;
        floor_total += ng * fl;
    }
    sched.missing = (int)((int64_t)n * bp.avg_budget - floor_total);
    const size_t smem = (M <= kBudShared ? (size_t)M * 12 : 0) + (p.units <= kBudShared ? (size_t)p.units * 4 : 0);
    static bool done[64] = {};
    cudaError_t e = allow_dynamic_smem((const void *)budgets_kernel, kBudShared * 16, done);
    if (e != cudaSuccess) return e;
    return launch_kernel(budgets_kernel, LaunchShape{dim3(1), kBudThreads, smem, 1}, st, d_erank, p.shape.B, p.shape.L,
                         p.shape.H, p.shape.N, p.shape.w, bp, sched, d_budgets, d_offsets, d_layer_group, d_layer_ctx, d_rank,
                         d_rem);
}

}  // namespace uncomp
