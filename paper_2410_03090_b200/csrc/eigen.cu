// Truncated matrix entropy of every unit from its partial Gram matrices (paper Section 3.1 - 3.2), in fp64.
//
// One CTA of 256 threads per unit:
//   1. C = sum_p G_p - s s^T / N with s = sum_p s_p (partials added in index order; the centring term is
//      dropped for the uncentred variant).  Eq. 1 without its 1/(N-1), which cancels in step 4.
//   2. Householder reduction of the 128 x 128 symmetric C to tridiagonal form, C in registers: lane t = lane & 15 of row
//      group i = 2 warp + lane / 16 holds the 64 entries C[i + 16 a][32 j + 2 t + e], a < 8, j < 4, e < 2.
//   3. The k largest eigenvalues by Sturm-count multi-section: a coarse round shared by all, then a team of lanes per
//      eigenvalue evaluates the division-free three-term recurrence of the characteristic polynomials at one interior point
//      each (8 lanes: 9-fold per round).  The recurrence is rescaled against underflow.  Few units: steps 3 and 4 are a
//      kernel of their own, where a cluster of CTAs shares the eigenvalues of a unit in larger teams.
//   4. p_i = lambda_i / sum (over the k kept, or the whole trace), H_k = -sum p_i ln p_i, erank_k = exp H_k.
//
// What bounds it: the chain of a step (a norm, a square root, a reciprocal, three shuffle reductions of two words a level,
// a barrier) and, while the matrix is large, the fp64 units (192 multiply-adds per thread and full step).  Shared
// memory delivers 128 bytes per cycle whatever the lanes have in common, so a layout with few columns per thread matters
// more than few shuffles: four lanes per row and 32 columns each took 4400 cycles per full step, 512 threads with 8 columns
// 3100, this form 2370, 1000 where almost nothing is left to
// update.  Row and column groups that are done drop out of the code (the step loop is unrolled over
// k / 16); inside the groups nothing is masked: reflectors and products are zero there.  With the matrix in shared
// memory, one warp forming the reflector and a warp per row for the product, 8 units took 543 us; now 140 (113 and 15 for the
// eigenvalues with a kernel of their own).
#include <cooperative_groups.h>

#include "common.cuh"
#include "newton.cuh"

namespace uncomp {

namespace {
constexpr int kEigThreads = 256;
constexpr int kValueThreads = 128;   // of a CTA of the eigenvalue kernel
constexpr int kEigWarps = kEigThreads / 32;
constexpr int n = kD;
template <typename T> struct __align__(2 * sizeof(T)) Pair { T x, y; };

struct EigenSmem {
    double x[2][n];   // row k + 1 before the update of step k
    double v[2][n];   // the step's reflector
    double p[2][n];   // minus the product of the matrix and the reflector
    double part[kEigWarps];
    double sd[n];     // column sums
    double trace;
};
struct ValueSmem {
    double dd[n];
    double ee[n];     // ee[i] couples i and i+1
    double2 de[n];    // (diagonal, -coupling^2) of the scaled matrix, the coupling to the entry before
    double lam[n];
    double scale;
    int cnt[2 * kEigThreads + 2];
    int not_converged;
};
// What the first kernel leaves for the eigenvalue kernel of few units, over the unit's own first partial, which it has consumed.
struct EigenBand64 {
    double dd[n], ee[n], trace;
};

// number of eigenvalues of the normalised tridiagonal matrix that are < x
__device__ __noinline__ int sturm_count_robust(const double2 *de, double x) {
    const double tiny = 0x1p-400, big = 0x1p+400;
    double p0 = 0.0, p1 = 1.0;
    bool neg1 = false;
    int count = 0;
    for (int i = 0; i < n; ++i) {
        double pn = (de[i].x - x) * p1 + de[i].y * p0;
        bool negn = pn < 0.0;
        if (pn == 0.0) {            // a zero takes the sign opposite to its predecessor
            negn = !neg1;
            pn = (negn ? -1.0 : 1.0) * fabs(p1) * 0x1p-100;
        }
        count += (negn != neg1);
        p0 = p1;
        p1 = pn;
        neg1 = negn;
        if (fabs(p1) < tiny) { p1 *= big; p0 *= big; }
    }
    return count;
}
// factor that brings |p| back near 1 (a power of two; p below 2^-831 is raised by 2^832)
__device__ __forceinline__ double rescale_of(double p) {
    const int ex = max(__double2hiint(p) & 0x7ff00000, 0x0c000000);
    return __hiloint2double(0x7fe00000 - ex, 0);
}
// The same for NP points without a branch per step, from both ends at once (half the chain): p over the leading, q over the
// trailing 64 rows.  With F = p_64 q_64 - e^2 p_63 q_63 (the whole determinant, e couples the halves) the count is the sign
// changes of p up to p_64, those of q up to q_63, and one more when F and p_64 q_63 differ in sign.  Sign bits are shifted
// into a word and the changes counted 32 at a time, the pairs are brought back near 1 every 8 steps (a step shrinks them by
// at most 2^-60 or so).  A zero adds one change whichever sign it gets as long as the coupling behind it is not zero;
// otherwise F is zero and the point is recounted.  Bound by the fp64 units and by the sign words (a funnel shift costs as
// much as an fp64 operation): with the next eight rows loaded ahead 8 warps take 3300 cycles (3900 from one end, 4 warps of
// two points).
template <int NP>
__device__ __forceinline__ void sturm_count(const double2 *de, const double (&x)[NP], int (&count)[NP]) {
    double p0[NP], p1[NP], q0[NP], q1[NP], me2 = 0.0;
    uint32_t lastp[NP], lastq[NP];
    double2 fn[8], gn[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) { fn[i] = de[i]; gn[i] = de[n - 1 - i]; }
#pragma unroll
    for (int c = 0; c < NP; ++c) { p0[c] = q0[c] = 0.0; p1[c] = q1[c] = 1.0; count[c] = 0; lastp[c] = lastq[c] = 0u; }
#pragma unroll 1
    for (int w = 0; w < 2; ++w) {
        uint32_t mp[NP], mq[NP];
#pragma unroll
        for (int c = 0; c < NP; ++c) mp[c] = mq[c] = 0u;
#pragma unroll 1
        for (int i0 = w * 32; i0 < w * 32 + 32; i0 += 8) {
            double2 f[8], g[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {              // the next eight entries are on their way
                f[i] = fn[i];
                g[i] = gn[i];
                fn[i] = de[(i0 + 8 + i) & (n - 1)];
                gn[i] = de[(n - 1 - i0 - 8 - i) & (n - 1)];
            }
#pragma unroll
            for (int i = 0; i < 8; ++i) {
#pragma unroll
                for (int c = 0; c < NP; ++c) {
                    const double pn = fma(f[i].x - x[c], p1[c], f[i].y * p0[c]), qn = fma(g[i].x - x[c], q1[c], me2 * q0[c]);
                    p0[c] = p1[c];
                    p1[c] = pn;
                    q0[c] = q1[c];
                    q1[c] = qn;
                    mp[c] = __funnelshift_l((uint32_t)__double2hiint(pn), mp[c], 1);
                    mq[c] = __funnelshift_l((uint32_t)__double2hiint(qn), mq[c], 1);
                }
                me2 = g[i].y;                          // couples row 127 - i0 - i to the one before
            }
#pragma unroll
            for (int c = 0; c < NP; ++c) {
                const double sp = rescale_of(p1[c]), sq = rescale_of(q1[c]);
                p0[c] *= sp;
                p1[c] *= sp;
                q0[c] *= sq;
                q1[c] *= sq;
            }
        }
#pragma unroll
        for (int c = 0; c < NP; ++c) {
            const uint32_t up = mp[c] ^ ((mp[c] >> 1) | (lastp[c] << 31));
            uint32_t dn = mq[c] ^ ((mq[c] >> 1) | (lastq[c] << 31));
            if (w == 1) dn &= ~1u;                     // q_64 belongs to F
            count[c] += __popc(up) + __popc(dn);
            lastp[c] = mp[c] & 1u;
            lastq[c] = w == 0 ? mq[c] & 1u : (mq[c] >> 1) & 1u;
        }
    }
#pragma unroll
    for (int c = 0; c < NP; ++c) {                     // me2: -e^2 between rows 63 and 64
        // the larger of a pair near 1: neither product leaves the range
        const double sp = rescale_of(fmax(fabs(p0[c]), fabs(p1[c]))), sq = rescale_of(fmax(fabs(q0[c]), fabs(q1[c])));
        const double F = fma(p1[c] * sp, q1[c] * sq, me2 * (p0[c] * sp) * (q0[c] * sq));
        count[c] += (int)(((uint32_t)__double2hiint(F) >> 31) ^ lastp[c] ^ lastq[c]);
        if (F == 0.0 || !isfinite(F)) count[c] = sturm_count_robust(de, x[c]);
    }
}

__device__ __forceinline__ double sum16(double v) {   // over the 16 lanes that share a row
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// 8 columns of a row vector, 32 (q / 2) + 2 t + q % 2, to shared memory
template <int J>
__device__ __forceinline__ void publish(const double (&row)[8], double *dst, int t) {
#pragma unroll
    for (int j = J; j < 4; ++j) *reinterpret_cast<double2 *>(dst + 32 * j + 2 * t) = make_double2(row[2 * j], row[2 * j + 1]);
}

// What a thread carries from step to step: the pending rank-2 update (v and -w for its columns and for its rows) and the row x
// the next reflector is made of, zero up to the diagonal.
struct Carry {
    double vc[8], wc[8], xc[8], vr[8], wr[8];
    double x0;         // entry k + 1 of x
};

// Householder steps k = 16 KA .. 16 KA + 15 (stopping at n - 3); row groups (16 rows) below KA and column groups (32
// columns) below J are done.
template <int KA>
__device__ __forceinline__ void householder_block(double (&A)[8][8], Carry &R, EigenSmem &S, ValueSmem &F, int lane, int warp) {
    constexpr int J = KA >> 1, JN = J < 3 ? J + 1 : 3, KN = KA < 7 ? KA + 1 : 7;
    constexpr bool kOdd = (KA & 1) != 0 && KA < 7;     // the block's end is also the end of a column group
    const int i = 2 * warp + (lane >> 4), t = lane & 15;
#pragma unroll 1
    for (int kt = 0; kt < 16; ++kt) {
        const int k = 16 * KA + kt;
        if (KA == 7 && k > n - 3) break;
        const bool end = KA < 7 && kt == 15;
        // ---- norm of x; meanwhile the pending update of step k - 1 and A x ----
        double sq[2] = {R.xc[2 * J] * R.xc[2 * J], R.xc[2 * J + 1] * R.xc[2 * J + 1]};
#pragma unroll
        for (int q = 2 * J + 2; q < 8; ++q) sq[q & 1] = fma(R.xc[q], R.xc[q], sq[q & 1]);
        const double sig = sum16(sq[0] + sq[1]);
        double y[8];
#pragma unroll
        for (int a = 0; a < 8; ++a) y[a] = 0.0;
#pragma unroll
        for (int a = KA; a < 8; ++a) {
#pragma unroll
            for (int q = 2 * J; q < 8; ++q) A[a][q] = fma(R.vr[a], R.wc[q], fma(R.wr[a], R.vc[q], A[a][q]));
#pragma unroll
            for (int q = 2 * J; q < 8; ++q) y[a] = fma(A[a][q], R.xc[q], y[a]);
        }
        // ---- -p = -beta A v, v = x - alpha e_{k+1}: the product starts from x, what alpha adds sits in one group ----
        double *xs = S.x[k & 1], *ps = S.p[k & 1], *vs = S.v[k & 1];
        const bool flat = !(sig > 1e-290);             // the row is reduced already: beta = 0
        const double root = sqrt_newton(sig);
        const double minus_alpha = flat ? -R.x0 : (R.x0 >= 0.0 ? root : -root);
        const double minus_beta = flat ? 0.0 : -recip_newton(fma(fabs(R.x0), root, sig));         // -2 / (v^T v)
        const double vk = R.x0 + minus_alpha;          // v_{k+1}
        if (threadIdx.x == 0) F.ee[k] = -minus_alpha;
        if (kOdd && end) {                             // column k + 1 is the first of the next group
            const double d0 = t == 0 ? minus_alpha : 0.0;
#pragma unroll
            for (int a = KA; a < 8; ++a) y[a] = fma(A[a][2 * JN], d0, y[a]);
            R.xc[2 * JN] += d0;
        } else {
            const int at = k + 1 - 32 * J - 2 * t;
            const double d0 = at == 0 ? minus_alpha : 0.0, d1 = at == 1 ? minus_alpha : 0.0;
#pragma unroll
            for (int a = KA; a < 8; ++a) y[a] = fma(A[a][2 * J], d0, fma(A[a][2 * J + 1], d1, y[a]));
            R.xc[2 * J] += d0;
            R.xc[2 * J + 1] += d1;
        }
        if (i == ((k + 1) & 15)) {                     // 16 lanes of one warp
            if (end) publish<J>(A[KN], xs, t);
            else publish<J>(A[KA], xs, t);
            publish<J>(R.xc, vs, t);
        }
        // over the 16 lanes of a row: three transposing levels and a plain one; lane t ends up with row group t / 2
        const bool up8 = (t & 8) != 0, up4 = (t & 4) != 0, up2 = (t & 2) != 0;
        double s4[4], s2[2];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            if (a + 4 < KA) { s4[a] = 0.0; continue; }
            s4[a] = (up8 ? y[a + 4] : y[a]) + __shfl_xor_sync(0xffffffffu, up8 ? y[a] : y[a + 4], 8);
        }
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            if (a + 6 < KA) { s2[a] = 0.0; continue; }
            s2[a] = (up4 ? s4[a + 2] : s4[a]) + __shfl_xor_sync(0xffffffffu, up4 ? s4[a] : s4[a + 2], 4);
        }
        double z = (up2 ? s2[1] : s2[0]) + __shfl_xor_sync(0xffffffffu, up2 ? s2[0] : s2[1], 2);
        z += __shfl_xor_sync(0xffffffffu, z, 1);
        if ((t & 1) == 0 && (t >> 1) >= KA) ps[i + 16 * (t >> 1)] = minus_beta * z;
        __syncthreads();
        // ---- -w = -p + (beta/2 v^T p) v, then row k + 1 after this step's update: the next x ----
#pragma unroll
        for (int j = J; j < 4; ++j) {
            const double2 q = *reinterpret_cast<const double2 *>(ps + 32 * j + 2 * t);
            R.wc[2 * j] = q.x;
            R.wc[2 * j + 1] = q.y;
            R.vc[2 * j] = R.xc[2 * j];
            R.vc[2 * j + 1] = R.xc[2 * j + 1];
        }
        double dot[2] = {R.vc[2 * J] * R.wc[2 * J], R.vc[2 * J + 1] * R.wc[2 * J + 1]};
#pragma unroll
        for (int q = 2 * J + 2; q < 8; ++q) dot[q & 1] = fma(R.vc[q], R.wc[q], dot[q & 1]);
        const double kk = 0.5 * minus_beta * sum16(dot[0] + dot[1]);            // beta/2 v^T p
        const double wk = fma(kk, vk, ps[k + 1]);
        if (threadIdx.x == 0) F.dd[k + 1] = fma(2.0 * vk, wk, xs[k + 1]);
#pragma unroll
        for (int j = J; j < 4; ++j) {
            const double2 row = *reinterpret_cast<const double2 *>(xs + 32 * j + 2 * t);
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int q = 2 * j + e;
                R.wc[q] = fma(kk, R.vc[q], R.wc[q]);
                R.xc[q] = fma(vk, R.wc[q], fma(wk, R.vc[q], e ? row.y : row.x));
            }
        }
        {                                              // columns up to k + 1 are zero
            const int at = k + 1 - 32 * J - 2 * t;
            if (at >= 0) R.xc[2 * J] = 0.0;
            if (at >= 1) R.xc[2 * J + 1] = 0.0;
            if (kOdd && end && t == 0) R.xc[2 * JN] = 0.0;
        }
        {                                              // entry k + 2 of the new x for everybody
            const int c = k + 2;
            const bool next = kOdd && kt >= 14;        // it lies in the next column group
            const double lo = next ? R.xc[2 * JN] : R.xc[2 * J], hi = next ? R.xc[2 * JN + 1] : R.xc[2 * J + 1];
            R.x0 = __shfl_sync(0xffffffffu, (c & 1) ? hi : lo, (lane & 16) + ((c >> 1) & 15));
        }
#pragma unroll
        for (int a = KA; a < 8; ++a) {
            R.vr[a] = vs[i + 16 * a];
            R.wr[a] = fma(kk, R.vr[a], ps[i + 16 * a]);
        }
    }
}

// Steps 3 and 4 of unit u, its tridiagonal matrix in S.dd and S.ee, by a block of NT threads; TEAM lanes look for an eigenvalue.
// CLUSTER: the CTAs of the cluster share the eigenvalues, the first of them collects.
template <int NT, int TEAM, bool CLUSTER>
__device__ __forceinline__ void finish_unit64(ValueSmem &S, int u, double trace, int k_trunc, int norm, int max_iters,
                                              float *__restrict__ entropy, float *__restrict__ erank,
                                              double *__restrict__ spectrum, uint32_t *__restrict__ status) {
    constexpr int kCoarse = 2 * NT;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    double *lam = S.lam;
    int *not_converged = &S.not_converged, rank = 0, ctas = 1;
    if constexpr (CLUSTER) {
        cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
        rank = (int)cluster.block_rank();
        ctas = (int)cluster.num_blocks();
        lam = cluster.map_shared_rank(S.lam, 0);
        not_converged = cluster.map_shared_rank(&S.not_converged, 0);
        cluster.sync();                                // the first CTA runs and has cleared its flag
    }
    // ---- 3. k largest eigenvalues by multi-section ------------------------------------------------
    if (wid == 0) {
        double rad = 0.0;   // Gershgorin radius as the scale
        for (int i = lane; i < n; i += 32) {
            const double left = i > 0 ? fabs(S.ee[i - 1]) : 0.0;
            const double right = i < n - 1 ? fabs(S.ee[i]) : 0.0;
            rad = fmax(rad, fabs(S.dd[i]) + left + right);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) rad = fmax(rad, __shfl_xor_sync(0xffffffffu, rad, o));
        if (lane == 0) S.scale = rad > 0.0 ? rad : 1.0;
    }
    __syncthreads();
    const double scale = S.scale, inv_scale = 1.0 / scale;
    if (tid < n) {
        const double e = tid > 0 ? S.ee[tid - 1] * inv_scale : 0.0;
        S.de[tid] = make_double2(S.dd[tid] * inv_scale, -e * e);
    }
    __syncthreads();

    // coarse round: counts at 2 NT interior points of [lo0, hi0], shared by all eigenvalues (C is positive semi-definite:
    // what rounding leaves below lo0 is a zero eigenvalue)
    const double lo0 = -0x1p-10, hi0 = 1.0 + 0x1p-40, step0 = (hi0 - lo0) / (double)(kCoarse + 1);
    {
        const double x[2] = {lo0 + step0 * (double)(2 * tid + 1), lo0 + step0 * (double)(2 * tid + 2)};
        int c[2];
        sturm_count<2>(S.de, x, c);
        S.cnt[2 * tid + 1] = c[0];
        S.cnt[2 * tid + 2] = c[1];
    }
    if (tid == 0) { S.cnt[0] = 0; S.cnt[kCoarse + 1] = n; }
    __syncthreads();

    // Teams of TEAM lanes, a point each, refine one eigenvalue.  A round is at least 9-fold and there is one more than asked
    // for: at least what as many rounds give after a coarse round of 512 points.
    static_assert(TEAM >= 8 && 9 * kCoarse >= 512, "");
    const int k = min(k_trunc, n);
    const int iters = (max_iters > 0 ? max_iters : 14) + 1;
    const double tol = 1e-13;
    const int sub = tid % TEAM, team0 = lane & ~(TEAM - 1);
    const unsigned team_mask = (0xffffffffu >> (32 - TEAM)) << team0;
    for (int j0 = rank * (NT / TEAM); j0 < k; j0 += ctas * (NT / TEAM)) {
        const int j = j0 + tid / TEAM;              // this team looks for the j-th largest
        const bool active = j < k;
        const int idx = n - 1 - (active ? j : 0);   // its 0-based rank from below
        int lo_i = 0, hi_i = kCoarse + 1;       // cnt[lo_i] <= idx < cnt[hi_i]
        while (hi_i - lo_i > 1) {
            const int mid = (lo_i + hi_i) >> 1;
            if (S.cnt[mid] > idx) hi_i = mid; else lo_i = mid;
        }
        double lo = lo0 + step0 * (double)lo_i, hi = lo0 + step0 * (double)hi_i;
        for (int it = 0; it < iters; ++it) {
            const double width = (hi - lo) * (1.0 / (TEAM + 1));
            const bool done = hi - lo <= tol;
            if (__all_sync(0xffffffffu, done)) break;
            const double x[1] = {lo + width * (double)(sub + 1)};
            int c[1];
            sturm_count<1>(S.de, x, c);
            const unsigned above = (__ballot_sync(0xffffffffu, c[0] > idx) & team_mask) >> team0;
            if (!done) {
                const int f = above ? __ffs(above) - 1 : TEAM;          // first of the points above the eigenvalue
                const double base_lo = lo;
                if (f < TEAM) hi = base_lo + width * (double)(f + 1);
                if (f > 0) lo = base_lo + width * (double)f;
            }
        }
        if (active && sub == 0) {
            lam[j] = lo > 0.0 ? 0.5 * (lo + hi) * scale : 0.0;      // what cannot be told from zero is zero
            if (hi - lo > tol) atomicOr(not_converged, 1);
        }
    }
    if constexpr (CLUSTER) {
        cooperative_groups::this_cluster().sync();
        if (rank != 0) return;
    } else __syncthreads();

    // ---- 4. entropy -----------------------------------------------------------------------------
    if (wid == 0) {      // lane i takes eigenvalues i, i + 32, ...; fixed-order butterfly sums
        double total = trace;
        if (!norm) {
            total = 0.0;
            for (int i = lane; i < k; i += 32) total += S.lam[i] > 0.0 ? S.lam[i] : 0.0;
            total = warp_sum(total);
        }
        double h = 0.0;
        if (total > 0.0) {
            for (int i = lane; i < k; i += 32) {
                const double p = (S.lam[i] > 0.0 ? S.lam[i] : 0.0) / total;
                if (p > 0.0) h -= p * log(p);
            }
        }
        h = warp_sum(h);
        if (lane == 0) {
            entropy[u] = (float)h;
            if (erank) erank[u] = (float)exp(h);
            if (S.not_converged) atomicOr(status, UNCOMP_STATUS_NOT_CONVERGED);
        }
    }
    if (spectrum && tid < k) spectrum[(size_t)u * k + tid] = S.lam[tid];
}
}  // namespace

template <typename PartialT>
__global__ void __launch_bounds__(kEigThreads, 1)
eigen_entropy_kernel(PartialT *partials, int P, bool hand_over, int N, int k_trunc, int center, int norm,
                     int max_iters, float *__restrict__ entropy, float *__restrict__ erank,
                     double *__restrict__ spectrum, uint32_t *__restrict__ status) {
    __shared__ EigenSmem S;
    __shared__ ValueSmem F;
    const int u = blockIdx.x, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int row0 = tid >> 4, t = tid & 15;
    constexpr int len = n * n + n;
    PartialT *base = partials + (size_t)u * P * len;
    chain_wait();

    // ---- 1. assemble C in registers ----------------------------------------------------------------
    if (tid < n) {
        double s = 0.0;
        for (int p = 0; p < P; ++p) s += (double)base[(size_t)p * len + n * n + tid];
        S.sd[tid] = s;
    }
    if (tid == 0) F.not_converged = 0;
    double A[8][8];
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int e = 0; e < 8; ++e) A[a][e] = 0.0;
    for (int p = 0; p < P; ++p) {
#pragma unroll
        for (int a = 0; a < 8; ++a) {
            const Pair<PartialT> *row = reinterpret_cast<const Pair<PartialT> *>(base + (size_t)p * len + (row0 + 16 * a) * n + 2 * t);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const Pair<PartialT> x = row[16 * j];
                A[a][2 * j] += (double)x.x;
                A[a][2 * j + 1] += (double)x.y;
            }
        }
    }
    __syncthreads();
    double d = 0.0;                                    // this thread's diagonal entries
#pragma unroll
    for (int a = 0; a < 8; ++a) {
        const int r = row0 + 16 * a;
        const double sr = S.sd[r] / (double)N;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int c = 32 * j + 2 * t;
            if (center) {
                A[a][2 * j] -= sr * S.sd[c];
                A[a][2 * j + 1] -= sr * S.sd[c + 1];
            }
            if (c == r) d += A[a][2 * j];
            if (c + 1 == r) d += A[a][2 * j + 1];
        }
    }
    d = warp_sum(d);
    if (lane == 0) S.part[wid] = d;
    if (row0 == 0) publish<0>(A[0], S.x[1], t);
    __syncthreads();
    if (tid == 0) {
        double s = 0.0;
        for (int w = 0; w < kEigWarps; ++w) s += S.part[w];
        S.trace = s;
    }

    // ---- 2. Householder tridiagonalisation ---------------------------------------------------------
    {
        Carry R;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            R.vc[q] = R.wc[q] = R.vr[q] = R.wr[q] = 0.0;
            R.xc[q] = S.x[1][32 * (q >> 1) + 2 * t + (q & 1)];
        }
        R.x0 = S.x[1][1];
        if (tid == 0) F.dd[0] = S.x[1][0];
        if (t == 0) R.xc[0] = 0.0;
        householder_block<0>(A, R, S, F, lane, wid);
        householder_block<1>(A, R, S, F, lane, wid);
        householder_block<2>(A, R, S, F, lane, wid);
        householder_block<3>(A, R, S, F, lane, wid);
        householder_block<4>(A, R, S, F, lane, wid);
        householder_block<5>(A, R, S, F, lane, wid);
        householder_block<6>(A, R, S, F, lane, wid);
        householder_block<7>(A, R, S, F, lane, wid);
        if (tid == 0) { F.ee[n - 2] = R.x0; F.ee[n - 1] = 0.0; }
        if (row0 == 15 && t == 15)                     // entry (127, 127) after the last update
            F.dd[n - 1] = fma(R.vr[7], R.wc[7], fma(R.wr[7], R.vc[7], A[7][7]));
    }
    __syncthreads();

    if (hand_over) {
        EigenBand64 *out = reinterpret_cast<EigenBand64 *>(base);
        if (tid < n) { out->dd[tid] = F.dd[tid]; out->ee[tid] = F.ee[tid]; }
        if (tid == 0) out->trace = S.trace;
        return;
    }
    finish_unit64<kEigThreads, 8, false>(F, u, S.trace, k_trunc, norm, max_iters, entropy, erank, spectrum, status);
}

// Steps 3 and 4 of few units: a cluster of 8, 4 or 2 CTAs per unit.
template <int TEAM>
__global__ void __launch_bounds__(kValueThreads)
eigen_values64_kernel(const char *__restrict__ partials, int64_t unit_stride, int k_trunc, int norm, int max_iters,
                      float *__restrict__ entropy, float *__restrict__ erank, double *__restrict__ spectrum, uint32_t *__restrict__ status) {
    __shared__ ValueSmem F;
    const int u = blockIdx.x / cooperative_groups::this_cluster().num_blocks(), tid = threadIdx.x;
    chain_wait();
    chain_signal();
    const EigenBand64 &E = *reinterpret_cast<const EigenBand64 *>(partials + u * unit_stride);
    F.dd[tid] = E.dd[tid];
    F.ee[tid] = E.ee[tid];
    if (tid == 0) F.not_converged = 0;
    __syncthreads();
    finish_unit64<kValueThreads, TEAM, true>(F, u, E.trace, k_trunc, norm, max_iters, entropy, erank, spectrum, status);
}

// Sum of the chunk partials of every unit in chunk order: out[u] = [G (d*d) | s (d)] in fp64.
template <typename PartialT>
__global__ void gram_reduce_kernel(const PartialT *__restrict__ partials, int P, double *__restrict__ out) {
    constexpr int len = kD * kD + kD;
    const int u = blockIdx.y;
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= len) return;
    double g = 0.0;
    for (int p = 0; p < P; ++p) g += (double)partials[((size_t)u * P + p) * len + e];
    out[(size_t)u * len + e] = g;
}

cudaError_t launch_gram_reduce(const Plan &p, const void *d_partials, double *d_out, cudaStream_t st) {
    dim3 grid((kD * kD + kD + 255) / 256, p.units);
    if (p.shape.dtype == UNCOMP_FP32)
        gram_reduce_kernel<double><<<grid, 256, 0, st>>>((const double *)d_partials, p.gram_splits, d_out);
    else
        gram_reduce_kernel<float><<<grid, 256, 0, st>>>((const float *)d_partials, p.gram_splits, d_out);
    return cudaGetLastError();
}

cudaError_t launch_eigen_entropy(const Plan &p, void *d_partials, const uncomp_entropy_params &ep, float *d_entropy, float *d_erank,
                                 double *d_spectrum, uint32_t *d_status, cudaStream_t st) {
    // Few units: the eigenvalues in a kernel of their own, a cluster of CTAs per unit, while each CTA has an SM to itself.
    // In the first kernel they take 28 us of one SM per unit, here 15 with eight CTAs of 128 threads (19 with 256 threads: two
    // warps share a sub-partition's fp64 unit); passes of 8 / 32 / 64 units of 512 tokens 198 -> 186, 241 -> 232, 294 -> 287 us.
    int ctas = 1;
    while (ctas < 8 && p.units * ctas * 2 <= kTargetSms) ctas *= 2;
    const bool wide = p.shape.dtype == UNCOMP_FP32;    // fp64 partials
    const LaunchShape shape{dim3(p.units), kEigThreads, 0, 1};
    cudaError_t e;
    if (wide)
        e = launch_kernel(eigen_entropy_kernel<double>, shape, st, (double *)d_partials, p.gram_splits, ctas > 1, p.shape.N,
                          ep.k_trunc, ep.center, ep.norm, ep.max_iters, d_entropy, d_erank, d_spectrum, d_status);
    else
        e = launch_kernel(eigen_entropy_kernel<float>, shape, st, (float *)d_partials, p.gram_splits, ctas > 1, p.shape.N, ep.k_trunc,
                          ep.center, ep.norm, ep.max_iters, d_entropy, d_erank, d_spectrum, d_status);
    if (e != cudaSuccess || ctas == 1) return e;
    const int64_t stride = (int64_t)p.gram_splits * (n * n + n) * (wide ? sizeof(double) : sizeof(float));
    return launch_kernel(ctas == 8 ? eigen_values64_kernel<16> : eigen_values64_kernel<8>,
                         LaunchShape{dim3(p.units * ctas), kValueThreads, 0, (unsigned)ctas}, st, (const char *)d_partials, stride,
                         ep.k_trunc, ep.norm, ep.max_iters, d_entropy, d_erank, d_spectrum, d_status);
}

}  // namespace uncomp
