// Truncated matrix entropy of every unit from its partial Gram matrices (paper Section 3.1 - 3.2), in fp64.
//
// One CTA of 256 threads per unit:
//   1. C = sum_p G_p - s s^T / N with s = sum_p s_p (partials added in index order; the centring term is
//      dropped for the uncentred variant).  Eq. 1 without its 1/(N-1), which cancels in step 4.
//   2. Householder reduction of the 128 x 128 symmetric C to tridiagonal form, C in registers: lane t = lane & 15 of row
//      group i = 2 warp + lane / 16 holds the 64 entries C[i + 16 a][32 j + 2 t + e], a < 8, j < 4, e < 2.
//   3. The k largest eigenvalues by Sturm-count multi-section: a coarse round of 512 points, then 4 lanes per eigenvalue
//      evaluate the division-free three-term recurrence of the characteristic polynomials at 8 interior points, so the
//      bracket shrinks 9-fold per round.  The recurrence is rescaled against underflow.
//   4. p_i = lambda_i / sum (over the k kept, or the whole trace), H_k = -sum p_i ln p_i, erank_k = exp H_k.
//
// What bounds it: the chain of a step (a norm, a square root, a reciprocal, four shuffle reductions of two words a level,
// two barriers) and, while the matrix is large, the fp64 units (192 multiply-adds per thread and full step).  Shared
// memory delivers 128 bytes per cycle whatever the lanes have in common, so a layout with few columns per thread matters
// more than few shuffles: four lanes per row and 32 columns each took 4400 cycles per full step, 512 threads with 8 columns
// 3100, this form 2500.  Row and column groups that are done drop out of the code (the step loop is unrolled over
// k / 16); inside the groups nothing is masked: reflectors and products are zero there.  With the matrix in shared
// memory, one warp forming the reflector and a warp per row for the product, 8 units took 543 us; now 166 us.
#include "common.cuh"
#include "newton.cuh"

namespace uncomp {

namespace {
constexpr int kEigThreads = 256;
constexpr int kEigWarps = kEigThreads / 32;
constexpr int kTeamThreads = 128;
constexpr int kCoarse = 2 * kEigThreads;
constexpr int n = kD;
template <typename T> struct __align__(2 * sizeof(T)) Pair { T x, y; };

struct EigenSmem {
    double x[2][n];   // row k + 1 before the update of step k
    double v[2][n];   // the step's reflector
    double p[2][n];   // minus the product of the matrix and the reflector
    double part[kEigWarps];
    double sd[n];     // column sums
    double dd[n];
    double ee[n];     // ee[i] couples i and i+1
    double2 de[n];    // (diagonal, -coupling^2) of the scaled matrix, the coupling to the entry before
    double lam[n];
    double scale, trace;
    int cnt[kCoarse + 2];
    int flags[2];
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
// The same for NP points without a branch per step: sign bits are shifted into a word and the changes counted 32 at a
// time, the pair is brought back near 1 every 8 steps (a step shrinks it by at most 2^-60 or so).  A zero between non-zero
// neighbours adds one change whichever sign it gets; a zero that stays zero to the end is recounted.
template <int NP>
__device__ __forceinline__ void sturm_count(const double2 *de, const double (&x)[NP], int (&count)[NP]) {
    double p0[NP], p1[NP];
    uint32_t last[NP];
#pragma unroll
    for (int c = 0; c < NP; ++c) { p0[c] = 0.0; p1[c] = 1.0; count[c] = 0; last[c] = 0u; }
#pragma unroll 1
    for (int w = 0; w < n / 32; ++w) {
        uint32_t m[NP];
#pragma unroll
        for (int c = 0; c < NP; ++c) m[c] = 0u;
#pragma unroll 1
        for (int i0 = 0; i0 < 32; i0 += 8) {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const double2 q = de[w * 32 + i0 + i];
#pragma unroll
                for (int c = 0; c < NP; ++c) {
                    const double pn = fma(q.x - x[c], p1[c], q.y * p0[c]);
                    p0[c] = p1[c];
                    p1[c] = pn;
                    m[c] = __funnelshift_l((uint32_t)__double2hiint(pn), m[c], 1);
                }
            }
#pragma unroll
            for (int c = 0; c < NP; ++c) {
                const int ex = max(__double2hiint(p1[c]) & 0x7ff00000, 0x0c000000);     // at least 2^-831
                const double s = __hiloint2double(0x7fe00000 - ex, 0);
                p0[c] *= s;
                p1[c] *= s;
            }
        }
#pragma unroll
        for (int c = 0; c < NP; ++c) {
            count[c] += __popc(m[c] ^ ((m[c] >> 1) | (last[c] << 31)));
            last[c] = m[c] & 1u;
        }
    }
#pragma unroll
    for (int c = 0; c < NP; ++c)
        if (p1[c] == 0.0) count[c] = sturm_count_robust(de, x[c]);
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
__device__ __forceinline__ void householder_block(double (&A)[8][8], Carry &R, EigenSmem &S, int lane, int warp) {
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
        if (threadIdx.x == 0) S.ee[k] = -minus_alpha;
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
        if (threadIdx.x == 0) S.dd[k + 1] = fma(2.0 * vk, wk, xs[k + 1]);
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
}  // namespace

template <typename PartialT>
__global__ void __launch_bounds__(kEigThreads, 1)
eigen_entropy_kernel(const PartialT *__restrict__ partials, int P, int N, int k_trunc, int center, int norm,
                     int max_iters, float *__restrict__ entropy, float *__restrict__ erank,
                     double *__restrict__ spectrum, uint32_t *__restrict__ status) {
    __shared__ EigenSmem S;
    const int u = blockIdx.x, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int row0 = tid >> 4, t = tid & 15;
    constexpr int len = n * n + n;
    const PartialT *base = partials + (size_t)u * P * len;
    chain_wait();

    // ---- 1. assemble C in registers ----------------------------------------------------------------
    if (tid < n) {
        double s = 0.0;
        for (int p = 0; p < P; ++p) s += (double)base[(size_t)p * len + n * n + tid];
        S.sd[tid] = s;
    }
    if (tid == 0) S.flags[0] = 0;
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
        if (tid == 0) S.dd[0] = S.x[1][0];
        if (t == 0) R.xc[0] = 0.0;
        householder_block<0>(A, R, S, lane, wid);
        householder_block<1>(A, R, S, lane, wid);
        householder_block<2>(A, R, S, lane, wid);
        householder_block<3>(A, R, S, lane, wid);
        householder_block<4>(A, R, S, lane, wid);
        householder_block<5>(A, R, S, lane, wid);
        householder_block<6>(A, R, S, lane, wid);
        householder_block<7>(A, R, S, lane, wid);
        if (tid == 0) { S.ee[n - 2] = R.x0; S.ee[n - 1] = 0.0; }
        if (row0 == 15 && t == 15)                     // entry (127, 127) after the last update
            S.dd[n - 1] = fma(R.vr[7], R.wc[7], fma(R.wr[7], R.vc[7], A[7][7]));
    }
    __syncthreads();

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

    // coarse round: counts at 512 interior points of [lo0, hi0], shared by all eigenvalues (C is positive semi-definite:
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

    // teams of 4 lanes, two points each, refine one eigenvalue: 9-fold per round.  128 threads keep the fp64 units busy;
    // with more, the broadcast loads of the matrix would be the limit.
    const int k = min(k_trunc, n);
    const int iters = max_iters > 0 ? max_iters : 14;
    const double tol = 1e-13;
    const int sub = tid & 3;
    const unsigned team_mask = 0xfu << (lane & 28);
    for (int j0 = 0; tid < kTeamThreads && j0 < k; j0 += kTeamThreads / 4) {
        const int j = j0 + (tid >> 2);              // this team looks for the j-th largest
        const bool active = j < k;
        const int idx = n - 1 - (active ? j : 0);   // its 0-based rank from below
        int lo_i = 0, hi_i = kCoarse + 1;       // cnt[lo_i] <= idx < cnt[hi_i]
        while (hi_i - lo_i > 1) {
            const int mid = (lo_i + hi_i) >> 1;
            if (S.cnt[mid] > idx) hi_i = mid; else lo_i = mid;
        }
        double lo = lo0 + step0 * (double)lo_i, hi = lo0 + step0 * (double)hi_i;
        for (int it = 0; it < iters; ++it) {
            const double width = (hi - lo) * (1.0 / 9.0);
            const bool done = hi - lo <= tol;
            if (__all_sync(0xffffffffu, done)) break;
            const double x[2] = {lo + width * (double)(2 * sub + 1), lo + width * (double)(2 * sub + 2)};
            int c[2];
            sturm_count<2>(S.de, x, c);
            const unsigned above_a = (__ballot_sync(0xffffffffu, c[0] > idx) & team_mask) >> (lane & 28);
            const unsigned above_b = (__ballot_sync(0xffffffffu, c[1] > idx) & team_mask) >> (lane & 28);
            if (!done) {
                // first of the 8 points above the eigenvalue (points 2 s + 1 and 2 s + 2 sit in lane s)
                const int fa = above_a ? 2 * (__ffs(above_a) - 1) : 8, fb = above_b ? 2 * (__ffs(above_b) - 1) + 1 : 8;
                const int f = min(fa, fb);
                const double base_lo = lo;
                if (f < 8) hi = base_lo + width * (double)(f + 1);
                if (f > 0) lo = base_lo + width * (double)f;
            }
        }
        if (active && sub == 0) {
            S.lam[j] = 0.5 * (lo + hi) * scale;
            if (hi - lo > tol) atomicOr(&S.flags[0], 1);
        }
    }
    __syncthreads();

    // ---- 4. entropy -----------------------------------------------------------------------------
    if (wid == 0) {      // lane i takes eigenvalues i, i + 32, ...; fixed-order butterfly sums
        double total = S.trace;
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
            if (S.flags[0]) atomicOr(status, UNCOMP_STATUS_NOT_CONVERGED);
        }
    }
    if (spectrum && tid < k) spectrum[(size_t)u * k + tid] = S.lam[tid];
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

cudaError_t launch_eigen_entropy(const Plan &p, const void *d_partials, const uncomp_entropy_params &ep,
                                 float *d_entropy, float *d_erank, double *d_spectrum, uint32_t *d_status,
                                 cudaStream_t st) {
    const LaunchShape shape{dim3(p.units), kEigThreads, 0, 1, true};
    if (p.shape.dtype == UNCOMP_FP32)
        return launch_kernel(eigen_entropy_kernel<double>, shape, st, (const double *)d_partials, p.gram_splits, p.shape.N,
                             ep.k_trunc, ep.center, ep.norm, ep.max_iters, d_entropy, d_erank, d_spectrum, d_status);
    return launch_kernel(eigen_entropy_kernel<float>, shape, st, (const float *)d_partials, p.gram_splits, p.shape.N, ep.k_trunc,
                         ep.center, ep.norm, ep.max_iters, d_entropy, d_erank, d_spectrum, d_status);
}

}  // namespace uncomp
