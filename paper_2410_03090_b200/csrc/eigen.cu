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

struct EigenSmem {
    double x[n];      // row k of the matrix, zero up to the diagonal
    double x1[n];     // row k + 1
    double v[n];      // reflector
    double p[n];      // beta A v
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

// Row of the matrix to shared memory by the 16 lanes that hold it, zero up to column `upto`.
template <int J>
__device__ __forceinline__ void publish_row(const double (&row)[8], double *dst, int t, int upto) {
#pragma unroll
    for (int j = J; j < 4; ++j) {
        const int c = 32 * j + 2 * t;
        double a = row[2 * j], b = row[2 * j + 1];
        if (j <= J + 1) {                              // groups that can hold columns up to k + 1
            if (c <= upto) a = 0.0;
            if (c + 1 <= upto) b = 0.0;
        }
        *reinterpret_cast<double2 *>(dst + c) = make_double2(a, b);
    }
}
// ... and its diagonal entry
template <int J>
__device__ __forceinline__ void publish_diagonal(const double (&row)[8], double *dst, int t, int k) {
#pragma unroll
    for (int j = J; j < 4 && j <= J + 1; ++j) {
        if (32 * j + 2 * t == k) *dst = row[2 * j];
        if (32 * j + 2 * t + 1 == k) *dst = row[2 * j + 1];
    }
}

// Householder steps k = 16 KA .. 16 KA + 15 (stopping at n - 3); row groups (16 rows) below KA and column groups (32
// columns) below J are done.
template <int KA>
__device__ __forceinline__ void householder_block(double (&A)[8][8], EigenSmem &S, int lane, int warp) {
    constexpr int J = KA >> 1, KN = KA < 7 ? KA + 1 : 7;
    const int i = 2 * warp + (lane >> 4), t = lane & 15;
    const int mine = i + 16 * (t >> 1);                // the row this lane finishes: 2 lanes share it
#pragma unroll 1
    for (int kt = 0; kt < 16; ++kt) {
        const int k = 16 * KA + kt;
        if (KA == 7 && k > n - 3) break;
        // ---- norm of x; y = A x meanwhile ----
        const double x0 = S.x[k + 1];
        double sig;
        {
            const double2 a = *reinterpret_cast<const double2 *>(S.x + 4 * lane), b = *reinterpret_cast<const double2 *>(S.x + 4 * lane + 2);
            sig = fma(a.x, a.x, a.y * a.y) + fma(b.x, b.x, b.y * b.y);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sig += __shfl_xor_sync(0xffffffffu, sig, o);
        double y[8];
#pragma unroll
        for (int a = 0; a < 8; ++a) y[a] = 0.0;
#pragma unroll
        for (int j = J; j < 4; ++j) {
            const double2 x = *reinterpret_cast<const double2 *>(S.x + 32 * j + 2 * t);
#pragma unroll
            for (int a = KA; a < 8; ++a) y[a] = fma(A[a][2 * j], x.x, fma(A[a][2 * j + 1], x.y, y[a]));
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
        // ---- v = x - alpha e_{k+1}; p = beta A v = beta (y - alpha A e_{k+1}), and column k + 1 is row k + 1 ----
        double alpha = x0, beta = 0.0;
        if (sig > 1e-290) {                            // otherwise the row is reduced already: beta = 0
            const double root = sqrt_newton(sig);
            alpha = x0 >= 0.0 ? -root : root;
            beta = recip_newton(fma(fabs(x0), root, sig));            // 2 / (v^T v)
        }
        const double v = mine > k + 1 ? S.x[mine] : (mine == k + 1 ? x0 - alpha : 0.0);
        const double p = mine > k ? beta * fma(-alpha, S.x1[mine], z) : 0.0;
        double s = v * p;
#pragma unroll
        for (int o = 2; o < 32; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) S.part[warp] = s;
        if ((t & 1) == 0) { S.v[mine] = v; S.p[mine] = p; }
        if (mine == k + 1 && (t & 1) == 0) S.ee[k] = alpha;
        __syncthreads();
        // ---- kk = beta/2 v^T p; A -= v p^T + (p - 2 kk v) v^T ----
        double q[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
        for (int w = 0; w < kEigWarps; w += 4) {
            const double2 a = *reinterpret_cast<const double2 *>(S.part + w), b = *reinterpret_cast<const double2 *>(S.part + w + 2);
            q[0] += a.x; q[1] += a.y; q[2] += b.x; q[3] += b.y;
        }
        const double kk = beta * ((q[0] + q[1]) + (q[2] + q[3]));     // 2 kk
        double nv[8], nf[8];
#pragma unroll
        for (int a = KA; a < 8; ++a) {
            const double vr = S.v[i + 16 * a];
            nv[a] = -vr;
            nf[a] = fma(kk, vr, -S.p[i + 16 * a]);
        }
#pragma unroll
        for (int j = J; j < 4; ++j) {
            const double2 vc = *reinterpret_cast<const double2 *>(S.v + 32 * j + 2 * t), pc = *reinterpret_cast<const double2 *>(S.p + 32 * j + 2 * t);
#pragma unroll
            for (int a = KA; a < 8; ++a) {
                A[a][2 * j] = fma(nv[a], pc.x, fma(nf[a], vc.x, A[a][2 * j]));
                A[a][2 * j + 1] = fma(nv[a], pc.y, fma(nf[a], vc.y, A[a][2 * j + 1]));
            }
        }
        // ---- rows k + 1 and k + 2 for the next step ----
        if (i == ((k + 1) & 15)) {
            if (KA == 7 || kt < 15) {
                publish_row<J>(A[KA], S.x, t, k + 1);
                publish_diagonal<J>(A[KA], &S.dd[k + 1], t, k + 1);
            } else {
                publish_row<J>(A[KN], S.x, t, k + 1);
                publish_diagonal<J>(A[KN], &S.dd[k + 1], t, k + 1);
            }
        } else if (i == ((k + 2) & 15)) {
            if (KA == 7 || kt < 14) publish_row<J>(A[KA], S.x1, t, -1);
            else publish_row<J>(A[KN], S.x1, t, -1);
        }
        __syncthreads();
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
            const PartialT *row = base + (size_t)p * len + (row0 + 16 * a) * n + 2 * t;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                A[a][2 * j] += (double)row[32 * j];
                A[a][2 * j + 1] += (double)row[32 * j + 1];
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
    if (row0 == 0) {
        publish_row<0>(A[0], S.x, t, 0);
        if (t == 0) S.dd[0] = A[0][0];
    } else if (row0 == 1) {
        publish_row<0>(A[0], S.x1, t, -1);
    }
    __syncthreads();
    if (tid == 0) {
        double s = 0.0;
        for (int w = 0; w < kEigWarps; ++w) s += S.part[w];
        S.trace = s;
    }
    __syncthreads();                                   // the first step overwrites S.part

    // ---- 2. Householder tridiagonalisation ---------------------------------------------------------
    householder_block<0>(A, S, lane, wid);
    householder_block<1>(A, S, lane, wid);
    householder_block<2>(A, S, lane, wid);
    householder_block<3>(A, S, lane, wid);
    householder_block<4>(A, S, lane, wid);
    householder_block<5>(A, S, lane, wid);
    householder_block<6>(A, S, lane, wid);
    householder_block<7>(A, S, lane, wid);
    if (tid == 0) {                                    // the last 2 x 2 block was published by step n - 3
        S.ee[n - 2] = S.x[n - 1];
        S.dd[n - 1] = S.x1[n - 1];
        S.ee[n - 1] = 0.0;
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
    if (tid == 0) {
        double total = 0.0;
        if (norm) total = S.trace;
        else for (int i = 0; i < k; ++i) total += S.lam[i] > 0.0 ? S.lam[i] : 0.0;
        double h = 0.0;
        if (total > 0.0) {
            for (int i = 0; i < k; ++i) {
                const double p = (S.lam[i] > 0.0 ? S.lam[i] : 0.0) / total;
                if (p > 0.0) h -= p * log(p);
            }
        }
        entropy[u] = (float)h;
        if (erank) erank[u] = (float)exp(h);
        if (S.flags[0]) atomicOr(status, UNCOMP_STATUS_NOT_CONVERGED);
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
