// The k largest eigenvalues of the n x n scatter matrix of the wide entropy (k <= 64, n >= 384) without reducing the
// whole matrix: block Lanczos with full reorthogonalisation from 32 pseudo-random start vectors, then Sturm counts of
// the projected band matrix.
//
//   lanczos_kernel      one cooperative launch per segment of block steps.  A CTA owns 32 rows of the matrix and of every
//                       basis block.  Step j: W = C Q_j (fp32 FMA, the rows of C stream from L2), three passes of
//                       W -= Q (Q^T W) (the second and third with a Cholesky factorisation of W^T W in fp64), Q_{j+1} =
//                       what is left, normalised.  Partial products of the CTAs meet in global memory and are summed in
//                       fp64 in a fixed order, two grid barriers per pass.  The coefficients make up the projected
//                       matrix T, block tridiagonal with upper triangular couplings: half-bandwidth 32 exactly.
//   band_coarse_kernel  the spectrum's bound, and negative pivots of T - x at 1024 shifts that all eigenvalues share.
//   band_eigen_kernel   a cluster of four CTAs per wanted eigenvalue, 32 shifts at a time, 33-fold per round: a warp
//                       eliminates T - x row by row in fp64 (the trailing 32 x 32 window in its registers) and counts
//                       negative pivots.
//
// Why: the reduction column by column sweeps the whole trailing matrix n times (33 ms at n = 4096), although only k of n
// eigenvalues are wanted; here a step of 32 vectors reads the matrix once and 8 to 32 steps suffice (8192 x 4096 hidden
// states with a decaying spectrum, k = 32: 8 steps, 0.93 ms, and the counts 0.44 ms, 0.1 more with no shared round; an
// isotropic matrix, the slowest to converge, takes 32).  Accuracy is that of fp32 products summed in fp32 / fp64, as in the
// reduction.
// What bounds it: about 70 us of every step are grid barriers, sums over the CTAs and the two factorisations, whatever n;
// the product takes 17 us of fp32 multiply-adds at n = 4096.  The counts are bound by the latency of one warp: eight shifts
// per SM are one warp per scheduler, which issues every 3.4 cycles (1.4 of them wait for results of fixed latency, 0.3 for
// shared memory, 0.3 for columns of T, 0.2 at branches); 29 % of the issue slots, 23 % of the fp64 pipe and, next in line,
// 52 % of the shared-memory pipe are used, which is why a second warp per scheduler did not pay.
// Convergence is tested by how far an eigenvalue still moves: T_m contains T_{m-64}, so by interlacing the i-th eigenvalue
// has moved by less than delta over the last two blocks exactly if T_{m-64} has i eigenvalues above lambda_i - delta (its
// pivots are the first ones of T, so one of the last round's shifts tells).  delta is 2e-6 of the eigenvalue itself (1e-7 of
// the bound at most, 1e-11 at least), not of the largest one: with one direction 1e5 times the rest the others may be off by
// per cents and still move by less than 1e-7 of the largest.  A movement is not a bound of the error; the error is smaller
// than the last movement as long as the steps converge at least as fast as before, which block Lanczos does (isotropic
// matrices of n = 1024, the slowest: movements of 4e-3, 1e-5, 1e-9 over two blocks left errors of 4e-4, 1e-7 and less).
// What has not settled gets twice as many steps, in a second and a third launch; they leave at once when there is
// nothing to do.  Not settled after that, a block that loses rank, a cluster as large as the block (an eigenvalue that may
// have higher multiplicity than the block can show), or wanted eigenvalues further apart than kKryMaxRatio: the
// caller's full reduction runs instead.
#include <cooperative_groups.h>

#include "grid_barrier.cuh"
#include "newton.cuh"
#include "wide_krylov.cuh"

namespace uncomp {

namespace {
constexpr int kB = kKryBlock;
constexpr int kLT = 256;                          // threads of the Lanczos kernel
constexpr int kKC = 64;                           // columns of C per stage
constexpr int kStages = 4;
constexpr int kPitch = kKC + 4;                   // floats; rows 16 bytes apart in the banks
constexpr int kCached = 28;                       // basis blocks whose 32 rows stay in shared memory
constexpr int kHChunk = 16;                       // blocks of H staged at once

struct LanczosSmem {
    union {
        struct {
            float C[kStages][kB][kPitch];         // rows of C
            float Q[kStages][kB][kPitch];         // the same columns of the 32 vectors of Q_j
        };
        float H[kHChunk * kB * kB];
        float sum[8][kB * kB];
        double piv[2][3 * kB];                    // pivot row (64 columns) and pivot column of the factorisation
    };
    float tile[kCached][kB][kB];                  // this CTA's rows of the basis: tile[block][vector][row]
    float Wt[kB][kB + 4];                         // the CTA's rows of W, transposed: Wt[b][r]
    float Rinv[kB][kB];
    float R1[kB][kB], R2[kB][kB];
    double red[8][4][32];
    double diag[kB];
    int flag, bad;
};

__device__ __forceinline__ void cp16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp8(void *dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// A pseudo-random number in (-1, 1) from its place: three multiplications modulo 2^32, by the fractions of the golden ratio
// and of the roots of 2 and 3 made odd, each followed by its upper half folded into the lower.  It only has to be
// unrelated to the data: 32 vectors of 384 places have a condition number of 1.7, of 4096 places 1.2, like numpy's.
__device__ __forceinline__ float place_random(uint32_t i) {
    i = (i + 1u) * 0x9e3779b9u;
    i = (i ^ (i >> 16)) * 0x6a09e667u;
    i = (i ^ (i >> 15)) * 0xbb67ae85u;
    i ^= i >> 16;
    return (float)(int)i * 0x1p-31f;
}

// rows r0 .. r0 + 31 of vector `a` of basis block `blk`
__device__ __forceinline__ const float *basis_rows(const LanczosSmem &S, const float *Q, int n, int r0, int blk, int a) {
    return blk < kCached ? S.tile[blk][a] : Q + ((size_t)blk * kB + a) * n + r0;
}

// W tile (32 rows of this CTA x 32 vectors) = C[rows, :] Q_j, left transposed in S.Wt.  A warp takes 8 of the 64 columns
// of a stage; a lane 8 rows x 4 vectors, pairs of neighbouring columns in one packed multiply-add.  Four stages in
// flight cover the latency of L2.
__device__ __forceinline__ void block_product(LanczosSmem &S, const float *C, const float *Qj, int n, int r0) {
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, rg = lane >> 3, cg = lane & 7;
    const int stages = n / kKC;                   // n is a multiple of 64
    auto stage = [&](int s) {
        if (s < stages) {
#pragma unroll
            for (int i = 0; i < kB * (kKC / 4) / kLT; ++i) {
                const int e = tid + kLT * i, row = e / (kKC / 4), c = 4 * (e % (kKC / 4));
                cp16(&S.C[s % kStages][row][c], C + (size_t)(r0 + row) * n + s * kKC + c);
                cp16(&S.Q[s % kStages][row][c], Qj + (size_t)row * n + s * kKC + c);
            }
        }
        cp_commit();
    };
    f32x2 acc[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[i][c] = 0ull;
#pragma unroll
    for (int s = 0; s + 1 < kStages; ++s) stage(s);
    for (int s = 0; s < stages; ++s) {
        cp_wait<kStages - 2>();
        __syncthreads();                          // stage s has landed; everyone is done with stage s - 1
        stage(s + kStages - 1);
        const float(*Cs)[kPitch] = S.C[s % kStages];
        const float(*Qs)[kPitch] = S.Q[s % kStages];
#pragma unroll
        for (int kk = 8 * wid; kk < 8 * wid + 8; kk += 4) {
            ulonglong2 b[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) b[c] = *reinterpret_cast<const ulonglong2 *>(&Qs[cg + 8 * c][kk]);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const ulonglong2 a = *reinterpret_cast<const ulonglong2 *>(&Cs[rg + 4 * i][kk]);
#pragma unroll
                for (int c = 0; c < 4; ++c) acc[i][c] = fma2(a.y, b[c].y, fma2(a.x, b[c].x, acc[i][c]));
            }
        }
    }
    cp_wait<0>();
    __syncthreads();
    // the eight warps' sums, added in warp order
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int c = 0; c < 4; ++c) S.sum[wid][(cg + 8 * c) * kB + rg + 4 * i] = sum2(acc[i][c]);
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kB * kB / kLT; ++i) {
        const int e = tid + kLT * i;
        float v = S.sum[0][e];
#pragma unroll
        for (int w = 1; w < 8; ++w) v += S.sum[w][e];
        S.Wt[e / kB][e % kB] = v;
    }
    __syncthreads();
}

// partial products of this CTA's rows: blk < nq: Q_blk^T W, blk == nq: W^T W.  Thread: row a of the result, four columns.
__device__ __forceinline__ void partial_products(const LanczosSmem &S, const float *Q, int n, int r0, int nq, bool gram,
                                                 float *part) {
    const int tid = threadIdx.x, a = tid >> 3, b0 = tid & 7;
    f32x2 w[4][kB / 2];
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int r = 0; r < kB; r += 4) {
            const ulonglong2 x = *reinterpret_cast<const ulonglong2 *>(&S.Wt[b0 + 8 * c][r]);
            w[c][r / 2] = x.x;
            w[c][r / 2 + 1] = x.y;
        }
    for (int blk = 0; blk < nq; ++blk) {
        const ulonglong2 *q = reinterpret_cast<const ulonglong2 *>(basis_rows(S, Q, n, r0, blk, a));
        ulonglong2 x[kB / 4];
#pragma unroll
        for (int r = 0; r < kB / 4; ++r) x[r] = q[r];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            f32x2 s = mul2(x[0].x, w[c][0]);
            s = fma2(x[0].y, w[c][1], s);
#pragma unroll
            for (int r = 1; r < kB / 4; ++r) s = fma2(x[r].y, w[c][2 * r + 1], fma2(x[r].x, w[c][2 * r], s));
            part[(size_t)blk * (kB * kB) + a * kB + b0 + 8 * c] = sum2(s);
        }
    }
    if (gram) {
        ulonglong2 x[kB / 4];
#pragma unroll
        for (int r = 0; r < kB / 4; ++r) x[r] = *reinterpret_cast<const ulonglong2 *>(&S.Wt[a][4 * r]);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            double s = 0.0;                       // products of fp32 numbers are exact in fp64
#pragma unroll
            for (int r = 0; r < kB / 4; ++r) {
                float a0, a1, b0_, b1_;
                unpack2(x[r].x, a0, a1);
                unpack2(w[c][2 * r], b0_, b1_);
                s = fma((double)a0, (double)b0_, fma((double)a1, (double)b1_, s));
                unpack2(x[r].y, a0, a1);
                unpack2(w[c][2 * r + 1], b0_, b1_);
                s = fma((double)a0, (double)b0_, fma((double)a1, (double)b1_, s));
            }
            // high and low word of the sum, so that the total keeps more than fp32
            const float hi = (float)s;
            part[(size_t)nq * (kB * kB) + a * kB + b0 + 8 * c] = hi;
            part[(size_t)(nq + 1) * (kB * kB) + a * kB + b0 + 8 * c] = (float)(s - (double)hi);
        }
    }
}

// Sum over the CTAs, this CTA's slice of the entries: eight warps take every eighth CTA, added in warp order.
__device__ __forceinline__ void reduce_slice(LanczosSmem &S, const KrylovBuffers &B, int nq, bool gram, size_t part_stride,
                                             float *H) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, ctas = gridDim.x;
    const int entries = (nq + (gram ? 1 : 0)) * kB * kB;
    const int per = ((entries + ctas - 1) / ctas + 31) & ~31;
    const int e0 = min(entries, (int)blockIdx.x * per), e1 = min(entries, e0 + per);
    for (int base = e0; base < e1; base += 128) {
        double acc[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 4
        for (int c = wid; c < ctas; c += 8) {
            const float *p = B.part + (size_t)c * part_stride;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int e = base + 32 * q + lane;
                if (e < e1) {
                    acc[q] += (double)__ldcg(p + e);
                    if (e >= nq * kB * kB) acc[q] += (double)__ldcg(p + e + kB * kB);
                }
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) S.red[wid][q][lane] = acc[q];
        __syncthreads();
        if (wid < 4) {
            const int e = base + 32 * wid + lane;
            if (e < e1) {
                double v = 0.0;
#pragma unroll
                for (int w = 0; w < 8; ++w) v += S.red[w][wid][lane];
                if (e < nq * kB * kB) __stcg(H + e, (float)v);
                else __stcg(B.G + e - nq * kB * kB, v);
            }
        }
        __syncthreads();
    }
}

// G = L D L^T by elimination beside the identity; Rinv = L^-T D^-1/2 and R = D^1/2 L^T, so that W Rinv has orthonormal
// columns and W = (W Rinv) R.  Thread: column tid mod 64 of [G | I], eight rows in registers; a step publishes pivot row
// and pivot column, one barrier each.  A pivot that has lost all of its column's norm marks the block as broken.
__device__ __forceinline__ void factorise(LanczosSmem &S, const double *G, float (*R)[kB]) {
    const int tid = threadIdx.x, col = tid & 63, rq = tid >> 6;
    double v[kB / 4], top = 0.0;
#pragma unroll
    for (int q = 0; q < kB / 4; ++q) {
        const int i = rq + 4 * q;
        v[q] = col < kB ? __ldcg(G + i * kB + col) : (col - kB == i ? 1.0 : 0.0);
    }
    if (tid < kB) S.diag[tid] = __ldcg(G + tid * (kB + 1));
    if (tid == 0) S.bad = 0;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kB; ++i) top = fmax(top, S.diag[i]);
#pragma unroll
    for (int s = 0; s < kB; ++s) {
        double *row = S.piv[s & 1], *column = row + 2 * kB;      // column[8 rq + q]: rows rq + 4 q
        if (rq == (s & 3)) row[col] = v[s >> 2];
        if (col == s) {
#pragma unroll
            for (int q = 0; q < kB / 4; ++q) column[8 * rq + q] = v[q];
        }
        __syncthreads();
        const double d = row[s], u = row[col];
        const bool ok = d > 1e-14 * top;
        if (!ok && tid == 0) S.bad = 1;
        const double inv = ok ? recip_newton(d) : 0.0, f = -u * inv;
#pragma unroll
        for (int q = s >> 2; q < kB / 4; ++q)
            if (rq + 4 * q > s) v[q] = fma(column[8 * rq + q], f, v[q]);
        if (tid == s) S.diag[s] = d;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kB / 4; ++q) {
        const int i = rq + 4 * q;
        const double di = S.diag[i] > 0.0 ? rsqrt(S.diag[i]) : 0.0;
        if (col < kB) R[i][col] = i <= col ? (float)(v[q] * di) : 0.f;       // row i of D L^T is what the elimination left
        else S.Rinv[col - kB][i] = col - kB <= i ? (float)(v[q] * di) : 0.f;  // L^-1[i][.]
    }
    __syncthreads();
}

// W -= Q H, then W <- W Rinv when `scale`.  Thread: row r = lane of the tile, columns 4 wid .. 4 wid + 3.
__device__ __forceinline__ void update_tile(LanczosSmem &S, const float *Q, int n, int r0, int nq, const float *H, bool scale) {
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    float acc[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[c] = S.Wt[4 * wid + c][lane];
    for (int b0 = 0; b0 < nq; b0 += kHChunk) {
        const int nb = min(kHChunk, nq - b0);
        for (int e = tid; e < nb * (kB * kB / 4); e += kLT) cp16(S.H + 4 * e, H + (size_t)b0 * kB * kB + 4 * e);
        cp_commit();
        cp_wait<0>();
        __syncthreads();
        for (int b = 0; b < nb; ++b) {
            const float *q = basis_rows(S, Q, n, r0, b0 + b, 0) + lane;
            const int step = b0 + b < kCached ? kB : n;
            const float4 *h4 = reinterpret_cast<const float4 *>(S.H + b * kB * kB) + wid;
#pragma unroll 16
            for (int a = 0; a < kB; ++a) {
                const float x = q[(size_t)a * step];
                const float4 h = h4[a * (kB / 4)];
                acc[0] = fmaf(-x, h.x, acc[0]);
                acc[1] = fmaf(-x, h.y, acc[1]);
                acc[2] = fmaf(-x, h.z, acc[2]);
                acc[3] = fmaf(-x, h.w, acc[3]);
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) S.Wt[4 * wid + c][lane] = acc[c];
    __syncthreads();
    if (!scale) return;
    float out[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 8
    for (int b = 0; b < kB; ++b) {
        const float w = S.Wt[b][lane];
        const float4 x = *reinterpret_cast<const float4 *>(&S.Rinv[b][4 * wid]);
        out[0] = fmaf(w, x.x, out[0]);
        out[1] = fmaf(w, x.y, out[1]);
        out[2] = fmaf(w, x.z, out[2]);
        out[3] = fmaf(w, x.w, out[3]);
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < 4; ++c) S.Wt[4 * wid + c][lane] = out[c];
    __syncthreads();
}

__global__ void __launch_bounds__(kLT, 1) lanczos_kernel(const float *__restrict__ C, int n, int k, int q_begin, int q_end,
                                                        int part_blocks, KrylovBuffers B, unsigned *bar,
                                                        uint32_t *__restrict__ status) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    LanczosSmem &S = *reinterpret_cast<LanczosSmem *>(smem_raw);
    if (B.state[1]) return;                       // the same answers in every CTA
    if (q_begin > 0 && (krylov_too_graded(B.lam, k) || krylov_done(B.state, B.lam, k))) return;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, r0 = blockIdx.x * kB;
    const size_t block = (size_t)kB * n, part_stride = (size_t)part_blocks * kB * kB;
    float *part = B.part + (size_t)blockIdx.x * part_stride;
    unsigned phase = 0;
    float a_sum[4];                               // T block (j, j): H of the first two passes (CTA 0)
    if (q_begin > 0) {                            // the basis so far
        for (int e = tid; e < min(q_begin + 1, kCached) * kB * (kB / 4); e += kLT) {
            const int vec = e / (kB / 4), c = 4 * (e % (kB / 4));
            *reinterpret_cast<float4 *>(&S.tile[0][0][0] + vec * kB + c) =
                __ldcg(reinterpret_cast<const float4 *>(B.Q + (size_t)vec * n + r0 + c));
        }
        __syncthreads();
    }

    for (int j = q_begin == 0 ? -1 : q_begin; j < q_end; ++j) {
        const int nq = j + 1;                     // blocks to be orthogonal to
        if (j < 0) {
#pragma unroll
            for (int c = 0; c < 4; ++c)
                S.Wt[4 * wid + c][lane] = place_random((uint32_t)((r0 + lane) * kB + 4 * wid + c));
            __syncthreads();
        } else {
            block_product(S, C, B.Q + j * block, n, r0);
        }
        // pass 0 removes the known directions, passes 1 and 2 what rounding left of them, and normalise
        for (int pass = j < 0 ? 1 : 0; pass < 3; ++pass) {
            const bool gram = pass > 0;
            partial_products(S, B.Q, n, r0, nq, gram, part);
            if (!grid_barrier(bar, phase, status, &S.flag)) return;
            float *H = B.H;
            reduce_slice(S, B, nq, gram, part_stride, H);
            if (!grid_barrier(bar, phase, status, &S.flag)) return;
            if (gram) {
                factorise(S, B.G, pass == 1 ? S.R1 : S.R2);
                if (S.bad) {                      // the same in every CTA
                    if (blockIdx.x == 0 && tid == 0) B.state[1] = 1;
                    return;
                }
            }
            if (blockIdx.x == 0 && j >= 0 && pass < 2) {
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const float h = __ldcg(H + (size_t)j * kB * kB + tid + kLT * c);
                    a_sum[c] = pass == 0 ? h : a_sum[c] + h;
                }
            }
            update_tile(S, B.Q, n, r0, nq, H, gram);
        }
        // the new block, rows r0 ..
        float *Qn = B.Q + (size_t)nq * block;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const float v = S.Wt[4 * wid + c][lane];
            __stcg(Qn + (size_t)(4 * wid + c) * n + r0 + lane, v);
            if (nq < kCached) S.tile[nq][4 * wid + c][lane] = v;
        }
        if (blockIdx.x == 0 && j >= 0) {
            // T: block (j, j) symmetrised, block (j + 1, j) = R2 R1 (upper triangular: the couplings of block j + 1)
            float *A = &S.Rinv[0][0];
            __syncthreads();
#pragma unroll
            for (int c = 0; c < 4; ++c) A[tid + kLT * c] = a_sum[c];
            __syncthreads();
            for (int e = tid; e < kB * kB; e += kLT) {
                const int r = e / kB, c = e % kB;
                if (r <= c) B.T[(size_t)(kB * j + c) * kKryBand + c - r] = 0.5 * ((double)A[r * kB + c] + (double)A[c * kB + r]);
                if (r <= c) {                     // entry (row r of block j + 1, column c of block j)
                    double s = 0.0;
                    for (int i = r; i <= c; ++i) s += (double)S.R2[r][i] * (double)S.R1[i][c];
                    B.T[(size_t)(kB * (j + 1) + r) * kKryBand + kB + r - c] = s;
                }
            }
        }
        if (!grid_barrier(bar, phase, status, &S.flag)) return;
    }
    if (blockIdx.x == 0 && tid == 0) B.state[0] = q_end;
}

// ---------------------------------------------------------------------------------------- eigenvalues of T
constexpr int kBT = 128;                          // 4 warps, two shifts each: 8 shifts per CTA
constexpr int kBandLead = 64;                     // rows that the leading block of the interlacing check lacks
constexpr int kBandCluster = 4;
constexpr int kCtaShifts = kBT / 16;
constexpr int kShifts = kBandCluster * kCtaShifts;   // 32 shifts per round

constexpr int kCoarseCtas = 128;                  // below the number of SMs: a CTA of the counts fills one
constexpr int kCoarse = kCoarseCtas * kCtaShifts; // shifts of the first round, for all eigenvalues together

constexpr int kRing = 8;                          // columns of T on their way per warp

struct BandSmem {
    double ring[kBT / 32][kRing][kKryBand];
    double row[kCtaShifts][kB];                   // per shift: the pivot row behind the pivot
    int count[2][kShifts];
    double red[kBT / 32];
};

// Negative pivots of T - x, rows 0 .. m - 1 (in lead: rows 0 .. m - kBandLead - 1), by half a warp per shift.  Lane i of the half-warp holds the window rows
// that are i and i + 16 modulo 32; register j is the column j places behind the pivot, so the window moves along by
// writing a multiply-add one register further down.  At row r the lane that owns it publishes the row; row and column
// r + 32 enter in its place.  Entries of a row at earlier columns are never read.
// Two rows per lane let one broadcast load of two entries feed four multiply-adds (with one row per lane and one shift
// per warp the shared-memory pipe was the limit: 740 cycles per row at 8 shifts per SM, now 570).  The next pivot is
// updated first, so its reciprocal is ready when the row is.
__device__ __forceinline__ int band_count(const double *__restrict__ T, int m, double x, double tiny, double *row,
                                          double (*ring)[kKryBand], int &lead) {
    const int lane = threadIdx.x & 31, h = lane & 15;
    double a[2][kB];
    // the first 32 columns: column c holds rows c - o
#pragma unroll
    for (int w = 0; w < 2; ++w)
#pragma unroll
        for (int c = 0; c < kB; ++c) {
            const int i = h + 16 * w;
            double v = i <= c ? __ldg(T + (size_t)c * kKryBand + c - i) : 0.0;
            if (i == c) v -= x;
            a[w][c] = v;
        }
    int count = 0;
    auto pivot = [&](double d) { return fabs(d) < tiny ? -tiny : d; };
    double d = pivot(__shfl_sync(0xffffffffu, a[0][0], lane & 16)), inv = recip_newton(d);
    // column r + 32 enters at row r; eight columns are on their way to the warp's ring (a row takes less time than L2)
    auto load = [&](int c) {
        if (c < m) {
            cp8(&ring[c % kRing][lane], T + (size_t)c * kKryBand + lane);
            if (lane == 0) cp8(&ring[c % kRing][kB], T + (size_t)c * kKryBand + kB);
        }
        cp_commit();
    };
    // rows h and h + 16 modulo 32 of it (offset 0 is row r + 32 itself), and its entry in row r
    double next[2], far;
    auto fetch = [&](int c) {
        const double *col = ring[c % kRing];
        next[0] = c < m ? col[(c - h) & 31] : 0.0;
        next[1] = c < m ? col[(c - h - 16) & 31] : 0.0;
        far = c < m ? col[kB] : 0.0;
    };
#pragma unroll 1
    for (int c = kB; c < kB + kRing; ++c) load(c);
    cp_wait<kRing - 1>();
    __syncwarp();
    fetch(kB);
    for (int r0 = 0; r0 < m; r0 += kB) {
        if (r0 == m - kBandLead) lead = count;
#pragma unroll
        for (int w = 0; w < 2; ++w) {
#pragma unroll 1
            for (int s = 0; s < 16; ++s) {
                const int r = r0 + 16 * w + s;
                const bool mine = h == s;
                if (mine) {
#pragma unroll
                    for (int j = 0; j + 2 < kB; j += 2) *reinterpret_cast<double2 *>(row + j) = make_double2(a[w][j + 1], a[w][j + 2]);
                    *reinterpret_cast<double2 *>(row + kB - 2) = make_double2(a[w][kB - 1], far);
                }
                const double enter[2] = {mine && w == 0 ? next[0] - x : next[0], mine && w == 1 ? next[1] - x : next[1]};
                const double u_far = far;
                load(r + kB + kRing);             // into the place of column r + 32, which everyone holds in registers
                cp_wait<kRing - 1>();
                __syncwarp();
                fetch(r + 1 + kB);
                count += d < 0.0;
                const double l0 = -row[(h - r - 1) & 31] * inv, l1 = -row[(h + 16 - r - 1) & 31] * inv;
                {
                    const double2 u = *reinterpret_cast<const double2 *>(row);
                    a[0][0] = fma(l0, u.x, a[0][1]);
                    a[1][0] = fma(l1, u.x, a[1][1]);
                    // the next pivot: row r + 1
                    const double dn = s < 15 ? a[w][0] : a[1 - w][0];
                    d = pivot(__shfl_sync(0xffffffffu, dn, (lane & 16) + ((s + 1) & 15)));
                    inv = recip_newton(d);
                    a[0][1] = fma(l0, u.y, a[0][2]);
                    a[1][1] = fma(l1, u.y, a[1][2]);
                }
#pragma unroll
                for (int j = 2; j + 2 < kB; j += 2) {
                    const double2 u = *reinterpret_cast<const double2 *>(row + j);
                    a[0][j] = fma(l0, u.x, a[0][j + 1]);
                    a[1][j] = fma(l1, u.x, a[1][j + 1]);
                    a[0][j + 1] = fma(l0, u.y, a[0][j + 2]);
                    a[1][j + 1] = fma(l1, u.y, a[1][j + 2]);
                }
                const double ux = row[kB - 2];
                a[0][kB - 2] = fma(l0, ux, a[0][kB - 1]);
                a[1][kB - 2] = fma(l1, ux, a[1][kB - 1]);
                a[0][kB - 1] = fma(l0, u_far, enter[0]);
                a[1][kB - 1] = fma(l1, u_far, enter[1]);
                __syncwarp();
            }
        }
    }
    cp_wait<0>();
    __syncwarp();
    return count;
}

__device__ __forceinline__ double band_low(double bound) { return -1e-6 * bound; }
__device__ __forceinline__ double band_high(double bound) { return bound * (1.0 + 1e-9); }

// To how much an eigenvalue of at least `lo` is bracketed: 2e-8 of itself, but no finer than 1e-13 and no coarser than 1e-9
// of the spectrum's bound.  It has settled when it moved by less than kSettled times that over the last two blocks.
constexpr double kSettled = 100.0;
__device__ __forceinline__ double band_tolerance(double lo, double bound) {
    return fmin(fmax(2e-8 * lo, 1e-13 * bound), 1e-9 * bound);
}

// The shared shifts, ascending: kCoarseLow of constant ratio up to 5 % of the bound, where the tolerance becomes a share
// of the eigenvalue itself, and equally spaced from there.  Both spacings are what four rounds bring to the tolerance
// (32 times 33^3 of it: 1.15e-3 of the bound, 2.3 % of the shift); below 6.6e-4 of the bound it takes two or three more.
constexpr int kCoarseLow = 194;
__device__ __forceinline__ double coarse_shift(int p, double bound) {
    if (p < kCoarseLow) return 0.05 * bound * exp(-0.02245 * (double)(kCoarseLow - 1 - p));
    return bound * (0.05 + 0.95 / (double)(kCoarse - kCoarseLow + 1) * (double)(p - kCoarseLow + 1));
}

// What the coarse round leaves for the eigenvalues, in the scratch of the products.
struct BandCoarse {
    double bound, trace;
    double shift[kCoarse];
    int count[kCoarse];
};

// The first round of the bisection: the bracket is the same for all eigenvalues, so they share 1024 shifts, eight per
// SM (what a round costs anyway), instead of 32 each: five rounds to the tolerance instead of six.
__global__ void __launch_bounds__(kBT, 1)
band_coarse_kernel(const float *__restrict__ C, int n, int q, KrylovBuffers B) {
    __shared__ BandSmem S;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, m = q * kB;
    // state[0] is q only if the Lanczos launch before this one ran
    if (B.state[1] || B.state[0] != q) return;    // uniform over the grid
    const double *T = B.T;
    BandCoarse *out = reinterpret_cast<BandCoarse *>(B.part);
    // Gershgorin bound of the spectrum (entries (i, c), i <= c, in column c) and the trace of the whole matrix
    double g = 0.0, tr = 0.0;
    for (int c = tid; c < m; c += kBT) {
        double s = 0.0;
        for (int o = 0; o <= kB && o <= c; ++o) s += fabs(__ldg(T + (size_t)c * kKryBand + o));
        for (int o = 1; o <= kB && c + o < m; ++o) s += fabs(__ldg(T + (size_t)(c + o) * kKryBand + o));
        g = fmax(g, s);
    }
    if (blockIdx.x == 0)
        for (int i = tid; i < n; i += kBT) tr += (double)C[(size_t)i * n + i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) g = fmax(g, __shfl_xor_sync(0xffffffffu, g, o));
    tr = warp_sum(tr);
    if (lane == 0) S.red[wid] = g;
    __syncthreads();
    double bound = 1e-280;
#pragma unroll
    for (int w = 0; w < kBT / 32; ++w) bound = fmax(bound, S.red[w]);
    __syncthreads();
    if (lane == 0) S.red[wid] = tr;
    __syncthreads();
    const int own = tid >> 4, p = blockIdx.x * kCtaShifts + own;
    const double x = coarse_shift(p, bound);
    int lead = 0;
    const int c = band_count(T, m, x, bound * 1e-19, S.row[own], S.ring[wid], lead);
    if ((lane & 15) == 0) {
        out->shift[p] = x;
        out->count[p] = c;
    }
    if (blockIdx.x == 0 && tid == 0) {
        double sum = 0.0;
#pragma unroll
        for (int w = 0; w < kBT / 32; ++w) sum += S.red[w];
        out->bound = bound;
        out->trace = sum;
    }
}

__global__ void __cluster_dims__(kBandCluster, 1, 1) __launch_bounds__(kBT, 1)
band_eigen_kernel(int k, int q, int max_iters, KrylovBuffers B, uint32_t *__restrict__ status) {
    namespace cg = cooperative_groups;
    __shared__ BandSmem S;
    __shared__ int s_first;
    cg::cluster_group cluster = cg::this_cluster();
    const int t = blockIdx.x / kBandCluster, rank = (int)cluster.block_rank();
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, m = q * kB;
    // flags and eigenvalues are read by the NEXT launch
    if (B.state[1] || B.state[0] != q) return;    // uniform over the grid
    const double *T = B.T;
    const BandCoarse *in = reinterpret_cast<const BandCoarse *>(B.part);
    const double bound = in->bound, tiny = bound * 1e-19;
    const int idx = m - 1 - t;                    // ascending index of the t-th largest
    double lo = band_low(bound), hi = band_high(bound);          // count(lo) <= idx < count(hi)
    if (tid == 0) s_first = kCoarse;
    __syncthreads();
    int first = kCoarse;                          // the first coarse shift above the eigenvalue
    for (int p = tid; p < kCoarse; p += kBT)
        if (in->count[p] > idx) first = min(first, p);
    atomicMin(&s_first, first);
    __syncthreads();
    first = s_first;
    if (first > 0) lo = in->shift[first - 1];
    if (first < kCoarse) hi = in->shift[first];
    // max_iters counts 257-fold rounds, as in the full reduction; these are 33-fold after the coarse 1025 intervals
    const int rounds = max_iters > 0 ? min(max((8 * max_iters - 6) / 5, 1), 7) : 7;
    bool last = false;
    for (int it = 0; it < rounds && !last; ++it) {
        const double tol = band_tolerance(lo, bound);
        last = hi - lo <= tol * (double)kShifts || it == rounds - 1;
        const int shifts = last ? kShifts - 1 : kShifts;
        const double step = (hi - lo) / (double)(shifts + 1);
        const int own = tid >> 4, p = rank * kCtaShifts + own;
        int lead = 0;
        const double x = p < shifts ? lo + step * (double)(p + 1) : hi - kSettled * tol;
        const int c = band_count(T, m, x, tiny, S.row[own], S.ring[wid], lead);
        if (p == shifts && (lane & 15) == 0) B.state[8 + t] = (m - kBandLead) - lead >= t + 1 ? 1 : 0;
        if ((lane & 15) < kBandCluster) cluster.map_shared_rank(&S, lane & 15)->count[it & 1][p] = c;
        cluster.sync();
        // the shifts whose count is still <= idx come first
        int nb = 0;
#pragma unroll
        for (int g0 = 0; g0 < kShifts; g0 += 32)
            nb += __popc(__ballot_sync(0xffffffffu, g0 + lane < shifts && S.count[it & 1][g0 + lane] <= idx));
        const double nl = nb > 0 ? lo + step * (double)nb : lo, nh = nb < shifts ? lo + step * (double)(nb + 1) : hi;
        lo = nl;
        hi = nh;
    }
    if (rank == 0 && tid == 0) {
        B.lam[t] = 0.5 * (lo + hi);
        if (hi - lo > band_tolerance(lo, bound)) atomicOr(status, (uint32_t)UNCOMP_STATUS_NOT_CONVERGED);
        if (t == 0) B.lam[k] = in->trace;
    }
    cluster.sync();                               // nobody leaves while another may still write its counts
}
}  // namespace

// More than kKryMaxK = 64 eigenvalues go to the reduction: the range that the tests hold against the oracle, not where the
// two sides meet.  That depends on the spectrum: 8192 x 4096 with 256 strong directions takes 2.2 ms here at k = 64, 5.0 at
// 128, 11.5 at 256, the reduction 35.8 whatever k; an isotropic matrix of n = 2048 12.8 ms at k = 64 against 11.3.
// kKryMinN: at n = 384 the buffers just hold the eight steps of k <= 32.
bool krylov_applies(int n, int k, int ctas) {
    return n >= kKryMinN && k <= kKryMaxK && krylov_steps(n) >= (k <= 32 ? 8 : 10) && n / kB <= ctas;
}

cudaError_t krylov_resident(int &ctas) {
    static bool done[64] = {};
    int dev = 0, sms = 0, per_sm = 0;
    cudaError_t e = allow_dynamic_smem((const void *)lanczos_kernel, sizeof(LanczosSmem), done);
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, lanczos_kernel, kLT, sizeof(LanczosSmem));
    ctas = sms * per_sm;
    return e;
}
int krylov_steps(int n) { return n < kKryMinN ? 0 : min(kKryMaxSteps, (n - 128) / kB); }

cudaError_t launch_krylov(const float *C, int n, int k, int max_iters, const KrylovBuffers &b, uint32_t *d_status,
                          cudaStream_t st) {
    cudaError_t e = cudaSuccess;
    const int most = krylov_steps(n);
    // Steps at first, and twice as many whenever some eigenvalue has not settled.  Nine spectra (256 strong directions, power
    // laws, exponential, 50 and 600 directions, isotropic; n = 1024 to 4096), k = 32, all nine together: from 6 steps 28.8 ms,
    // from 8 26.6, 10 32.1, 12 27.0, 16 32.8.  k = 64, the six of them that end here: from 8 29.8 ms, 10 24.8, 12 22.9,
    // 16 26.3; 10 is the best of the two with 256 strong directions (2.2 and 1.7 ms against 2.6 and 2.1 from 12).
    int part_blocks = most + 3, q0 = 0, q = k <= 32 ? 8 : 10, launch = 0;
    while (true) {
        unsigned *bar = b.bar + launch;
        KrylovBuffers B = b;
        void *args[] = {(void *)&C, (void *)&n, (void *)&k, (void *)&q0, (void *)&q, (void *)&part_blocks, (void *)&B,
                        (void *)&bar, (void *)&d_status};
        e = cudaLaunchCooperativeKernel((const void *)lanczos_kernel, dim3(n / kB), dim3(kLT), args, sizeof(LanczosSmem), st);
        if (e != cudaSuccess) return e;
        band_coarse_kernel<<<kCoarseCtas, kBT, 0, st>>>(C, n, q, b);
        band_eigen_kernel<<<k * kBandCluster, kBT, 0, st>>>(k, q, max_iters, b, d_status);
        if (q >= most || ++launch >= 3) break;
        q0 = q;
        q = min(most, 2 * q);
    }
    return cudaGetLastError();
}

}  // namespace uncomp
