// The k largest eigenvalues of the n x n scatter matrix of the wide entropy (k <= 64, n >= 384) without reducing the
// whole matrix: block Lanczos with full reorthogonalisation from 32 pseudo-random start vectors, then Sturm counts of
// the projected band matrix.
//
//   lanczos_kernel      one cooperative launch per segment of steps.  A CTA owns 32 rows of the matrix and of every
//                       basis block.  Step j: W = C Q_j (fp32 FMA, the rows of C stream from L2), two passes of
//                       W -= Q (Q^T W) with a Cholesky factorisation of W^T W (the first from its own sums, G - H^T H; where
//                       that says nothing any more, three passes), Q_{j+1} = what is left, normalised.  Partial products
//                       of the CTAs meet in global memory and are summed in fp64 in a fixed order, two grid barriers per
//                       pass.  The coefficients make up the projected matrix T, block tridiagonal with upper triangular
//                       couplings: half-bandwidth 32 exactly.
//   band_coarse_kernel  the spectrum's bound, and negative pivots of T - x at 512 shifts that all eigenvalues share.
//   band_eigen_kernel   a cluster of four CTAs per wanted eigenvalue, 15 shifts at a time: a warp eliminates T - x row by row
//                       in fp64 from both ends at once (the 32 x 32 windows behind the pivots in its registers) and counts
//                       negative pivots; their product, the determinant, tells where to put the next shifts.
//
// Why: the reduction column by column sweeps the whole trailing matrix n times (33 ms at n = 4096), although only k of n
// eigenvalues are wanted; here a step of 32 vectors reads the matrix once and 8 to 32 steps suffice (8192 x 4096 hidden
// states with a decaying spectrum, k = 32: 8 steps, 0.69 ms, and the counts 0.29 ms; an isotropic matrix, the slowest to
// converge, takes 32).  Accuracy is that of fp32 products summed in fp32 / fp64, as in the reduction.
// What bounds it, n = 4096, 85 us a step: the product 34 (1 MB per CTA from L2, 24 us without any arithmetic, and multiply-adds,
// 21 us at the 100 per SM and cycle that an outer product in registers reaches), five grid barriers and what they wait for 9,
// sums over the CTAs 6, the two factorisations 8 and 4, H^T H 5, partial products 7, updates 7.  Three passes, sums with one
// load in flight, all of T by one CTA and smaller register tiles took 114.  The counts are bound by the latency of one warp
// per scheduler (an instruction every 3.4 cycles); two warps per scheduler take 1000 cycles per row instead of 570 (8 x 8
// tiles of the window in place of two rows per lane: 1200), so rows are saved by eliminating from both ends and rounds by
// interpolation: 78 us at first and four rounds of 53, where 32 or 1024 shifts counted from one end took 101 and four of 82.
// Convergence is tested by how far an eigenvalue still moves: T_m contains T_{m-64}, so by interlacing the i-th eigenvalue
// has moved by less than delta over the last two blocks exactly if T_{m-64} has i eigenvalues above lambda_i - delta (its
// leading rows of T are the same, so one more shift tells).  delta is 2e-6 of the eigenvalue itself (1e-7 of
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
constexpr int kLWarps = kLT / 32;
constexpr int kKC = 64;                           // columns of C per stage
constexpr int kStages = 3;
constexpr int kPitch = kKC + 4;                   // floats; rows 16 bytes apart in the banks
constexpr int kCached = 17;                       // basis blocks whose 32 rows stay in shared memory
constexpr int kHChunk = 16;                       // blocks of H staged at once

struct LanczosSmem {
    union {
        struct {
            float C[2][kStages][kB][kPitch];      // of either group of warps: rows of C
            float Q[2][kStages][kKC][kB];         // the 32 vectors of Q_j at these columns
        };
        float H[kHChunk * kB * kB];
        float sum[8][kB * kB];
    };
    double piv[2][2][3 * kB];                     // two pivot rows (64 columns) and pivot columns of the factorisation
    double gram[kB * kB];                         // of the block before normalisation
    double V[kB * kB];                            // of the second factorisation: R - I
    float tile[kCached][kB][kB];                  // this CTA's rows of the basis: tile[block][vector][row]
    float Wt[kB][kB + 4];                         // the CTA's rows of W, transposed: Wt[b][r]
    float Rinv[kB][kB];
    float R1[kB][kB], R2[kB][kB];
    float A[kB * kB], A2[kB * kB];                // coefficients of the block before: first passes, last pass
    double red[8][4][32];
    double diag[kB], before[kB];
    int flag;
};
static_assert(sizeof(LanczosSmem) <= 227 * 1024, "shared memory of one CTA");

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

// W tile (32 rows of this CTA x 32 vectors) = C[rows, :] Q_j, left transposed in S.Wt.  Two groups of four warps take every
// other 64 columns, each with its own ring of stages and its own barrier, so that one group's loads and barrier overlap with
// the other's multiply-adds.  A lane takes 4 columns, 8 rows and 16 vectors of a stage: 24 loads of 16 bytes feed 256 packed
// multiply-adds.  The pairs are neighbouring vectors, so Q_j comes with a row's 32 vectors side by side (`rows_of`, the place
// of its rows 32 c ..).  The CTAs start at different columns: all of them read all of Q_j.
// 8 x 4 per lane over whole warps, then 8 x 8 over half-warps with pairs along the columns took 44 us a step at n = 4096, this
// 34.  Registers decide: what spills in this loop takes 55.
__device__ __forceinline__ void product_barrier(int group) { asm volatile("bar.sync %0, 128;" ::"r"(1 + group) : "memory"); }
__device__ __forceinline__ void block_product(LanczosSmem &S, const float *C, const float *rows_of, size_t rows_stride, int n, int r0) {
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, rg = lane & 3, cg = (lane >> 2) & 1, kq = lane >> 3;
    const int group = wid >> 2, gt = tid & (kLT / 2 - 1);
    const int all = n / kKC, stages = (all - group + 1) / 2;          // n is a multiple of 64
    const int turn = (int)((size_t)blockIdx.x * all / gridDim.x);
    const int row = gt >> 4, col = 4 * (gt & 15);                     // of this thread's copies of C: rows row + 8 i
    const float *pc = C + (size_t)(r0 + row) * n + col;
    const uint32_t down = 8u * (uint32_t)n;
    auto stage = [&](int st) {
        if (st < stages) {
            int s = 2 * st + group + turn;
            if (s >= all) s -= all;
            const float *fc = pc + s * kKC, *fq = rows_of + (size_t)(2 * s) * rows_stride + 4 * gt;
            float *tc = &S.C[group][st % kStages][row][col], *tq = &S.Q[group][st % kStages][0][0] + 4 * gt;
#pragma unroll
            for (int i = 0; i < kB / 8; ++i) cp16(tc + 8 * i * kPitch, fc + i * down);
            cp16(tq, fq);
            cp16(tq + 512, fq + 512);
            cp16(tq + 1024, fq + rows_stride);
            cp16(tq + 1536, fq + rows_stride + 512);
        }
        cp_commit();
    };
    f32x2 acc[8][8];                              // [row rg + 4 i][vectors 16 cg + 2 c, + 1]
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int c = 0; c < 8; ++c) acc[i][c] = 0ull;
#pragma unroll
    for (int s = 0; s + 1 < kStages; ++s) stage(s);
    for (int s = 0; s < stages; ++s) {
        cp_wait<kStages - 2>();
        product_barrier(group);                   // stage s has landed; the group is done with stage s - 1
        stage(s + kStages - 1);
        const int k0 = 16 * (wid & 3) + 4 * kq;
        const float *Cs = &S.C[group][s % kStages][rg][k0], *Qs = &S.Q[group][s % kStages][k0][16 * cg];
#pragma unroll 1
        for (int h = 0; h < 4; h += 2) {
            float2 a[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) a[i] = *reinterpret_cast<const float2 *>(Cs + 4 * i * kPitch + h);
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                f32x2 q[8];
#pragma unroll
                for (int c = 0; c < 8; c += 2) {
                    const ulonglong2 x = *reinterpret_cast<const ulonglong2 *>(Qs + (h + k) * kB + 2 * c);
                    q[c] = x.x;
                    q[c + 1] = x.y;
                }
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const f32x2 xx = k == 0 ? pack2(a[i].x, a[i].x) : pack2(a[i].y, a[i].y);
#pragma unroll
                    for (int c = 0; c < 8; ++c) acc[i][c] = fma2(xx, q[c], acc[i][c]);
                }
            }
        }
    }
    cp_wait<0>();
    __syncthreads();
    // the four column quarters of a warp: two transposing levels leave every lane two rows; then the eight warps, in order
    const bool up16 = (lane & 16) != 0, up8 = (lane & 8) != 0;
    f32x2 s4[4][8];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int c = 0; c < 8; ++c)
            s4[i][c] = add2(up16 ? acc[i + 4][c] : acc[i][c], __shfl_xor_sync(0xffffffffu, up16 ? acc[i][c] : acc[i + 4][c], 16));
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            float lo, hi;
            unpack2(add2(up8 ? s4[i + 2][c] : s4[i][c], __shfl_xor_sync(0xffffffffu, up8 ? s4[i][c] : s4[i + 2][c], 8)), lo, hi);
            const int at = (16 * cg + 2 * c) * kB + rg + 4 * (i + (up8 ? 2 : 0) + (up16 ? 4 : 0));
            S.sum[wid][at] = lo;
            S.sum[wid][at + kB] = hi;
        }
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

// Sum over the CTAs of this CTA's share of the entries, 32 entries (a group) at a time: eight warps take every eighth CTA,
// added in a fixed order.  The loads of up to four groups and 16 CTAs each are in flight together, without a branch or a
// condition between them: one after another they took 7 us of a pass, now 3.
__device__ __forceinline__ void reduce_slice(LanczosSmem &S, const KrylovBuffers &B, int nq, bool gram, size_t part_stride,
                                             float *H) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, ctas = gridDim.x;
    constexpr int kGroups = kB * kB / 32;         // of a block
    const int groups = (nq + (gram ? 1 : 0)) * kGroups, most = (groups + ctas - 1) / ctas;
    for (int g0 = 0; g0 < most; g0 += 4) {
        double acc[4] = {0.0, 0.0, 0.0, 0.0};
        const int g[4] = {(int)blockIdx.x + g0 * ctas, (int)blockIdx.x + (g0 + 1) * ctas, (int)blockIdx.x + (g0 + 2) * ctas,
                          (int)blockIdx.x + (g0 + 3) * ctas};
        for (int c0 = 0; c0 < ctas; c0 += 128) {
            float x[4][16];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                if (g[q] < groups) {              // uniform over the CTA
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        x[q][i] = __ldcg(B.part + (size_t)min(c0 + 8 * i + wid, ctas - 1) * part_stride + 32 * g[q] + lane);
                }
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                if (g[q] < groups) {
#pragma unroll
                    for (int i = 0; i < 16; ++i) acc[q] += c0 + 8 * i + wid < ctas ? (double)x[q][i] : 0.0;
                }
            }
#pragma unroll 1
            for (int q = 0; q < 4; ++q) {         // the low words of the block's Gram matrix
                if (g[q] >= nq * kGroups && g[q] < groups) {
                    float y[16];
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        y[i] = __ldcg(B.part + (size_t)min(c0 + 8 * i + wid, ctas - 1) * part_stride + 32 * (g[q] + kGroups) + lane);
                    double low = 0.0;
#pragma unroll
                    for (int i = 0; i < 16; ++i) low += c0 + 8 * i + wid < ctas ? (double)y[i] : 0.0;
                    if (q == 0) acc[0] += low;
                    else if (q == 1) acc[1] += low;
                    else if (q == 2) acc[2] += low;
                    else acc[3] += low;
                }
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) S.red[wid][q][lane] = acc[q];
        __syncthreads();
        const int mine = (int)blockIdx.x + (g0 + wid) * ctas;
        if (wid < 4 && mine < groups) {
            double v = 0.0;
#pragma unroll
            for (int w = 0; w < 8; ++w) v += S.red[w][wid][lane];
            if (mine < nq * kGroups) __stcg(H + 32 * mine + lane, (float)v);
            else __stcg(B.G + 32 * (mine - nq * kGroups) + lane, v);
        }
        __syncthreads();
    }
}

// blocks b0 .. b0 + nb - 1 of H to shared memory
__device__ __forceinline__ void stage_coefficients(LanczosSmem &S, const float *H, int b0, int nb) {
    for (int e = threadIdx.x; e < nb * (kB * kB / 4); e += kLT) cp16(S.H + 4 * e, H + (size_t)b0 * kB * kB + 4 * e);
    cp_commit();
    cp_wait<0>();
    __syncthreads();
}
__device__ __forceinline__ void load_gram(LanczosSmem &S, const double *G) {
    for (int e = threadIdx.x; e < kB * kB; e += kLT) S.gram[e] = __ldcg(G + e);
    __syncthreads();
}
// S.gram -= H^T H: the Gram matrix of W - Q H where H = Q^T W.  In fp32 like H: what rounding leaves in it (3e-7 of the norms
// before) is removed by the pass that follows.  Thread: 4 x 4 entries over every fourth row of H, the quarters added in order.
// H stays staged when one chunk holds it.
__device__ __forceinline__ void project_gram(LanczosSmem &S, const float *H, int nq) {
    const int tid = threadIdx.x, part = tid >> 6, ty = (tid >> 3) & 7, tx = tid & 7;
    double acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.0;
    for (int b0 = 0; b0 < nq; b0 += kHChunk) {
        const int nb = min(kHChunk, nq - b0);
        if (b0 > 0) __syncthreads();
        stage_coefficients(S, H, b0, nb);
#pragma unroll 4
        for (int r = part; r < nb * kB; r += 4) {
            const float4 x = *reinterpret_cast<const float4 *>(S.H + r * kB + 4 * ty), y = *reinterpret_cast<const float4 *>(S.H + r * kB + 4 * tx);
            const double xs[4] = {x.x, x.y, x.z, x.w}, ys[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fma(xs[i], ys[j], acc[i][j]);
        }
    }
    for (int p = 0; p < 4; ++p) {
        if (part == p) {
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) S.gram[(4 * ty + i) * kB + 4 * tx + j] -= acc[i][j];
        }
        __syncthreads();
    }
}

// S.gram = L D L^T by elimination beside the identity; Rinv = L^-T D^-1/2 and R = D^1/2 L^T, so that W Rinv has orthonormal
// columns and W = (W Rinv) R.  Thread: column tid mod 64 of [G | I], eight rows in registers.  Two pivots at a time: one
// barrier, one exchange and one reciprocal on the chain where single pivots take two (5.7 us, now 3.4); the second pivot's
// reciprocal comes from their determinant, but the rows are eliminated one after the other.  (With the inverse of the 2 x 2
// block, whose entries grow with one over the ratio of its pivots, a block of which one direction is 1e10 times the others
// lost the others, and matrices of rank 33 ended in the full reduction.)  False when a pivot is below `share` of what
// its column was (its entry of `before`, or of the diagonal): the column depends on those before it as far as the Gram matrix
// can tell.  Not of the largest column: a matrix whose rank is used up leaves a block whose columns differ by 1e8 in length,
// and its short columns are as good as the long ones.  (Against the largest 200 of 297 matrices with 33 to 300 features in
// use ended in the full reduction, 36 ms instead of 1.3 at n = 4096; now none.)
__device__ __forceinline__ bool factorise(LanczosSmem &S, float (*R)[kB], const double *before, double share) {
    const int tid = threadIdx.x, col = tid & 63, rq = tid >> 6;
    double v[kB / 4];
#pragma unroll
    for (int q = 0; q < kB / 4; ++q) {
        const int i = rq + 4 * q;
        v[q] = col < kB ? S.gram[i * kB + col] : (col - kB == i ? 1.0 : 0.0);
    }
    bool good = true;
#pragma unroll
    for (int s = 0; s < kB; s += 2) {
        double(*P)[3 * kB] = S.piv[(s >> 1) & 1];                 // [pivot]: row (64 columns), column
        if (rq == (s & 3)) P[0][col] = v[s >> 2];
        if (rq == ((s + 1) & 3)) P[1][col] = v[s >> 2];
        if (col == s || col == s + 1) {
            double *column = P[col - s] + 2 * kB;                 // column[8 rq + q]: rows rq + 4 q
#pragma unroll
            for (int q = 0; q < kB / 4; ++q) column[8 * rq + q] = v[q];
        }
        __syncthreads();
        const double a = P[0][s], b = P[1][s], c = P[1][s + 1], u0 = P[0][col], u1 = P[1][col];
        const double lim0 = share * (before ? before[s] : S.gram[s * (kB + 1)]);
        const double lim1 = share * (before ? before[s + 1] : S.gram[(s + 1) * (kB + 1)]);
        const double det = fma(a, c, -b * b);                     // a times the second pivot
        const bool ok = a > lim0 && det > lim1 * a;               // the same in every thread
        good = good && ok;
        const double ia = ok ? recip_newton(a) : 0.0, id = ok ? recip_newton(det) : 0.0;
        const double l = -b * ia, w1 = fma(l, u0, u1), f0 = -u0 * ia, f1 = -w1 * (a * id);      // w1: row s + 1 without row s
#pragma unroll
        for (int q = s >> 2; q < kB / 4; ++q)
            if (rq + 4 * q > s + 1) {
                const double p0 = P[0][2 * kB + 8 * rq + q];
                v[q] = fma(fma(l, p0, P[1][2 * kB + 8 * rq + q]), f1, fma(p0, f0, v[q]));
            }
        if (rq == ((s + 1) & 3)) v[s >> 2] = w1;
        if (tid == s) S.diag[s] = a;
        if (tid == s + 1) S.diag[s + 1] = det * ia;
    }
    __syncthreads();
    if (!good) return false;
#pragma unroll
    for (int q = 0; q < kB / 4; ++q) {
        const int i = rq + 4 * q;
        const double di = rsqrt(S.diag[i]);
        if (col < kB) R[i][col] = i <= col ? (float)(v[q] * di) : 0.f;       // row i of D L^T is what the elimination left
        else S.Rinv[col - kB][i] = col - kB <= i ? (float)(v[q] * di) : 0.f;  // L^-1[i][.]
    }
    __syncthreads();
    return true;
}

// The same for a Gram matrix within 1e-4 of the identity, I + E: with U = upper(E), the diagonal halved, R = I + U - upper(U^T U)
// and Rinv = I - V + V V, V = R - I, up to E^3, which is 3e-8 at most.  (That is what a block's first normalisation leaves as
// a rule.)  U and V^T take the place of the Gram matrix; a thread 2 x 2 entries, so that two loads of 16 bytes feed four
// multiply-adds (1 x 4: 3 us more, shared memory).
__device__ __forceinline__ bool nearly_orthonormal(LanczosSmem &S) {
    bool near = true;
    for (int e = threadIdx.x; e < kB * kB; e += kLT) near = near && fabs(S.gram[e] - (e / kB == e % kB ? 1.0 : 0.0)) < 1e-4;
    return __syncthreads_and(near) != 0;
}
__device__ __forceinline__ void factorise_near(LanczosSmem &S, float (*R)[kB]) {
    const int tid = threadIdx.x, r0 = 2 * (tid >> 4), c0 = 2 * (tid & 15);  // entries (r0, c0) .. (r0 + 1, c0 + 1)
    double *U = S.gram, *Vt = S.gram;
    auto pair = [](const double *at) { return *reinterpret_cast<const double2 *>(at); };
    double own[2][2], v[2][2] = {{0.0, 0.0}, {0.0, 0.0}}, w[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            const int r = r0 + a, c = c0 + b;
            own[a][b] = r < c ? U[r * kB + c] : (r == c ? 0.5 * (U[r * kB + c] - 1.0) : 0.0);
            U[r * kB + c] = own[a][b];
        }
    __syncthreads();
    if (c0 >= r0) {
#pragma unroll 4
        for (int i = 0; i <= r0 + 1; ++i) {       // U^T U
            const double2 x = pair(U + i * kB + r0), y = pair(U + i * kB + c0);
            v[0][0] = fma(x.x, y.x, v[0][0]); v[0][1] = fma(x.x, y.y, v[0][1]);
            v[1][0] = fma(x.y, y.x, v[1][0]); v[1][1] = fma(x.y, y.y, v[1][1]);
        }
    }
    __syncthreads();                              // U has been read
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            const int r = r0 + a, c = c0 + b;
            v[a][b] = r < c ? own[a][b] - v[a][b] : (r == c ? own[a][b] - 0.5 * v[a][b] : 0.0);
            R[r][c] = (float)(v[a][b] + (r == c ? 1.0 : 0.0));
            S.V[r * kB + c] = v[a][b];
            Vt[c * kB + r] = v[a][b];
        }
    __syncthreads();
    if (c0 >= r0) {
#pragma unroll 4
        for (int i = r0; i <= c0 + 1; ++i) {      // V V
            const double2 x = pair(Vt + i * kB + r0), y = pair(S.V + i * kB + c0);
            w[0][0] = fma(x.x, y.x, w[0][0]); w[0][1] = fma(x.x, y.y, w[0][1]);
            w[1][0] = fma(x.y, y.x, w[1][0]); w[1][1] = fma(x.y, y.y, w[1][1]);
        }
    }
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b) S.Rinv[r0 + a][c0 + b] = (float)(w[a][b] - v[a][b] + (r0 + a == c0 + b ? 1.0 : 0.0));
    __syncthreads();
}

// W -= Q H, then W <- W Rinv when `scale`.  A warp takes every eighth row of H, a lane 4 rows of the tile x 8 vectors: three
// loads of 16 bytes feed 32 multiply-adds (one row x 4 vectors per thread and all rows of H took three times the loads).
// The warps' sums are added in warp order.
__device__ __forceinline__ void update_tile(LanczosSmem &S, const float *Q, int n, int r0, int nq, const float *H, bool staged,
                                            bool scale) {
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, tr = 4 * (lane & 7), tc = 8 * (lane >> 3);
    if (nq > 0) {
        float acc[8][4];
#pragma unroll
        for (int c = 0; c < 8; ++c)
#pragma unroll
            for (int r = 0; r < 4; ++r) acc[c][r] = 0.f;
        for (int b0 = 0; b0 < nq; b0 += kHChunk) {
            const int nb = min(kHChunk, nq - b0);
            if (!staged) stage_coefficients(S, H, b0, nb);
            for (int b = 0; b < nb; ++b) {
                const float *q = basis_rows(S, Q, n, r0, b0 + b, 0) + tr;
                const int step = b0 + b < kCached ? kB : n;
#pragma unroll
                for (int i = 0; i < kB / kLWarps; ++i) {
                    const int a = wid + kLWarps * i;
                    const float4 x = *reinterpret_cast<const float4 *>(q + (size_t)a * step);
                    const float *h = S.H + (b * kB + a) * kB + tc;
                    const float4 h0 = *reinterpret_cast<const float4 *>(h), h1 = *reinterpret_cast<const float4 *>(h + 4);
                    const float hs[8] = {h0.x, h0.y, h0.z, h0.w, h1.x, h1.y, h1.z, h1.w};
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        acc[c][0] = fmaf(x.x, hs[c], acc[c][0]);
                        acc[c][1] = fmaf(x.y, hs[c], acc[c][1]);
                        acc[c][2] = fmaf(x.z, hs[c], acc[c][2]);
                        acc[c][3] = fmaf(x.w, hs[c], acc[c][3]);
                    }
                }
            }
            __syncthreads();
        }
#pragma unroll
        for (int c = 0; c < 8; ++c)
            *reinterpret_cast<float4 *>(&S.sum[wid][(tc + c) * kB + tr]) = make_float4(acc[c][0], acc[c][1], acc[c][2], acc[c][3]);
        __syncthreads();
#pragma unroll
        for (int i = 0; i < kB * kB / kLT; ++i) {
            const int e = tid + kLT * i;
            float v = S.sum[0][e];
#pragma unroll
            for (int w = 1; w < kLWarps; ++w) v += S.sum[w][e];
            S.Wt[e / kB][e % kB] -= v;
        }
        __syncthreads();
    }
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
    // the last block of a CTA's partial products holds its rows of the newest basis block, a row's 32 vectors side by side
    const float *rows_of = B.part + (size_t)(part_blocks - 1) * kB * kB;
    unsigned phase = 0;
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
            block_product(S, C, rows_of, part_stride, n, r0);
        }
        // The first pass removes the known directions and normalises what is left by its Gram matrix G - H^T H, which needs
        // no sum of its own; where that difference says nothing any more (a pivot below 1e-5 of what it was), it only
        // removes, and a further pass forms the Gram matrix anew.  The last pass removes what rounding left and normalises.
        bool first = j >= 0;
        for (int pass = first ? 0 : 1; pass < 3; ++pass) {
            partial_products(S, B.Q, n, r0, nq, true, part);
            if (!grid_barrier(bar, phase, status, &S.flag)) return;
            float *H = B.H;
            reduce_slice(S, B, nq, true, part_stride, H);
            if (!grid_barrier(bar, phase, status, &S.flag)) return;
            load_gram(S, B.G);
            bool scale = true;
            if (first) {
                if (tid < kB) S.before[tid] = S.gram[tid * (kB + 1)];
                project_gram(S, H, nq);
                scale = factorise(S, S.R1, S.before, 1e-5);
            } else if (pass == 2 && nearly_orthonormal(S)) {
                factorise_near(S, S.R2);
            } else if (!factorise(S, pass == 1 ? S.R1 : S.R2, nullptr, 1e-14)) {      // the same in every CTA
                if (blockIdx.x == 0 && tid == 0) B.state[1] = 1;
                return;
            }
            if (j >= 0) {                         // for T's diagonal block
                float *out = pass == 2 ? S.A2 : S.A;
                for (int e = tid; e < kB * kB; e += kLT) {
                    const float h = __ldcg(H + (size_t)j * kB * kB + e);
                    out[e] = first || pass == 2 ? h : out[e] + h;
                }
            }
            update_tile(S, B.Q, n, r0, nq, H, first && nq <= kHChunk, scale);
            if (first && scale) pass = 1;
            first = false;
        }
        // the new block, rows r0 ..
        float *Qn = B.Q + (size_t)nq * block;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const float v = S.Wt[4 * wid + c][lane];
            __stcg(Qn + (size_t)(4 * wid + c) * n + r0 + lane, v);
            if (nq < kCached) S.tile[nq][4 * wid + c][lane] = v;
        }
        {
            const int row = tid >> 3, v0 = 4 * (tid & 7);
            __stcg(reinterpret_cast<float4 *>(part + (size_t)(part_blocks - 1) * kB * kB + row * kB + v0),
                   make_float4(S.Wt[v0][row], S.Wt[v0 + 1][row], S.Wt[v0 + 2][row], S.Wt[v0 + 3][row]));
        }
        // T: block (j, j) symmetrised, A + A2 R1, and block (j + 1, j) = R2 R1 (upper triangular: the couplings of block
        // j + 1).  Every CTA knows all of it and writes a few entries (by one CTA it took 2 us that the others waited for).
        const int e = tid * (int)gridDim.x + (int)blockIdx.x;
        if (j >= 0 && e < kB * kB && e / kB <= e % kB) {
            const int r = e / kB, c = e % kB;
            double up = (double)S.A[r * kB + c], low = (double)S.A[c * kB + r], s = 0.0;
            for (int i = 0; i <= c; ++i) up += (double)S.A2[r * kB + i] * (double)S.R1[i][c];
            for (int i = 0; i <= r; ++i) low += (double)S.A2[c * kB + i] * (double)S.R1[i][r];
            for (int i = r; i <= c; ++i) s += (double)S.R2[r][i] * (double)S.R1[i][c];
            B.T[(size_t)(kB * j + c) * kKryBand + c - r] = 0.5 * (up + low);
            B.Trev[(size_t)(kB * j + r) * kKryBand + c - r] = 0.5 * (up + low);
            B.T[(size_t)(kB * (j + 1) + r) * kKryBand + kB + r - c] = s;      // row r of block j + 1, column c of block j
            B.Trev[(size_t)(kB * j + c) * kKryBand + kB + r - c] = s;
        }
        if (!grid_barrier(bar, phase, status, &S.flag)) return;
    }
    if (blockIdx.x == 0 && tid == 0) B.state[0] = q_end;
}

// ---------------------------------------------------------------------------------------- eigenvalues of T
constexpr int kBT = 128;                          // 4 warps, a shift each
constexpr int kBandLead = 64;                     // rows that the leading block of the interlacing check lacks
constexpr int kBandCluster = 4;
constexpr int kCtaShifts = kBT / 32;
constexpr int kShifts = kBandCluster * kCtaShifts - 1;   // 15 shifts per round and the leading block

constexpr int kCoarseCtas = 128;                  // below the number of SMs: a CTA of the counts fills one
constexpr int kCoarse = kCoarseCtas * kCtaShifts; // shifts of the first round, for all eigenvalues together

constexpr int kRing = 8;                          // columns on their way per half-warp

struct BandSmem {
    double ring[kBT / 32][2][kRing][kKryBand];    // the halves' columns; then the middle block's upper triangle
    double row[kBT / 32][2][kB];                  // per half: the pivot row behind the pivot
    int count[2][kShifts + 1], expo[2][kShifts + 1];
    double mant[2][kShifts + 1];                  // of the determinant: mant 2^expo
    double shift[2][kShifts + 1];
    double red[kBT / 32];
};
static_assert(2 * kRing * kKryBand >= kB * (kB + 1) / 2, "the middle block takes the rings' place");

// Elimination of T - x by half a warp, row by row.  Lane h of the half-warp holds the window rows that are h and h + 16 modulo
// 32; a[..][j] is the column j places behind the pivot, so the window moves along by writing a multiply-add one register
// further down.  At row r the lane that owns it publishes the row; row and column r + 32 enter in its place.  Entries of a
// row at earlier columns are never read.  Two rows per lane let one broadcast load of two entries feed four multiply-adds.
// The next pivot is updated first, so its reciprocal is ready when the row is.
struct BandWindow {
    double a[2][kB], d, inv;
    double mant;                                  // product of the pivots so far: mant 2^expo, 1 <= |mant| < 2
    int expo, count;
};
__device__ __forceinline__ void take_pivot(BandWindow &W) {
    W.count += W.d < 0.0;
    W.mant *= W.d;
    const int hi = __double2hiint(W.mant);
    W.expo += ((hi >> 20) & 0x7ff) - 1023;
    W.mant = __hiloint2double((hi & 0x800fffff) | 0x3ff00000, __double2loint(W.mant));
}
__device__ __forceinline__ double band_pivot(double d, double tiny) { return fabs(d) < tiny ? -tiny : d; }
__device__ __forceinline__ void first_pivot(BandWindow &W, double tiny) {
    W.d = band_pivot(__shfl_sync(0xffffffffu, W.a[0][0], threadIdx.x & 16), tiny);
    W.inv = recip_newton(W.d);
}
// 16 `halves` rows.  ENTER: column c of this half's matrix (entry (c - o, c) at [o]) lies at col + c step, c < m.
template <bool ENTER>
__device__ __forceinline__ void band_sweep(BandWindow &W, int halves, const double *__restrict__ col, int step, int m, double x, double tiny,
                                           double *row, double (*ring)[kKryBand]) {
    const int lane = threadIdx.x & 31, h = lane & 15;
    // column r + 32 enters at row r; eight columns are on their way to the half-warp's ring (a row takes less time than L2)
    auto load = [&](int c) {
        if (c < m) {
            const double *src = col + (int64_t)c * step + h;
            cp8(&ring[c % kRing][h], src);
            cp8(&ring[c % kRing][h + 16], src + 16);
            if (h == 0) cp8(&ring[c % kRing][kB], src + kB);
        }
        cp_commit();
    };
    // rows h and h + 16 modulo 32 of it (offset 0 is row r + 32 itself), and its entry in row r
    double next[2] = {0.0, 0.0}, far = 0.0;
    auto fetch = [&](int c) {
        const double *at = ring[c % kRing];
        next[0] = c < m ? at[(c - h) & 31] : 0.0;
        next[1] = c < m ? at[(c - h - 16) & 31] : 0.0;
        far = c < m ? at[kB] : 0.0;
    };
    if (ENTER) {
#pragma unroll 1
        for (int c = kB; c < kB + kRing; ++c) load(c);
        cp_wait<kRing - 1>();
        __syncwarp();
        fetch(kB);
        __syncwarp();                             // row 0 loads column kB + kRing into the place of column kB
    }
#pragma unroll 1
    for (int r0 = 0; r0 < 16 * halves; r0 += kB) {
#pragma unroll
        for (int w = 0; w < 2; ++w) {
            if (w == 1 && r0 + 16 >= 16 * halves) break;
#pragma unroll 1
            for (int s = 0; s < 16; ++s) {
                const int r = r0 + 16 * w + s;
                const bool mine = h == s;
                if (mine) {
#pragma unroll
                    for (int j = 0; j + 2 < kB; j += 2) *reinterpret_cast<double2 *>(row + j) = make_double2(W.a[w][j + 1], W.a[w][j + 2]);
                    *reinterpret_cast<double2 *>(row + kB - 2) = make_double2(W.a[w][kB - 1], far);
                }
                const double enter[2] = {mine && w == 0 ? next[0] - x : next[0], mine && w == 1 ? next[1] - x : next[1]};
                const double u_far = far;
                if (ENTER) {
                    load(r + kB + kRing);         // into the place of column r + 32, which everyone holds in registers
                    cp_wait<kRing - 1>();
                }
                __syncwarp();
                if (ENTER) fetch(r + 1 + kB);
                take_pivot(W);
                const double l0 = -row[(h - r - 1) & 31] * W.inv, l1 = -row[(h + 16 - r - 1) & 31] * W.inv;
                {
                    const double2 u = *reinterpret_cast<const double2 *>(row);
                    W.a[0][0] = fma(l0, u.x, W.a[0][1]);
                    W.a[1][0] = fma(l1, u.x, W.a[1][1]);
                    // the next pivot: row r + 1
                    const double dn = s < 15 ? W.a[w][0] : W.a[1 - w][0];
                    W.d = band_pivot(__shfl_sync(0xffffffffu, dn, (lane & 16) + ((s + 1) & 15)), tiny);
                    W.inv = recip_newton(W.d);
                    W.a[0][1] = fma(l0, u.y, W.a[0][2]);
                    W.a[1][1] = fma(l1, u.y, W.a[1][2]);
                }
#pragma unroll
                for (int j = 2; j + 2 < kB; j += 2) {
                    const double2 u = *reinterpret_cast<const double2 *>(row + j);
                    W.a[0][j] = fma(l0, u.x, W.a[0][j + 1]);
                    W.a[1][j] = fma(l1, u.x, W.a[1][j + 1]);
                    W.a[0][j + 1] = fma(l0, u.y, W.a[0][j + 2]);
                    W.a[1][j + 1] = fma(l1, u.y, W.a[1][j + 2]);
                }
                const double ux = row[kB - 2];
                W.a[0][kB - 2] = fma(l0, ux, W.a[0][kB - 1]);
                W.a[1][kB - 2] = fma(l1, ux, W.a[1][kB - 1]);
                W.a[0][kB - 1] = fma(l0, u_far, enter[0]);
                W.a[1][kB - 1] = fma(l1, u_far, enter[1]);
                __syncwarp();
            }
        }
    }
    if (ENTER) cp_wait<0>();
    __syncwarp();
}

// Eigenvalues below x of the leading m rows of T (m a multiple of 32, 96 at least): negative pivots of T - x.  One half of the
// warp eliminates the rows from the top, the other from the bottom (columns of Trev backwards are columns of the reversed
// matrix); 32 rows in the middle remain, to which both add what their eliminations left, and those are eliminated last: m / 2
// + 16 rows one after another instead of m.  mant 2^expo: the determinant.
__device__ __forceinline__ int band_count(const double *__restrict__ T, const double *__restrict__ Trev, int m, double x, double tiny,
                                          double (*rows)[kB], double (*rings)[kRing][kKryBand], double &mant, int &expo) {
    const int lane = threadIdx.x & 31, h = lane & 15, half = lane >> 4, halves = (m - kB) / 32, p = 16 * halves;
    const double *col = half ? Trev + (int64_t)(m - 1) * kKryBand : T;
    const int step = half ? -kKryBand : kKryBand;
    BandWindow W;
    W.count = W.expo = 0;
    W.mant = 1.0;
    // the first 32 columns: column c holds rows c - o
#pragma unroll
    for (int w = 0; w < 2; ++w)
#pragma unroll
        for (int c = 0; c < kB; ++c) {
            const int i = h + 16 * w;
            double v = i <= c ? __ldg(col + (int64_t)c * step + c - i) : 0.0;
            if (i == c) v -= x;
            W.a[w][c] = v;
        }
    first_pivot(W, tiny);
    band_sweep<true>(W, halves, col, step, m, x, tiny, rows[half], rings[half]);
    // the middle block, rows p .. p + 31: both windows hold it, each with its own side taken off, so T - x itself comes off once
    double *mid = &rings[0][0][0];                // row i of the upper triangle starts at i (65 - i) / 2
    auto at = [](int i, int j) { return i * (2 * kB + 1 - i) / 2 + j - i; };
    if (half == 0) {
#pragma unroll
        for (int w = 0; w < 2; ++w) {
            const int i = (h + 16 * w - p) & 31;
#pragma unroll
            for (int j = 0; j < kB; ++j)
                if (j >= i) mid[at(i, j)] = W.a[w][j];
        }
    }
    __syncwarp();
    if (half == 1) {
#pragma unroll
        for (int w = 0; w < 2; ++w) {
            const int i = (h + 16 * w - p) & 31;  // of the reversed matrix: entry (i, j) is (31 - j, 31 - i)
#pragma unroll
            for (int j = 0; j < kB; ++j)
                if (j >= i) {
                    const double t = __ldg(T + (int64_t)(p + 31 - i) * kKryBand + j - i) - (j == i ? x : 0.0);
                    mid[at(31 - j, 31 - i)] += W.a[w][j] - t;
                }
        }
    }
    __syncwarp();
#pragma unroll
    for (int w = 0; w < 2; ++w)
#pragma unroll
        for (int c = 0; c < kB; ++c) W.a[w][c] = h + 16 * w <= c ? mid[at(h + 16 * w, c)] : 0.0;
    __syncwarp();
    const int sides = W.count + __shfl_xor_sync(0xffffffffu, W.count, 16);
    const double sides_mant = W.mant * __shfl_xor_sync(0xffffffffu, W.mant, 16);
    const int sides_expo = W.expo + __shfl_xor_sync(0xffffffffu, W.expo, 16);
    W.count = W.expo = 0;
    W.mant = 1.0;
    first_pivot(W, tiny);
    band_sweep<false>(W, 2, nullptr, 0, 0, x, tiny, rows[half], nullptr);      // both halves, the same numbers
    mant = sides_mant * W.mant;
    expo = sides_expo + W.expo;
    return sides + W.count;
}

__device__ __forceinline__ double band_low(double bound) { return -1e-6 * bound; }
__device__ __forceinline__ double band_high(double bound) { return bound * (1.0 + 1e-9); }

// To how much an eigenvalue of at least `lo` is bracketed: 2e-8 of itself, but no finer than 1e-13 and no coarser than 1e-9
// of the spectrum's bound.  It has settled when it moved by less than kSettled times that over the last two blocks.
constexpr double kSettled = 100.0;
// Rounds of equal spacing, 16-fold each: six between two shared shifts (2.3e-3 of the bound to 1e-9 of it, 4.6 % of a shift to
// 2e-8), nine below the lowest of them (6.8e-4 of the bound to 1e-13), where an eigenvalue beyond the matrix's rank lies.
constexpr int kBandRounds = 9;
__device__ __forceinline__ double band_tolerance(double lo, double bound) {
    return fmin(fmax(2e-8 * lo, 1e-13 * bound), 1e-9 * bound);
}

// The shared shifts, ascending: kCoarseLow of constant ratio up to 5 % of the bound, where the tolerance becomes a share
// of the eigenvalue itself, and equally spaced from there (2.3e-3 of the bound, 4.6 % of the shift).
constexpr int kCoarseLow = 97;
__device__ __forceinline__ double coarse_shift(int p, double bound) {
    if (p < kCoarseLow) return 0.05 * bound * exp(-0.0449 * (double)(kCoarseLow - 1 - p));
    return bound * (0.05 + 0.95 / (double)(kCoarse - kCoarseLow + 1) * (double)(p - kCoarseLow + 1));
}

// What the coarse round leaves for the eigenvalues, in the scratch of the products.
struct BandCoarse {
    double bound, trace;
    double shift[kCoarse];
    int count[kCoarse];
};

// The first round of the bisection: the bracket is the same for all eigenvalues, so they share 512 shifts, four per
// SM (what a round costs anyway).
__global__ void __launch_bounds__(kBT, 1)
band_coarse_kernel(const float *__restrict__ C, int n, int q, KrylovBuffers B) {
    __shared__ BandSmem S;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, m = q * kB;
    chain_wait();
    // state[0] is q only if the Lanczos launch before this one ran
    if (B.state[1] || B.state[0] != q) return;    // uniform over the grid
    const double *T = B.T;
    BandCoarse *out = reinterpret_cast<BandCoarse *>(B.part);
    // Gershgorin bound of the spectrum (column c of T above the diagonal, row c to its right) and the trace of the whole
    // matrix; a warp per column
    double g = 0.0, tr = 0.0;
#pragma unroll 8
    for (int c = wid; c < m; c += kBT / 32) {
        const double *up = T + (size_t)c * kKryBand, *right = B.Trev + (size_t)c * kKryBand;
        double s = lane <= c ? fabs(__ldg(up + lane)) : 0.0;
        if (lane == 0 && c >= kB) s += fabs(__ldg(up + kB));
        if (c + lane + 1 < m) s += fabs(__ldg(right + lane + 1));
        g = fmax(g, warp_sum(s));
    }
    if (blockIdx.x == 0)
        for (int i = tid; i < n; i += kBT) tr += (double)C[(size_t)i * n + i];
    tr = warp_sum(tr);
    if (lane == 0) S.red[wid] = g;
    __syncthreads();
    double bound = 1e-280;
#pragma unroll
    for (int w = 0; w < kBT / 32; ++w) bound = fmax(bound, S.red[w]);
    __syncthreads();
    if (lane == 0) S.red[wid] = tr;
    __syncthreads();
    const int p = blockIdx.x * kCtaShifts + wid;
    const double x = coarse_shift(p, bound);
    double mant;
    int expo;
    const int c = band_count(T, B.Trev, m, x, bound * 1e-19, S.row[wid], S.ring[wid], mant, expo);
    if (lane == 0) {
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
    chain_wait();
    // flags and eigenvalues are read by the NEXT launch
    if (B.state[1] || B.state[0] != q) return;    // uniform over the grid
    cluster.barrier_arrive();                     // waited for before anybody's shared memory is written
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
    cluster.barrier_wait();                       // every CTA runs
    if (first > 0) lo = in->shift[first - 1];
    if (first < kCoarse) hi = in->shift[first];
    int c_lo = first > 0 ? in->count[first - 1] : 0, c_hi = first < kCoarse ? in->count[first] : m;
    // max_iters counts 257-fold rounds, as in the full reduction; these are 16-fold after the coarse 513 intervals
    const int rounds = max_iters > 0 ? min(max((8 * max_iters - 6) / 4, 1), kBandRounds) : kBandRounds;
    bool settled = false, done = false, guided = false;
    double guess = 0.0, width = 0.0;              // a guess of the eigenvalue, and the bracket it was made for
    // a guided round that has not earned as much as one of equal spacing does not count; one of those follows it
    for (int it = 0, spent = 0; spent < rounds && !done; ++it) {
        const double tol = band_tolerance(lo, bound), step = (hi - lo) / (double)(kShifts + 1);
        // Shifts: equally spaced, or seven on either side of the guess at distances that grow from half the tolerance to a
        // quarter of the bracket, and the guess itself.
        width = hi - lo;
        const double near = 0.45 * tol, grow = guided ? exp(log(fmax(0.25 * width / near, 1.0)) * (1.0 / 6.0)) : 1.0;
        const int p = rank * kCtaShifts + wid;
        // beside them the leading block: have t + 1 of its eigenvalues come this far?
        const bool lead = p == kShifts;
        const int rows = lead ? m - kBandLead : m;
        double x;
        if (lead) {
            x = guided ? guess - 0.84 * kSettled * tol : hi - kSettled * tol;
        } else if (guided) {
            double far = p == kShifts / 2 ? 0.0 : near;
            for (int i = 1; i < abs(p - kShifts / 2); ++i) far *= grow;
            x = guess + (p < kShifts / 2 ? -far : far);
        } else {
            x = lo + step * (double)(p + 1);
        }
        double mant;
        int expo;
        const int c = band_count(T, B.Trev, rows, x, tiny, S.row[wid], S.ring[wid], mant, expo);
        if (lane < kBandCluster) {
            BandSmem *R = cluster.map_shared_rank(&S, lane);
            R->count[it & 1][p] = lead ? rows - c : c;
            R->mant[it & 1][p] = mant;
            R->expo[it & 1][p] = expo;
            R->shift[it & 1][p] = x;
        }
        cluster.sync();
        const int *count = S.count[it & 1];
        const double *shift = S.shift[it & 1];
        // the shifts whose count is still <= idx come first; those outside the bracket say nothing new
        int nb = 0, last_in = kShifts;
        for (int q = 0; q < kShifts; ++q) {
            const double y = shift[q];
            if (y <= lo || (y < hi && count[q] <= idx)) nb = q + 1;
            if (y >= hi) last_in = min(last_in, q);
        }
        const double old_lo = lo, old_hi = hi;
        if (nb > 0 && shift[nb - 1] > old_lo) { lo = shift[nb - 1]; c_lo = count[nb - 1]; }
        if (nb < last_in && shift[nb] < old_hi) { hi = shift[nb]; c_hi = count[nb]; }
        done = hi - lo <= band_tolerance(lo, bound);
        settled = count[kShifts] >= t + 1;
        // The next guess: inverse interpolation of the determinant through the four shifts around the eigenvalue, when it is
        // the only one in the bracket and all four lie in the old bracket.
        const bool earned = hi - lo <= (1.0 / 16.0) * width;
        spent += !guided || earned;
        const int i0 = min(max(nb - 2, 0), kShifts - 4);
        bool usable = c_hi - c_lo == 1 && (!guided || earned);
        double xs[4], fs[4];
        int top = INT_MIN;
        for (int i = 0; i < 4; ++i) top = max(top, S.expo[it & 1][i0 + i]);
        for (int i = 0; i < 4; ++i) {
            xs[i] = shift[i0 + i];
            fs[i] = ldexp(S.mant[it & 1][i0 + i], max(S.expo[it & 1][i0 + i] - top, -2000));
            usable = usable && xs[i] > old_lo && xs[i] < old_hi;
        }
        for (int w = 1; w < 4; ++w)
            for (int i = 0; i + w < 4; ++i) {
                const double df = fs[i + w] - fs[i];
                usable = usable && df != 0.0;
                xs[i] = (fs[i + w] * xs[i] - fs[i] * xs[i + 1]) / df;
            }
        usable = usable && xs[0] > lo && xs[0] < hi;
        guess = xs[0];
        guided = usable;
    }
    if (rank == 0 && tid == 0) {
        B.lam[t] = 0.5 * (lo + hi);
        B.state[8 + t] = done && settled ? 1 : 0;
        if (!done) atomicOr(status, (uint32_t)UNCOMP_STATUS_NOT_CONVERGED);
        if (t == 0) B.lam[k] = in->trace;
    }
    cluster.sync();                               // nobody leaves while another may still write its counts
}
}  // namespace

// More than kKryMaxK = 64 eigenvalues go to the reduction: the range that the tests hold against the oracle, not where the
// two sides meet.  That depends on the spectrum: 8192 x 4096 with 256 strong directions takes 1.6 ms here at k = 64, 4.8 at
// 128, 7.4 at 256, the reduction 35.5 whatever k; an isotropic matrix of n = 2048 7.6 ms at k = 64 against 11.3.
// kKryMinN: at n = 384 the buffers just hold the eight steps of k <= 32.  256 strong directions take 0.94 ms there (the
// reduction 1.6), isotropic matrices, which leave the steps unsettled, 2.5; from n = 768 on those are faster here as well (3.2
// and 3.3 ms; n = 1024 4.4 and 4.6, 4096 5.7 and 35.6).
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
    // Steps at first, and twice as many whenever some eigenvalue has not settled.  Ten spectra (256 strong directions, power
    // laws, exponential, 50 and 600 directions, isotropic; n = 1024 to 4096), all together: k = 32 from 6 steps 22.1 ms, from 8
    // 19.7, 10 20.7, 12 20.7, 16 24.6; k = 64 from 6 41.0, 8 38.2, 10 32.3, 12 32.0, 16 35.8, without the two isotropic ones
    // 10 19.3 and 12 20.1.
    int part_blocks = most + 3, q0 = 0, q = k <= 32 ? 8 : 10, launch = 0;
    while (true) {
        unsigned *bar = b.bar + launch;
        KrylovBuffers B = b;
        void *args[] = {(void *)&C, (void *)&n, (void *)&k, (void *)&q0, (void *)&q, (void *)&part_blocks, (void *)&B,
                        (void *)&bar, (void *)&d_status};
        e = cudaLaunchCooperativeKernel((const void *)lanczos_kernel, dim3(n / kB), dim3(kLT), args, sizeof(LanczosSmem), st);
        if (e != cudaSuccess) return e;
        e = launch_kernel(band_coarse_kernel, LaunchShape{dim3(kCoarseCtas), kBT, 0, 1}, st, C, n, q, b);
        if (e != cudaSuccess) return e;
        e = launch_kernel(band_eigen_kernel, LaunchShape{dim3(k * kBandCluster), kBT, 0, 1}, st, k, q, max_iters, b, d_status);
        if (e != cudaSuccess) return e;
        if (q >= most || ++launch >= 3) break;
        q0 = q;
        q = min(most, 2 * q);
    }
    return cudaSuccess;
}

}  // namespace uncomp
