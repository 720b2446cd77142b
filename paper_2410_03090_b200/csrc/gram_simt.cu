// Per-unit Gram matrix G = X^T X and column sums s = X^T 1 on the CUDA cores.
//
// Used for fp32 keys, which need fp64 accumulation: with 1e-3 noise under a unit-scale low-rank signal
// the small eigenvalues of the covariance (Eq. 1 of the paper) sit near 2e-8 of the largest one, below
// what an fp32 Gram entry resolves.  bf16 keys take the tensor-core kernel in gram_tc.cu; the second kernel
// here also accepts them (fp32 accumulation) and is the known-good path the tensor-core kernel is tested
// against.
//
// Each token chunk writes its own partial [d*d + d]; the eigen kernel adds the partials in a fixed order, so results do
// not depend on scheduling.
#include "common.cuh"

namespace uncomp {

// fp32 keys.  Grid: (units x 10 tile pairs I <= J of 32 x 32 entries, token chunks): the symmetric half, and enough CTAs
// for calls of few units and few tokens (one CTA per unit and chunk took 126 us for 8 units of 512 tokens, this 13 us).
// A quarter of the CTA takes every fourth token; a thread owns 4 x 4 entries, so four 16-byte loads feed 16 fp64
// multiply-adds.  The columns are two neighbours in each half of the block: eight lanes read 128 contiguous bytes (four
// neighbours are a two-way bank conflict and made shared memory the bound, at 77 % of its rate with the fp64 pipe at 23 %).
// With the column sums spread over the warps: 8 units of 512 tokens 15.2 -> 12.8 us, the pass of 32 units of 8192 tokens
// 926 -> 840.
__global__ void __launch_bounds__(256) gram_f64_kernel(const float *__restrict__ K, UnitAddr addr, int N, int chunk,
                                                      double *__restrict__ partials, int P) {
    constexpr int TT = 32;
    __shared__ __align__(16) double smem[2 * 2 * TT * 32];          // [buffer][I or J][token][32], later the quarters' sums
    const int pair = blockIdx.x % 10, p = blockIdx.y, u = blockIdx.x / 10;
    const int I = pair < 4 ? 0 : (pair < 7 ? 1 : (pair < 9 ? 2 : 3));
    const int J = pair - (I == 0 ? 0 : (I == 1 ? 3 : (I == 2 ? 5 : 6)));
    const int tid = threadIdx.x, g = tid >> 6, ty = (tid >> 3) & 7, tx = tid & 7;
    const float *X = K + addr.base(u);
    const int t0 = p * chunk, t1 = min(N, t0 + chunk);
    // a stage is 32 tokens x (32 + 32) features: two 16-byte loads per thread, converted on the way to shared memory
    float4 pre[2];
    auto fetch = [&](int t) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int e = tid + 256 * i, tok = e >> 4, c = e & 15;       // c: 8 vectors of block I, 8 of block J
            const int col = c < 8 ? 32 * I + 4 * c : 32 * J + 4 * (c - 8);
            pre[i] = t + tok < t1 ? *reinterpret_cast<const float4 *>(X + (int64_t)(t + tok) * addr.sN + col)
                                  : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    };
    auto store = [&](int b) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int e = tid + 256 * i, tok = e >> 4, c = e & 15;
            double *dst = smem + ((b * 2 + (c >> 3)) * TT + tok) * 32 + 4 * (c & 7);
            *reinterpret_cast<double2 *>(dst) = make_double2((double)pre[i].x, (double)pre[i].y);
            *reinterpret_cast<double2 *>(dst + 2) = make_double2((double)pre[i].z, (double)pre[i].w);
        }
    };
    chain_wait();
    double acc[4][4], colsum = 0.0;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.0;
    fetch(t0);
    store(0);
    __syncthreads();
    for (int t = t0, b = 0; t < t1; t += TT, b ^= 1) {
        if (t + TT < t1) fetch(t + TT);
        const double *tI = smem + b * 2 * TT * 32, *tJ = tI + TT * 32;
#pragma unroll
        for (int k = 0; k < TT / 4; ++k) {
            const int tok = 4 * k + g;
            const double2 a0 = *reinterpret_cast<const double2 *>(tI + tok * 32 + 4 * ty), a1 = *reinterpret_cast<const double2 *>(tI + tok * 32 + 4 * ty + 2);
            const double2 b0 = *reinterpret_cast<const double2 *>(tJ + tok * 32 + 2 * tx), b1 = *reinterpret_cast<const double2 *>(tJ + tok * 32 + 16 + 2 * tx);
            const double a[4] = {a0.x, a0.y, a1.x, a1.y}, c[4] = {b0.x, b0.y, b1.x, b1.y};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fma(a[i], c[j], acc[i][j]);
        }
        if (I == J) {                                  // a warp per four tokens, a lane per column
#pragma unroll
            for (int i = 0; i < TT / 8; ++i) colsum += tI[((tid >> 5) * (TT / 8) + i) * 32 + (tid & 31)];
        }
        if (t + TT < t1) store(b ^ 1);
        __syncthreads();
    }
    // the four quarters, added in order
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) smem[(g * 32 + 4 * ty + i) * 32 + 2 * tx + (j & 1) + 8 * (j & 2)] = acc[i][j];
    __syncthreads();
    double *out = partials + ((size_t)u * P + p) * (kD * kD + kD);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int e = tid + 256 * q, i = e >> 5, j = e & 31;
        const double v = ((smem[e] + smem[1024 + e]) + smem[2048 + e]) + smem[3072 + e];
        out[(32 * I + i) * kD + 32 * J + j] = v;
        if (I != J) out[(32 * J + j) * kD + 32 * I + i] = v;
    }
    if (I == J) {
        __syncthreads();
        smem[tid] = colsum;
        __syncthreads();
        if (tid < 32) {
            double sum = 0.0;
#pragma unroll
            for (int i = 0; i < 8; ++i) sum += smem[32 * i + tid];
            out[kD * kD + 32 * I + tid] = sum;
        }
    }
}

// Grid: (P token chunks, units).  A CTA of 256 threads streams its chunk in tiles of 32 tokens through shared memory;
// thread (ty, tx) owns the 8 x 8 outputs {ty + 16 i} x {tx + 16 j}.
template <typename T, typename Acc>
__global__ void __launch_bounds__(256) gram_simt_kernel(const T *__restrict__ K, UnitAddr addr, int N, int chunk,
                                                        Acc *__restrict__ partials, int P) {
    constexpr int TT = 32;
    __shared__ Acc tile[TT][kD];
    const int p = blockIdx.x, u = blockIdx.y;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const T *X = K + addr.base(u);
    const int t0 = p * chunk;
    const int t1 = min(N, t0 + chunk);

    Acc acc[8][8];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = Acc(0);
    Acc colsum = Acc(0);  // threads 0..127 own one column each

    for (int t = t0; t < t1; t += TT) {
        const int nt = min(TT, t1 - t);
        for (int e = tid; e < TT * kD; e += 256) {
            const int r = e >> 7, c = e & 127;
            tile[r][c] = r < nt ? Acc(to_float(X[(int64_t)(t + r) * addr.sN + c])) : Acc(0);
        }
        __syncthreads();
        if (tid < kD) {
#pragma unroll 8
            for (int r = 0; r < TT; ++r) colsum += tile[r][tid];
        }
#pragma unroll 4
        for (int r = 0; r < TT; ++r) {
            Acc a[8], b[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) { a[i] = tile[r][ty + 16 * i]; b[i] = tile[r][tx + 16 * i]; }
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int j = 0; j < 8; ++j) acc[i][j] += a[i] * b[j];
        }
        __syncthreads();
    }
    Acc *out = partials + ((size_t)u * P + p) * (kD * kD + kD);
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) out[(ty + 16 * i) * kD + tx + 16 * j] = acc[i][j];
    if (tid < kD) out[kD * kD + tid] = colsum;
}

cudaError_t launch_gram_simt(const Plan &p, const void *dK, const UnitAddr &addr, void *d_partials, cudaStream_t st) {
    if (p.shape.dtype == UNCOMP_FP32) {
        return launch_kernel(gram_f64_kernel, LaunchShape{dim3(10 * p.units, p.gram_splits), 256, 0, 1}, st, (const float *)dK, addr,
                             p.shape.N, p.gram_chunk, (double *)d_partials, p.gram_splits);
    } else {
        dim3 grid(p.gram_splits, p.units);
        gram_simt_kernel<__nv_bfloat16, float><<<grid, 256, 0, st>>>((const __nv_bfloat16 *)dK, addr, p.shape.N,
                                                                    p.gram_chunk, (float *)d_partials,
                                                                    p.gram_splits);
    }
    return cudaGetLastError();
}

}  // namespace uncomp
