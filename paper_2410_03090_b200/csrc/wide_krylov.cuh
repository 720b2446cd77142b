// The k largest eigenvalues of a large symmetric matrix by block Lanczos (see wide_krylov.cu).
#pragma once

#include "common.cuh"

namespace uncomp {

constexpr int kKryBlock = 32;        // vectors per block
constexpr int kKryMaxK = 64;         // eigenvalues wanted at most
constexpr int kKryMaxSteps = 40;     // block steps at most
constexpr int kKryMinN = 384;        // smaller matrices: the column-by-column reduction is as fast

// Scratch of one matrix (device pointers), and what the kernels leave there.
struct KrylovBuffers {
    float *Q;            // [steps + 1][32][n] orthonormal blocks, a vector contiguous
    float *part;         // [n / 32][steps + 1][1024] partial products of the CTAs
    float *H;            // [steps][1024] their sums
    double *G;           // [1024] Gram matrix of the new block
    double *T;           // [32 steps + 32][kKryBand] projected matrix, column c: entry (c - o, c) at [c][o], o <= 32
    double *Trev;        // [the same] row r: entry (r, r + o) at [r][o]; read backwards, the columns of T reversed
    double *lam;         // [k + 1] eigenvalues descending, then the trace
    int *state;          // [0] steps in Q, [1] broken, [2] all settled (set by the reduction's kernel); [8 ..] settled, each
    unsigned *bar;       // grid barrier counters, one per launch, zero at the start
};
constexpr int kKryBand = 34;
constexpr int kKryStateInts = 8 + kKryMaxK;

// Largest ratio of the k wanted eigenvalues.  Rounding of the product is a share of the largest one.  Relative to the
// eigenvalue itself (root mean square over 32, six matrices each, n = 1024 and 2048) it comes to 0.4e-6 to 0.7e-6 at ratios
// up to 1000 and 1.0e-6 to 1.2e-6 at 3000, as in the full reduction, but 2.8e-6 to 7.3e-6 at 30000, where the reduction has
// 2.2e-6 to 5.7e-6: beyond this the reduction runs.
constexpr double kKryMaxRatio = 4096.0;

__device__ __forceinline__ bool krylov_too_graded(const double *lam, int k) { return !(lam[0] <= kKryMaxRatio * lam[k - 1]); }

// true when all k eigenvalues have converged (every kernel behind the first asks this before it does anything).  Called by
// whole warps, the answer is the same in all of them.
__device__ __forceinline__ bool krylov_done(const int *state, const double *lam, int k) {
    const int lane = threadIdx.x & 31;
    bool ok = !state[1] && !krylov_too_graded(lam, k);
    for (int i = lane; i < k; i += 32) ok = ok && state[8 + i];
    // a block of 32 start vectors shows an eigenvalue at most 32 times: a cluster of that size may be larger
    for (int i = lane; i + kKryBlock <= k - 1; i += 32) ok = ok && lam[i] - lam[i + kKryBlock - 1] > 1e-6 * lam[0];
    return __all_sync(0xffffffffu, ok);
}

// `ctas`: how many CTAs of the Lanczos kernel the device holds at once (they wait for one another, n / 32 of them)
bool krylov_applies(int n, int k, int ctas);
cudaError_t krylov_resident(int &ctas);
int krylov_steps(int n);             // blocks the buffers hold besides the first
cudaError_t launch_krylov(const float *C, int n, int k, int max_iters, const KrylovBuffers &b, uint32_t *d_status, cudaStream_t st);

}  // namespace uncomp
