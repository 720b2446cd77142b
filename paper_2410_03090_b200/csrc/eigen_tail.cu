// Second half of the eigenvalue stage for bf16 keys: the last 64 x 64 of the Householder reduction, the k largest
// eigenvalues and the entropy (paper Section 3.1 - 3.2; see eigen_f32.cu for the first half).
//
// Why a kernel of its own: at half the size the matrix fits the registers of ONE warp (lane t = lane & 7 of row class
// i = lane / 8 holds the 128 entries M[i + 4 a][4 t + 32 j + e], a < 16, j < 2, e < 4, as packed pairs), so a step needs
// no block barrier, and eight units share an SM where the whole matrix allows two.  The steps are the first kernel's
// (one exchange through shared memory, the rank-2 update one step late) with a warp barrier.
// Bound by the chain of a step (three shuffle reductions, a square root, a reciprocal); two warps per SM sub-partition, what
// the registers admit, use half of its issue slots (1024 units: 49 %, an instruction of a warp every 3.4 cycles).
#include "eigen_common.cuh"

namespace uncomp {

namespace {
constexpr int kT = 128;
constexpr int n = kD, m = kTailN;

struct StepSmem {                    // of one unit
    float p[2][m];                   // minus the product of the matrix and the step's reflector
    float2 pd[2][m];                 // the same, every value twice
    float x[2][m];                   // row k + 1 before the update of step k
    float2 vd[2][m];                 // the step's reflector, every value twice
};
// 8 columns of a row vector into an array that holds every entry twice: the factor of a row as a packed pair
template <int J>
__device__ __forceinline__ void store_twice(const f32x2 (&v)[4], float2 *dst, int t) {
#pragma unroll
    for (int q = 2 * J; q < 4; ++q) {
        float v0, v1;
        unpack2(v[q], v0, v1);
        *reinterpret_cast<float4 *>(dst + 4 * t + 32 * (q >> 1) + 2 * (q & 1)) = make_float4(v0, v0, v1, v1);
    }
}
template <int J>
__device__ __forceinline__ void store_row(const f32x2 (&row)[4], float *x, int t) {
#pragma unroll
    for (int j = J; j < 2; ++j)
        *reinterpret_cast<ulonglong2 *>(x + 4 * t + 32 * j) = make_ulonglong2(row[2 * j], row[2 * j + 1]);
}

// What a lane carries from step to step: the pending rank-2 update (v and -w for its columns; for its rows v and -p lie in
// shared memory and kk makes -w of them) and the row x the next reflector is made of, zero up to the diagonal.
struct Carry {
    f32x2 vc[4], wc[4], xc[4];
    float kk, x0;                    // x0: entry k + 1 of x
};

// Householder steps k = 16 KA .. 16 KA + 15 (stopping at m - 3) of the 64 x 64 matrix: row groups below 4 KA (4 rows each)
// and column groups below J (32 columns) are done.
template <int KA>
__device__ __forceinline__ void warp_householder(f32x2 (&A)[16][4], Carry &R, StepSmem &S, SturmSmem &out, int lane) {
    constexpr int J = KA >> 1, R0 = 4 * KA;
    constexpr bool kOdd = KA == 1;                     // the block's end is also the end of a column group
    const int t = lane & 7, i = lane >> 3;
#pragma unroll 1
    for (int kt = 0; kt < 16; ++kt) {
        const int k = 16 * KA + kt;
        if (KA == 3 && k > m - 3) break;
        const bool end = kOdd && kt == 15;
        // ---- norm of x ----
        f32x2 sq0 = mul2(R.xc[2 * J], R.xc[2 * J]), sq1 = mul2(R.xc[2 * J + 1], R.xc[2 * J + 1]);
        if (J == 0) {
            sq0 = fma2(R.xc[2], R.xc[2], sq0);
            sq1 = fma2(R.xc[3], R.xc[3], sq1);
        }
        const float sig = sum8(sum2(add2(sq0, sq1)));
        // ---- meanwhile the pending update of step k - 1 and A x ----
        const float2 *vd_old = S.vd[(k + 1) & 1] + i, *pd_old = S.pd[(k + 1) & 1] + i;
        const f32x2 kk_old = pack2(R.kk, R.kk);
        f32x2 acc[16];
#pragma unroll
        for (int a = R0; a < 16; ++a) {
            const f32x2 vr = *reinterpret_cast<const f32x2 *>(vd_old + 4 * a);
            const f32x2 wr = fma2(kk_old, vr, *reinterpret_cast<const f32x2 *>(pd_old + 4 * a));
#pragma unroll
            for (int q = 2 * J; q < 4; ++q) A[a][q] = fma2(vr, R.wc[q], fma2(wr, R.vc[q], A[a][q]));
            acc[a] = mul2(A[a][2 * J], R.xc[2 * J]);
#pragma unroll
            for (int q = 2 * J + 1; q < 4; ++q) acc[a] = fma2(A[a][q], R.xc[q], acc[a]);
        }
        float *xs = S.x[k & 1], *ps = S.p[k & 1];
        float2 *vd = S.vd[k & 1], *pd = S.pd[k & 1];
        if (i == ((k + 1) & 3)) {                      // the 8 lanes that hold row k + 1
            switch ((kt + 1) >> 2) {
                case 0: store_row<J>(A[R0], xs, t); break;
                case 1: store_row<J>(A[R0 + 1], xs, t); break;
                case 2: store_row<J>(A[R0 + 2], xs, t); break;
                case 3: store_row<J>(A[R0 + 3], xs, t); break;
                default: store_row<J>(A[R0 + 4 < 16 ? R0 + 4 : 15], xs, t); break;
            }
        }
        // a row whose norm is below 1e-15 of the trace counts as reduced (beta = 0: the step changes nothing)
        const bool flat = !(sig > 1e-30f);
        const float root = sqrt_newton(sig);
        const float minus_alpha = flat ? -R.x0 : (R.x0 >= 0.f ? root : -root);
        const float minus_beta = flat ? 0.f : -recip_newton(fmaf(fabsf(R.x0), root, sig));        // -2 / (v^T v)
        const float vk = R.x0 + minus_alpha;           // v_{k+1}
        if (lane == 0) out.ee[64 + k] = -minus_alpha;
        // ---- v = x - alpha e_{k+1} ----
        float part[16];
#pragma unroll
        for (int a = 0; a < R0; ++a) part[a] = 0.f;
        if (end) {                                     // column k + 1 is the first of the next group
            const f32x2 d0 = pack2(t == 0 ? minus_alpha : 0.f, 0.f);
#pragma unroll
            for (int a = R0; a < 16; ++a) part[a] = sum2(fma2(A[a][2], d0, acc[a]));
            R.xc[2] = add2(R.xc[2], d0);
        } else {
            const int at = k + 1 - 32 * J - 4 * t;
            const f32x2 d0 = pack2(at == 0 ? minus_alpha : 0.f, at == 1 ? minus_alpha : 0.f);
            const f32x2 d1 = pack2(at == 2 ? minus_alpha : 0.f, at == 3 ? minus_alpha : 0.f);
#pragma unroll
            for (int a = R0; a < 16; ++a) part[a] = sum2(fma2(A[a][2 * J], d0, fma2(A[a][2 * J + 1], d1, acc[a])));
            R.xc[2 * J] = add2(R.xc[2 * J], d0);
            R.xc[2 * J + 1] = add2(R.xc[2 * J + 1], d1);
        }
        // ---- -p = -beta A v: sum the 16 rows over the 8 lanes; lane t ends up with row groups 2 t and 2 t + 1 ----
        const bool up4 = (t & 4) != 0, up2 = (t & 2) != 0, up1 = (t & 1) != 0;
        float s8[8], s4[4], s2[2];
#pragma unroll
        for (int a = 0; a < 8; ++a) {
            if (a + 8 < R0) { s8[a] = 0.f; continue; }
            s8[a] = (up4 ? part[a + 8] : part[a]) + __shfl_xor_sync(0xffffffffu, up4 ? part[a] : part[a + 8], 4);
        }
#pragma unroll
        for (int a = 0; a < 4; ++a) s4[a] = (up2 ? s8[a + 4] : s8[a]) + __shfl_xor_sync(0xffffffffu, up2 ? s8[a] : s8[a + 4], 2);
#pragma unroll
        for (int a = 0; a < 2; ++a) s2[a] = (up1 ? s4[a + 2] : s4[a]) + __shfl_xor_sync(0xffffffffu, up1 ? s4[a] : s4[a + 2], 1);
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            const float mp = minus_beta * s2[a];
            ps[i + 8 * t + 4 * a] = mp;
            pd[i + 8 * t + 4 * a] = make_float2(mp, mp);
        }
        if (i == 3 - ((k + 1) & 3)) store_twice<J>(R.xc, vd, t);         // any 8 lanes; not the ones that store the row
        __syncwarp();
        // ---- -w = -p + (beta/2 v^T p) v, then row k + 1 after this step's update: the next x ----
        f32x2 row[4];
#pragma unroll
        for (int j = J; j < 2; ++j) {
            const ulonglong2 p = *reinterpret_cast<const ulonglong2 *>(ps + 4 * t + 32 * j);
            const ulonglong2 r = *reinterpret_cast<const ulonglong2 *>(xs + 4 * t + 32 * j);
            R.wc[2 * j] = p.x;
            R.wc[2 * j + 1] = p.y;
            row[2 * j] = r.x;
            row[2 * j + 1] = r.y;
            R.vc[2 * j] = R.xc[2 * j];
            R.vc[2 * j + 1] = R.xc[2 * j + 1];
        }
        f32x2 dot0 = mul2(R.vc[2 * J], R.wc[2 * J]), dot1 = mul2(R.vc[2 * J + 1], R.wc[2 * J + 1]);
        if (J == 0) {
            dot0 = fma2(R.vc[2], R.wc[2], dot0);
            dot1 = fma2(R.vc[3], R.wc[3], dot1);
        }
        R.kk = 0.5f * minus_beta * sum8(sum2(add2(dot0, dot1)));         // beta/2 v^T p
        const float wk = fmaf(R.kk, vk, ps[k + 1]);
        const f32x2 kk2 = pack2(R.kk, R.kk), vk2 = pack2(vk, vk), wk2 = pack2(wk, wk);
        if (lane == 0) out.dd[64 + k + 1] = fmaf(2.f * vk, wk, xs[k + 1]);
#pragma unroll
        for (int q = 2 * J; q < 4; ++q) {
            R.wc[q] = fma2(kk2, R.vc[q], R.wc[q]);
            R.xc[q] = fma2(vk2, R.wc[q], fma2(wk2, R.vc[q], row[q]));
        }
        {                                              // columns up to k + 1 are zero
            const int at = k + 1 - 32 * J - 4 * t;
            float v0, v1, v2, v3;
            unpack2(R.xc[2 * J], v0, v1);
            unpack2(R.xc[2 * J + 1], v2, v3);
            R.xc[2 * J] = pack2(at >= 0 ? 0.f : v0, at >= 1 ? 0.f : v1);
            R.xc[2 * J + 1] = pack2(at >= 2 ? 0.f : v2, at >= 3 ? 0.f : v3);
            if (end) {
                unpack2(R.xc[2], v0, v1);
                R.xc[2] = pack2(t == 0 ? 0.f : v0, v1);
            }
        }
        {                                              // entry k + 2 of the new x for everybody
            const int c = k + 2;
            const bool next = kOdd && kt >= 14;        // it lies in the next column group
            float a0, a1, a2, a3;
            unpack2(next ? R.xc[2] : R.xc[2 * J], a0, a1);
            unpack2(next ? R.xc[3] : R.xc[2 * J + 1], a2, a3);
            const float lo = (c & 1) ? a1 : a0, hi = (c & 1) ? a3 : a2;
            R.x0 = __shfl_sync(0xffffffffu, (c & 2) ? hi : lo, (lane & 24) + ((c >> 2) & 7));
        }
    }
}
}  // namespace

// a warp per unit; nothing synchronises the block
__global__ void __launch_bounds__(kT, 2)
eigen_tail_kernel(const float *__restrict__ partials, int64_t unit_stride, int units, int k_trunc, int norm, int max_iters,
                  float *__restrict__ entropy, float *__restrict__ erank, double *__restrict__ spectrum,
                  uint32_t *__restrict__ status) {
    __shared__ StepSmem steps[kT / 32];
    __shared__ SturmSmem sturm[kT / 32];
    // warp id by shuffle: uniform for the compiler too (without it every shuffle below costs a convergence check)
    const int lane = threadIdx.x & 31, wid = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0);
    const int u = blockIdx.x * (kT / 32) + wid;
    if (u >= units) return;
    chain_wait();
    const EigenTail &E = *reinterpret_cast<const EigenTail *>(partials + u * unit_stride);
    SturmSmem &S = sturm[wid];

    // ---- 1. the last 62 Householder steps ----------------------------------------------------------
    for (int i = lane; i < m; i += 32) { S.dd[i] = E.dd[i]; S.ee[i] = E.ee[i]; }
    if (lane == 0) S.not_converged = 0;
    {
        StepSmem &P = steps[wid];
        const int t = lane & 7, i = lane >> 3;
        f32x2 A[16][4];
#pragma unroll
        for (int a = 0; a < 16; ++a)
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const ulonglong2 q = *reinterpret_cast<const ulonglong2 *>(&E.M[i + 4 * a][4 * t + 32 * j]);
                A[a][2 * j] = q.x;
                A[a][2 * j + 1] = q.y;
            }
        Carry R;
        R.kk = 0.f;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const ulonglong2 q = *reinterpret_cast<const ulonglong2 *>(&E.M[0][4 * t + 32 * j]);
            R.xc[2 * j] = q.x;
            R.xc[2 * j + 1] = q.y;
            R.vc[2 * j] = R.vc[2 * j + 1] = R.wc[2 * j] = R.wc[2 * j + 1] = 0ull;
        }
        for (int e = lane; e < m; e += 32) P.vd[1][e] = P.pd[1][e] = make_float2(0.f, 0.f);
        R.x0 = E.M[0][1];
        if (lane == 0) S.dd[m] = E.M[0][0];
        if (t == 0) {
            float v0, v1;
            unpack2(R.xc[0], v0, v1);
            R.xc[0] = pack2(0.f, v1);
        }
        __syncwarp();
        warp_householder<0>(A, R, P, S, lane);
        warp_householder<1>(A, R, P, S, lane);
        warp_householder<2>(A, R, P, S, lane);
        warp_householder<3>(A, R, P, S, lane);
        if (lane == 0) { S.ee[n - 2] = R.x0; S.ee[n - 1] = 0.f; }
        if (lane == 31) {                              // entry (63, 63) after the last update (step m - 3)
            const f32x2 vr = *reinterpret_cast<const f32x2 *>(&P.vd[(m - 3) & 1][m - 1]);
            const f32x2 wr = fma2(pack2(R.kk, R.kk), vr, *reinterpret_cast<const f32x2 *>(&P.pd[(m - 3) & 1][m - 1]));
            float lo, hi;
            unpack2(fma2(vr, R.wc[3], fma2(wr, R.vc[3], A[15][3])), lo, hi);
            S.dd[n - 1] = hi;
        }
    }
    __syncwarp();
    finish_unit<32, 1, false>(S, u, lane, true, E.trace, k_trunc, norm, max_iters, entropy, erank, spectrum, status);
}

cudaError_t launch_eigen_tail(int units, float *d_partials, int partials_per_unit, const uncomp_entropy_params &ep,
                              float *d_entropy, float *d_erank, double *d_spectrum, uint32_t *d_status, cudaStream_t st) {
    const int64_t stride = (int64_t)partials_per_unit * (kD * kD + kD);
    return launch_kernel(eigen_tail_kernel, LaunchShape{dim3((units + kT / 32 - 1) / (kT / 32)), kT, 0, 1}, st, d_partials, stride,
                         units, ep.k_trunc, ep.norm, ep.max_iters, d_entropy, d_erank, d_spectrum, d_status);
}

}  // namespace uncomp
