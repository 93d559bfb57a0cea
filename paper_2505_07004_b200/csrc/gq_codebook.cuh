// Codebook step of the layer-wise quantiser (Section 4.2, Eq. 8; the codebook steps of Algorithm 2): for every
// output channel j of group k, with the assignment matrix P in {0,1}^{d_in x m} given by the codes Q,
//
//     c^(j) = (P^T H_k P + lambda I)^-1  P^T H_k w_j .
//
// The d_in^2-sized contractions and their sums by level are one tensor-core kernel (gq_codebook_gemm.cuh).  The kernels
// here prepare its W operand, solve the m x m systems by Cholesky in fp64 and write W_hat.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "gq_ptx.cuh"

namespace gq {

constexpr int CB_MAX_LEVELS = 16;

// W [d_out][d_in] -> bf16 hi + lo of W^T [d_in][d_out] (lo = what hi leaves, 2^-17 |w| is dropped).  Tiles of 32
// coordinates x 64 channels, so that both sides move whole 128-byte segments (one bf16 per lane and 64-byte segments took
// 57 us for 4096 x 4096 where the bytes need 20).
__global__ void __launch_bounds__(256)
cb_transpose_kernel(const float *W, int d_in, int d_out, __nv_bfloat16 *W0, __nv_bfloat16 *W1)
{
    __shared__ float tw[64][33];
    griddep_launch();
    griddep_wait();
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int i0 = blockIdx.x * 32, j0 = blockIdx.y * 64;
#pragma unroll
    for (int r = 0; r < 64; r += 8) {
        const int j = j0 + r + ty, i = i0 + tx;
        tw[r + ty][tx] = (j < d_out && i < d_in) ? W[static_cast<size_t>(j) * d_in + i] : 0.0f;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 32; r += 8) {
        const int i = i0 + r + ty, j = j0 + 2 * tx;          // d_out is a multiple of 8: pairs are inside or outside
        if (i < d_in && j < d_out) {
            const float a = tw[2 * tx][r + ty], b = tw[2 * tx + 1][r + ty];
            const __nv_bfloat162 hi = __floats2bfloat162_rn(a, b);
            const __nv_bfloat162 lo = __floats2bfloat162_rn(a - __low2float(hi), b - __high2float(hi));
            const size_t o = static_cast<size_t>(i) * d_out + j;
            *reinterpret_cast<__nv_bfloat162 *>(W0 + o) = hi;
            *reinterpret_cast<__nv_bfloat162 *>(W1 + o) = lo;
        }
    }
}

// (G + lambda I) c = r by Cholesky in fp64; G is symmetrised first (its two triangles come from different sums).  Sixteen lanes per channel, lane q holds row q (rows from m on
// are those of the identity).  A pivot that is not positive (possible only through rounding) is replaced by lambda-sized
// regularisation so that the solve always completes.  With one thread per channel and its matrix in local memory 4096
// channels took 89 us.
__global__ void __launch_bounds__(128)
cb_solve_kernel(const double *G, const double *R, int d_out, int m, double lambda,
                float *codebook)
{
    constexpr int M = CB_MAX_LEVELS;
    griddep_launch();
    griddep_wait();
    const int q = threadIdx.x & 15;
    const int jj = blockIdx.x * 8 + (threadIdx.x >> 4);
    const int j = jj < d_out ? jj : d_out - 1;           // all lanes take part in the shuffles
    const double *g = G + static_cast<size_t>(j) * M * M;
    double a[M], b = q < m ? R[static_cast<size_t>(j) * M + q] : 0.0, diag = 1.0;
#pragma unroll
    for (int t = 0; t < M; ++t) {
        a[t] = (q < m && t < m) ? 0.5 * (g[q * M + t] + g[t * M + q]) : 0.0;
        if (t == q) a[t] = q < m ? a[t] + lambda : 1.0;
    }
    auto from = [](double v, int lane) { return __shfl_sync(0xffffffffu, v, lane, 16); };
#pragma unroll
    for (int t = 0; t < M; ++t) {                        // column t of L; a[t] of lane q > t becomes L[q][t]
        double d = from(a[t], t);
        if (!(d > 0.0)) d = lambda > 0.0 ? lambda : 1e-300;
        const double root = sqrt(d);
        if (q == t) diag = root;
        const double l = q > t ? a[t] / root : 0.0;
        a[t] = l;
#pragma unroll
        for (int s = t + 1; s < M; ++s) a[s] -= l * from(l, s);
        const double y = from(b, t) / root;              // L y = r alongside
        b = q == t ? y : b - l * y;
    }
#pragma unroll
    for (int t = M - 1; t >= 0; --t) {                   // L^T c = y
        double sum = q > t ? a[t] * b : 0.0;             // lanes above t hold their c already
#pragma unroll
        for (int off = 8; off > 0; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off, 16);
        if (q == t) b = (b - sum) / diag;
    }
    if (jj < d_out && q < m) codebook[static_cast<size_t>(j) * m + q] = static_cast<float>(b);
}

// What[j][i] = codebook[j][Q[j][i]], one block per channel, four codes per thread.  Q 4-byte aligned.
__global__ void __launch_bounds__(256)
cb_apply_kernel(const float *codebook, const uint8_t *Q, int d_in, int m, float *What)
{
    __shared__ float cb[CB_MAX_LEVELS];
    griddep_launch();
    griddep_wait();
    const size_t j = blockIdx.x;
    if (threadIdx.x < m) cb[threadIdx.x] = codebook[j * m + threadIdx.x];
    __syncthreads();
    const uchar4 *src = reinterpret_cast<const uchar4 *>(Q + j * d_in);
    float4 *dst = reinterpret_cast<float4 *>(What + j * d_in);
    for (int c = threadIdx.x; c < d_in / 4; c += 256) {
        const uchar4 q = src[c];
        dst[c] = make_float4(cb[min(static_cast<int>(q.x), m - 1)], cb[min(static_cast<int>(q.y), m - 1)],
                             cb[min(static_cast<int>(q.z), m - 1)], cb[min(static_cast<int>(q.w), m - 1)]);
    }
}

}  // namespace gq
