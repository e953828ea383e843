// Surrogate network for screening local-search neighbours: training and
// inference kernels. BF16 weights, per-position features as BF16 hi + lo
// pairs (about 16 significant bits), FP32 activations and accumulation.
// The products of layers 1 and 2, forward and backward, run on the tensor
// cores (mlp_tc.cu, with the output layer and the loss in their epilogue); this
// file holds the rest: the output layer's gradient, the layer-2 bias gradient
// and Adam.
//
// Architecture (width H = 256):
//   per position k of a tour:  phi_k = (x, y, mu / Q, sd / Q, frac(cum_k / Q))
//                              (coordinates / 1000; cum_k = expected load of
//                               positions 1..k along the tour)
//   layer 1 (per position):    h_k = relu(W1 phi_k + b1)            H x 5
//   pooling:                   z = mean_k h_k
//   tour-length feature:       t = (c(0,s_1) + D[n] + c(s_n,0) - m) / sd, with (m, sd)
//                              set by the caller (default m = 0, sd = 500 n)
//   layer 2:                   u = relu(W2 [z; t] + b2)              H x (H+1)
//   layer 3:                   y = w3 . u + b3
// Parameters are one fp32 vector (layout in mlp.h); the kernels read bf16
// copies of the weight matrices. The backward pass recomputes layer 1 from the
// tour instead of storing an activation per position.
#include <cuda_bf16.h>
#include <stdint.h>

#include "mlp.h"
#include "tcgen05.h"

namespace cvrpsd {

// ---------------------------------------------------------------- layer 3 backward

// dU[b][j] = dy_b w3_j [u_bj > 0]; g_w3[j] += sum_b dy_b u_bj; g_b3 += sum_b
// dy_b; g_b2[j] += sum_b dU[b][j]. A block takes 16 rows, eight at a time in
// flight, and one atomic per column and sum (with two rows a block and the
// last sum in a kernel of its own: 7.4 + 6.8 us for 1024 rows).
constexpr int kOutRows = 16;

__global__ void __launch_bounds__(kMlpH) mlp_out_backward_kernel(const float *U, int B, const float *dy,
                                                                 const __nv_bfloat16 *w3, float *dU, float *gw3,
                                                                 float *gb3, float *gb2)
{
    const int j = threadIdx.x;                // kMlpH threads
    float acc = 0.0f, accb = 0.0f, accu = 0.0f;
    const float wj = __bfloat162float(w3[j]);
    const int b0 = blockIdx.x * kOutRows, b1 = min(B, b0 + kOutRows);
#pragma unroll 8
    for (int b = b0; b < b1; ++b) {
        const float u = U[(long long)b * kMlpH + j];
        const float d = dy[b];
        acc += d * u;
        accb += d;
        const float du = u > 0.0f ? d * wj : 0.0f;
        accu += du;
        dU[(long long)b * kMlpH + j] = du;
    }
    atomicAdd(gw3 + j, acc);
    atomicAdd(gb2 + j, accu);
    if (j == 0) atomicAdd(gb3, accb);
}

// ---------------------------------------------------------------- Adam

// The BF16 copies of parameter i: the flat one, and for W2 and b2 their place
// in the head's operand.
__device__ __forceinline__ void store_bf16(long long i, float v, __nv_bfloat16 *q, unsigned char *w2b)
{
    const __nv_bfloat16 b = __float2bfloat16_rn(v);
    q[i] = b;
    if (i < kOffW2 || i >= kOffW3) return;
    const int e = (int)(i - kOffW2), o = i < kOffB2 ? e / kMlpIn2 : (int)(i - kOffB2);
    const int k = i < kOffB2 ? e - o * kMlpIn2 : kMlpIn2;
    *reinterpret_cast<__nv_bfloat16 *>(w2b + (size_t)(o / kL2M) * kL2Tile + tc::kmajor_offset(o % kL2M, k, kL2Kc)) = b;
}

__global__ void adam_kernel(float *p, const float *g, float *m, float *v, long long P, float lr, float b1, float b2,
                            float eps, float c1, float c2, __nv_bfloat16 *q, unsigned char *w2b)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < P; i += (long long)gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.0f - b1) * gi;
        const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        const float pi = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
        p[i] = pi;
        store_bf16(i, pi, q, w2b);
    }
}

__global__ void to_bf16_kernel(const float *p, __nv_bfloat16 *q, unsigned char *w2b, long long P)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < P; i += (long long)gridDim.x * blockDim.x)
        store_bf16(i, p[i], q, w2b);
}

// ---------------------------------------------------------------- host launchers


cudaError_t mlp_forward(const MlpLayer1Args &l1, const MlpWeights &wt, float *U, float *y, const float *target,
                        float *dy, float *loss, cudaStream_t st)
{
    const int T = l1.T;
    cudaError_t e = mlp_layer1_tc(l1, l1.sm_count > 0 ? l1.sm_count : 1, st);
    if (e != cudaSuccess) return e;
    return mlp_head(MlpHeadArgs{l1.z_hi, l1.z_lo, wt.w2b, wt.w3, wt.b3, T, U, y, target, dy, loss, l1.err}, st);
}

cudaError_t mlp_backward(const MlpLayer1Args &l1, const MlpWeights &wt, const float *U, const float *dy, float *dU,
                         float *dzt, float *grad, cudaStream_t st)
{
    const int T = l1.T;
    float *gw1 = grad + kOffW1, *gb1 = grad + kOffB1, *gw2 = grad + kOffW2, *gb2 = grad + kOffB2;
    float *gw3 = grad + kOffW3, *gb3 = grad + kOffB3;
    mlp_out_backward_kernel<<<(unsigned)((T + kOutRows - 1) / kOutRows), kMlpH, 0, st>>>(U, T, dy, wt.w3, dU, gw3, gb3, gb2);
    cudaError_t e = mlp_grad_w2_tc(dU, l1.zt, T, gw2, l1.err, st);
    if (e != cudaSuccess) return e;
    e = mlp_grad_zt_tc(dU, T, wt.w2, dzt, l1.err, st);
    if (e != cudaSuccess) return e;
    MlpLayer1Args b = l1;
    b.dzt = dzt;
    b.gw1 = gw1;
    b.gb1 = gb1;
    e = mlp_layer1_bwd_tc(b, l1.sm_count > 0 ? l1.sm_count : 1, st);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

cudaError_t mlp_adam(float *p, const float *g, float *m, float *v, __nv_bfloat16 *pb, unsigned char *w2b, float lr,
                     int step, cudaStream_t st)
{
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    const float c1 = 1.0f - powf(b1, (float)step), c2 = 1.0f - powf(b2, (float)step);
    adam_kernel<<<266, 256, 0, st>>>(p, g, m, v, kMlpParams, lr, b1, b2, eps, c1, c2, pb, w2b);
    return cudaGetLastError();
}

cudaError_t mlp_to_bf16(const float *p, __nv_bfloat16 *pb, unsigned char *w2b, cudaStream_t st)
{
    to_bf16_kernel<<<266, 256, 0, st>>>(p, pb, w2b, kMlpParams);
    return cudaGetLastError();
}

}  // namespace cvrpsd
