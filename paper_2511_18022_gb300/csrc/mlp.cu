// Surrogate network for screening local-search neighbours: training and
// inference kernels. BF16 weights, per-position features as BF16 hi + lo
// pairs (about 16 significant bits), FP32 activations and accumulation.
// The layers run on the tensor cores, forward and backward (mlp_tc.cu); this
// file holds Adam, the BF16 copies and the order of the launches.
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

cudaError_t mlp_backward(const MlpLayer1Args &l1, const MlpWeights &wt, const float *U, const float *dy, float *dzt,
                         float *grad, cudaStream_t st)
{
    cudaError_t e = mlp_grad(MlpGradArgs{U, dy, wt.w3, wt.w2, l1.zt, l1.T, dzt, grad + kOffW2, grad + kOffW3,
                                         grad + kOffB2, grad + kOffB3, l1.err}, st);
    if (e != cudaSuccess) return e;
    MlpLayer1Args b = l1;
    b.dzt = dzt;
    b.gw1 = grad + kOffW1;
    b.gb1 = grad + kOffB1;
    return mlp_layer1_bwd_tc(b, l1.sm_count > 0 ? l1.sm_count : 1, st);
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
