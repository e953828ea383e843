// Internal interface of the surrogate network kernels (mlp.cu).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace cvrpsd {

constexpr int kMlpH = 256;                 // hidden width
constexpr int kMlpIn1 = 5;                 // per-position features
constexpr int kMlpIn2 = kMlpH + 1;         // pooled features + tour length

// Offsets into the flat parameter vector: W1 [H][5], b1 [H], W2 [H][H+1],
// b2 [H], w3 [H], b3 [1].
constexpr long long kOffW1 = 0;
constexpr long long kOffB1 = kOffW1 + (long long)kMlpH * kMlpIn1;
constexpr long long kOffW2 = kOffB1 + kMlpH;
constexpr long long kOffB2 = kOffW2 + (long long)kMlpH * kMlpIn2;
constexpr long long kOffW3 = kOffB2 + kMlpH;
constexpr long long kOffB3 = kOffW3 + kMlpH;
constexpr long long kMlpParams = kOffB3 + 1;

// Operands of the head (layer 2 on the tensor cores) in their shared-memory
// layout (tc::kmajor_offset): tiles of 128 rows x 272 BF16 columns, of which
// 257 are inputs, one is the bias and the rest are zero. Layer 1 writes the
// pooled inputs' hi and lo parts (a row per tour), the weight update W2' (two
// tiles of 128 units).
constexpr int kL2K = 272;                 // 257 inputs + 1 (bias) padded
constexpr int kL2Kc = kL2K / 8;           // 16-byte core-matrix columns per row group
constexpr int kL2M = 128;                 // rows of a tile
constexpr size_t kL2Tile = (size_t)kL2M * kL2K * 2;
inline size_t mlp_tile_bytes(long long T) { return (size_t)((T + kL2M - 1) / kL2M) * kL2Tile; }

struct MlpWeights {                        // bf16 views into one vector
    const __nv_bfloat16 *w1, *b1, *w2, *b2, *w3, *b3;
    const unsigned char *w2b;              // W2 and b2 as the head's operand
};

struct MlpLayer1Args {
    const int32_t *tours;                  // device [T][n]
    int T, n;
    const float *cust;                     // device [n][4]: x/1000, y/1000, mu/Q, sd/Q of customer k at k-1
    const int32_t *dist;                   // device (n+1)^2
    const __nv_bfloat16 *w1, *b1;
    float len_mean, len_inv_sd;            // tour-length feature t = (length - len_mean) * len_inv_sd
    float *zt;                             // device [T][H+1]: pooled features and tour length, or nullptr
    unsigned char *z_hi, *z_lo;            // device: the same as the head's operands (mlp_tile_bytes(T) each)
    const float *dzt;                      // backward: gradient of the pooled features, [T][H]
    float *gw1, *gb1;                      // backward: accumulated gradients
    float *loss;                           // forward: cleared for the head that follows, or nullptr
    unsigned int *err;                     // device word: set if a tensor-core wait gave up
    int sm_count;                          // SMs of the device (grid of the tensor-core kernel)
};

struct MlpHeadArgs {
    const unsigned char *z_hi, *z_lo;      // layer 1's output
    const unsigned char *w2b;              // W2' (two tiles)
    const __nv_bfloat16 *w3, *b3;
    int T;
    float *U;                              // device [T][H] or nullptr: layer 2's output
    float *y;                              // device [T]
    const float *target;                   // device [T] or nullptr
    float *dy, *loss;                      // with target: dy = 2 (y - target) / T; loss += mean squared error
    unsigned int *err;
};

// Layer 1 forward (features, W1, ReLU, mean pool; writes zt) on the tensor
// cores: tcgen05 MMAs with the accumulators in tensor memory (mlp_tc.cu).
cudaError_t mlp_layer1_tc(const MlpLayer1Args &l1, int sm_count, cudaStream_t st);
// Layer 1 backward (dW1, db1 from dzt) on the tensor cores (mlp_tc.cu).
cudaError_t mlp_layer1_bwd_tc(const MlpLayer1Args &l1, int sm_count, cudaStream_t st);
// Layers 2 and 3 and the loss, U = relu(zt W2^T + b2), y = w3 . U + b3
// (mlp_tc.cu).
cudaError_t mlp_head(const MlpHeadArgs &a, cudaStream_t st);

// Gradients of layers 2 and 3 from U and dy, and dZ for layer 1.
struct MlpGradArgs {
    const float *U, *dy;                       // T x 256 (rows 16-byte aligned), T
    const __nv_bfloat16 *w3, *w2;
    const float *zt;                           // T x 257: pooled features and tour length
    int T;
    float *dzt;                                // T x 256, written
    float *gw2, *gw3, *gb2, *gb3;              // added to
    unsigned int *err;
};
cudaError_t mlp_grad(const MlpGradArgs &g, cudaStream_t st);

cudaError_t mlp_forward(const MlpLayer1Args &l1, const MlpWeights &wt, float *U, float *y, const float *target,
                        float *dy, float *loss, cudaStream_t st);
cudaError_t mlp_backward(const MlpLayer1Args &l1, const MlpWeights &wt, const float *U, const float *dy, float *dzt,
                         float *grad, cudaStream_t st);
// Both write the BF16 copies: pb (flat) and W2' in w2b (whose padding the
// caller has zeroed once).
cudaError_t mlp_adam(float *p, const float *g, float *m, float *v, __nv_bfloat16 *pb, unsigned char *w2b, float lr,
                     int step, cudaStream_t st);
cudaError_t mlp_to_bf16(const float *p, __nv_bfloat16 *pb, unsigned char *w2b, cudaStream_t st);

}  // namespace cvrpsd
