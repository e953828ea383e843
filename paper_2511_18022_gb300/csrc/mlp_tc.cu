// The surrogate network's matrix products on the tensor cores (tcgen05,
// TMEM). Layer 1, forward:
//
// Per tour the layer is a small matrix product: the pre-activations of the
// H = 256 hidden units at the n positions are W1' (H x 16) times F' (16 x n),
// one MMA step of kind::f16 with BF16 operands. F' holds each of the five
// per-position features as two BF16 numbers, hi = bf16(v) in columns 0-4 and
// lo = bf16(v - hi) in columns 6-10, with a constant 1 in column 5; W1' holds
// W1 in columns 0-4 and again in 6-10, and the bias b1 in column 5. So the
// product keeps about 16 significant bits of the features against the exact
// BF16 weights, at no extra MMA: K = 16 has room. The accumulators land in tensor
// memory as FP32, hidden units on the 128 TMEM lanes and positions on the
// columns, so the mean-pooling over positions is a sum along each thread's
// own row: ReLU and sum in registers, no cross-thread reduction.
//
// One persistent CTA per SM holds two lines that take its tours in turn. A
// line's warps have roles, so that the features of later chunks, the MMAs of
// the next piece and the pooling of this one overlap:
//   - four producer warps, each a tour of its own at a time: per 32 positions
//     (one per lane) a warp gathers the features (a step ahead), forms the
//     cumulative expected load by a scan and writes F' into one of its four
//     stages of shared memory, 128 positions each;
//   - one thread issues the MMAs of a stage (hidden units 0-127 and 128-255)
//     into the line's half of tensor memory;
//   - eight pooling warps read it (tcgen05.ld 32x32b) and accumulate, position
//     after position.
// The stages are handed on by mbarriers, with waits that give up after a fixed
// number of polls (all roles then stop and an error is recorded). Operands lie in the canonical K-major layout without swizzle
// (8-row x 16-byte core matrices; 128 bytes between the two core matrices
// along K, 256 bytes between 8-row groups).
//
// What bounds it: the pooling's two operations per (unit, position), 210 M
// pairs for 4096 tours of n = 200 (10.8 us at one ALU-pipe maximum per two
// clocks; a tcgen05.ld takes about 175 clocks and an addition waits 4 for the
// one before, which four pooling warps on a scheduler hide). 81 us with one
// chunk at a time per CTA, each step behind the one before it. The producers'
// 1000 clocks a step are latency, so a producer's stages hold a tour or more;
// a stage's way through the waits of the three roles takes about 1250 clocks
// beside its pooling, so one stage of 128 positions per line (34 us) beats two
// of 64 (40 us).
#include <cuda_bf16.h>
#include <stdint.h>

#include "mlp.h"
#include "tcgen05.h"

namespace cvrpsd {

namespace {

constexpr int kTcThreads = 256;          // eight warps
constexpr int kTcK = 16;                 // one kind::f16 MMA step
constexpr uint32_t kTmemCols = 512;      // two 128 x 256 FP32 accumulators

constexpr int kF1Piece = 128;            // positions per stage
constexpr int kF1Lines = 2;
constexpr int kF1Pool = 8;               // pooling warps of a line: 0-7 and 8-15
constexpr int kF1Prod = 4;               // producer warps of a line: 16-19 and 20-23
// F' stages of a producer, and their size (backward: with FP32 features after
// the operand). 128 KB either way: one CTA per SM.
template <bool BWD> constexpr int f1_depth = BWD ? 2 : 4;
template <bool BWD> constexpr size_t f1_stage = kF1Piece * kTcK * 2 + (BWD ? kF1Piece * 32 : 0);
constexpr size_t kF1Smem = kF1Lines * kF1Prod * f1_depth<false> * f1_stage<false>;
static_assert(kF1Smem == kF1Lines * kF1Prod * f1_depth<true> * f1_stage<true>, "same stages' total");
constexpr int kF1Threads = 32 * kF1Lines * (kF1Pool + kF1Prod + 1);   // MMA warps 24 and 25

__device__ __forceinline__ uint32_t pack_bf16x2(__nv_bfloat16 a, __nv_bfloat16 b)
{
    return (uint32_t)__bfloat16_as_ushort(a) | ((uint32_t)__bfloat16_as_ushort(b) << 16);
}

// W1' = [W1 | b1 | W1 | 0] in shared memory: row h, columns 0..4 and 6..10
// weights, 5 bias, 11..15 zero.
__device__ __forceinline__ void stage_w1(const MlpLayer1Args &a, unsigned char *s_w1, int tid, int threads)
{
    for (int e = tid; e < kMlpH * kTcK; e += threads) {
        const int h = e / kTcK, k = e % kTcK;
        __nv_bfloat16 v = __float2bfloat16_rn(0.0f);
        if (k < kMlpIn1) v = a.w1[h * kMlpIn1 + k];
        else if (k == kMlpIn1) v = a.b1[h];
        else if (k < 2 * kMlpIn1 + 1) v = a.w1[h * kMlpIn1 + k - kMlpIn1 - 1];
        *reinterpret_cast<__nv_bfloat16 *>(s_w1 + tc::kmajor_offset(h, k, 2)) = v;
    }
}

// The 16 columns of F' for one position: feature pairs and the bias's 1.
__device__ __forceinline__ void feature_row(bool valid, const float4 &cu, float cum, __nv_bfloat16 (&f)[kTcK])
{
#pragma unroll
    for (int q = 0; q < kTcK; ++q) f[q] = __float2bfloat16_rn(0.0f);
    if (valid) {
        const float v[kMlpIn1] = {cu.x, cu.y, cu.z, cu.w, cum - floorf(cum)};
#pragma unroll
        for (int q = 0; q < kMlpIn1; ++q) {
            f[q] = __float2bfloat16_rn(v[q]);
            f[q + kMlpIn1 + 1] = __float2bfloat16_rn(v[q] - __bfloat162float(f[q]));
        }
        f[kMlpIn1] = __float2bfloat16_rn(1.0f);
    }
}

// Row j of F': two 16-byte halves (k 0..7 and 8..15).
__device__ __forceinline__ void store_feature_row(unsigned char *s_f, int j, const __nv_bfloat16 (&f)[kTcK])
{
#pragma unroll
    for (int half_k = 0; half_k < 2; ++half_k) {
        const __nv_bfloat16 *p = f + half_k * 8;
        *reinterpret_cast<uint4 *>(s_f + tc::kmajor_offset(j, half_k * 8, 2)) =
            make_uint4(pack_bf16x2(p[0], p[1]), pack_bf16x2(p[2], p[3]), pack_bf16x2(p[4], p[5]), pack_bf16x2(p[6], p[7]));
    }
}

// What a producer lane gathers for its position: loads a step ahead of the
// ids' use, two ahead of the values'.
struct FeatureItem {
    int c, nx;         // customer there and the next one, as the tour has them
    float4 cu;         // its features
    int edge, first;   // length of the edge to the next one (the depot after the last), from the depot
};

__device__ __forceinline__ void item_ids(const MlpLayer1Args &a, long long t, int k, FeatureItem &x)
{
    const int32_t *tour = a.tours + (t < a.T ? t : 0) * a.n;
    x.c = __ldg(tour + min(k, a.n - 1));
    x.nx = __ldg(tour + min(k + 1, a.n - 1));
}
__device__ __forceinline__ void item_gather(const MlpLayer1Args &a, int k, FeatureItem &x)
{
    const int c = min(max(x.c, 1), a.n), nx = k + 1 < a.n ? min(max(x.nx, 1), a.n) : 0;
    x.cu = __ldg(reinterpret_cast<const float4 *>(a.cust) + c - 1);
    x.edge = __ldg(a.dist + (long long)c * (a.n + 1) + nx);
    x.first = __ldg(a.dist + c);
}

// (a, b) += m * (x, y) as one packed operation.
__device__ __forceinline__ void fma2(unsigned long long &ab, unsigned long long m2, unsigned long long xy)
{
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(ab) : "l"(m2), "l"(xy));
}
__device__ __forceinline__ float2 unpack2(unsigned long long v)
{
    return make_float2(__uint_as_float((uint32_t)v), __uint_as_float((uint32_t)(v >> 32)));
}

// BWD: layer 1's backward pass in the same roles. With m_hk = [pre_hk > 0] the
// ReLU mask of hidden unit h at position k, the gradient of tour t is
//     dW1[h][:] += (dz_th / n) * sum_k m_hk F[k][:]    (F with the bias's 1)
// so the pooling warps recompute the pre-activations as the forward pass does
// (no per-position activations are stored) and add the feature rows where the
// mask is set: a broadcast of the row from shared memory and three packed FP32
// multiply-adds per (unit, position). Each thread scales its unit's six sums by
// dz_th / n after a tour; the sums reach the gradient once per CTA.
template <bool BWD>
__global__ void __launch_bounds__(kF1Threads, 1) mlp_layer1_tc_kernel(MlpLayer1Args a)
{
    constexpr int kF1Depth = f1_depth<BWD>;
    constexpr size_t kF1StageBytes = f1_stage<BWD>, kF1Rows = kF1Piece * kTcK * 2;   // FP32 rows' offset in a stage
    __shared__ __align__(128) unsigned char s_w1[kMlpH * kTcK * 2];                    // W1' (H x 16), 8 KB
    __shared__ __align__(8) unsigned long long s_full[kF1Lines][kF1Prod][kF1Depth], s_empty[kF1Lines][kF1Prod][kF1Depth];
    __shared__ __align__(8) unsigned long long s_tfull[kF1Lines], s_tempty[kF1Lines];        // TMEM halves
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort;
    __shared__ float s_gw[BWD ? kMlpIn1 + 1 : 1][kMlpH];
    extern __shared__ __align__(128) unsigned char s_f[];   // F' (128 x 16), 4 KB each: [line][producer][stage]

    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int n = a.n;
    auto bar = [](unsigned long long &b) { return (uint32_t)__cvta_generic_to_shared(&b); };

    stage_w1(a, s_w1, tid, kF1Threads);
    if (tid == 0) {
        if (!BWD && a.loss && blockIdx.x == 0) *a.loss = 0.0f;
        for (int l = 0; l < kF1Lines; ++l) {
            for (int p = 0; p < kF1Prod; ++p)
                for (int k = 0; k < kF1Depth; ++k) {
                    tc::mbar_init_count(bar(s_full[l][p][k]), 1);
                    tc::mbar_init_count(bar(s_empty[l][p][k]), BWD ? 1 + kF1Pool : 1);
                }
            tc::mbar_init_count(bar(s_tfull[l]), 1);
            tc::mbar_init_count(bar(s_tempty[l]), kF1Pool);
        }
        tc::mbar_init_fence();
        s_abort = 0;
    }
    if (w == 0) tc::tmem_alloc((uint32_t)__cvta_generic_to_shared(&s_tmem), kTmemCols);
    tc::fence_operands();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = s_tmem;

    // A line's tours: blockIdx.x + line * gridDim.x, and on by twice the grid.
    const long long step = (long long)kF1Lines * gridDim.x;
    if (w < kF1Lines * kF1Pool) {
        // pooling: this warp's TMEM rows are lanes 32 (w % 4) .. +31 of one of the line's two accumulators
        const int line = w >> 3, half = (w >> 2) & 1, h = half * 128 + 32 * (w & 3) + lane;
        const uint32_t row = tmem + ((uint32_t)(32 * (w & 3)) << 16) + (uint32_t)(line * 256 + half * kF1Piece);
        int q = 0;                                           // stage number within the line
        int p = 0;                                           // producer of this tour, and its next stage in bits 4 p ..
        uint32_t slot = 0;
        float gw[kMlpIn1 + 1] = {0, 0, 0, 0, 0, 0};
        for (long long t = blockIdx.x + (long long)line * gridDim.x; t < a.T; t += step, p = (p + 1) % kF1Prod) {
            float acc = 0.0f;
            unsigned long long s01 = 0, s23 = 0, s45 = 0;
            bool ok = true;
            for (int p0 = 0; p0 < n; p0 += kF1Piece, ++q) {
                ok = __all_sync(0xffffffffu, tc::mbar_wait_role(bar(s_tfull[line]), (uint32_t)q & 1u, &s_abort, a.err));
                if (!ok) break;
                tc::fence_after_sync();
                // columns past n hold 0 up to the next multiple of 32
                const int cols = (min(kF1Piece, n - p0) + 31) / 32 * 32;
                for (int col = 0; col < cols; col += 32) {
                    uint32_t r[32];
                    tc::tmem_ld32_issue(row + (uint32_t)col, r);
                    tc::tmem_ld_wait(r);
                    if (col + 32 >= cols) {                  // all of the stage is in registers
                        tc::fence_before_sync();
                        __syncwarp();
                        if (lane == 0) tc::mbar_arrive(bar(s_tempty[line]));
                    }
                    if (BWD) {
                        const uint32_t f_s = (uint32_t)((slot >> (4 * p)) & (kF1Depth - 1));
                        const ulonglong2 *f = reinterpret_cast<const ulonglong2 *>(
                            s_f + ((line * kF1Prod + p) * kF1Depth + f_s) * kF1StageBytes + kF1Rows) + 2 * col;
#pragma unroll
                        for (int k = 0; k < 32; ++k) {
                            const ulonglong2 f03 = f[2 * k];
                            const unsigned long long f45 = f[2 * k + 1].x;
                            const uint32_t m = __uint_as_float(r[k]) > 0.0f ? 0x3f800000u : 0u;
                            const unsigned long long m2 = ((unsigned long long)m << 32) | m;
                            fma2(s01, m2, f03.x);
                            fma2(s23, m2, f03.y);
                            fma2(s45, m2, f45);
                        }
                    } else {
#pragma unroll
                        for (int k = 0; k < 32; ++k) acc += fmaxf(__uint_as_float(r[k]), 0.0f);
                    }
                }
                if (BWD) {                                   // the stage's feature rows are read
                    __syncwarp();
                    if (lane == 0) tc::mbar_arrive(bar(s_empty[line][p][(slot >> (4 * p)) & (kF1Depth - 1)]));
                    slot = (slot + (1u << (4 * p))) & (0x1111u * (kF1Depth - 1));
                }
            }
            if (!ok) break;
            if (BWD) {
                const float g = a.dzt[t * kMlpH + h] / (float)n;
                const float2 u01 = unpack2(s01), u23 = unpack2(s23), u45 = unpack2(s45);
                gw[0] += g * u01.x;
                gw[1] += g * u01.y;
                gw[2] += g * u23.x;
                gw[3] += g * u23.y;
                gw[4] += g * u45.x;
                gw[5] += g * u45.y;
                continue;
            }
            const float z = acc / (float)n;
            if (a.zt) a.zt[t * kMlpIn2 + h] = z;
            const size_t off = (size_t)(t / kL2M) * kL2Tile + tc::kmajor_offset((int)(t % kL2M), h, kL2Kc);
            const __nv_bfloat16 hi = __float2bfloat16_rn(z);
            *reinterpret_cast<__nv_bfloat16 *>(a.z_hi + off) = hi;
            *reinterpret_cast<__nv_bfloat16 *>(a.z_lo + off) = __float2bfloat16_rn(z - __bfloat162float(hi));
        }
        if (BWD) {
            // the lines' sums together, once to the gradient
            if (line == 1) {
#pragma unroll
                for (int k = 0; k < kMlpIn1 + 1; ++k) s_gw[k][h] = gw[k];
            }
            asm volatile("barrier.cta.sync 1, %0;" ::"n"(32 * kF1Lines * kF1Pool) : "memory");
            if (line == 0) {
#pragma unroll
                for (int k = 0; k < kMlpIn1; ++k) atomicAdd(a.gw1 + h * kMlpIn1 + k, gw[k] + s_gw[k][h]);
                atomicAdd(a.gb1 + h, gw[kMlpIn1] + s_gw[kMlpIn1][h]);
            }
        }
    } else if (w < kF1Lines * (kF1Pool + kF1Prod)) {
        // producer p takes the line's tours p, p + 4, ...
        const int pw = w - kF1Lines * kF1Pool, line = pw / kF1Prod, p = pw % kF1Prod;
        const long long stride = step * kF1Prod;
        unsigned char *stages = s_f + pw * kF1Depth * kF1StageBytes;
        long long t = blockIdx.x + (long long)line * gridDim.x + p * step;
        long long t1 = t;                                    // (t1, k1): the step after this one
        int k1 = lane;
        auto next = [&](long long &tt, int &kk) {
            kk += 32;
            if (kk - lane >= n) {
                kk = lane;
                tt += stride;
            }
        };
        FeatureItem x, y;                                    // this step's, the next one's
        item_ids(a, t, lane, x);
        item_gather(a, lane, x);
        next(t1, k1);
        item_ids(a, t1, k1, y);
        int q = 0;                                           // stage number of this warp
        bool ok = true;
        for (; t < a.T && ok; t += stride) {
            float carry = 0.0f, len = 0.0f;
            for (int k0 = 0; k0 < n; k0 += 32) {
                const int k = k0 + lane;
                FeatureItem z;
                long long t2 = t1;
                int k2 = k1;
                next(t2, k2);
                item_ids(a, t2, k2, z);
                item_gather(a, k1, y);
                const bool valid = k < n;
                float v = valid ? x.cu.z : 0.0f;
                if (valid) len += (float)x.edge;
                if (k == 0) len += (float)x.first;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const float u = __shfl_up_sync(0xffffffffu, v, o);
                    if (lane >= o) v += u;
                }
                const float cum = carry + v;
                carry = __shfl_sync(0xffffffffu, cum, 31);
                __nv_bfloat16 f[kTcK];
                feature_row(valid, x.cu, cum, f);
                const int s = q % kF1Depth, in = k0 % kF1Piece;
                if (in == 0)
                    ok = __all_sync(0xffffffffu, tc::mbar_wait_role(bar(s_empty[line][p][s]), ((uint32_t)(q / kF1Depth) & 1u) ^ 1u,
                                                                    &s_abort, a.err));
                if (!ok) break;
                store_feature_row(stages + s * kF1StageBytes, in + lane, f);
                if (BWD) {                                   // the pairs' values, as the forward operand has them
                    float v6[8] = {0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll
                    for (int o = 0; o < kMlpIn1; ++o) v6[o] = __bfloat162float(f[o]) + __bfloat162float(f[o + kMlpIn1 + 1]);
                    v6[kMlpIn1] = __bfloat162float(f[kMlpIn1]);
                    float4 *rows = reinterpret_cast<float4 *>(stages + s * kF1StageBytes + kF1Rows) + 2 * (in + lane);
                    rows[0] = make_float4(v6[0], v6[1], v6[2], v6[3]);
                    rows[1] = make_float4(v6[4], v6[5], 0.0f, 0.0f);
                }
                if (in + 32 == kF1Piece || k0 + 32 >= n) {
                    tc::fence_operands();
                    __syncwarp();
                    if (lane == 0) tc::mbar_arrive(bar(s_full[line][p][s]));
                    ++q;
                }
                x = y;
                y = z;
                t1 = t2;
                k1 = k2;
            }
            if (!ok) break;
            if constexpr (!BWD) {
                // tour length: sum over the warp; the rest of row t of the head's operand
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) len += __shfl_xor_sync(0xffffffffu, len, o);
                if (lane == 0) {
                    const float u = (len - a.len_mean) * a.len_inv_sd;
                    if (a.zt) a.zt[t * kMlpIn2 + kMlpH] = u;
                    const size_t off = (size_t)(t / kL2M) * kL2Tile + tc::kmajor_offset((int)(t % kL2M), kMlpH, kL2Kc);
                    const __nv_bfloat16 hi = __float2bfloat16_rn(u), one = __float2bfloat16_rn(1.0f);
                    const __nv_bfloat16 lo = __float2bfloat16_rn(u - __bfloat162float(hi)), none = __float2bfloat16_rn(0.0f);
                    *reinterpret_cast<uint4 *>(a.z_hi + off) = make_uint4(pack_bf16x2(hi, one), 0u, 0u, 0u);
                    *reinterpret_cast<uint4 *>(a.z_hi + off + 128) = make_uint4(0u, 0u, 0u, 0u);
                    *reinterpret_cast<uint4 *>(a.z_lo + off) = make_uint4(pack_bf16x2(lo, none), 0u, 0u, 0u);
                    *reinterpret_cast<uint4 *>(a.z_lo + off + 128) = make_uint4(0u, 0u, 0u, 0u);
                }
            }
        }
    } else {
        if (lane == 0) {
            // Everything that does not change with the piece is formed before the
            // loop: this thread's chain of waits and issues is on every piece's way.
            const int line = w - kF1Lines * (kF1Pool + kF1Prod);
            const uint32_t w1_s = (uint32_t)__cvta_generic_to_shared(s_w1);
            const uint64_t a_desc0 = tc::smem_desc(w1_s, 128, 256);
            const uint64_t a_desc1 = tc::smem_desc(w1_s + 16 * 256, 128, 256);   // hidden units 128..255
            const uint64_t b_desc0 = tc::smem_desc((uint32_t)__cvta_generic_to_shared(s_f + line * (kF1Smem / kF1Lines)), 128, 256);
            constexpr uint64_t kStageDesc = kF1StageBytes >> 4;                   // between stages, in the descriptor
            static_assert(kF1Prod * kF1Depth <= 32 && kF1Depth <= 8, "a phase bit per stage, four bits per producer's next stage");
            const uint32_t full = bar(s_full[line][0][0]), empty = bar(s_empty[line][0][0]);
            const uint32_t tfull = bar(s_tfull[line]), tempty = bar(s_tempty[line]);
            const uint32_t acc = tmem + (uint32_t)(line * 256);
            const uint32_t idesc = tc::instr_desc(kF1Piece), idesc_last = tc::instr_desc((uint32_t)(((n - 1) % kF1Piece) / 32 * 32 + 32));
            uint32_t phase = 0, slot = 0;                    // full[p][s]'s parity in bit kF1Depth p + s; producer p's s in bits 4 p ..
            uint32_t tphase = 1;
            int p = 0;
            bool ok = true;
            for (long long t = blockIdx.x + (long long)line * gridDim.x; t < a.T && ok; t += step, p = (p + 1) % kF1Prod) {
                for (int left = n; left > 0; left -= kF1Piece) {
                    const uint32_t x = kF1Depth * p + ((slot >> (4 * p)) & (kF1Depth - 1));
                    ok = tc::mbar_wait_role(full + 8u * x, (phase >> x) & 1u, &s_abort, a.err) &&
                         tc::mbar_wait_role(tempty, tphase, &s_abort, a.err);
                    if (!ok) break;
                    tc::fence_after_sync();
                    const uint64_t bd = b_desc0 + kStageDesc * x;
                    const uint32_t id = left > kF1Piece ? idesc : idesc_last;
                    tc::mma_bf16(acc, a_desc0, bd, id, false);
                    tc::mma_bf16(acc + kF1Piece, a_desc1, bd, id, false);
                    tc::mma_commit(tfull);
                    tc::mma_commit(empty + 8u * x);
                    phase ^= 1u << x;
                    slot = (slot + (1u << (4 * p))) & (0x1111u * (kF1Depth - 1));
                    tphase ^= 1u;
                }
            }
        }
        __syncwarp();
    }
    tc::fence_before_sync();
    __syncthreads();
    if (w == 0) tc::tmem_dealloc(tmem, kTmemCols);
}

// ---------------------------------------------------------------- the head
//
// Layer 2, layer 3 and the loss for a tile of 128 tours:
// U = relu([z; t] W2^T + b2), y = w3 . U + b3. M = 128 tours, N = 256 hidden
// units in two halves, K = 257 inputs + 1 (the bias rides in W2' as column 257
// against a constant 1) padded to 272 = 17 MMA steps. The pooled inputs are
// FP32, split by layer 1 into BF16 hi + lo parts (hi = bf16(v), lo =
// bf16(v - hi)); both products are accumulated, so the result keeps about 16
// significant bits of the inputs against the exact BF16 weights: the FP32
// layer's accuracy on the tensor cores. Layer 1 writes its parts, and the
// weight update W2', in the operands' own layout, so a CTA fetches them with
// three bulk copies (the second half of W2' with a fourth, once the first
// half's MMAs have read its room); a thread owns a tour's row of the
// accumulator, so the output is a sum in registers.
//
// What bounds it: copying 272 KB into a CTA, then latency (one CTA per 128
// tours: 32 for 4096). Before, with FP32 inputs converted element by element
// and the output layer apart: 20.6 + 7.1 us for 4096 tours.
constexpr size_t kHeadSmem = 3 * kL2Tile;          // A hi, A lo, half of W2'
constexpr uint32_t kHeadTmemCols = 256;

__global__ void __launch_bounds__(kTcThreads, 1) mlp_head_kernel(MlpHeadArgs a)
{
    extern __shared__ __align__(128) unsigned char smem[];   // A hi | A lo | B
    __shared__ __align__(8) unsigned long long s_load[2], s_mma[2];
    __shared__ uint32_t s_tmem;
    __shared__ float s_w3[kMlpH];
    const int j = threadIdx.x, lane = j & 31, w = j >> 5;
    const long long tile = blockIdx.x;
    auto bar = [](unsigned long long &b) { return (uint32_t)__cvta_generic_to_shared(&b); };
    const uint32_t sa = (uint32_t)__cvta_generic_to_shared(smem);
    const uint32_t sb = sa + 2 * (uint32_t)kL2Tile;
    if (j == 0) {
        for (int k = 0; k < 2; ++k) {
            tc::mbar_init_count(bar(s_load[k]), 1);
            tc::mbar_init_count(bar(s_mma[k]), 1);
        }
        tc::mbar_init_fence();
        tc::mbar_expect(bar(s_load[0]), 3 * (uint32_t)kL2Tile);
        tc::bulk_load(sa, a.z_hi + tile * kL2Tile, (uint32_t)kL2Tile, bar(s_load[0]));
        tc::bulk_load(sa + (uint32_t)kL2Tile, a.z_lo + tile * kL2Tile, (uint32_t)kL2Tile, bar(s_load[0]));
        tc::bulk_load(sb, a.w2b, (uint32_t)kL2Tile, bar(s_load[0]));
    }
    s_w3[j] = __bfloat162float(a.w3[j]);
    if (w == 0) tc::tmem_alloc((uint32_t)__cvta_generic_to_shared(&s_tmem), kHeadTmemCols);
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = s_tmem;
    if (j == 0) {
        bool ok = true;
        for (int half = 0; half < 2 && ok; ++half) {
            if (half == 1) {
                // the first half's MMAs have read its weights
                ok = tc::mbar_wait(bar(s_mma[0]), 0);
                if (!ok) break;
                tc::mbar_expect(bar(s_load[1]), (uint32_t)kL2Tile);
                tc::bulk_load(sb, a.w2b + kL2Tile, (uint32_t)kL2Tile, bar(s_load[1]));
            }
            // (a copy under way is waited for in any case)
            ok = tc::mbar_wait(bar(s_load[half]), 0);
            if (!ok) break;
            tc::fence_after_sync();
            const uint32_t idesc = tc::instr_desc(128), sbo = kL2Kc * 128;
            for (int step = 0; step < kL2K / 16; ++step) {
                const uint32_t koff = (uint32_t)step * 256;     // two 16-byte core-matrix columns per step
                const uint64_t bd = tc::smem_desc(sb + koff, 128, sbo);
                tc::mma_bf16(tmem + half * 128, tc::smem_desc(sa + koff, 128, sbo), bd, idesc, step > 0);
                tc::mma_bf16(tmem + half * 128, tc::smem_desc(sa + (uint32_t)kL2Tile + koff, 128, sbo), bd, idesc, true);
            }
            tc::mma_commit(bar(s_mma[half]));
        }
        if (!ok) atomicOr(a.err, 1u);
    }
    __syncwarp();
    // warps 0-3 take the first half's units, 4-7 the second's; lane = tour
    const int half = w >> 2, row = 32 * (w & 3) + lane;
    const long long t = tile * kL2M + row;
    const bool ok = __all_sync(0xffffffffu, tc::mbar_wait(bar(s_mma[half]), 0));
    tc::fence_after_sync();
    // w3 . u as 32 sums of every 32nd product, then their sum by halves: the
    // second half's threads go on from the first half's sums (through shared
    // memory, over the operands that both halves' MMAs have read).
    float *s_sum = reinterpret_cast<float *>(smem);          // [32][128]
    float d[32];
    auto products = [&]() {
        const uint32_t at = tmem + ((uint32_t)(32 * (w & 3)) << 16) + (uint32_t)(half * 128);
#pragma unroll 1
        for (int c = 0; c < 128; c += 32) {
            float r[32];
            tc::tmem_ld32(at + c, r);
#pragma unroll
            for (int k = 0; k < 32; ++k) r[k] = fmaxf(r[k], 0.0f);
            const float *w3 = s_w3 + half * 128 + c;
#pragma unroll
            for (int k = 0; k < 32; ++k) d[k] = fmaf(r[k], w3[k], d[k]);
            if (a.U && t < a.T) {
                float *out = a.U + t * kMlpH + half * 128 + c;
#pragma unroll
                for (int k = 0; k < 32; k += 4)
                    *reinterpret_cast<float4 *>(out + k) = make_float4(r[k], r[k + 1], r[k + 2], r[k + 3]);
            }
        }
    };
#pragma unroll
    for (int k = 0; k < 32; ++k) d[k] = 0.0f;
    if (ok && half == 0) products();
    const bool all_ok = __syncthreads_and(ok);               // both halves' MMAs are done
    if (all_ok && half == 0) {
#pragma unroll
        for (int k = 0; k < 32; ++k) s_sum[k * kL2M + row] = d[k];
    }
    __syncthreads();
    if (all_ok && half == 1) {
#pragma unroll
        for (int k = 0; k < 32; ++k) d[k] = s_sum[k * kL2M + row];
        products();
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int k = 0; k < o; ++k) d[k] += d[k + o];
        float loss = 0.0f;
        if (t < a.T) {
            const float y = d[0] + __bfloat162float(a.b3[0]);
            a.y[t] = y;
            if (a.target) {
                const float e = y - a.target[t];
                a.dy[t] = 2.0f * e / (float)a.T;
                loss = e * e / (float)a.T;
            }
        }
        if (a.target) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, o);
            if (lane == 0) atomicAdd(a.loss, loss);
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    if (w == 0) tc::tmem_dealloc(tmem, kHeadTmemCols);
}

// ---------------------------------------------------------------- gradients behind layer 1
//
// With dU[b][j] = dy_b w3_j [u_bj > 0], formed from U where it is staged:
//   dZ (T x 256) = dU (T x 256) W2[:, 0..255]   (the tour length has no
//                                                gradient to pass on)
//   gW2 (256 x 257) += dU^T (256 x T) ZT (T x 257), in slabs of 128 tours
//   gw3_j += sum_b dy_b u_bj, gb2_j += sum_b dU[b][j], gb3 += sum_b dy_b
// in one launch, whose first blocks take 128 x 64 tiles of dZ and the others 128 x
// 80 tiles of gW2; those of the first columns also add up the three sums, over the
// slab that they stage anyway. FP32 operands are split into BF16 hi and lo parts
// (hi = bf16(v), lo = bf16(v - hi)); a product of two split operands takes
// hi*hi + hi*lo + lo*hi (the lo*lo term, at most 2^-18 of the product, is the
// order of the pair's own rounding and is left out), one with an exact BF16
// operand hi*B + lo*B.
//
// What bounds it: latency. A tile's chain is two rounds of loads per operand and
// chunk of K = 128, the MMAs, their commit and the epilogue, and there are
// fewer tiles than SMs at the usual 1024 tours; so a thread has 32 words and
// more in flight, and the accumulators go through shared memory to full rows.
// 13.3 us for 1024 tours; as an elementwise kernel and two products, one after
// the other: 10.9 + 17.3 + 23.2. 80 columns, not 96: two blocks fit an SM.
constexpr int kGM = 128;                       // rows of a tile
constexpr int kGNz = 64, kGNw = 80;            // its columns: dZ, gW2
constexpr int kGK = 128;                       // K per staged chunk
constexpr int kGKc = kGK / 8;                  // 16-byte core-matrix columns per row group
constexpr size_t kGA = (size_t)kGM * kGK * 2;  // one BF16 A part
constexpr size_t kGB = (size_t)kGNw * kGK * 2; // one BF16 B part
constexpr size_t kGSmem = 2 * kGA + 2 * kGB;   // A hi, A lo, B hi, B lo; then the tile of C
static_assert((size_t)kGM * (kGNw + 1) * 4 <= kGSmem, "the tile of C takes the operands' place");
constexpr uint32_t kGTmemCols = 128;
constexpr int kGwTiles = (kMlpIn2 + kGNw - 1) / kGNw;
static_assert(kMlpH == 2 * kGM && kMlpH == kTcThreads && kMlpH % kGNz == 0, "tiles of the two products");

// Eight values along K as BF16 hi and lo parts.
__device__ __forceinline__ void split8(const float (&v)[8], uint4 &hi, uint4 &lo)
{
    uint32_t h[4], l[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const __nv_bfloat16 h0 = __float2bfloat16_rn(v[2 * q]), h1 = __float2bfloat16_rn(v[2 * q + 1]);
        h[q] = pack_bf16x2(h0, h1);
        l[q] = pack_bf16x2(__float2bfloat16_rn(v[2 * q] - __bfloat162float(h0)),
                           __float2bfloat16_rn(v[2 * q + 1] - __bfloat162float(h1)));
    }
    hi = make_uint4(h[0], h[1], h[2], h[3]);
    lo = make_uint4(l[0], l[1], l[2], l[3]);
}

__device__ __forceinline__ float relu_grad(float u, float d, float w) { return u > 0.0f ? d * w : 0.0f; }

// dZ: rows m0.. of A, all K in two chunks. s_d holds dy of the tile's rows.
__device__ __forceinline__ void stage_dz(const MlpGradArgs &g, unsigned char *smem, const float *s_d, const float *s_w3,
                                         int m0, int n0, int kc0)
{
    unsigned char *a_hi = smem, *a_lo = smem + kGA, *b_hi = smem + 2 * kGA;
    const int j = threadIdx.x, lane = j & 31, w = j >> 5;
    // an eighth of a warp reads a whole line of a row, and eight rows make a core matrix
#pragma unroll
    for (int half = 0; half < 2; ++half) {
        float4 x[4][2];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int it = w * 8 + half * 4 + i, m = m0 + (it >> 2) * 8 + (lane & 7), gk = (it & 3) * 4 + (lane >> 3);
            const float4 *src = reinterpret_cast<const float4 *>(g.U + (long long)m * kMlpH + kc0 + 8 * gk);
            const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
            x[i][0] = m < g.T ? __ldg(src) : zero;
            x[i][1] = m < g.T ? __ldg(src + 1) : zero;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int it = w * 8 + half * 4 + i, r = (it >> 2) * 8 + (lane & 7), gk = (it & 3) * 4 + (lane >> 3);
            const float d = s_d[r], *w3 = s_w3 + kc0 + 8 * gk;
            const float u[8] = {x[i][0].x, x[i][0].y, x[i][0].z, x[i][0].w, x[i][1].x, x[i][1].y, x[i][1].z, x[i][1].w};
            float v[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = relu_grad(u[q], d, w3[q]);
            uint4 hi, lo;
            split8(v, hi, lo);
            const uint32_t off = tc::kmajor_offset(r, 8 * gk, kGKc);
            *reinterpret_cast<uint4 *>(a_hi + off) = hi;
            *reinterpret_cast<uint4 *>(a_lo + off) = lo;
        }
    }
    // B(n, k) = W2[k][n0 + n], neighbouring threads on neighbouring columns
    const int r = j % kGNz;
    unsigned short b[4][8];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int q = 0; q < 8; ++q)
            b[i][q] = __ldg(reinterpret_cast<const unsigned short *>(g.w2) +
                            (kc0 + 8 * (j / kGNz + 4 * i) + q) * kMlpIn2 + n0 + r);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        uint32_t p[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) p[q] = (uint32_t)b[i][2 * q] | (uint32_t)b[i][2 * q + 1] << 16;
        *reinterpret_cast<uint4 *>(b_hi + tc::kmajor_offset(r, 8 * (j / kGNz + 4 * i), kGKc)) =
            make_uint4(p[0], p[1], p[2], p[3]);
    }
}

// gW2: hidden units m0.. over the slab of tours from kc0. s_d holds the slab's dy (0 past T).
__device__ __forceinline__ void stage_gw2(const MlpGradArgs &g, unsigned char *smem, const float *s_d, const float *s_w3,
                                          int m0, int n0, int kc0)
{
    unsigned char *a_hi = smem, *a_lo = smem + kGA, *b_hi = smem + 2 * kGA, *b_lo = smem + 2 * kGA + kGB;
    const int j = threadIdx.x, r = j % kGM;
    const float w3 = s_w3[m0 + r];
    float sum = 0.0f, sumu = 0.0f;
#pragma unroll
    for (int half = 0; half < 2; ++half) {
        float x[4][8];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int b = kc0 + 8 * (j / kGM + 2 * (half * 4 + i)) + q;
                x[i][q] = b < g.T ? __ldg(g.U + (long long)b * kMlpH + m0 + r) : 0.0f;
            }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int gk = j / kGM + 2 * (half * 4 + i);
            float v[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const float d = s_d[8 * gk + q];
                v[q] = relu_grad(x[i][q], d, w3);
                sum += d * x[i][q];
                sumu += v[q];
            }
            uint4 hi, lo;
            split8(v, hi, lo);
            const uint32_t off = tc::kmajor_offset(r, 8 * gk, kGKc);
            *reinterpret_cast<uint4 *>(a_hi + off) = hi;
            *reinterpret_cast<uint4 *>(a_lo + off) = lo;
        }
    }
    if (n0 == 0) {
        atomicAdd(g.gw3 + m0 + r, sum);
        atomicAdd(g.gb2 + m0 + r, sumu);
        if (m0 == 0 && j < 32) {
            float d = (s_d[j] + s_d[j + 32]) + (s_d[j + 64] + s_d[j + 96]);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
            if (j == 0) atomicAdd(g.gb3, d);
        }
    }
    float x[5][8];
#pragma unroll
    for (int i = 0; i < 5; ++i)
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int e = j + i * kTcThreads, n = n0 + e % kGNw, b = kc0 + 8 * (e / kGNw) + q;
            x[i][q] = n < kMlpIn2 && b < g.T ? __ldg(g.zt + (long long)b * kMlpIn2 + n) : 0.0f;
        }
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        const int e = j + i * kTcThreads;
        uint4 hi, lo;
        split8(x[i], hi, lo);
        const uint32_t off = tc::kmajor_offset(e % kGNw, 8 * (e / kGNw), kGKc);
        *reinterpret_cast<uint4 *>(b_hi + off) = hi;
        *reinterpret_cast<uint4 *>(b_lo + off) = lo;
    }
}
static_assert(kGNw * kGKc == 5 * kTcThreads && kGNz * kGKc == 4 * kTcThreads && kGM * kGKc == 8 * kTcThreads,
              "items per thread of the staging loops");

template <bool DZ>
__device__ __forceinline__ void grad_tile(const MlpGradArgs &g, unsigned char *smem, uint32_t tmem, uint32_t mbar,
                                          float *s_d, const float *s_w3, int m0, int n0, int b0)
{
    constexpr int N = DZ ? kGNz : kGNw, kChunks = DZ ? kMlpH / kGK : 1;
    const int j = threadIdx.x, lane = j & 31, w = j >> 5;
    if (j < kGM) s_d[j] = b0 + j < g.T ? __ldg(g.dy + b0 + j) : 0.0f;
    __syncthreads();
    bool ok = true;
#pragma unroll 1
    for (int c = 0; c < kChunks && ok; ++c) {
        if (DZ) stage_dz(g, smem, s_d, s_w3, m0, n0, c * kGK);
        else stage_gw2(g, smem, s_d, s_w3, m0, n0, b0);
        tc::fence_operands();
        tc::fence_before_sync();
        __syncthreads();
        tc::fence_after_sync();
        if (j == 0) {
            const uint32_t idesc = tc::instr_desc(N), sbo = kGKc * 128;
            const uint32_t ah = (uint32_t)__cvta_generic_to_shared(smem), al = ah + kGA, bh = al + kGA, bl = bh + kGB;
            for (int step = 0; step < kGK / 16; ++step) {
                const uint32_t ko = (uint32_t)step * 256;
                const uint64_t dah = tc::smem_desc(ah + ko, 128, sbo), dal = tc::smem_desc(al + ko, 128, sbo);
                const uint64_t dbh = tc::smem_desc(bh + ko, 128, sbo);
                tc::mma_bf16(tmem, dah, dbh, idesc, c > 0 || step > 0);
                tc::mma_bf16(tmem, dal, dbh, idesc, true);
                if (!DZ) tc::mma_bf16(tmem, dah, tc::smem_desc(bl + ko, 128, sbo), idesc, true);
            }
            tc::mma_commit(mbar);
        }
        // the operands are overwritten next (by the next chunk, then by the tile): wait for the MMAs
        ok = tc::mbar_wait(mbar, (uint32_t)c & 1u);
        if (!ok && lane == 0) atomicOr(g.err, 1u);
        tc::fence_after_sync();
        ok = __syncthreads_and(ok);
    }
    float *tile = reinterpret_cast<float *>(smem);
    if (ok && w < 4) {
#pragma unroll
        for (int c = 0; c < N; c += 32) {                     // the last load may run past N, within the allocation
            float r[32];
            tc::tmem_ld32(tmem + ((uint32_t)(32 * w) << 16) + c, r);
#pragma unroll
            for (int q = 0; q < 32; ++q)
                if (c + q < N) tile[(32 * w + lane) * (N + 1) + c + q] = r[q];
        }
    }
    __syncthreads();
    if (!ok) return;
#pragma unroll 4
    for (int e = j; e < kGM * N; e += kTcThreads) {
        const int r = e / N, c = e % N;
        const float v = tile[r * (N + 1) + c];
        if (DZ) {
            if (m0 + r < g.T) g.dzt[(long long)(m0 + r) * kMlpH + n0 + c] = v;
        } else if (n0 + c < kMlpIn2) {
            atomicAdd(g.gw2 + (long long)(m0 + r) * kMlpIn2 + n0 + c, v);
        }
    }
}

__global__ void __launch_bounds__(kTcThreads, 2) mlp_grad_kernel(MlpGradArgs g)
{
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ __align__(8) unsigned long long s_mbar;
    __shared__ uint32_t s_tmem;
    __shared__ float s_w3[kMlpH], s_d[kGM];
    const int j = threadIdx.x, w = j >> 5;
    const uint32_t mbar = (uint32_t)__cvta_generic_to_shared(&s_mbar);
    if (j == 0) tc::mbar_init(mbar);
    if (w == 0) tc::tmem_alloc((uint32_t)__cvta_generic_to_shared(&s_tmem), kGTmemCols);
    s_w3[j] = __bfloat162float(g.w3[j]);
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = s_tmem;
    const int slabs = (g.T + kGM - 1) / kGM;                   // of 128 tours, in both products
    const int b = blockIdx.x, dz = slabs * (kMlpH / kGNz);
    if (b < dz) {
        const int m0 = b / (kMlpH / kGNz) * kGM, n0 = b % (kMlpH / kGNz) * kGNz;
        grad_tile<true>(g, smem, tmem, mbar, s_d, s_w3, m0, n0, m0);
    } else {
        const int t = b - dz, m0 = (t & 1) * kGM, n0 = (t >> 1) % kGwTiles * kGNw, b0 = (t >> 1) / kGwTiles * kGM;
        grad_tile<false>(g, smem, tmem, mbar, s_d, s_w3, m0, n0, b0);
    }
    tc::fence_before_sync();
    __syncthreads();
    if (w == 0) tc::tmem_dealloc(tmem, kGTmemCols);
}

}  // namespace

cudaError_t mlp_head(const MlpHeadArgs &a, cudaStream_t st)
{
    cudaError_t e = cudaFuncSetAttribute(mlp_head_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kHeadSmem);
    if (e != cudaSuccess) return e;
    mlp_head_kernel<<<(unsigned)((a.T + kL2M - 1) / kL2M), kTcThreads, kHeadSmem, st>>>(a);
    return cudaGetLastError();
}

template <bool BWD>
static cudaError_t layer1(const MlpLayer1Args &l1, int sm_count, cudaStream_t st)
{
    cudaError_t e = cudaFuncSetAttribute(mlp_layer1_tc_kernel<BWD>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kF1Smem);
    if (e != cudaSuccess) return e;
    const int grid = l1.T < sm_count ? l1.T : sm_count;
    mlp_layer1_tc_kernel<BWD><<<grid, kF1Threads, kF1Smem, st>>>(l1);
    return cudaGetLastError();
}

cudaError_t mlp_layer1_tc(const MlpLayer1Args &l1, int sm_count, cudaStream_t st) { return layer1<false>(l1, sm_count, st); }
cudaError_t mlp_layer1_bwd_tc(const MlpLayer1Args &l1, int sm_count, cudaStream_t st) { return layer1<true>(l1, sm_count, st); }

cudaError_t mlp_grad(const MlpGradArgs &g, cudaStream_t st)
{
    cudaError_t e = cudaFuncSetAttribute(mlp_grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGSmem);
    if (e != cudaSuccess) return e;
    const long long slabs = ((long long)g.T + kGM - 1) / kGM;
    mlp_grad_kernel<<<(unsigned)(slabs * (kMlpH / kGNz + 2 * kGwTiles)), kTcThreads, kGSmem, st>>>(g);
    return cudaGetLastError();
}

}  // namespace cvrpsd
