// Seeded scenario generator: fills a [n][ld] demand matrix on the device.
//
// Random words come from Philox4x32-10 (Salmon, Moraes, Dror, Shaw, "Parallel
// random numbers: as easy as 1, 2, 3", SC 2011), keyed by the 64-bit seed and
// counted by (scenario, index, domain, 0), so every entry is a pure function
// of its coordinates. Standard normals are Box-Muller draws in float64 from
// the first two words. Each float64 operation is written with an explicit
// round-to-nearest intrinsic so that no multiply-add is fused and the result
// is the one a plain IEEE evaluation in the written order gives.
#include <stdint.h>

#include "kernels.h"

namespace cvrpsd {

// Round multipliers and Weyl key increments of Philox4x32.
constexpr uint32_t kPhiloxM0 = 0xD2511F53u, kPhiloxM1 = 0xCD9E8D57u;
constexpr uint32_t kPhiloxW0 = 0x9E3779B9u, kPhiloxW1 = 0xBB67AE85u;

__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint32_t k0, uint32_t k1)
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        if (r > 0) { k0 += kPhiloxW0; k1 += kPhiloxW1; }
        const uint32_t lo0 = kPhiloxM0 * c.x, hi0 = __umulhi(kPhiloxM0, c.x);
        const uint32_t lo1 = kPhiloxM1 * c.z, hi1 = __umulhi(kPhiloxM1, c.z);
        c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
    }
    return c;
}

__device__ __forceinline__ double std_normal(uint32_t s, uint32_t index, uint32_t domain,
                                             uint32_t k0, uint32_t k1)
{
    const uint4 w = philox4x32_10(make_uint4(s, index, domain, 0u), k0, k1);
    const double inv32 = 2.3283064365386963e-10;   // 2^-32
    const double two_pi = 6.283185307179586;
    const double u1 = __dmul_rn(__dadd_rn((double)w.x, 0.5), inv32);
    const double u2 = __dmul_rn((double)w.y, inv32);
    const double r = sqrt(__dmul_rn(-2.0, log(u1)));
    return __dmul_rn(r, cos(__dmul_rn(two_pi, u2)));
}

// One demand by the recipe in float64: what every entry is defined by.
template <typename DT>
__device__ __noinline__ DT demand_f64(const GenParams &g, uint32_t s, int row)
{
    const uint32_t k0 = (uint32_t)g.seed, k1 = (uint32_t)(g.seed >> 32);
    const double dmax = sizeof(DT) == 2 ? 32767.0 : 2147483647.0;
    const double mu = (double)g.mu[row];
    double x;
    if (g.kind == 1) {
        const double f = std_normal(s, (uint32_t)(g.region[row] & 3), 1u, k0, k1);
        const double e = std_normal(s, (uint32_t)row, 0u, k0, k1);
        const double y = __dadd_rn(__dmul_rn(0.6, f), __dmul_rn(0.8, e));
        x = __dmul_rn(mu, exp(__dsub_rn(__dmul_rn(0.3, y), 0.045)));
    } else {
        const double z = std_normal(s, (uint32_t)row, 2u, k0, k1);
        x = __dadd_rn(mu, __dmul_rn(__dmul_rn(0.3, mu), z));
    }
    double rnd = floor(x);
    if (__dsub_rn(x, rnd) >= 0.5) rnd = __dadd_rn(rnd, 1.0);   // half away from zero
    rnd = fmin(fmax(rnd, 0.0), dmax);
    return (DT)(long long)rnd;
}

// The same standard normal in float32, with a bound `err` on its distance
// from the float64 value. From the documented errors of the intrinsics
// (__logf 2^-21.41 absolute on [0.5, 2] and 3 ulp elsewhere, rsqrtf 2 ulp,
// __cosf 2^-21.19 absolute on [-pi, pi]) and the roundings of u1 (2^-23) and
// of the angle (3 * 2^-24 * pi):
//   t = -2 ln u1:  |dt| <= 1.0e-6 + 4.0e-7 t
//   r = sqrt(t):   |dr| <= |dt| / r + 3.1e-7 r
//   z = r cos:     |dz| <= |dr| + 1.05e-6 r  <=  1.0e-6 / r + 1.8e-6 r
// A t below 1e-4 (5e-5 of all draws: u1 near 1, where the square root
// amplifies dt) reports an infinite bound and z = 0.
__device__ __forceinline__ float std_normal_f32(uint32_t wx, uint32_t wy, float &err)
{
    const float u1 = ((float)wx + 0.5f) * 2.3283064365386963e-10f;
    const float t = -2.0f * __logf(u1);
    const float ri = rsqrtf(t), r = t * ri;
    const float z = r * __cosf((float)(int32_t)wy * 1.4629180792671596e-9f);   // pi 2^-31
    const bool ok = t > 1e-4f;
    err = ok ? fmaf(1.0e-6f, ri, 1.8e-6f * r) : __int_as_float(0x7f800000);
    return ok ? z : 0.0f;
}

// What bounds it: the float64 pipe when every entry goes through it (GB300
// issues one float64 warp instruction every 16 clocks per SM: 3784 us for
// n = 200, S = 100,000, 10.6 GB/s of output). So each entry is evaluated in
// float32 with a rigorous error bound first; when every value inside the
// bound rounds to the same integer that integer is the float64 result. The
// others (about 1e-4 of the entries at means of 5 to 30; all of them above
// about 1e5, where float32 cannot decide) go through the float64 recipe:
// collected in shared memory and evaluated densely after the block's rows, or
// on the spot when the list is full. What bounds it now: the ten Philox
// rounds and four special-function operations per entry.
constexpr int kGenThreads = 256;
constexpr int kGenList = 512;
constexpr float kGenMax = 1.0e6f;                // float32 decides nothing above
constexpr float kGenMagic = 12582912.0f;         // 1.5 * 2^23: adding it rounds to an integer

template <typename DT, int KIND>
__global__ void __launch_bounds__(kGenThreads) gen_demand_kernel(GenParams g, int rows_per_block)
{
    __shared__ uint32_t s_list[kGenList];
    __shared__ int s_count;
    const long long s_block = (long long)blockIdx.x * kGenThreads;
    const long long s = s_block + threadIdx.x;
    const uint32_t k0 = (uint32_t)g.seed, k1 = (uint32_t)(g.seed >> 32);
    const int r0 = blockIdx.y * rows_per_block;
    const int r1 = min(g.n, r0 + rows_per_block);
    const float dmax = sizeof(DT) == 2 ? 32767.0f : 2147483648.0f;
    if (threadIdx.x == 0) s_count = 0;
    __syncthreads();
    DT *out = reinterpret_cast<DT *>(g.out);
    if (s < g.S) {
        float f[4] = {0.0f, 0.0f, 0.0f, 0.0f}, ef = 0.0f;
        if (KIND == 1) {
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const uint4 w = philox4x32_10(make_uint4((uint32_t)s, (uint32_t)r, 1u, 0u), k0, k1);
                float e;
                f[r] = 0.6f * std_normal_f32(w.x, w.y, e);
                ef = fmaxf(ef, 0.18f * e);
            }
            ef += 2.0e-6f;   // roundings of the exponent (|0.3 y| <= 2.9) and the products, __expf (5 ulp)
        }
#pragma unroll 2
        for (int row = r0; row < r1; ++row) {
            const float mu = (float)g.mu[row];
            const uint4 w = philox4x32_10(make_uint4((uint32_t)s, (uint32_t)row, KIND == 1 ? 0u : 2u, 0u), k0, k1);
            float e, x, err;
            const float z = std_normal_f32(w.x, w.y, e);
            if (KIND == 1) {
                const int reg = g.region[row] & 3;
                const float fr = reg == 0 ? f[0] : reg == 1 ? f[1] : reg == 2 ? f[2] : f[3];
                x = mu * __expf(fmaf(0.3f, fmaf(0.8f, z, fr), -0.045f));
                err = x * fmaf(0.24f, e, ef);
            } else {
                x = fmaf(0.3f * mu, z, mu);
                err = mu * fmaf(0.3f, e, 1.0e-6f + 3.0e-7f * fabsf(z));
            }
            // nearest integers of both ends (an end on a tie is within the
            // bound of it, so the other end rounds elsewhere or the list is
            // only entered needlessly), clamped as the result is
            const float lo = (fmaxf(x - err, 0.0f) + kGenMagic), hi = (fmaxf(x + err, 0.0f) + kGenMagic);
            if (x < kGenMax && err < 1.0f && lo == hi) {
                out[(long long)row * g.ld + s] = (DT)(int)fminf(lo - kGenMagic, dmax);
            } else {
                const int at = atomicAdd(&s_count, 1);
                if (at < kGenList) s_list[at] = ((uint32_t)(row - r0) << 8) | threadIdx.x;
                else out[(long long)row * g.ld + s] = demand_f64<DT>(g, (uint32_t)s, row);
            }
        }
    }
    __syncthreads();
    const int count = min(s_count, kGenList);
    for (int k = threadIdx.x; k < count; k += kGenThreads) {
        const int row = r0 + (int)(s_list[k] >> 8);
        const long long c = s_block + (s_list[k] & 255u);
        out[(long long)row * g.ld + c] = demand_f64<DT>(g, (uint32_t)c, row);
    }
}

template <typename TI, typename TO>
__global__ void convert_demand_kernel(const TI *in, long long ld_in, TO *out, long long ld_out, int n, long long S,
                                      unsigned int *saturated)
{
    const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= S) return;
    for (int r = blockIdx.y; r < n; r += gridDim.y) {
        const long long v = (long long)in[(long long)r * ld_in + s];
        if (sizeof(TO) == 2 && (v > 32767 || v < -32768)) atomicOr(saturated, 1u);
        out[(long long)r * ld_out + s] = (TO)(v > 32767 && sizeof(TO) == 2 ? 32767 : v);
    }
}

cudaError_t launch_convert_demand(const void *in, int esize_in, long long ld_in, void *out, int esize_out,
                                  long long ld_out, int n, long long S, unsigned int *saturated,
                                  cudaStream_t stream)
{
    if (S == 0 || n == 0) return cudaSuccess;
    dim3 grid((unsigned)((S + 255) / 256), (unsigned)(n < 64 ? n : 64));
    if (esize_in == 2 && esize_out == 2)
        convert_demand_kernel<int16_t, int16_t><<<grid, 256, 0, stream>>>((const int16_t *)in, ld_in, (int16_t *)out,
                                                                          ld_out, n, S, saturated);
    else if (esize_in == 2)
        convert_demand_kernel<int16_t, int32_t><<<grid, 256, 0, stream>>>((const int16_t *)in, ld_in, (int32_t *)out,
                                                                          ld_out, n, S, saturated);
    else if (esize_out == 2)
        convert_demand_kernel<int32_t, int16_t><<<grid, 256, 0, stream>>>((const int32_t *)in, ld_in, (int16_t *)out,
                                                                          ld_out, n, S, saturated);
    else
        convert_demand_kernel<int32_t, int32_t><<<grid, 256, 0, stream>>>((const int32_t *)in, ld_in, (int32_t *)out,
                                                                          ld_out, n, S, saturated);
    return cudaGetLastError();
}

cudaError_t launch_gen_demand(const GenParams &g, int esize, cudaStream_t stream)
{
    if (g.S == 0 || g.n == 0) return cudaSuccess;
    const long long bx = (g.S + kGenThreads - 1) / kGenThreads;
    // 64 rows a block spread the four factor draws of a column thin; fewer
    // where that leaves less than four blocks of 256 for each of 152 SMs.
    int rows = 64;
    while (rows > 8 && bx * ((g.n + rows - 1) / rows) < 4 * 152) rows >>= 1;
    const dim3 grid((unsigned)bx, (unsigned)((g.n + rows - 1) / rows));
    if (esize == 2) {
        if (g.kind == 1) gen_demand_kernel<int16_t, 1><<<grid, kGenThreads, 0, stream>>>(g, rows);
        else gen_demand_kernel<int16_t, 0><<<grid, kGenThreads, 0, stream>>>(g, rows);
    } else {
        if (g.kind == 1) gen_demand_kernel<int32_t, 1><<<grid, kGenThreads, 0, stream>>>(g, rows);
        else gen_demand_kernel<int32_t, 0><<<grid, kGenThreads, 0, stream>>>(g, rows);
    }
    return cudaGetLastError();
}

}  // namespace cvrpsd
