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

// The recipe's last step in float64: half away from zero, clamped at 0 and at
// the type's maximum.
template <typename DT>
__device__ __forceinline__ DT round_demand(double x)
{
    const double dmax = sizeof(DT) == 2 ? 32767.0 : 2147483647.0;
    double rnd = floor(x);
    if (__dsub_rn(x, rnd) >= 0.5) rnd = __dadd_rn(rnd, 1.0);
    rnd = fmin(fmax(rnd, 0.0), dmax);
    return (DT)(long long)rnd;
}

__device__ __forceinline__ double correlated_f64(double mu, double f, double e)
{
    const double y = __dadd_rn(__dmul_rn(0.6, f), __dmul_rn(0.8, e));
    return __dmul_rn(mu, exp(__dsub_rn(__dmul_rn(0.3, y), 0.045)));
}

// One demand by the recipe in float64: what every entry is defined by.
template <typename DT>
__device__ __noinline__ DT demand_f64(const GenParams &g, uint32_t s, int row)
{
    const uint32_t k0 = (uint32_t)g.seed, k1 = (uint32_t)(g.seed >> 32);
    const double mu = (double)g.mu[row];
    if (g.kind == 1)
        return round_demand<DT>(correlated_f64(mu, std_normal(s, (uint32_t)(g.region[row] & 3), 1u, k0, k1),
                                               std_normal(s, (uint32_t)row, 0u, k0, k1)));
    return round_demand<DT>(__dadd_rn(mu, __dmul_rn(__dmul_rn(0.3, mu), std_normal(s, (uint32_t)row, 2u, k0, k1))));
}

__device__ __forceinline__ float lg2_ftz(float x)
{
    float r;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float ex2_ftz(float x)
{
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float rsqrt_ftz(float x)
{
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float cos_ftz(float x)
{
    float r;
    asm("cos.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// The same standard normal in float32, with a bound `err` on its distance
// from the float64 value. From the documented errors of the PTX instructions
// (lg2 2^-22 absolute on (0.5, 2) and relative elsewhere, rsqrt 2^-22.9
// relative, cos 2^-20.5 absolute on [-pi, pi]) and the roundings of u1
// (2^-23 relative, 2 * 2^-23 of t), of the products (2^-24 each) and of the
// angle (3 * 2^-24 * pi):
//   t = -2 ln u1:  |dt| <= 1.0e-6 + 4.0e-7 t
//   r = sqrt(t):   |dr| <= |dt| / r + 3.1e-7 r
//   z = r cos:     |dz| <= |dr| + 1.3e-6 r  <=  1.0e-6 / r + 2.1e-6 r
// below t = 1e-4 (5e-5 of all draws: u1 near 1, where the square root
// amplifies dt) the bound does not hold and `ok` says so (NaN included).
__device__ __forceinline__ float std_normal_f32(uint32_t wx, uint32_t wy, float &err, bool &ok)
{
    const float u1 = ((float)wx + 0.5f) * 2.3283064365386963e-10f;
    const float t = -1.3862943611198906f * lg2_ftz(u1);                        // -2 ln 2
    const float ri = rsqrt_ftz(t), r = t * ri;
    ok = t > 1e-4f;
    err = fmaf(1.0e-6f, ri, 2.1e-6f * r);
    return r * cos_ftz((float)(int32_t)wy * 1.4629180792671596e-9f);           // pi 2^-31
}

// The parts of Philox4x32-10 at counter (s, row, domain, 0) that depend on
// (s, domain) alone: the first two rounds and half of the third. A thread
// walks the rows of one scenario, so they are formed once.
struct PhiloxColumn {
    uint32_t k0, k1, a, b, c, d, hi, lo;
    __device__ __forceinline__ PhiloxColumn(uint32_t s, uint32_t domain, uint32_t key0, uint32_t key1)
        : k0(key0), k1(key1)
    {
        a = __umulhi(kPhiloxM1, domain) ^ k0;                                  // ^ row: round 0's x
        const uint32_t z0 = __umulhi(kPhiloxM0, s) ^ k1;
        c = kPhiloxM0 * s ^ (k1 + kPhiloxW1);                                  // ^ hi(M0 x): round 1's z
        b = kPhiloxM1 * z0;                                                    // round 1's y
        const uint32_t x1 = __umulhi(kPhiloxM1, z0) ^ (kPhiloxM1 * domain) ^ (k0 + kPhiloxW0);
        hi = __umulhi(kPhiloxM0, x1) ^ (k1 + 2u * kPhiloxW1);                  // ^ w: round 2's z
        lo = kPhiloxM0 * x1;                                                   // round 2's w
        d = b ^ (k0 + 2u * kPhiloxW0);                                         // ^ hi(M1 z): round 2's x
    }
    __device__ __forceinline__ uint2 at(uint32_t row) const
    {
        const uint32_t x0 = a ^ row;                                           // the same for all threads
        const uint32_t z1 = __umulhi(kPhiloxM0, x0) ^ c;
        uint32_t x = __umulhi(kPhiloxM1, z1) ^ d, y = kPhiloxM1 * z1, z = (kPhiloxM0 * x0) ^ hi, w = lo;
#pragma unroll
        for (int r = 3; r < 10; ++r) {
            const uint32_t lo0 = kPhiloxM0 * x, hi0 = __umulhi(kPhiloxM0, x);
            const uint32_t lo1 = kPhiloxM1 * z, hi1 = __umulhi(kPhiloxM1, z);
            x = hi1 ^ y ^ (k0 + (uint32_t)r * kPhiloxW0);
            y = lo1;
            z = hi0 ^ w ^ (k1 + (uint32_t)r * kPhiloxW1);
            w = lo0;
        }
        return make_uint2(x, y);
    }
};

// What bounds it: the float64 pipe when every entry goes through it (GB300
// issues one float64 warp instruction every 16 clocks per SM: 3784 us for
// n = 200, S = 100,000, 10.6 GB/s of output). So each entry is evaluated in
// float32 with a rigorous error bound first; when both ends of the bound
// round to the same integer that integer is the float64 result. The others
// (about 2e-4 of the entries at means of 5 to 30) go through the float64
// recipe: collected in shared memory and evaluated densely after the block's
// rows, or on the spot when the list is full. SKIP: rows of means from `dense`
// on are left to gen_dense_kernel. What bounds it now: issue of the Philox rounds
// (14 wide multiplies) and the four special functions of an entry, 153 clocks
// of a scheduler per 32 entries. 110 us at n = 200, S = 100,000 (1.01 ms at
// n = 1000, S = 2^18); 132 us before the draws' common Philox rounds, the
// bare special-function instructions and the paired float64 tail. Four blocks
// a SM (64 registers): 123 us at one block, 119 us at six.
constexpr int kGenThreads = 256;
constexpr int kGenList = 512;
constexpr int kGenRows = 64;                     // most rows of a block
constexpr float kGenMax = 1.0e6f;                // float32 decides nothing above
constexpr float kGenMagic = 12582912.0f;         // 1.5 * 2^23: adding it rounds to an integer

template <typename DT, int KIND, bool SKIP>
__global__ void __launch_bounds__(kGenThreads, 4) gen_demand_kernel(GenParams g, int rows_per_block, float dense)
{
    __shared__ uint32_t s_list[kGenList];
    __shared__ int s_count;
    __shared__ float s_f[4][kGenThreads];        // 0.6 F of the block's columns
    __shared__ float2 s_row[kGenRows];           // mean, and the region's offset in s_f
    const long long s_block = (long long)blockIdx.x * kGenThreads;
    const int tid = threadIdx.x;
    const long long s = s_block + tid;
    const uint32_t k0 = (uint32_t)g.seed, k1 = (uint32_t)(g.seed >> 32);
    const int r0 = blockIdx.y * rows_per_block;
    const int rows = min(g.n - r0, rows_per_block);
    if (tid == 0) s_count = 0;
    for (int k = tid; k < rows; k += kGenThreads)
        s_row[k] = make_float2((float)g.mu[r0 + k], __int_as_float(KIND == 1 ? (g.region[r0 + k] & 3) * kGenThreads : 0));
    __syncthreads();
    DT *out = reinterpret_cast<DT *>(g.out) + (long long)r0 * g.ld + s;
    if (s < g.S) {
        float ef = 0.0f;
        if (KIND == 1) {
            bool fine = true;
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const uint4 w = philox4x32_10(make_uint4((uint32_t)s, (uint32_t)r, 1u, 0u), k0, k1);
                float e;
                bool ok;
                const float f = std_normal_f32(w.x, w.y, e, ok);
                s_f[r][tid] = ok ? 0.6f * f : 0.0f;
                fine &= ok;
                ef = fmaxf(ef, 0.18f * e);
            }
            // + roundings of the exponent (|0.3 y| <= 2.9) and of the products, ex2 (2^-22)
            ef = fine ? ef + 2.0e-6f : __int_as_float(0x7f800000);
        }
        const PhiloxColumn px((uint32_t)s, KIND == 1 ? 0u : 2u, k0, k1);
#pragma unroll 2
        for (int k = 0; k < rows; ++k, out += g.ld) {
            const float2 rw = s_row[k];
            const float mu = rw.x;
            if (SKIP && mu >= dense) continue;               // the same for all threads
            const uint2 w = px.at((uint32_t)(r0 + k));
            float e, x, err;
            bool ok;
            const float z = std_normal_f32(w.x, w.y, e, ok);
            float lo, hi;
            if (KIND == 1) {
                const float y = fmaf(0.8f, z, (&s_f[0][0])[__float_as_int(rw.y) + tid]);
                x = mu * ex2_ftz(fmaf(0.3f * 1.4426950408889634f, y, -0.045f * 1.4426950408889634f));
                err = x * fmaf(0.24f, e, ef);
                lo = x - err;
                hi = x + err;
            } else {
                x = fmaf(0.3f * mu, z, mu);
                err = mu * fmaf(0.3f, e, 1.0e-6f + 3.0e-7f * fabsf(z));
                lo = fmaxf(x - err, 0.0f);
                hi = fmaxf(x + err, 0.0f);
            }
            // nearest integers of both ends (an infinite or NaN bound makes them differ)
            lo += kGenMagic;
            hi += kGenMagic;
            if (ok && x < kGenMax && lo == hi) {
                const int v = __float_as_int(lo) - __float_as_int(kGenMagic);
                *out = (DT)(sizeof(DT) == 2 ? min(v, 32767) : v);
            } else {
                const int at = atomicAdd(&s_count, 1);
                if (at < kGenList) s_list[at] = ((uint32_t)k << 8) | (uint32_t)tid;
                else *out = demand_f64<DT>(g, (uint32_t)s, r0 + k);
            }
        }
    }
    __syncthreads();
    // Two neighbouring lanes share an entry of a correlated matrix: one draws
    // the customer's normal, the other the region's, which halves the serial
    // float64 chain that a block ends with.
    const int count = min(s_count, kGenList), half = tid & 1;
    for (int k0_ = 0; k0_ < count; k0_ += kGenThreads / 2) {
        const int k = k0_ + (tid >> 1);
        const uint32_t item = s_list[min(k, count - 1)];
        const int row = r0 + (int)(item >> 8);
        const long long c = s_block + (item & 255u);
        const uint32_t index = KIND == 1 && half ? (uint32_t)(g.region[row] & 3) : (uint32_t)row;
        const double z = std_normal((uint32_t)c, index, KIND == 1 ? (half ? 1u : 0u) : 2u, k0, k1);
        const double mu = (double)g.mu[row];
        double x;
        if (KIND == 1) x = correlated_f64(mu, __shfl_xor_sync(0xffffffffu, z, 1), z);
        else x = __dadd_rn(mu, __dmul_rn(__dmul_rn(0.3, mu), z));
        if (!half && k < count) reinterpret_cast<DT *>(g.out)[(long long)row * g.ld + c] = round_demand<DT>(x);
    }
}

// Rows of large means, where float32 decides so few of a warp's entries that
// the draws behind the others (two normals for each of a correlated matrix)
// take longer: the recipe in float64 for every entry, a column's four factors
// once per block. Bound by the float64 pipe.
template <typename DT, int KIND>
__global__ void __launch_bounds__(kGenThreads) gen_dense_kernel(GenParams g, int rows_per_block, float dense)
{
    const long long s = (long long)blockIdx.x * kGenThreads + threadIdx.x;
    if (s >= g.S) return;
    const uint32_t k0 = (uint32_t)g.seed, k1 = (uint32_t)(g.seed >> 32);
    const int r0 = blockIdx.y * rows_per_block, r1 = min(g.n, r0 + rows_per_block);
    DT *out = reinterpret_cast<DT *>(g.out) + (long long)r0 * g.ld + s;
    double f[4] = {0.0, 0.0, 0.0, 0.0};
    bool drawn = false;
    for (int row = r0; row < r1; ++row, out += g.ld) {
        if ((float)g.mu[row] < dense) continue;              // the same for all threads
        const double mu = (double)g.mu[row], z = std_normal((uint32_t)s, (uint32_t)row, KIND == 1 ? 0u : 2u, k0, k1);
        if (KIND == 1) {
            if (!drawn) {
#pragma unroll
                for (int r = 0; r < 4; ++r) f[r] = std_normal((uint32_t)s, (uint32_t)r, 1u, k0, k1);
                drawn = true;
            }
            const int reg = g.region[row] & 3;
            *out = round_demand<DT>(correlated_f64(mu, reg == 0 ? f[0] : reg == 1 ? f[1] : reg == 2 ? f[2] : f[3], z));
        } else {
            *out = round_demand<DT>(__dadd_rn(mu, __dmul_rn(__dmul_rn(0.3, mu), z)));
        }
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

template <typename DT, int KIND>
static cudaError_t launch_gen(const GenParams &g, cudaStream_t stream)
{
    const long long bx = (g.S + kGenThreads - 1) / kGenThreads;
    // 64 rows a block spread the four factor draws of a column thin; fewer
    // where that leaves less than four blocks of 256 for each of 152 SMs (two in float64).
    const auto block_rows = [&](int blocks) {
        int rows = kGenRows;
        while (rows > 8 && bx * ((g.n + rows - 1) / rows) < blocks) rows >>= 1;
        return rows;
    };
    const int rows = block_rows(4 * 152), rows64 = block_rows(2 * 152);
    // Means from here on go through float64 throughout. By float32 first and in
    // float64, us: correlated, n = 200, S = 100,000, means of 10,000 3565 and 3775,
    // 14,000 4365 and 3777, 10^6 6076 and 3772; in shorter blocks more of a row's
    // entries fit the list (n = 200, S = 4000, 8 rows a block: 50,000 217 and 239,
    // 10^5 295 and 238). Normal: 10^5 2902 and 2937, 10^6 3010 and 2937.
    const float dense = KIND == 1 ? 7.0e5f / (float)rows : 1.0e5f;
    const dim3 grid((unsigned)bx, (unsigned)((g.n + rows - 1) / rows));
    if ((float)g.mu_max < dense) {
        gen_demand_kernel<DT, KIND, false><<<grid, kGenThreads, 0, stream>>>(g, rows, dense);
        return cudaGetLastError();
    }
    if ((float)g.mu_min < dense) gen_demand_kernel<DT, KIND, true><<<grid, kGenThreads, 0, stream>>>(g, rows, dense);
    gen_dense_kernel<DT, KIND><<<dim3((unsigned)bx, (unsigned)((g.n + rows64 - 1) / rows64)), kGenThreads, 0, stream>>>(
        g, rows64, dense);
    return cudaGetLastError();
}

cudaError_t launch_gen_demand(const GenParams &g, int esize, cudaStream_t stream)
{
    if (g.S == 0 || g.n == 0) return cudaSuccess;
    if (esize == 2) return g.kind == 1 ? launch_gen<int16_t, 1>(g, stream) : launch_gen<int16_t, 0>(g, stream);
    return g.kind == 1 ? launch_gen<int32_t, 1>(g, stream) : launch_gen<int32_t, 0>(g, stream);
}

}  // namespace cvrpsd
