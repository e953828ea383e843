// Batched Split on the second deque walk (split_deque2.cuh): the persistent
// item loop of split_batch.cu (blocks take (tour, tile of T scenarios) items
// from an atomic counter, longest tours first, and copy a tour's table into
// shared memory when they move to it), with each thread walking its scenario
// by the second walk's rules: int16 demands read unclamped, tests of the
// route length and of ring overflow once per span of 8 positions, no
// frozen flag in the tests, front walks that read only keys, back-pop skip
// bits and a vote-free first back step. The table differs from the
// single-tour walk's only in where it lives: shared memory instead of the
// launch parameters, with the skip bit and the block flag derived while it
// is copied. One scenario per thread, rings of 16 or more,
// keys that cannot wrap (the host checks every tour). int32 demands keep the
// second walk's clamp and running maximum.
#include "split_deque2.cuh"

namespace cvrpsd {

// The tour's table in shared memory: the demand rows of its positions, their
// C_i, both up to the next multiple of 4 (the last row and 0 again), so that a
// prefetch block of 4 positions reads each in one load (1084 -> 1048 us for 64
// tours of n = 200 under 65,536 scenarios against pairs read per position); and
// a word of flags for every span of two prefetch blocks (8 positions): bit u
// where no scenario can pop the back at the span's position u (kTab2NoBack of
// the parameter table), bit 8 + m where its prefetch block m holds some C_i <= 0
// with i < n.
//
// All threads of a block read the same entries, but a load from shared memory
// gives the compiler no way to know that. The flags (and the tour's
// parameters, below) therefore pass through a warp reduction of equal values,
// whose result it keeps in uniform registers: branches on them are uniform,
// and the walk takes 40 registers instead of 48, six blocks of 256 on an SM
// instead of five.
__device__ __forceinline__ int4 lds4(uint32_t a)
{
    int4 v;
    asm volatile("ld.shared.v4.s32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
    return v;
}
__device__ __forceinline__ int lane4(const int4 &v, int u) { return u == 0 ? v.x : u == 1 ? v.y : u == 2 ? v.z : v.w; }

struct TabShared2 {
    uint32_t a;       // shared-window address of the rows
    uint32_t c;       // of the C_i
    uint32_t f;       // of the flags
    static constexpr int kCap = 1 << 30;
    using Costs = int4;
    using Rows = int4;
    __device__ __forceinline__ int4 costs(int i0) const { return lds4(c + (uint32_t)(i0 - 1) * 4u); }
    __device__ __forceinline__ int cost(const int4 &v, int, int u) const { return lane4(v, u); }
    __device__ __forceinline__ int4 rows(int i0) const { return lds4(a + (uint32_t)(i0 - 1) * 4u); }
    __device__ __forceinline__ uint32_t row_at(const int4 &v, int, int u) const { return (uint32_t)lane4(v, u); }
    __device__ __forceinline__ uint32_t span(int i0) const
    {
        return __reduce_or_sync(0xffffffffu, (uint32_t)lds1(f + (uint32_t)((i0 - 1) >> 3) * 4u));
    }
    __device__ __forceinline__ bool general(uint32_t fl, int, int at) const { return (fl >> (8 + at / kPrefetch2)) & 1u; }
    __device__ __forceinline__ bool noback(uint32_t fl, int, int u) const { return (fl >> u) & 1u; }
};
static_assert(kPrefetch2 == 4, "a span's flags are for two blocks of four positions");

__device__ __forceinline__ uint32_t uniform(uint32_t x) { return __reduce_or_sync(0xffffffffu, x); }

// Blocks an SM holds (and the registers a thread may take): shared memory for
// the rings and a table of a few hundred positions, or 2048 threads. 256
// threads with rings of 16: six blocks of 40 registers (64 tours of n = 200
// under 65,536 scenarios 1116 -> 1096 us, 64 tours of 100 to 1000 under 8192
// 464 -> 453 us against five of 48; at n = 1000 the table leaves room for five).
template <int R, int T>
constexpr int b2_min_blocks()
{
    constexpr int by_smem = 233472 / (R * T * 8 + 4096 + 1024);
    constexpr int by_threads = 2048 / T;
    constexpr int m = by_smem < by_threads ? by_smem : by_threads;
    return m < 1 ? 1 : (m > 32 ? 32 : m);
}

// SMOOTH: the walk of smooth tours (see smooth_table), a kernel of its own: both
// walks in one kernel cost the other one registers (64 tours of n = 100..1000
// under 8192 scenarios 434 -> 443 us; out of line worse). Where the host has
// the tables it launches one of the two; where they were built on the device
// both are launched and the blocks of the one that does not apply exit.
template <typename DT, int R, int T, bool LCAP, bool SMOOTH>
__global__ void __launch_bounds__(T, b2_min_blocks<R, T>()) split_batch2_kernel(BatchParams b)
{
    if (b.smooth < 0 && (2 * b.acc[BACC_SMOOTH] > (unsigned long long)b.T) != SMOOTH) return;
    extern __shared__ __align__(16) unsigned char smem[];   // rings [R][T], then the table
    __shared__ int s_item;
    __shared__ long long s_sum[T / 32];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const uint32_t rs = (uint32_t)__cvta_generic_to_shared(smem);
    const int cap = (b.max_n + 3) / 4 * 4;
    int32_t *rowp = reinterpret_cast<int32_t *>(smem + (size_t)R * T * 8), *costp = rowp + cap;
    uint32_t *flagp = reinterpret_cast<uint32_t *>(costp + cap);
    const uint32_t row_s = rs + (uint32_t)R * T * 8;
    const TabShared2 tab{row_s, row_s + 4u * cap, row_s + 8u * cap};
    unsigned long long *tacc = b.acc + BACC_WORDS;
    unsigned long long *status = b.acc + BACC_STATUS;
    int cur = -1;
    for (;;) {
        __syncthreads();                          // the previous item is finished everywhere
        if (tid == 0) s_item = (int)atomicAdd(reinterpret_cast<unsigned int *>(b.acc + BACC_COUNTER), 1u);
        __syncthreads();
        const int item = s_item;
        if (item >= b.n_items) break;
        const int2 it = b.items ? b.items[item] : make_int2(item / b.tiles, item % b.tiles);
        if (!index_ok(it.x >= 0 && it.y >= 0 && (long long)it.y * T < b.S, status)) continue;
        const TourDev td = b.tours[it.x];
        const int t = it.x;
        if (t != cur) {   // block-uniform; the loop-top barrier has retired the previous item
            for (int k = tid; k < (td.n + 3) / 4 * 4; k += T) {
                const TourStep e = td.tab[min(k, td.n - 1)];
                rowp[k] = e.row & kRowMask;
                costp[k] = k < td.n ? e.c : 0;
            }
            for (int m = tid; m < (td.n + 7) / 8; m += T) {
                uint32_t fl = 0;
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int k = 8 * m + u;
                    if (k >= td.n) break;
                    const int ck = td.tab[k].c, cp = k ? td.tab[k - 1].c : 0;
                    // position k + 1 >= 2 with C_k > 0 and C_{k+1} > C_k: no back pops
                    if (cp > 0 && ck > cp) fl |= 1u << u;
                    if (k < td.n - 1 && ck <= 0) fl |= 1u << (8 + u / kPrefetch2);
                }
                flagp[m] = fl;
            }
            __syncthreads();
            cur = t;
        }
        Walk2Params p{};
        p.demand = td.demand;
        p.S = b.S;
        p.n = (int)uniform((uint32_t)td.n);
        p.Q = (int)uniform((uint32_t)td.Q);
        p.L = (int)uniform((uint32_t)td.L);
        p.g0 = td.g0;
        p.K = uniform(td.K);
        p.pitch = uniform((uint32_t)(td.ld * (int)sizeof(DT)));
        p.status = status;
        const long long s = (long long)it.y * T + tid;
        bool aside = false;
        const int c = walk2_scenario<DT, R, T, LCAP, true, SMOOTH>(p, tab, s, rs, (uint32_t)tid * 8u, aside);
        long long sum = 0;
        if (s < b.S) {
            if (aside) {
                const unsigned long long idx = atomicAdd(b.acc + BACC_LIST, 1ull);
                if ((long long)idx < b.list_cap) b.list[idx] = make_int2(t, (int)s);
                else atomicOr(status, (unsigned long long)BST_LIST_FULL);
            } else {
                sum = c;
                if (td.out_cost) td.out_cost[s] = c;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if (lane == 0) s_sum[w] = sum;
        __syncthreads();
        if (tid == 0) {
            long long tot = 0;
#pragma unroll
            for (int k = 0; k < T / 32; ++k) tot += s_sum[k];
            if (tot) atomicAdd(tacc + 3 * t, (unsigned long long)tot);
        }
    }
}

template <typename DT, int R, int T, bool LCAP, bool SMOOTH>
static cudaError_t launch2_one(const BatchParams &b, const DequeShape &shape, int grid, bool configure_only,
                               int *blocks_per_sm, cudaStream_t stream)
{
    auto kern = split_batch2_kernel<DT, R, T, LCAP, SMOOTH>;
    const size_t smem = split_batch_smem(b.max_n, shape);
    if (configure_only) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        return blocks_per_sm ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, kern, T, smem)
                             : cudaSuccess;
    }
    kern<<<grid, T, smem, stream>>>(b);
    return cudaGetLastError();
}

// Shapes of the batch kernel's list with one scenario per thread.
#define CVRPSD_BATCH2_SHAPES(X)                                                                 \
    X(32, 16) X(32, 32) X(32, 64) X(64, 16) X(64, 32) X(64, 64) X(128, 16) X(128, 32)            \
    X(128, 64) X(256, 16) X(256, 32) X(512, 16)

// 32-bit demands: the library's own shapes (64 tours of n = 200 under 65,536
// scenarios 1451 us by the first walk, 1152; in strips 1703, 1553).
#define CVRPSD_BATCH2_SHAPES_I32(X) X(64, 16) X(128, 16) X(256, 16) X(512, 16)

template <typename DT, bool LCAP>
static cudaError_t dispatch2(BatchParams b, const DequeShape &s, int grid, bool configure_only,
                             int *blocks_per_sm, cudaStream_t st)
{
    if (b.smooth != 0 && batch2_smooth_compiled(s)) {
        const cudaError_t e = s.threads == 256
            ? launch2_one<DT, 16, 256, LCAP, true>(b, s, grid, configure_only, blocks_per_sm, st)
            : launch2_one<DT, 16, 512, LCAP, true>(b, s, grid, configure_only, blocks_per_sm, st);
        if (e != cudaSuccess || b.smooth > 0) return e;
    } else {
        b.smooth = 0;
    }
#define CVRPSD_CASE(T_, R_)                                                            \
    if (s.threads == T_ && s.spt == 1 && s.ring == R_)                                \
        return launch2_one<DT, R_, T_, LCAP, false>(b, s, grid, configure_only, blocks_per_sm, st);
    if constexpr (sizeof(DT) == 2) {
        CVRPSD_BATCH2_SHAPES(CVRPSD_CASE)
    } else {
        CVRPSD_BATCH2_SHAPES_I32(CVRPSD_CASE)
    }
#undef CVRPSD_CASE
    return cudaErrorInvalidValue;
}

#if CVRPSD_BATCH2_PART == 0
bool batch2_shape_compiled(const DequeShape &s, int esize)
{
#define CVRPSD_CASE(T_, R_) if (s.threads == T_ && s.spt == 1 && s.ring == R_) return true;
    if (esize == 2) {
        CVRPSD_BATCH2_SHAPES(CVRPSD_CASE)
    } else {
        CVRPSD_BATCH2_SHAPES_I32(CVRPSD_CASE)
    }
#undef CVRPSD_CASE
    return false;
}

cudaError_t launch_split_batch2(const BatchParams &b, int esize, bool lcap, const DequeShape &shape, int grid,
                                bool configure_only, int *blocks_per_sm, cudaStream_t stream)
{
    if (esize == 2)
        return lcap ? launch_split_batch2_cap(b, shape, grid, configure_only, blocks_per_sm, stream)
                    : launch_split_batch2_nocap(b, shape, grid, configure_only, blocks_per_sm, stream);
    return lcap ? launch_split_batch2_i32_cap(b, shape, grid, configure_only, blocks_per_sm, stream)
                : launch_split_batch2_i32_nocap(b, shape, grid, configure_only, blocks_per_sm, stream);
}

cudaError_t launch_split_batch2_cap(const BatchParams &b, const DequeShape &shape, int grid, bool configure_only,
                                    int *blocks_per_sm, cudaStream_t stream)
{
    return dispatch2<int16_t, true>(b, shape, grid, configure_only, blocks_per_sm, stream);
}
#elif CVRPSD_BATCH2_PART == 1
cudaError_t launch_split_batch2_nocap(const BatchParams &b, const DequeShape &shape, int grid, bool configure_only,
                                      int *blocks_per_sm, cudaStream_t stream)
{
    return dispatch2<int16_t, false>(b, shape, grid, configure_only, blocks_per_sm, stream);
}
#elif CVRPSD_BATCH2_PART == 2
cudaError_t launch_split_batch2_i32_cap(const BatchParams &b, const DequeShape &shape, int grid, bool configure_only,
                                        int *blocks_per_sm, cudaStream_t stream)
{
    return dispatch2<int32_t, true>(b, shape, grid, configure_only, blocks_per_sm, stream);
}
#else
cudaError_t launch_split_batch2_i32_nocap(const BatchParams &b, const DequeShape &shape, int grid, bool configure_only,
                                          int *blocks_per_sm, cudaStream_t stream)
{
    return dispatch2<int32_t, false>(b, shape, grid, configure_only, blocks_per_sm, stream);
}
#endif

}  // namespace cvrpsd
