// Transition-parallel Split: one warp evaluates one scenario (the second
// level of parallelism of Section 3: the candidate predecessors of a position). For each position i the 32 lanes take the
// candidates p of the feasible window [mask(i), i-1] of Eq. 2/3 in a strided
// pattern and a warp min-reduction picks the best, so the cost per position
// is O(|window| / 32 + log 32) and no candidate bound is needed. It serves the
// scenarios the deque kernel sets aside, and any tour when forced.
//
// Per warp, shared memory holds the scenario's prefix loads P[0..n] (demands
// loaded by all lanes at once, then a warp scan) and the values
// g[0..n] with g(p) = f(p) + c(0, sigma_{p+1}) - D[p+1] (see split_deque.cuh).
// The window start mask(i) is the smallest p >= i - L with
// P(i) - P(p) <= Q, tracked by a pointer that only moves forward.
//
// Windows of at most 64 candidates (all of them when L <= 64) take the
// register walk (warp_walk_scenario): the last 64 values g live in two
// registers per lane, and the walk goes four positions at a time. The window
// starts do not depend on g, so the minima of the four windows over the
// values already known are four independent warp reductions, and what is
// left in sequence is three minima and four additions on uniform values.
#include <stdint.h>

#include "kernels.h"
#include "split_deque.cuh"
#include "tour_table.h"

namespace cvrpsd {

struct WarpResult {
    int cost;      // f(n), INT32_MAX if infeasible
    bool bad;      // some demand > Q
    bool neg;      // some demand < 0
    bool wide;     // register walk only: a window longer than kWalkWidth, no cost
};

constexpr int kWalkWidth = 64;       // candidates held in registers
constexpr int kWalkRing = 128;       // prefix loads kept: 32 of this chunk, 65 before it

// One warp's shared memory of the register walk.
struct __align__(16) WalkSmem {
    int P[kWalkRing];                // prefix loads of positions i, slot i mod 128
    int lo[32], c[32];               // window start and C_i of the chunk's positions
};

// The recursion over the positions i0 .. min(n, i0 + 31) of a chunk, four to
// a step. The value of position p lives in lane (p - 1) mod 32: v0 the latest
// there (position pl), v1 the one 32 positions earlier. The window starts do
// not depend on g, so the minima of a step's four windows over the values
// known before it are four independent warp reductions; the values of the
// step itself are added on uniform registers. PLAIN: no window of the chunk
// is longer than 32 positions or starts inside its own step.
template <bool PLAIN>
__device__ __forceinline__ void walk_chunk(const WalkSmem &w, int n, int i0, int &v0, int &v1, int &pl)
{
    constexpr int kNone = INT32_MAX;
    constexpr unsigned kAll = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const bool odd = lane & 1, high = lane & 2;
    const int4 *lo = reinterpret_cast<const int4 *>(w.lo), *c = reinterpret_cast<const int4 *>(w.c);
    int4 l4 = lo[0], c4 = c[0];
#pragma unroll
    for (int b = 0; b < 8; ++b) {
        const int ib = i0 + 4 * b;
        if (b > 0 && ib > n) break;
        const int4 ln = lo[(b + 1) & 7], cn = c[(b + 1) & 7];
        int m0 = pl >= l4.x ? v0 : kNone, m1 = pl >= l4.y ? v0 : kNone;
        int m2 = pl >= l4.z ? v0 : kNone, m3 = pl >= l4.w ? v0 : kNone;
        if (!PLAIN) {
            const int pe = pl - 32;
            m0 = min(m0, pe >= l4.x ? v1 : kNone);
            m1 = min(m1, pe >= l4.y ? v1 : kNone);
            m2 = min(m2, pe >= l4.z ? v1 : kNone);
            m3 = min(m3, pe >= l4.w ? v1 : kNone);
        }
        m0 = __reduce_min_sync(kAll, m0);
        m1 = __reduce_min_sync(kAll, m1);
        m2 = __reduce_min_sync(kAll, m2);
        m3 = __reduce_min_sync(kAll, m3);
        // the previous position is always in the window
        const int ga = c4.x + m0;
        const int gb = c4.y + min(m1, ga);
        const int ab = min(ga, gb);
        const int gc = c4.z + min(m2, PLAIN ? ab : min(gb, l4.z <= ib ? ga : kNone));
        const int gd = c4.w + min(m3, PLAIN ? min(ab, gc)
                                            : min(gc, l4.w <= ib ? ab : l4.w <= ib + 1 ? gb : kNone));
        const int mine = high ? (odd ? gd : gc) : (odd ? gb : ga);
        if ((lane >> 2) == b) {
            v1 = v0;
            v0 = mine;
            pl = i0 + lane;
        }
        l4 = ln;
        c4 = cn;
    }
}

// Evaluates scenario s of one tour with the calling (full) warp, 32
// positions (one per lane) to a chunk: the chunk's demands (loaded a chunk
// ahead) are scanned to prefix loads, each lane finds its position's window
// start by bisection over the prefix loads kept in shared memory, and the
// recursion follows.
//
// What bounds it: the chain of a step (select, 18 clocks of reduction, four
// additions and minima, insertion) while few warps run, issue of the ALU pipe
// when many do.
template <typename DT>
__device__ __forceinline__ WarpResult warp_walk_scenario(const TourStep *__restrict__ tab, int n, int Q, int L, int g0,
                                                         const DT *__restrict__ dem, long long ld, long long s,
                                                         WalkSmem &w, unsigned long long *status)
{
    constexpr unsigned kAll = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    WarpResult r{INT32_MAX, false, false, false};
    const TourStep none{0, 0};
    auto step_of = [&](int i) { return i <= n ? tab[i - 1] : none; };
    auto demand_of = [&](const TourStep &t, int i) {
        const int row = t.row & kRowMask;
        return i <= n && index_ok(row < n && s >= 0 && s < ld, status) ? (int)__ldg(dem + (long long)row * ld + s) : 0;
    };
    TourStep t0 = step_of(1 + lane), t1 = step_of(33 + lane);
    int q = demand_of(t0, 1 + lane);
    int v0 = lane == 31 ? g0 : INT32_MAX, v1 = INT32_MAX, pl = lane == 31 ? 0 : -kWalkWidth;
    int carry = 0;
    bool neg = false, bad = false;
    __syncwarp();                                              // the previous scenario's readers are done
    if (lane == 0) w.P[0] = 0;
    for (int i0 = 1; i0 <= n; i0 += 32) {
        const int i = i0 + lane;
        const TourStep t2 = step_of(i + 64);
        const int qn = demand_of(t1, i + 32);
        neg |= q < 0;
        bad |= q > Q;
        int P = max(q, 0);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(kAll, P, o);
            if (lane >= o) P += u;
        }
        P += carry;
        carry = __shfl_sync(kAll, P, 31);
        w.P[i & (kWalkRing - 1)] = P;
        __syncwarp();
        const int first = max(0, i - L);                       // the route-length limit's start
        const int before = i - kWalkWidth - 1;
        const bool wide = i <= n && before >= first && P - w.P[before & (kWalkRing - 1)] <= Q;
        // a scenario with a demand above Q has no cost; one with a longer window is not for this walk
        if (__any_sync(kAll, wide | bad)) {
            r.bad = __any_sync(kAll, bad);
            r.wide = !r.bad;
            break;
        }
        int lo = max(first, i - kWalkWidth), hi = i - 1;       // hi is always in the window
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const int mid = (lo + hi) >> 1;
            const bool in = P - w.P[mid & (kWalkRing - 1)] <= Q;
            hi = in ? mid : hi;
            lo = in ? lo : mid + 1;
        }
        const bool plain = i > n || (i - lo <= 32 && lo <= i - (lane & 3));
        // positions past n (the last chunk) have an empty window
        w.lo[lane] = i <= n ? lo : INT32_MAX;
        w.c[lane] = t0.c;
        __syncwarp();
        if (__all_sync(kAll, plain)) walk_chunk<true>(w, n, i0, v0, v1, pl);
        else walk_chunk<false>(w, n, i0, v0, v1, pl);
        t0 = t1;
        t1 = t2;
        q = qn;
    }
    if (r.bad)                                                 // a negative demand anywhere is still reported
        for (int i = 1 + lane; i <= n; i += 32) neg |= demand_of(step_of(i), i) < 0;
    r.neg = __any_sync(kAll, neg);
    const int cost = __shfl_sync(kAll, v0, (n - 1) & 31);
    if (!r.bad && !r.wide) r.cost = cost;
    return r;
}

// Evaluates scenario s of one tour with the calling (full) warp. P and g are
// this warp's shared arrays of n + 1 ints each.
template <typename DT>
__device__ WarpResult warp_split_scenario(const TourStep *tab, int n, int Q, int L, int g0, const DT *dem,
                                          long long ld, long long s, int *P, int *g, unsigned long long *status,
                                          int16_t *pred = nullptr, long long ldp = 0)
{
    const int lane = threadIdx.x & 31;
    // Demands in tour order, clamped to Q+1 (anything above Q is infeasible).
    bool neg = false, bad = false;
    for (int i = 1 + lane; i <= n; i += 32) {
        const int row = tab[i - 1].row & kRowMask;
        int q = index_ok(row < n && s >= 0 && s < ld, status) ? (int)dem[(long long)row * ld + s] : 0;
        if (q < 0) { neg = true; q = 0; }
        if (q > Q) { bad = true; q = Q + 1; }
        P[i] = q;
    }
    __syncwarp();
    // Inclusive prefix sums, 32 positions at a time.
    int carry = 0;
    for (int b = 1; b <= n; b += 32) {
        const int i = b + lane;
        int v = i <= n ? P[i] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, v, o);
            if (lane >= o) v += t;
        }
        if (i <= n) P[i] = v + carry;
        carry += __shfl_sync(0xffffffffu, v, 31);
    }
    if (lane == 0) { P[0] = 0; g[0] = g0; }
    WarpResult r{};
    r.neg = __any_sync(0xffffffffu, neg);
    r.bad = __any_sync(0xffffffffu, bad);
    __syncwarp();
    r.cost = INT32_MAX;
    if (!r.bad) {
        int lo = 0;
        for (int i = 1; i <= n; ++i) {
            const int Pi = P[i];
            if (i - lo > L) lo = i - L;
            while (Pi - P[lo] > Q) ++lo;            // same on every lane
            int m = INT32_MAX, at = INT32_MAX;
            for (int c = lo + lane; c < i; c += 32) {
                const int v = g[c];
                if (v < m) { m = v; at = c; }          // first (smallest) c of this lane's minimum
            }
            const int mm = __reduce_min_sync(0xffffffffu, m);
            const int gi = tab[i - 1].c + mm;
            if (pred) {                                 // smallest optimal predecessor
                const int p = __reduce_min_sync(0xffffffffu, m == mm ? at : INT32_MAX);
                if (lane == 0) pred[(long long)(i - 1) * ldp + s] = (int16_t)p;
            }
            if (lane == 0) g[i] = gi;
            __syncwarp();
        }
        r.cost = g[n];
    }
    __syncwarp();
    return r;
}

template <typename DT>
__global__ void __launch_bounds__(128) split_warp_kernel(SplitParams p, const int32_t *list,
                                                         const unsigned long long *count)
{
    extern __shared__ __align__(16) int wsmem[];
    __shared__ WalkSmem s_walk[4];
    const int n = p.n;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, wpb = blockDim.x >> 5;
    int *P = wsmem + (size_t)w * 2 * (n + 1);
    int *g = P + (n + 1);
    const long long total = list ? (long long)*count : p.S;
    const DT *dem = reinterpret_cast<const DT *>(p.demand);

    long long sum = 0;
    unsigned inf = 0, status = 0;
    for (long long item = (long long)blockIdx.x * wpb + w; item < total;
         item += (long long)gridDim.x * wpb) {
        const long long s = list ? (long long)list[item] : item;
        if (!index_ok(s >= 0 && s < p.S, p.acc + ACC_STATUS)) continue;   // warp-uniform
        WarpResult r{};
        r.wide = true;
        if (!p.pred) r = warp_walk_scenario<DT>(p.tab, n, p.Q, p.L, p.g0, dem, p.ld, s, s_walk[w], p.acc + ACC_STATUS);
        if (r.wide)
            r = warp_split_scenario<DT>(p.tab, n, p.Q, p.L, p.g0, dem, p.ld, s, P, g, p.acc + ACC_STATUS, p.pred,
                                        p.ldp);
        if (lane == 0) {
            if (r.neg) status |= ST_NEGATIVE_DEMAND;
            if (r.bad) ++inf; else sum += r.cost;
            if (p.out_cost) p.out_cost[s] = r.cost;
        }
    }
    if (lane == 0) {
        if (sum) atomicAdd(p.acc + ACC_SUM, (unsigned long long)sum);
        if (inf) atomicAdd(p.acc + ACC_INFEASIBLE, (unsigned long long)inf);
        if (status) {
            atomicOr(p.acc + ACC_STATUS, (unsigned long long)status);
            atomicOr(p.sticky, (unsigned long long)status);
        }
    }
}

// The register walk alone, one scenario per warp: a scenario with a window
// longer than kWalkWidth goes on the list (for split_warp_kernel).
constexpr int kWalkWarps = 4;

template <typename DT>
__global__ void __launch_bounds__(32 * kWalkWarps) split_walk_kernel(SplitParams p)
{
    __shared__ WalkSmem s_walk[kWalkWarps];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const long long s = (long long)blockIdx.x * kWalkWarps + w;
    long long sum = 0;
    unsigned inf = 0, status = 0;
    if (s < p.S) {
        const WarpResult r = warp_walk_scenario<DT>(p.tab, p.n, p.Q, p.L, p.g0, reinterpret_cast<const DT *>(p.demand),
                                                    p.ld, s, s_walk[w], p.acc + ACC_STATUS);
        if (lane == 0) {
            if (r.wide) {
                p.ovf_list[atomicAdd(p.acc + ACC_OVERFLOW, 1ull)] = (int32_t)s;
            } else {
                if (r.neg) status = ST_NEGATIVE_DEMAND;
                if (r.bad) inf = 1; else sum = r.cost;
                if (p.out_cost) p.out_cost[s] = r.cost;
            }
        }
    }
    if (status) atomicOr(p.sticky, (unsigned long long)status);
    block_accumulate(sum, inf, status, p.acc);
    block_finish(p.acc, p.done);
}

cudaError_t launch_split_walk(const SplitParams &p, int esize, cudaStream_t stream)
{
    const unsigned grid = (unsigned)((p.S + kWalkWarps - 1) / kWalkWarps);
    if (esize == 2) split_walk_kernel<int16_t><<<grid, 32 * kWalkWarps, 0, stream>>>(p);
    else split_walk_kernel<int32_t><<<grid, 32 * kWalkWarps, 0, stream>>>(p);
    return cudaGetLastError();
}

// Set-aside (tour, scenario) pairs of a batch; per-tour sums, infeasible
// counts and status words follow the batch header in `acc`.
template <typename DT>
__global__ void __launch_bounds__(128) split_warp_batch_kernel(BatchParams b)
{
    extern __shared__ __align__(16) int wsmem[];
    __shared__ WalkSmem s_walk[4];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, wpb = blockDim.x >> 5;
    int *P = wsmem + (size_t)w * 2 * (b.max_n + 1);
    int *g = P + (b.max_n + 1);
    const unsigned long long cnt = b.acc[BACC_LIST];
    const long long total = (long long)(cnt < (unsigned long long)b.list_cap ? cnt : (unsigned long long)b.list_cap);
    unsigned long long *tacc = b.acc + BACC_WORDS;
    for (long long item = (long long)blockIdx.x * wpb + w; item < total;
         item += (long long)gridDim.x * wpb) {
        const int2 e = b.list[item];
        if (!index_ok(e.x >= 0 && e.y >= 0 && e.y < b.S, b.acc + BACC_STATUS)) continue;   // warp-uniform
        const TourDev td = b.tours[e.x];
        const DT *dem = reinterpret_cast<const DT *>(td.demand);
        WarpResult r = warp_walk_scenario<DT>(td.tab, td.n, td.Q, td.L, td.g0, dem, td.ld, e.y, s_walk[w],
                                              b.acc + BACC_STATUS);
        if (r.wide)
            r = warp_split_scenario<DT>(td.tab, td.n, td.Q, td.L, td.g0, dem, td.ld, e.y, P, g, b.acc + BACC_STATUS);
        if (lane == 0) {
            if (r.neg) atomicOr(tacc + 3 * e.x + 2, (unsigned long long)ST_NEGATIVE_DEMAND);
            if (r.bad) atomicAdd(tacc + 3 * e.x + 1, 1ull);
            else atomicAdd(tacc + 3 * e.x, (unsigned long long)r.cost);
            if (td.out_cost) td.out_cost[e.y] = r.cost;
        }
    }
}

// Warps of a block whose prefix loads and values fit beside the register
// walk's static arrays.
static int warps_for(size_t per_warp, int max_smem)
{
    int warps = 4;
    max_smem -= (int)(4 * sizeof(WalkSmem)) + 1024;
    while (warps > 1 && (size_t)warps * per_warp > (size_t)max_smem) --warps;
    return per_warp > (size_t)max_smem ? 0 : warps;
}

cudaError_t launch_split_warp(const SplitParams &p, int esize, const int32_t *list,
                              const unsigned long long *count, int grid_ctas, int max_smem,
                              cudaStream_t stream)
{
    const size_t per_warp = split_warp_smem_per_warp(p.n);
    const int warps = warps_for(per_warp, max_smem);
    if (!warps) return cudaErrorInvalidValue;
    const int threads = 32 * warps;
    const size_t smem = (size_t)warps * per_warp;
    if (esize == 2) {
        auto k = split_warp_kernel<int16_t>;
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        k<<<grid_ctas, threads, smem, stream>>>(p, list, count);
    } else {
        auto k = split_warp_kernel<int32_t>;
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        k<<<grid_ctas, threads, smem, stream>>>(p, list, count);
    }
    return cudaGetLastError();
}

cudaError_t launch_split_warp_batch(const BatchParams &b, int esize, int grid_ctas, int max_smem, bool configure_only,
                                    cudaStream_t stream)
{
    const size_t per_warp = split_warp_smem_per_warp(b.max_n);
    const int warps = warps_for(per_warp, max_smem);
    if (!warps) return cudaErrorInvalidValue;
    const size_t smem = (size_t)warps * per_warp;
    auto k = esize == 2 ? split_warp_batch_kernel<int16_t> : split_warp_batch_kernel<int32_t>;
    if (configure_only)
        return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    k<<<grid_ctas, 32 * warps, smem, stream>>>(b);
    return cudaGetLastError();
}

cudaError_t launch_split_deque(const SplitParams &p, int esize, const DequeShape &shape,
                               cudaStream_t stream)
{
    const bool cap = p.L < p.n;
    if (esize == 2) return cap ? launch_split_deque_i16_cap(p, shape, stream)
                               : launch_split_deque_i16_nocap(p, shape, stream);
    return cap ? launch_split_deque_i32_cap(p, shape, stream)
               : launch_split_deque_i32_nocap(p, shape, stream);
}

cudaError_t launch_split_host(const SplitParams &p, int esize, cudaStream_t stream)
{
    const bool cap = p.L < p.n;
    if (esize == 2) return cap ? launch_split_host_i16_cap(p, stream) : launch_split_host_i16_nocap(p, stream);
    return cap ? launch_split_host_i32_cap(p, stream) : launch_split_host_i32_nocap(p, stream);
}

}  // namespace cvrpsd
