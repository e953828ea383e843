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
__device__ __forceinline__ void walk_chunk(const int *lo32, const int *c32, int n, int i0, int &v0, int &v1, int &pl)
{
    constexpr int kNone = INT32_MAX;
    constexpr unsigned kAll = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const bool odd = lane & 1, high = lane & 2;
    const int4 *lo = reinterpret_cast<const int4 *>(lo32), *c = reinterpret_cast<const int4 *>(c32);
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

// One scenario's positions prepared by a (full) warp, 32 at a time, one per
// lane: demands (loaded a chunk ahead) are scanned to prefix loads, and each
// lane finds its position's window start by bisection over the prefix loads
// kept in shared memory.
template <typename DT>
struct WalkPrep {
    static constexpr unsigned kAll = 0xffffffffu;
    const TourStep *__restrict__ tab;
    int n, Q, L;
    const DT *__restrict__ dem;
    long long ld, s;
    unsigned long long *status;
    int *P;                                                    // kWalkRing prefix loads, this warp's
    TourStep t0, t1;                                           // table entries of this chunk and the next
    int q, carry;
    bool neg, bad;

    __device__ __forceinline__ TourStep step_of(int i) const
    {
        const TourStep none{0, 0};
        return i <= n ? tab[i - 1] : none;
    }
    __device__ __forceinline__ int demand_of(const TourStep &t, int i) const
    {
        const int row = t.row & kRowMask;
        return i <= n && index_ok(row < n && s >= 0 && s < ld, status) ? (int)__ldg(dem + (long long)row * ld + s) : 0;
    }
    __device__ __forceinline__ void start()
    {
        const int lane = threadIdx.x & 31;
        t0 = step_of(1 + lane);
        t1 = step_of(33 + lane);
        q = demand_of(t0, 1 + lane);
        carry = 0;
        neg = bad = false;
        __syncwarp();                                          // the previous scenario's readers are done
        if (lane == 0) P[0] = 0;
    }
    // The chunk from i0: window starts to lo, C_i to c. False (uniformly) if the
    // scenario has no cost (bad) or a window longer than kWalkWidth.
    __device__ __forceinline__ bool chunk(int i0, int *lo_out, int *c_out, bool &plain)
    {
        const int lane = threadIdx.x & 31, i = i0 + lane;
        const TourStep t2 = step_of(i + 64);
        const int qn = demand_of(t1, i + 32);
        neg |= q < 0;
        bad |= q > Q;
        int p = max(q, 0);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(kAll, p, o);
            if (lane >= o) p += u;
        }
        p += carry;
        carry = __shfl_sync(kAll, p, 31);
        P[i & (kWalkRing - 1)] = p;
        __syncwarp();
        const int first = max(0, i - L);                       // the route-length limit's start
        const int before = i - kWalkWidth - 1;
        const bool wide = i <= n && before >= first && p - P[before & (kWalkRing - 1)] <= Q;
        // a scenario with a demand above Q has no cost; one with a longer window is not for this walk
        if (__any_sync(kAll, wide | bad)) return false;
        int lo = max(first, i - kWalkWidth), hi = i - 1;       // hi is always in the window
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const int mid = (lo + hi) >> 1;
            const bool in = p - P[mid & (kWalkRing - 1)] <= Q;
            hi = in ? mid : hi;
            lo = in ? lo : mid + 1;
        }
        // positions past n (the last chunk) have an empty window
        lo_out[lane] = i <= n ? lo : INT32_MAX;
        c_out[lane] = t0.c;
        plain = __all_sync(kAll, i > n || (i - lo <= 32 && lo <= i - (lane & 3)));
        t0 = t1;
        t1 = t2;
        q = qn;
        return true;
    }
    // After the last chunk, or the one that ended the walk.
    __device__ __forceinline__ void finish(bool ended, bool &any_neg, bool &any_bad)
    {
        any_bad = __any_sync(kAll, bad);
        if (ended && any_bad)                                  // a negative demand anywhere is still reported
            for (int i = 1 + (threadIdx.x & 31); i <= n; i += 32) neg |= demand_of(step_of(i), i) < 0;
        any_neg = __any_sync(kAll, neg);
    }
};

// Evaluates scenario s of one tour with the calling (full) warp: 32 positions
// are prepared, then walked.
//
// What bounds it: the chain of a step (select, 18 clocks of reduction, four
// additions and minima, insertion) while few warps run, issue of the ALU pipe
// when many do.
template <typename DT>
__device__ __forceinline__ WarpResult warp_walk_scenario(const TourStep *__restrict__ tab, int n, int Q, int L, int g0,
                                                         const DT *__restrict__ dem, long long ld, long long s,
                                                         WalkSmem &w, unsigned long long *status)
{
    const int lane = threadIdx.x & 31;
    WarpResult r{INT32_MAX, false, false, false};
    WalkPrep<DT> pr{tab, n, Q, L, dem, ld, s, status, w.P};
    pr.start();
    int v0 = lane == 31 ? g0 : INT32_MAX, v1 = INT32_MAX, pl = lane == 31 ? 0 : -kWalkWidth;
    bool ended = false;
    for (int i0 = 1; i0 <= n; i0 += 32) {
        bool plain;
        if (!pr.chunk(i0, w.lo, w.c, plain)) {
            ended = true;
            break;
        }
        __syncwarp();
        if (plain) walk_chunk<true>(w.lo, w.c, n, i0, v0, v1, pl);
        else walk_chunk<false>(w.lo, w.c, n, i0, v0, v1, pl);
    }
    pr.finish(ended, r.neg, r.bad);
    r.wide = ended && !r.bad;
    const int cost = __shfl_sync(0xffffffffu, v0, (n - 1) & 31);
    if (!ended) r.cost = cost;
    return r;
}

// A set-aside scenario with the calling (full) warp: a demand above Q, which
// takes no walk, is looked for first, with its loads in flight together (n = 200,
// 108,613 of 120,000 infeasible: 451 -> 267 us per call; 3 % more where a batch
// sets many feasible ones aside, 1529 -> 1575 us).
template <typename DT>
__device__ __forceinline__ WarpResult warp_aside_scenario(const TourStep *__restrict__ tab, int n, int Q, int L, int g0,
                                                          const DT *__restrict__ dem, long long ld, long long s,
                                                          WalkSmem &w, unsigned long long *status)
{
    bool neg = false, bad = false;
#pragma unroll 4
    for (int i = threadIdx.x & 31; i < n; i += 32) {
        const int row = tab[i].row & kRowMask;
        const int q = index_ok(row < n && s >= 0 && s < ld, status) ? (int)__ldg(dem + (long long)row * ld + s) : 0;
        neg |= q < 0;
        bad |= q > Q;
    }
    if (__any_sync(0xffffffffu, bad)) return WarpResult{INT32_MAX, true, (bool)__any_sync(0xffffffffu, neg), false};
    return warp_walk_scenario<DT>(tab, n, Q, L, g0, dem, ld, s, w, status);
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
        if (list && s < 0) continue;                         // settled by split_list_kernel (warp-uniform)
        if (!index_ok(s >= 0 && s < p.S, p.acc + ACC_STATUS)) continue;   // warp-uniform
        WarpResult r{};
        r.wide = true;
        if (!p.pred) r = warp_aside_scenario<DT>(p.tab, n, p.Q, p.L, p.g0, dem, p.ld, s, s_walk[w], p.acc + ACC_STATUS);
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

// The register walk with a second warp that prepares the next 32 positions
// while the first walks these: a block is one scenario, and the two meet at a
// barrier per chunk.
//
// What bounds it: the walking warp's chain (see above), which one warp alone
// interrupts for the 37 % of its time that a chunk's preparation takes. A call
// with n = 1000, S = 37 takes 67 us, 78 without the second warp.
__device__ __forceinline__ void pair_sync() { asm volatile("bar.sync 1, 64;" ::: "memory"); }

template <typename DT>
__global__ void __launch_bounds__(64) split_walk_pair_kernel(SplitParams p)
{
    __shared__ int s_prefix[kWalkRing];
    __shared__ __align__(16) int s_lo[2][32], s_c[2][32];
    __shared__ int s_mode[2];                                  // 0 ended, 1 general, 2 plain
    __shared__ int s_flags;                                    // 1 negative demand, 2 demand above Q
    const int lane = threadIdx.x & 31, n = p.n;
    const long long s = blockIdx.x;
    const bool prepares = threadIdx.x >= 32;
    const int chunks = (n + 31) >> 5;
    int v0 = lane == 31 ? p.g0 : INT32_MAX, v1 = INT32_MAX, pl = lane == 31 ? 0 : -kWalkWidth;
    bool ended = false;
    if (prepares) {
        WalkPrep<DT> pr{p.tab, n, p.Q, p.L, reinterpret_cast<const DT *>(p.demand), p.ld, s, p.acc + ACC_STATUS, s_prefix};
        pr.start();
        for (int k = 0; k < chunks && !ended; ++k) {
            bool plain = false;
            ended = !pr.chunk(1 + 32 * k, s_lo[k & 1], s_c[k & 1], plain);
            if (lane == 0) s_mode[k & 1] = ended ? 0 : plain ? 2 : 1;
            pair_sync();                                       // chunk k is there, chunk k - 1 walked
        }
        bool neg, bad;
        pr.finish(ended, neg, bad);
        if (lane == 0) s_flags = (neg ? 1 : 0) | (bad ? 2 : 0);
    } else {
        for (int k = 0; k < chunks; ++k) {
            pair_sync();
            const int mode = s_mode[k & 1];
            if (mode == 2) walk_chunk<true>(s_lo[k & 1], s_c[k & 1], n, 1 + 32 * k, v0, v1, pl);
            else if (mode == 1) walk_chunk<false>(s_lo[k & 1], s_c[k & 1], n, 1 + 32 * k, v0, v1, pl);
            else {
                ended = true;
                break;
            }
        }
    }
    __syncthreads();
    const int cost = __shfl_sync(0xffffffffu, v0, (n - 1) & 31);
    long long sum = 0;
    unsigned inf = 0, status = 0;
    if (threadIdx.x == 0) {
        const int flags = s_flags;
        if (ended && !(flags & 2)) {                           // a long window: set aside
            const unsigned long long idx = atomicAdd(p.acc + ACC_OVERFLOW, 1ull);
            if (index_ok(idx < (unsigned long long)p.S, p.acc + ACC_STATUS)) p.ovf_list[idx] = (int32_t)s;
        } else {
            if (flags & 1) status = ST_NEGATIVE_DEMAND;
            if (ended) inf = 1; else sum = cost;
            if (p.out_cost) p.out_cost[s] = ended ? INT32_MAX : cost;
        }
    }
    if (status) atomicOr(p.sticky, (unsigned long long)status);
    block_accumulate(sum, inf, status, p.acc);
    block_finish(p.acc, p.done);
}

cudaError_t launch_split_walk(const SplitParams &p, int esize, int sm_count, cudaStream_t stream)
{
    // Pairs while each scenario can have a walking warp's scheduler to itself;
    // more of them fill the preparation's gaps with other scenarios (n = 1000, us
    // per call alone / in pairs: S = 600 78.9, 69.9; 1000 82, 82; 2000 96.7, 100).
    if (p.S <= 4LL * sm_count) {
        if (esize == 2) split_walk_pair_kernel<int16_t><<<(unsigned)p.S, 64, 0, stream>>>(p);
        else split_walk_pair_kernel<int32_t><<<(unsigned)p.S, 64, 0, stream>>>(p);
        return cudaGetLastError();
    }
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
        WarpResult r = warp_aside_scenario<DT>(td.tab, td.n, td.Q, td.L, td.g0, dem, td.ld, e.y, s_walk[w],
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

// A part of a tour table as a launch's parameters (at most 32764 bytes).
constexpr int kTabPart = 2040;
struct TabPart {
    TourStep e[kTabPart];
};

__global__ void store_table_kernel(const __grid_constant__ TabPart part, TourStep *out, int count)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < count) out[k] = part.e[k];
}

cudaError_t launch_store_table(const TourStep *tab, int n, TourStep *d_tab, cudaStream_t stream)
{
    static thread_local TabPart part;
    for (int at = 0; at < n; at += kTabPart) {
        const int count = n - at < kTabPart ? n - at : kTabPart;
        for (int k = 0; k < count; ++k) part.e[k] = tab[at + k];
        store_table_kernel<<<(count + 127) / 128, 128, 0, stream>>>(part, d_tab + at, count);
    }
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

cudaError_t launch_split_list(const SplitParams &p, long long count, int esize, cudaStream_t stream)
{
    const bool cap = p.L < p.n;
    if (esize == 2) return cap ? launch_split_list_i16_cap(p, count, stream) : launch_split_list_i16_nocap(p, count, stream);
    return cap ? launch_split_list_i32_cap(p, count, stream) : launch_split_list_i32_nocap(p, count, stream);
}

}  // namespace cvrpsd
