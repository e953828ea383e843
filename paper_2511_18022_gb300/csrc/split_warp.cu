// Transition-parallel Split: one warp evaluates one scenario (the second
// level of parallelism of Section 3: the candidate predecessors of a position). For each position i the 32 lanes take the
// candidates p of the feasible window [mask(i), i-1] of Eq. 2/3 in a strided
// pattern and a warp min-reduction picks the best, so the cost per position
// is O(|window| / 32 + log 32) and no candidate bound is needed. It serves
// calls of up to 8192 scenarios, the scenarios the deque kernel sets aside, and any
// tour when forced.
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
// Where L and n allow longer windows, the walk of a whole call (split_walk_*)
// also keeps the prefix loads and values of older positions in shared memory,
// the values as suffix minima of their 32 positions, and adds the minimum of
// a window's older part to each reduction (see WalkPrep).
#include <stdint.h>

#include "kernels.h"
#include "split_deque.cuh"
#include "tour_table.h"

namespace cvrpsd {

struct WarpResult {
    int cost;      // f(n), INT32_MAX if infeasible
    bool bad;      // some demand > Q
    bool neg;      // some demand < 0
    bool wide;     // register walk only: a window longer than it holds, no cost
};

constexpr int kWalkWidth = 64;       // candidates held in registers
constexpr int kWalkRing = 128;       // prefix loads kept: 32 of this chunk, 65 before it

// One warp's shared memory of the register walk.
struct __align__(16) WalkSmem {
    int P[kWalkRing];                // prefix loads of positions i, slot i mod 128
    int lo[32], c[32];               // window start and C_i of the chunk's positions
};

// What a walk reads and writes there. FAR walks, whose windows may be longer
// than kWalkWidth, have rings of `ring` prefix loads and values (slot i & mask),
// and the minima of the chunk's windows before the values in registers.
struct WalkStore {
    int *P, *lo, *c;
    int *a, *g;
    WalkRing ring;
};

// How a prepared chunk is walked.
enum WalkMode { WALK_ENDED, WALK_GENERAL, WALK_PLAIN, WALK_FAR, WALK_SCAN };

// The recursion over the positions i0 .. min(n, i0 + 31) of a chunk, four to
// a step. The value of position p lives in lane (p - 1) mod 32: v0 the latest
// there (position pl), v1 the one 32 positions earlier. The window starts do
// not depend on g, so the minima of a step's four windows over the values
// known before it are four independent warp reductions; the values of the
// step itself are added on uniform registers. PLAIN: no window of the chunk
// is longer than 32 positions or starts inside its own step. FAR: some window
// is longer than kWalkWidth; a32 holds the minima of the positions' windows
// up to i0 - 33, and the registers always reach back to i0 - 36 or further.
template <int MODE>
__device__ __forceinline__ void walk_chunk(const int *lo32, const int *c32, const int *a32, int n, int i0, int &v0,
                                           int &v1, int &pl)
{
    constexpr bool PLAIN = MODE == WALK_PLAIN, FAR = MODE == WALK_FAR;
    constexpr int kNone = INT32_MAX;
    constexpr unsigned kAll = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const bool odd = lane & 1, high = lane & 2;
    const int4 *lo = reinterpret_cast<const int4 *>(lo32), *c = reinterpret_cast<const int4 *>(c32);
    const int4 *a = reinterpret_cast<const int4 *>(a32);
    int4 l4 = lo[0], c4 = c[0], a4 = FAR ? a[0] : make_int4(0, 0, 0, 0);
#pragma unroll
    for (int b = 0; b < 8; ++b) {
        const int ib = i0 + 4 * b;
        if (b > 0 && ib > n) break;
        const int4 ln = lo[(b + 1) & 7], cn = c[(b + 1) & 7], an = FAR ? a[(b + 1) & 7] : a4;
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
        if (FAR) {
            m0 = min(m0, a4.x);
            m1 = min(m1, a4.y);
            m2 = min(m2, a4.z);
            m3 = min(m3, a4.w);
        }
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
        a4 = an;
    }
}

// The same for a chunk whose windows all start at i0 or before: with A_i the
// minimum of position i's window before i0 and m_i that of the chunk's values up
// to i, m_i = min(m_{i-1} + min(C_i, 0), A_i + C_i): a warp scan of such pairs
// gives all positions at once, for a fifth of the instructions of eight steps
// (calls with n = 1000, windows of 70: S = 8192 288 us by steps, 199 by scans;
// S = 1000 108, 88; S = 37, where the preparing warp is the slower one, 81, 77).
__device__ __forceinline__ void scan_chunk(const WalkStore &w, int i0, int &v0, int &v1, int &pl)
{
    constexpr int kFar = 1 << 30;                              // above all values; sums with C_i stay in range
    constexpr unsigned kAll = 0xffffffffu;
    const int lane = threadIdx.x & 31, lo = w.lo[lane], c = w.c[lane];
    int m = v0;                                                // position i0 - 32 + lane
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_down_sync(kAll, m, o);
        if (lane + o < 32) m = min(m, u);
    }
    m = __shfl_sync(kAll, m, max(lo - (i0 - 32), 0) & 31);
    const int A = min(kFar, min(w.a[lane], lo < i0 ? m : kFar));
    int shift = min(c, 0), best = A + c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int us = __shfl_up_sync(kAll, shift, o), ub = __shfl_up_sync(kAll, best, o);
        if (lane >= o) {
            best = min(best, ub + shift);
            shift += us;
        }
    }
    const int before = __shfl_up_sync(kAll, best, 1);
    v1 = v0;
    v0 = c + (lane ? min(A, before) : A);
    pl = i0 + lane;
}

// A chunk in the mode its preparation found, and (FAR) its values to the ring.
template <bool FAR>
__device__ __forceinline__ void walk_chunk(int mode, const WalkStore &w, int n, int i0, int &v0, int &v1, int &pl)
{
    if (mode == WALK_PLAIN) walk_chunk<WALK_PLAIN>(w.lo, w.c, w.a, n, i0, v0, v1, pl);
    else if (!FAR || mode == WALK_GENERAL) walk_chunk<WALK_GENERAL>(w.lo, w.c, w.a, n, i0, v0, v1, pl);
    else if (mode == WALK_SCAN) scan_chunk(w, i0, v0, v1, pl);
    else walk_chunk<WALK_FAR>(w.lo, w.c, w.a, n, i0, v0, v1, pl);
    if (FAR) w.g[(i0 + (int)(threadIdx.x & 31)) & w.ring.mask] = v0;
}

// One scenario's positions prepared by a (full) warp, 32 at a time, one per
// lane: demands (loaded a chunk ahead) are scanned to prefix loads, and each
// lane finds its position's window start by bisection over the prefix loads
// kept in shared memory.
//
// FAR: where a chunk holds a window longer than kWalkWidth, the values of
// positions up to i0 - 33 (the walk of the chunk before this one may still be
// under way) are turned into suffix minima of their chunks of 32, each chunk
// once, and a lane's minimum over its window there is the suffix from the
// window's start and the minima of the whole chunks after it.
template <typename DT, bool FAR>
struct WalkPrep {
    static constexpr unsigned kAll = 0xffffffffu;
    const TourStep *__restrict__ tab;
    int n, Q, L;
    const DT *__restrict__ dem;
    long long ld, s;
    unsigned long long *status;
    WalkStore w;
    TourStep t0, t1;                                           // table entries of this chunk and the next
    int q, carry;
    int suffixes;                                              // chunks before this one hold suffix minima
    bool neg, bad;

    __device__ __forceinline__ int slot(int p) const { return p & (FAR ? w.ring.mask : kWalkRing - 1); }
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
        suffixes = -1;
        neg = bad = false;
        __syncwarp();                                          // the previous scenario's readers are done
        if (lane == 0) w.P[0] = 0;
    }
    // Minimum of the window from lo (INT32_MAX: none) over the positions up to i0 - 33.
    __device__ __forceinline__ int older(int i0, int lo)
    {
        const int lane = threadIdx.x & 31, last = ((i0 - 1) >> 5) - 2;
        const int from = (__shfl_sync(kAll, lo, 0) - 1) >> 5;  // window starts never move back
        for (int k = max(suffixes, from); k <= last; ++k) {
            const int p = 32 * k + 1 + lane;                   // chunk -1 holds position 0 alone
            int v = p >= 0 ? w.g[slot(p)] : INT32_MAX;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_down_sync(kAll, v, o);
                if (lane + o < 32) v = min(v, u);
            }
            if (p >= 0) w.g[slot(p)] = v;
        }
        suffixes = last + 1;
        __syncwarp();
        int m = lo <= i0 - 33 ? w.g[slot(lo)] : INT32_MAX;
        for (int k = from + 1; k <= last; ++k) {
            const int whole = w.g[slot(32 * k + 1)];
            if (k > (lo - 1) >> 5) m = min(m, whole);
        }
        return m;
    }
    // The chunk from i0: window starts, C_i and (FAR) older minima to shared memory.
    // WALK_ENDED (uniformly) if the scenario has no cost (bad) or a window too long.
    __device__ __forceinline__ int chunk(int i0)
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
        w.P[slot(i)] = p;
        __syncwarp();
        const int first = max(0, i - L);                       // the route-length limit's start
        const auto beyond = [&](int width) {                   // the window is longer than width
            const int before = i - width - 1;
            return i <= n && before >= first && p - w.P[slot(before)] <= Q;
        };
        const bool wide = beyond(kWalkWidth);
        // a scenario with a demand above Q has no cost; one with a longer window is not for this walk
        bool far = __any_sync(kAll, wide | bad);
        if (far && (!FAR || __any_sync(kAll, bad || beyond(w.ring.width)))) return WALK_ENDED;
        int lo = max(first, i - (far ? w.ring.width : kWalkWidth)), hi = i - 1;       // hi is always in the window
        const auto halve = [&]() {
            const int mid = (lo + hi) >> 1;
            const bool in = p - w.P[slot(mid)] <= Q;
            hi = in ? mid : hi;
            lo = in ? lo : mid + 1;
        };
        if (far)
            for (int k = 32 - __clz(w.ring.width); k > 6; --k) halve();
#pragma unroll
        for (int k = 0; k < 6; ++k) halve();
        // positions past n (the last chunk) have an empty window
        if (i > n) lo = INT32_MAX;
        w.lo[lane] = lo;
        w.c[lane] = t0.c;
        const bool plain = __all_sync(kAll, i > n || (i - lo <= 32 && lo <= i - (lane & 3)));
        const bool scan = FAR && !plain && __all_sync(kAll, i > n || lo <= i0);
        if (far || scan) w.a[lane] = older(i0, lo);
        t0 = t1;
        t1 = t2;
        q = qn;
        return scan ? WALK_SCAN : far ? WALK_FAR : plain ? WALK_PLAIN : WALK_GENERAL;
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
template <typename DT, bool FAR>
__device__ __forceinline__ WarpResult warp_walk_scenario(const TourStep *__restrict__ tab, int n, int Q, int L, int g0,
                                                         const DT *__restrict__ dem, long long ld, long long s,
                                                         const WalkStore &w, unsigned long long *status)
{
    const int lane = threadIdx.x & 31;
    WarpResult r{INT32_MAX, false, false, false};
    WalkPrep<DT, FAR> pr{tab, n, Q, L, dem, ld, s, status, w};
    pr.start();
    if (FAR && lane == 0) w.g[0] = g0;
    int v0 = lane == 31 ? g0 : INT32_MAX, v1 = INT32_MAX, pl = lane == 31 ? 0 : -kWalkWidth;
    bool ended = false;
    for (int i0 = 1; i0 <= n; i0 += 32) {
        const int mode = pr.chunk(i0);
        if (mode == WALK_ENDED) {
            ended = true;
            break;
        }
        __syncwarp();
        walk_chunk<FAR>(mode, w, n, i0, v0, v1, pl);
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
    return warp_walk_scenario<DT, false>(tab, n, Q, L, g0, dem, ld, s, WalkStore{w.P, w.lo, w.c}, status);
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

// Whether the scenarios of a warp's lanes (s < 0: none) hold a demand above Q, one
// lane each: the rows in tour order, so that all warps read the same few rows at
// a time and neighbours on the list share their sectors.
template <typename DT>
__device__ __forceinline__ void scan_lanes(const TourStep *__restrict__ tab, int n, int Q, const DT *__restrict__ dem,
                                           long long ld, long long s, bool &neg, bool &bad, unsigned long long *status)
{
    neg = bad = false;
    if (s < 0) return;
#pragma unroll 8
    for (int i = 0; i < n; ++i) {
        const int row = tab[i].row & kRowMask;
        const int q = index_ok(row < n && s < ld, status) ? (int)__ldg(dem + (long long)row * ld + s) : 0;
        neg |= q < 0;
        bad |= q > Q;
    }
}

// A warp's share of the list from which its lanes look for demands above Q, each in
// a scenario of its own, once the first of the share has one (why a scenario is
// listed, that or a long deque, the list doesn't say). Calls that enqueue, scenarios
// listed for such a demand, a warp each and by lanes: n = 1000, S = 500,000, 136,017
// listed 3404 us, 1251; S = 200,000, 54,320 1116, 597; n = 200, S = 1,000,000,
// 126,039 563, 400. Four a warp: n = 1000, S = 500,000, 17,300 listed 1134, 1113;
// n = 200, S = 140,000, 17,318 106, 113. Listed for their deques, n = 1000: 476,146
// of 500,000 14.0 ms, 12.5; 133,460 of 140,000 3297 us, 3534.
constexpr int kScanItems = 6;

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
    const auto settle = [&](long long s, WarpResult r) {     // r.wide: not walked yet
        if (r.wide)
            r = warp_split_scenario<DT>(p.tab, n, p.Q, p.L, p.g0, dem, p.ld, s, P, g, p.acc + ACC_STATUS, p.pred,
                                        p.ldp);
        if (lane == 0) {
            if (r.neg) status |= ST_NEGATIVE_DEMAND;
            if (r.bad) ++inf; else sum += r.cost;
            if (p.out_cost) p.out_cost[s] = r.cost;
        }
    };
    const long long warps = (long long)gridDim.x * wpb, first = (long long)blockIdx.x * wpb + w;
    const long long share = (total + warps - 1) / warps;
    if (list && !p.pred && share >= kScanItems) {
        const long long rounds = (share + 31) / 32;
        const int items = (int)((share + rounds - 1) / rounds);
        // a block's warps take neighbours at the same time: they share sectors
        for (long long base = (long long)blockIdx.x * wpb * items; base < total; base += warps * items) {
            const long long at = base + lane * wpb + w;
            long long mine = lane < items && at < total ? (long long)list[at] : -1;
            if (!index_ok(mine < p.S, p.acc + ACC_STATUS)) mine = -1;
            unsigned left = __ballot_sync(0xffffffffu, mine >= 0);
            bool begun = false, scan = false, scanned = false;
            while (left) {
                if (scan && !scanned) {
                    bool neg, bad;
                    scan_lanes<DT>(p.tab, n, p.Q, dem, p.ld, (left >> lane) & 1u ? mine : -1, neg, bad, p.acc + ACC_STATUS);
                    if (neg) status |= ST_NEGATIVE_DEMAND;
                    if (bad) {
                        ++inf;
                        if (p.out_cost) p.out_cost[mine] = INT32_MAX;
                    }
                    left &= ~__ballot_sync(0xffffffffu, bad);
                    scanned = true;
                    continue;
                }
                const long long s = __shfl_sync(0xffffffffu, mine, __ffs(left) - 1);
                left &= left - 1;
                const WarpResult r = scanned ? warp_walk_scenario<DT, false>(p.tab, n, p.Q, p.L, p.g0, dem, p.ld, s,
                                                   WalkStore{s_walk[w].P, s_walk[w].lo, s_walk[w].c}, p.acc + ACC_STATUS)
                                             : warp_aside_scenario<DT>(p.tab, n, p.Q, p.L, p.g0, dem, p.ld, s, s_walk[w],
                                                                       p.acc + ACC_STATUS);
                if (!begun) scan = r.bad;
                begun = true;
                settle(s, r);
            }
        }
    } else {
        for (long long item = first; item < total; item += warps) {
            const long long s = list ? (long long)list[item] : item;
            if (list && s < 0) continue;                     // settled by split_list_kernel (warp-uniform)
            if (!index_ok(s >= 0 && s < p.S, p.acc + ACC_STATUS)) continue;   // warp-uniform
            WarpResult r{};
            r.wide = true;
            if (!p.pred) r = warp_aside_scenario<DT>(p.tab, n, p.Q, p.L, p.g0, dem, p.ld, s, s_walk[w], p.acc + ACC_STATUS);
            settle(s, r);
        }
    }
    inf = __reduce_add_sync(0xffffffffu, inf);
    status = __reduce_or_sync(0xffffffffu, status);
    if (lane == 0) {
        if (sum) atomicAdd(p.acc + ACC_SUM, (unsigned long long)sum);
        if (inf) atomicAdd(p.acc + ACC_INFEASIBLE, (unsigned long long)inf);
        if (status) {
            atomicOr(p.acc + ACC_STATUS, (unsigned long long)status);
            atomicOr(p.sticky, (unsigned long long)status);
        }
    }
    if (p.done) {
        __syncthreads();                                     // the block's additions are done
        block_finish(p.acc, p.done, true);
    }
}

// The register walk alone, one scenario per warp: a scenario with a window
// longer than it holds goes on the list (for split_warp_kernel). FAR: windows
// of up to ring.width, with the rings in dynamic shared memory.
constexpr int kWalkWarps = 4;

template <typename DT, bool FAR>
__global__ void __launch_bounds__(32 * kWalkWarps) split_walk_kernel(SplitParams p, WalkRing ring)
{
    extern __shared__ __align__(16) int wsmem[];
    __shared__ __align__(16) int s_P[FAR ? 1 : kWalkWarps][FAR ? 4 : kWalkRing];
    __shared__ __align__(16) int s_lo[kWalkWarps][32], s_c[kWalkWarps][32], s_a[FAR ? kWalkWarps : 1][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const long long s = (long long)blockIdx.x * kWalkWarps + w;
    int *far = wsmem + (FAR ? w * 2 * ring.size : 0);
    const WalkStore store{FAR ? far : s_P[FAR ? 0 : w], s_lo[w], s_c[w], s_a[FAR ? w : 0], far + ring.size, ring};
    long long sum = 0;
    unsigned inf = 0, status = 0;
    if (s < p.S) {
        const WarpResult r = warp_walk_scenario<DT, FAR>(p.tab, p.n, p.Q, p.L, p.g0, reinterpret_cast<const DT *>(p.demand),
                                                         p.ld, s, store, p.acc + ACC_STATUS);
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

template <typename DT, bool FAR>
__global__ void __launch_bounds__(64) split_walk_pair_kernel(SplitParams p, WalkRing ring)
{
    extern __shared__ __align__(16) int wsmem[];
    __shared__ int s_prefix[FAR ? 1 : kWalkRing];
    __shared__ __align__(16) int s_lo[2][32], s_c[2][32], s_a[FAR ? 2 : 1][32];
    __shared__ int s_mode[2];                                  // WalkMode
    __shared__ int s_flags;                                    // 1 negative demand, 2 demand above Q
    const int lane = threadIdx.x & 31, n = p.n;
    const long long s = blockIdx.x;
    const bool prepares = threadIdx.x >= 32;
    const int chunks = (n + 31) >> 5;
    const auto store = [&](int k) {
        return WalkStore{FAR ? wsmem : s_prefix, s_lo[k & 1], s_c[k & 1], s_a[FAR ? k & 1 : 0], wsmem + ring.size, ring};
    };
    int v0 = lane == 31 ? p.g0 : INT32_MAX, v1 = INT32_MAX, pl = lane == 31 ? 0 : -kWalkWidth;
    bool ended = false;
    if (prepares) {
        WalkPrep<DT, FAR> pr{p.tab, n, p.Q, p.L, reinterpret_cast<const DT *>(p.demand), p.ld, s, p.acc + ACC_STATUS,
                             store(0)};
        pr.start();
        for (int k = 0; k < chunks && !ended; ++k) {
            pr.w = store(k);
            const int mode = pr.chunk(1 + 32 * k);
            ended = mode == WALK_ENDED;
            if (lane == 0) s_mode[k & 1] = mode;
            pair_sync();                                       // chunk k is there, chunk k - 1 walked
        }
        bool neg, bad;
        pr.finish(ended, neg, bad);
        if (lane == 0) s_flags = (neg ? 1 : 0) | (bad ? 2 : 0);
    } else {
        if (FAR && lane == 0) wsmem[ring.size] = p.g0;
        for (int k = 0; k < chunks; ++k) {
            pair_sync();
            const int mode = s_mode[k & 1];
            if (mode == WALK_ENDED) {
                ended = true;
                break;
            }
            walk_chunk<FAR>(mode, store(k), n, 1 + 32 * k, v0, v1, pl);
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

// Pairs while each scenario can have a walking warp's scheduler to itself;
// more of them fill the preparation's gaps with other scenarios (n = 1000, us
// per call alone / in pairs: S = 600 78.9, 69.9; 1000 82, 82; 2000 96.7, 100).
static bool walk_in_pairs(long long S, int sm_count) { return S <= 4LL * sm_count; }

// All positions (no slot is used twice) or a power of two that holds a window,
// the chunk being prepared and the one being walked, whichever is less; where
// that leaves fewer than kWalkResident scenarios resident, the largest power of two
// that does not. Six blocks of four warps hold 1004 positions: n = 1000, L = n and
// windows of 13 then take 131 us at S = 4096 (120 with the registers alone, whose
// 13 resident blocks cannot finish a longer window) and 194 (182) at S = 8192.
constexpr int kWalkResident = 3600;

WalkRing walk_ring(int n, int L, long long S, int sm_count)
{
    const int reach = n < L ? n : L, all = (n + 31) / 32 * 32 + 4, warps = walk_in_pairs(S, sm_count) ? 1 : kWalkWarps;
    if (reach <= kWalkWidth) return WalkRing{0, 0, kWalkWidth};
    const auto fits = [&](int size) {
        const size_t block = warps * 2 * (size_t)size * sizeof(int) + 3072;
        return (long long)(233472 / block) * sm_count * warps >= (S < kWalkResident ? S : kWalkResident);
    };
    int size = kWalkRing;
    while (size < reach + kWalkWidth) size *= 2;
    if (all <= size && fits(all)) return WalkRing{all, -1, n};
    while (size > kWalkRing && !fits(size)) size /= 2;
    return WalkRing{size, size - 1, size - kWalkWidth};
}

template <bool FAR>
static cudaError_t launch_walk(const SplitParams &p, int esize, const WalkRing &ring, bool pairs, cudaStream_t stream)
{
    const size_t smem = FAR ? (pairs ? 1 : kWalkWarps) * 2 * (size_t)ring.size * sizeof(int) : 0;
    const unsigned grid = pairs ? (unsigned)p.S : (unsigned)((p.S + kWalkWarps - 1) / kWalkWarps);
    auto k = pairs ? (esize == 2 ? split_walk_pair_kernel<int16_t, FAR> : split_walk_pair_kernel<int32_t, FAR>)
                   : (esize == 2 ? split_walk_kernel<int16_t, FAR> : split_walk_kernel<int32_t, FAR>);
    if (smem > 40 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    k<<<grid, pairs ? 64 : 32 * kWalkWarps, smem, stream>>>(p, ring);
    return cudaGetLastError();
}

cudaError_t launch_split_walk(const SplitParams &p, int esize, int sm_count, cudaStream_t stream)
{
    const WalkRing ring = walk_ring(p.n, p.L, p.S, sm_count);
    const bool pairs = walk_in_pairs(p.S, sm_count);
    return ring.size ? launch_walk<true>(p, esize, ring, pairs, stream) : launch_walk<false>(p, esize, ring, pairs, stream);
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

int store_table_launches(int n) { return (n + kTabPart - 1) / kTabPart; }

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
