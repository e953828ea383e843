// Internal interface of the second deque walk (split_deque2.cuh): its
// parameter blocks and launcher.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "kernels.h"
#include "tour_table.h"

namespace cvrpsd {

// Table capacities of the kernel-parameter tour table: 8 KB for tours up to
// 1024 customers, and the largest that fits the 32 KB parameter space.
constexpr int kTab2Small = 1024;
constexpr int kTab2Large = 4032;

// Tour positions per prefetch block of the second walk: its demands are
// loaded one block ahead (at full occupancy four positions hide the load
// latency, and the walk then fits 32 registers).
constexpr int kPrefetch2 = 4;

// Table entry of position i (index i - 1): x = the demand row of sigma_i in
// the low bits, plus kTab2NoBack when no scenario can pop the deque's back
// at i (C_{i-1} > 0 and C_i > C_{i-1}, see split_deque2.cuh); y = C_i. Bit m
// of nonpos marks prefetch block m (positions 1 + m * kPrefetch2 ...) as
// holding some C_i <= 0 with i < n.
constexpr uint32_t kTab2NoBack = 1u << 31;
constexpr uint32_t kTab2RowMask = kTab2NoBack - 1u;

// Positions of a smooth tour: the last three C_i rose. Along a tour whose
// neighbours are close together (as a search makes it) C_i follows the
// distance to the depot, rises over many positions and the deques get long;
// in a random order one position in 24 is like that. Above one in 8 the walk
// is compiled for spans that need the exact per-position tests often:
// 64 strip-ordered tours of n = 200 under 65,536 scenarios 1886 -> 1471 us,
// the same tours in random order 1140 -> 1157 us.
__host__ __device__ inline bool rising(int c0, int c1, int c2, int c3) { return c1 > c0 && c2 > c1 && c3 > c2; }
__host__ __device__ inline bool smooth_table(int rises, int n) { return 8 * rises > n; }

template <int CAP>
struct TabParam {
    uint2 e[CAP];
    uint32_t nonpos[(CAP / kPrefetch2 + 31) / 32];
    static constexpr int kCap = CAP;
#ifdef __CUDACC__
    // The walk's view of a table (see TabShared2 for the batch kernel's).
    __device__ __forceinline__ uint32_t row(int i) const { return e[i - 1].x & kTab2RowMask; }
    // Flags of the span of two prefetch blocks from i0: read where they are used.
    __device__ __forceinline__ uint32_t span(int i0) const { return 0; }
    __device__ __forceinline__ bool general(uint32_t, int i0, int) const
    {
        const int m = (i0 - 1) / kPrefetch2;
        return (nonpos[m >> 5] >> (m & 31)) & 1u;
    }
    __device__ __forceinline__ bool noback(uint32_t, int i, int) const { return (e[i - 1].x & kTab2NoBack) != 0; }
    // C_i and demand rows of a prefetch block's positions.
    struct Costs {};
    __device__ __forceinline__ Costs costs(int) const { return {}; }
    __device__ __forceinline__ int cost(const Costs &, int i, int) const { return (int)e[i - 1].y; }
    struct Rows {};
    __device__ __forceinline__ Rows rows(int) const { return {}; }
    __device__ __forceinline__ uint32_t row_at(const Rows &, int i, int) const { return row(i); }
#endif
};

struct Walk2Params {
    const void *demand;        // device [n][ld]
    long long S;               // scenarios
    long long stride;          // grid * T: scenario step between a thread's rounds
    int32_t n, Q, L, g0;       // L > n: no route-length limit
    uint32_t K;                // key scale: power of two > n
    uint32_t pitch;            // bytes between demand rows
    int32_t *out_cost;         // device [S] or nullptr
    unsigned long long *acc;   // device [ACC_WORDS]
    int32_t *ovf_list;         // device [S]
    unsigned long long *status;   // device word for index-check status bits
    unsigned long long *done;     // see SplitParams
    int16_t *pred;             // device [n][ldp] or nullptr
    long long ldp;
};

// Whether the second walk can run this Split (otherwise the first walk runs):
// n <= kTab2Large, demand rows addressable with
// 32-bit byte offsets, and for int16 demands Q < 32768 (a negative demand
// read as unsigned then exceeds Q). Predecessors: int16 demands, keys that
// cannot wrap, n <= kTab2Small, and the library's choice of shape.
bool deque2_supported(const SplitParams &p, int esize);

// Launch it. `tab` is the host copy of the tour table (TourStep rows with
// the block flag); rounds = 0 gives one scenario per thread, rounds >= 1 a
// grid of ceil(tiles / rounds) blocks, each walking up to `rounds` tiles of
// T scenarios. shape.threads = 0: the library's choice. *shape_ran receives the (threads, ring) actually launched.
cudaError_t launch_split_deque2(const SplitParams &p, const TourStep *tab, int esize, const DequeShape &shape,
                                int rounds, int sm_count, DequeShape *shape_ran, cudaStream_t stream);

}  // namespace cvrpsd
