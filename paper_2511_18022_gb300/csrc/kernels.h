// Internal interface between the C ABI (api.cu) and the CUDA kernels.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace cvrpsd {

// Accumulator words written by the Split kernels (device). The first
// ACC_WORDS are zeroed per call; ACC_STICKY collects the status bits of every
// call until the host reads and clears it (cvrpsd_check_inputs), so that a
// call that returned without waiting still has its input errors reported.
//
// A call that returns host outputs and runs one kernel uses a second set of
// these words that is zero between calls: the kernel's last block (by
// ACC_TICKET) hands the totals to the host and clears them again, so the call
// is that one launch (see block_finish).
enum AccWord { ACC_SUM = 0, ACC_INFEASIBLE = 1, ACC_OVERFLOW = 2, ACC_STATUS = 3, ACC_WORDS = 4, ACC_STICKY = 4,
               ACC_TICKET = 5, ACC_ALLOC_WORDS = 8 };

// Device status bits (ACC_STATUS, and a batch's BACC_STATUS).
enum StatusBits { ST_NEGATIVE_DEMAND = 1, ST_INDEX = 2 };

// Checked build (compile with -DCVRPSD_CHECKED=1): every index a Split kernel
// forms from data (table rows, scenario columns, list entries) is compared
// with its buffer before use; a bad one sets ST_INDEX in `status` and the
// access is skipped. Nothing traps. The regular build compiles the checks
// away.
#ifndef CVRPSD_CHECKED
#define CVRPSD_CHECKED 0
#endif
#ifdef __CUDACC__
__device__ __forceinline__ bool index_ok(bool ok, unsigned long long *status)
{
#if CVRPSD_CHECKED
    if (!ok) atomicOr(status, (unsigned long long)ST_INDEX);
    return ok;
#else
    (void)status;
    (void)ok;
    return true;
#endif
}
#endif

// One tour position as the kernels read it: the demand row of sigma_i and the
// scenario-independent cost term C_i (see api.cu: C_i = c(sigma_i,0) +
// c(0,sigma_{i+1}) - c(sigma_i,sigma_{i+1}) for i < n, and for i = n the full
// tail D[n] + c(sigma_n, 0)).
struct TourStep {
    int32_t row;
    int32_t c;
};

struct SplitParams {
    const TourStep *tab;          // device [n]
    const void *demand;           // device [n][ld]
    int64_t ld;                   // row pitch, elements
    int64_t S;                    // scenarios
    int32_t n, Q, L;              // L > n means no route-length limit
    int32_t g0;                   // c(0, sigma_1)
    uint32_t K;                   // key scale: power of two > n
    int32_t *out_cost;            // device [S] or nullptr
    unsigned long long *acc;      // device [ACC_WORDS]
    unsigned long long *sticky;   // device word that collects status bits over calls
    unsigned long long *done;     // page-locked host [ACC_WORDS] for the totals, or nullptr (acc keeps them)
    int32_t *ovf_list;            // device [S]: scenarios the deque could not hold
    int16_t *pred;                // device [n][ldp] or nullptr: optimal predecessor of each position
    long long ldp;
};

struct DequeShape {
    int threads;    // 64, 128, 256
    int spt;        // 1, 2
    int ring;       // 16, 32, 64
};

// Deque kernel, one thread per `spt` scenarios. esize = 2 or 4.
cudaError_t launch_split_deque(const SplitParams &p, int esize, const DequeShape &shape,
                               cudaStream_t stream);
cudaError_t launch_split_deque_i16_cap(const SplitParams &p, const DequeShape &s, cudaStream_t st);
cudaError_t launch_split_deque_i16_nocap(const SplitParams &p, const DequeShape &s, cudaStream_t st);
cudaError_t launch_split_deque_i32_cap(const SplitParams &p, const DequeShape &s, cudaStream_t st);
cudaError_t launch_split_deque_i32_nocap(const SplitParams &p, const DequeShape &s, cudaStream_t st);

// The scenarios of p.ovf_list (count of them, known to the host) by rings of 32;
// entries that are settled become -1, and ACC_TICKET (0 before) counts the others.
cudaError_t launch_split_list(const SplitParams &p, long long count, int esize, cudaStream_t stream);
cudaError_t launch_split_list_i16_cap(const SplitParams &p, long long count, cudaStream_t st);
cudaError_t launch_split_list_i16_nocap(const SplitParams &p, long long count, cudaStream_t st);
cudaError_t launch_split_list_i32_cap(const SplitParams &p, long long count, cudaStream_t st);
cudaError_t launch_split_list_i32_nocap(const SplitParams &p, long long count, cudaStream_t st);

// The same walk for scenarios in page-locked host memory (device addresses of
// it in p): 1 KB windows of the rows staged through shared memory, rings of 16.
cudaError_t launch_split_host(const SplitParams &p, int esize, cudaStream_t stream);
cudaError_t launch_split_host_i16_cap(const SplitParams &p, cudaStream_t st);
cudaError_t launch_split_host_i16_nocap(const SplitParams &p, cudaStream_t st);
cudaError_t launch_split_host_i32_cap(const SplitParams &p, cudaStream_t st);
cudaError_t launch_split_host_i32_nocap(const SplitParams &p, cudaStream_t st);

// Writes a tour table of n entries to d_tab, from the launches' own parameters:
// `tab` is free again when this returns, also under stream capture.
cudaError_t launch_store_table(const TourStep *tab, int n, TourStep *d_tab, cudaStream_t stream);
int store_table_launches(int n);

// Dynamic shared memory of the deque kernel: its rings ([spt][ring][threads] int2).
inline size_t split_deque_smem(const SplitParams &p, const DequeShape &shape)
{
    (void)p;
    return (size_t)shape.spt * shape.ring * shape.threads * 8;
}

// Blocks per SM of the pass over set-aside scenarios (four warps each; its
// registers and tours of a few hundred positions let eight be resident). 64
// tours of n = 200 in strips under 65,536 scenarios, many set aside: two blocks
// 2579 us, four 2145, eight 2024; none set aside: 0.3 us more to start them.
constexpr int kAsideBlocks = 8;

// Warp-per-scenario kernel. If `list` is non-null it evaluates the scenarios
// named in list[0 .. *count) (count lives on the device); otherwise all S.
// `max_smem` is the device's opt-in shared memory per block.
cudaError_t launch_split_warp(const SplitParams &p, int esize, const int32_t *list,
                              const unsigned long long *count, int grid_ctas, int max_smem,
                              cudaStream_t stream);
// The register walk's memory of older positions: entries of its two rings (0:
// none, no window can be longer than 64), a slot's mask, the longest window.
struct WalkRing {
    int size, mask, width;
};
WalkRing walk_ring(int n, int L, long long S, int sm_count);
// One scenario per warp by the register walk; scenarios with a window longer
// than walk_ring's go on p.ovf_list (count in ACC_OVERFLOW) for launch_split_warp.
cudaError_t launch_split_walk(const SplitParams &p, int esize, int sm_count, cudaStream_t stream);
inline size_t split_warp_smem_per_warp(int n) { return (size_t)2 * (n + 1) * sizeof(int); }
// Blocks of that pass over one tour's list: no more than are resident, since the
// list is dealt out evenly and a second wave would start when the first ends (n =
// 1000, six fit: S = 140,000 with 37,906 listed 682 -> 621 us). A batch's pass, whose tours
// differ, keeps all eight (8 tours, n = 1000, S = 200,000 in strips 41.7 ms, 44.1 by six).
inline int aside_grid(int n, int sm_count)
{
    const int fit = (int)(233472 / (4 * split_warp_smem_per_warp(n) + 4096));
    return (sm_count > 0 ? sm_count : 152) * (fit < 1 ? 1 : fit < kAsideBlocks ? fit : kAsideBlocks);
}

// ---- batches of tours (one persistent launch) ----

// One tour of a batch, as the batch kernels read it.
struct TourDev {
    const TourStep *tab;          // device [n]
    const void *demand;           // device [n][ld]
    long long ld;
    int32_t *out_cost;            // device [S] or nullptr
    int32_t n, Q, L, g0;          // L > n: no route-length limit
    uint32_t K;
    int32_t pad;
};

// Batch accumulator header; per tour three words follow: sum, infeasible
// count, status bits.
enum BatchAccWord { BACC_COUNTER = 0, BACC_LIST = 1, BACC_STATUS = 2, BACC_SMOOTH = 3, BACC_WORDS = 4 };
enum BatchStatusBits { BST_LIST_FULL = 1 };   // shares its word with ST_INDEX (2)

struct BatchParams {
    const TourDev *tours;         // device [T]
    const int2 *items;            // device [n_items]: (tour, scenario tile), in processing order;
                                  // nullptr: item = tour * tiles + tile
    int n_items;
    int tiles;                    // scenario tiles per tour (with items == nullptr)
    long long S;                  // scenarios per tour
    unsigned long long *acc;      // device [BACC_WORDS + 3 T]
    int2 *list;                   // device [list_cap]: set-aside (tour, scenario)
    long long list_cap;
    int max_n;                    // largest tour
    int walk2;                    // keys that cannot wrap in every tour (and 32-bit pitches): the
                                  // second walk runs the one-scenario-per-thread shapes
    int T;                        // tours
    int smooth;                   // second walk: 1 if most tours are smooth (smooth_table), 0 if not, -1 if only
                                  // the device knows (their number in BACC_SMOOTH)
};

// Dynamic shared memory of the batch kernel: rings, then the current tour's
// table and (second walk) a word of flags for every 8 positions.
inline size_t split_batch_smem(int max_n, const DequeShape &shape)
{
    return (size_t)shape.spt * shape.ring * shape.threads * 8 + (size_t)((max_n + 3) / 4 * 4) * sizeof(TourStep) +
           (size_t)((max_n + 7) / 8) * 4;
}
// Launch shape without a request, rings of 16: the smallest blocks that hold all
// scenarios at once (even shares for the SMs: 64 tours of 100 to 1000 customers
// under 1000 scenarios 212 us with 64 threads, 250 with 256; 8 tours under 8192
// 192 against 220), else the one with the most resident threads beside its
// table (under 8192 scenarios 428 us with 512 threads, 452 with 256, whose
// tables leave room for five blocks).
inline DequeShape batch_default_shape(int max_n, long long scenarios, int sm_count)
{
    DequeShape best{256, 1, 16};
    int most = 0;
    for (int threads : {64, 128, 256, 512}) {
        const DequeShape s{threads, 1, 16};
        const int by_smem = (int)(233472 / (split_batch_smem(max_n, s) + 1024)), by_threads = 2048 / threads;
        const int resident = (by_smem < by_threads ? by_smem : by_threads) * threads;
        if (scenarios <= (long long)resident * sm_count) return s;
        if (resident > most || (resident == most && threads <= 256)) {
            most = resident;
            best = s;
        }
    }
    return best;
}
// Persistent deque kernel over all work items; with configure_only it only
// sets the kernel's shared-memory limit (call before stream capture) and
// reports blocks per SM in *blocks_per_sm.
cudaError_t launch_split_batch(const BatchParams &b, int esize, bool lcap, const DequeShape &shape, int grid,
                               bool configure_only, int *blocks_per_sm, cudaStream_t stream);
// Shapes that the second walk has for smooth tours too: the library's own where the
// scenarios outgrow the device (n > 64), and those a tuner picks. In blocks of 64 or
// 128 threads, for scenarios that fit at once, it does not pay: batches in strips
// of 64 tours, n = 200, S = 3000 118 us by the other walk, 119; of 16 tours,
// n = 500, S = 4000 327, 317; candidate tours, whose order only the device knows,
// pay for a second launch: 64 in random order, n = 200, S = 3000 133, 141.
inline bool batch2_smooth_compiled(const DequeShape &s)
{
    return s.spt == 1 && s.ring == 16 && (s.threads == 256 || s.threads == 512);
}
// The batch kernel on the second walk (split_batch2.cu), which
// launch_split_batch picks where b.walk2 is set and the shape has one
// scenario per thread.
bool batch2_shape_compiled(const DequeShape &s, int esize);
cudaError_t launch_split_batch2(const BatchParams &b, int esize, bool lcap, const DequeShape &shape, int grid,
                                bool configure_only, int *blocks_per_sm, cudaStream_t stream);
cudaError_t launch_split_batch2_cap(const BatchParams &b, const DequeShape &shape, int grid, bool configure_only,
                                    int *blocks_per_sm, cudaStream_t stream);
cudaError_t launch_split_batch2_nocap(const BatchParams &b, const DequeShape &shape, int grid, bool configure_only,
                                      int *blocks_per_sm, cudaStream_t stream);
cudaError_t launch_split_batch2_i32_cap(const BatchParams &b, const DequeShape &shape, int grid, bool configure_only,
                                        int *blocks_per_sm, cudaStream_t stream);
cudaError_t launch_split_batch2_i32_nocap(const BatchParams &b, const DequeShape &shape, int grid, bool configure_only,
                                          int *blocks_per_sm, cudaStream_t stream);
// Whether every key K (P + Q) + p of a walk stays below 2^31 (int16 demands are
// read unclamped: one bad demand may add up to 65535 before the walk freezes;
// int32 ones add Q at most).
inline bool batch2_keys_fit(long long n, long long Q, long long K)
{
    return K * (n * Q + 65535 + Q) + n < (1LL << 31);
}
cudaError_t launch_split_batch_i16_cap(const BatchParams &b, const DequeShape &shape, int grid, bool configure_only,
                                       int *blocks_per_sm, cudaStream_t stream);
cudaError_t launch_split_batch_i16_nocap(const BatchParams &b, const DequeShape &shape, int grid, bool configure_only,
                                         int *blocks_per_sm, cudaStream_t stream);
cudaError_t launch_split_batch_i32_cap(const BatchParams &b, const DequeShape &shape, int grid, bool configure_only,
                                       int *blocks_per_sm, cudaStream_t stream);
cudaError_t launch_split_batch_i32_nocap(const BatchParams &b, const DequeShape &shape, int grid, bool configure_only,
                                         int *blocks_per_sm, cudaStream_t stream);
// Whether the batch kernel is compiled for this (threads, spt, ring).
bool batch_shape_compiled(const DequeShape &s);
cudaError_t launch_split_warp_batch(const BatchParams &b, int esize, int grid_ctas, int max_smem, bool configure_only,
                                    cudaStream_t stream);

// Sequence-parallel Split for few scenarios (seqpar.cu).
struct SeqParParams {
    const TourStep *tab;          // device [n]
    const void *demand;           // device [n][ld]
    long long ld;
    int S, n, Q, L, g0;
    int blocks;                   // ceil(n / block)
    int32_t *lo;                  // scratch [S][n]: window starts
    int32_t *flags;               // scratch [S]: nonzero = hand to the warp kernel
    int32_t *mats;                // scratch [S][blocks][W][W]: block transfer matrices
    int32_t *out_cost;            // device [S] or nullptr
    unsigned long long *acc;      // device [ACC_WORDS]
    int32_t *list;                // device [S]: scenarios for the warp kernel
};
cudaError_t launch_seqpar(const SeqParParams &a, int esize, cudaStream_t st);
int seqpar_blocks(int n);
int seqpar_width();

// Local search on the device (search.cu).
cudaError_t launch_neighbors(const int32_t *base, int n, const int32_t *moves, int M, int32_t *out, cudaStream_t st);
cudaError_t launch_tour_tables(const int32_t *tours, int T, int n, const int32_t *dist, int32_t *D_out,
                               TourStep *tabs, TourDev *descs, const void *demand, long long ld, int Q, int L,
                               uint32_t K, unsigned long long *smooth, cudaStream_t st);
cudaError_t launch_tour_means(const unsigned long long *acc, int T, long long S, double *mean, long long *sum,
                              long long *inf, cudaStream_t st);
cudaError_t launch_topk(const float *scores, int M, int k, int32_t *idx_out, cudaStream_t st);
cudaError_t launch_gather_rows(const int32_t *in, int rows, int n, const int32_t *idx, int R, int32_t *out,
                               cudaStream_t st);
cudaError_t launch_accept_best(const int32_t *tours, int T, int n, const double *cost, int32_t *cur,
                               double *cur_cost, double *trace, cudaStream_t st);

// Copy a [n][ld_in] demand matrix into a [n][ld_out] one of another element
// type (first S columns); values outside int16 set *saturated (device flag).
cudaError_t launch_convert_demand(const void *in, int esize_in, long long ld_in, void *out, int esize_out,
                                  long long ld_out, int n, long long S, unsigned int *saturated,
                                  cudaStream_t stream);

// Scenario generator.
struct GenParams {
    uint64_t seed;
    int32_t kind;
    const int32_t *mu;            // device [n]
    const int32_t *region;        // device [n]
    int32_t n;
    int64_t S, ld;
    void *out;
    int32_t mu_min, mu_max;       // of mu
};
cudaError_t launch_gen_demand(const GenParams &g, int esize, cudaStream_t stream);

}  // namespace cvrpsd
