// Threshold tuning on the divergences a verification call returns (Section "Selecting T": the
// threshold is tuned on a small development set by looking at the speed each candidate gives;
// Discussion: the FSD decision is deterministic given the divergences, so token-level labels can
// be dumped).  The accepted length of a row at threshold T is the index of its first position
// that fails D cmp T (NaN never passes); the speed proxy is the mean accepted length.
//
// With P[b, k] = max(D[b, 0..k]) (NaN once a NaN has been seen) the accepted length of row b is
// the number of k with P[b, k] cmp T, so
//   * a sweep counts, for every candidate threshold, the prefix maxima that pass, and
//   * the smallest T that reaches a wanted mean accepted length is an order statistic of the
//     multiset {P[b, k]}: the ceil(target * B)-th smallest value v (T = v under <=, the next
//     float above v under <).  It is found by a most-significant-digit-first radix selection on
//     the float bit patterns (monotone for non-negative floats): 12, 10 and 9 bits below the sign;
//     when the first digit leaves few candidates they are ranked directly.  The first digit is wide because divergences sit in few binades: with 16 bins a binade the
//     lanes of a warp seldom add to the same one.
//
// What bounds these kernels is latency: 4096 x 8 divergences are 128 KB.  Neither call has a
// workspace, so the blocks that share a job are a cluster (8 blocks): one for the calibration, one
// for every few thresholds of a sweep; few rows take single blocks.  A block's rows come to shared
// memory by bulk copies and, where they all fit, stay there for every walk; a thread walks a row
// in the widest loads its length allows, which also keeps lanes that walk neighbouring rows off one
// another's banks.  What the blocks tell one another is pushed (st.async, bulk copies between the
// blocks' shared memories) and counted in on the receiver's barrier: a cluster barrier orders all
// memory first, and reading eight histograms back from the peers took longer than all the rest.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "fsd_pair_stream.cuh"

namespace fsd {

constexpr int kTuneThreads = 512;             // at most; a sweep over few rows takes fewer
constexpr int kTuneCluster = 8;               // the portable size
constexpr int kTuneBins = 4096;               // of the first digit; 1024 and 512 of the others
constexpr int kTuneTileBytes = 72 * 1024;     // a tile of rows; two are in shared memory
constexpr int kSweepFew = 4, kSweepMany = 16; // thresholds a thread counts for in one walk over its rows (many: where a cluster has more than eight)
constexpr uint64_t kTuneLost = ~0ull;         // in the place of a count: a wait ran out
constexpr uint32_t kKeyInf = 0x7f800000u;     // keys above this are NaN (or negative): never accepted

// Sortable key of a prefix maximum: divergences are >= 0, so the bit pattern orders them; -0 and
// negative inputs count as 0, NaN as "never".
__device__ __forceinline__ uint32_t tune_key(float p) {
    if (p != p) return 0xffffffffu;
    return p <= 0.f ? 0u : __float_as_uint(p);
}

__device__ __forceinline__ void bulk_push(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "r"(smem_u32(src)), "r"(bytes), "r"(bar) : "memory");
}
// Bounded; what it waits for are copies already started or pushes of peers that run.  `lost` remembers, for the
// thread, that one has run out (the results are NaN then) and ends further waits.
struct TuneWait {
    bool lost;
    bool short_limit;                     // (test aid)
    __device__ __forceinline__ void operator()(uint64_t* bar, uint32_t parity) { if (!lost && !thread_wait(bar, parity, short_limit ? kInjectedWaitNs : 0)) lost = true; }
};
#ifdef FSD_DEBUG_CHECKS
#define FSD_TUNE_SILENT (silent != 0)
#else
#define FSD_TUNE_SILENT false
#endif

// These kernels are a few microseconds each and follow one another: all are launched with programmatic stream
// serialization.  What is in front of a kernel in its stream has ended (or it is waited for here, before global memory
// is touched); what comes behind it may be set up meanwhile.
__device__ __forceinline__ void launch_in_turn() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// ---- a block's rows [row0, row1) of the divergence matrix, tile by tile ---------------------
// Two tiles are in shared memory at most; a block whose rows are no more than that copies them once.
struct TuneRows {
    const float* D;
    int G, row0, rows, tile, tiles;       // rows a tile has (a multiple of four, so that tiles start 16 bytes apart like D), and tiles
    int off;                              // words between a 16-byte boundary and D
    bool staged;                          // (rows so long that a tile has too few for the threads are walked where they are)
    float* buf;
    uint64_t* bar;                        // [2]
    int seq, issued;                      // tiles walked and asked for so far, over all walks
    TuneWait wait;
};
__device__ __forceinline__ void tune_issue(TuneRows& t) {         // one thread
    const int i = t.issued % t.tiles, slot = t.issued & 1, n = min(t.tile, t.rows - i * t.tile);
    const uintptr_t first = reinterpret_cast<uintptr_t>(t.D + static_cast<size_t>(t.row0 + i * t.tile) * t.G);
    const uintptr_t a = first & ~uintptr_t(15), e = (first + static_cast<size_t>(n) * t.G * 4 + 15) & ~uintptr_t(15);
    float* dst = t.buf + slot * (kTuneTileBytes / 4);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    mbar_arrive_expect_tx(&t.bar[slot], static_cast<uint32_t>(e - a));
    bulk_g2s(dst, reinterpret_cast<const void*>(a), static_cast<uint32_t>(e - a), &t.bar[slot]);
}
// Rows of block `rank` of `cs`; starts the first copies.  `bar`: two barriers, initialised (count 1).
__device__ __forceinline__ TuneRows tune_rows(const float* D, int B, int G, int rank, int cs, float* buf, uint64_t* bar, bool short_limit) {
    TuneRows t;
    t.wait = TuneWait{false, short_limit};
    const int quads = (B + 3) / 4, base = quads / cs, rem = quads % cs;
    t.D = D; t.G = G; t.buf = buf; t.bar = bar; t.seq = 0; t.issued = 0;
    t.row0 = 4 * (rank * base + min(rank, rem));
    t.rows = max(0, min(4 * (base + (rank < rem ? 1 : 0)), B - t.row0));
    const long long quad_bytes = 16ll * G;
    // A thread walks a row, so a tile of few rows leaves the block's other threads idle: where it has less than half of what
    // they could take, the rows are read through L1 instead (300 rows of 1000, calibration 3863 us from tiles of 16 rows).
    const int fit = 4 * static_cast<int>((kTuneTileBytes - 16) / quad_bytes);
    t.staged = fit > 0 && 2 * fit >= min(t.rows, static_cast<int>(blockDim.x));
    t.tile = t.staged ? fit : t.rows;
    t.tiles = t.staged ? (t.rows + t.tile - 1) / t.tile : (t.rows > 0 ? 1 : 0);
    t.off = static_cast<int>((reinterpret_cast<uintptr_t>(D) & 15) / 4);
    if (t.staged)
        for (; t.issued < 2 && t.issued < t.tiles; ++t.issued)
            if (threadIdx.x == 0) tune_issue(t);
    return t;
}
// One thread's walk along one row: step(d) for every position in order, until stop() says that the rest does not matter.
template <int W, typename F, typename S>
__device__ __forceinline__ void walk_row(const float* row, int G, F step, S stop) {
    for (int k = 0; k < G && !stop(); k += W) {
        float d[W];
        if constexpr (W == 4) { const float4 v = *reinterpret_cast<const float4*>(row + k); d[0] = v.x; d[1] = v.y; d[2] = v.z; d[3] = v.w; }
        else if constexpr (W == 2) { const float2 v = *reinterpret_cast<const float2*>(row + k); d[0] = v.x; d[1] = v.y; }
        else d[0] = row[k];
#pragma unroll
        for (int q = 0; q < W; ++q) step(d[q]);
    }
}
// One walk over all of the block's rows: begin() / step(d) until stop() / end() per row.  All threads of the block take part.
template <typename Begin, typename Step, typename Stop, typename End>
__device__ __forceinline__ void tune_walk(TuneRows& t, Begin begin, Step step, Stop stop, End end) {
    for (int i = 0; i < t.tiles; ++i) {
        const int slot = t.seq & 1, n = min(t.tile, t.rows - i * t.tile);
        const bool resident = t.tiles <= 2;
        const float* base = t.D + static_cast<size_t>(t.row0 + i * t.tile) * t.G;
        const int width = t.off == 0 && t.G % 4 == 0 ? 4 : t.off % 2 == 0 && t.G % 2 == 0 ? 2 : 1;
        if (t.staged) {
            // a resident tile i is in slot i for good; others take turns
            const int s = resident ? i : slot;
            t.wait(&t.bar[s], resident ? 0 : (t.seq >> 1) & 1);
            base = t.buf + s * (kTuneTileBytes / 4) + t.off;
        }
        for (int r = threadIdx.x; r < n; r += blockDim.x) {
            const float* row = base + static_cast<size_t>(r) * t.G;
            begin();
            if (width == 4) walk_row<4>(row, t.G, step, stop);
            else if (width == 2) walk_row<2>(row, t.G, step, stop);
            else walk_row<1>(row, t.G, step, stop);
            end();
        }
        ++t.seq;
        if (t.staged && !resident) {
            __syncthreads();                          // everybody is through with the slot
            if (threadIdx.x == 0) tune_issue(t);      // (the walk after this one starts over: its first tiles are asked for too)
            ++t.issued;
        }
    }
}
// No copy may still be on its way into a block that leaves.
__device__ __forceinline__ void tune_drain(TuneRows& t) {
    if (!t.staged) return;
    if (t.tiles <= 2) {
        for (int i = 0; i < t.tiles; ++i) t.wait(&t.bar[i], 0);
    } else {
        for (int q = t.seq; q < t.issued; ++q) t.wait(&t.bar[q & 1], (q >> 1) & 1);
    }
}

// ---- sweep: a cluster (or a block) per group of candidate thresholds ---------------------------
// Each block counts for its rows and pushes its counts to the cluster's first block.  On a B200, 64
// thresholds: 4096 x 8 13.5 -> 4.6 us, 32768 x 20 245 -> 24 us (a block per threshold before, its
// threads walking rows in global memory one dependent load at a time).
template <int CS, int AT>
__global__ void __launch_bounds__(kTuneThreads) fsd_threshold_sweep_kernel(const float* __restrict__ D, int B, int G,
                                                                           const float* __restrict__ thresholds, int n_thresholds, int cmp,
                                                                           float* __restrict__ mean_len, float* __restrict__ frac, int silent) {
    extern __shared__ __align__(16) float tune_buf[];
    __shared__ uint64_t bar[2], link[2];
    __shared__ unsigned int part[kTuneThreads / 32][AT];
    __shared__ uint64_t got[2][kTuneCluster][AT];      // (B * positions fits an int); kTuneLost: not to be relied on
    __shared__ int lost;                              // a wait of some thread of this block has run out
    const int rank = CS == 1 ? 0 : static_cast<int>(cg::this_cluster().block_rank());
    const int n_clusters = static_cast<int>(gridDim.x) / CS, cid = static_cast<int>(blockIdx.x) / CS;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) {
        lost = 0;
        for (int k = 0; k < 2; ++k) { mbar_init(&bar[k], 1); mbar_init(&link[k], 1); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if constexpr (CS > 1) cg::this_cluster().barrier_arrive();   // "this block's barriers are ready": waited for before the first push
    launch_in_turn();
    TuneRows rows = tune_rows(D, B, G, rank, CS, tune_buf, bar, FSD_TUNE_SILENT);
    // thresholds cid, cid + n_clusters, ...: AT of them in one walk
    int turn = 0;
    for (int t0 = cid; t0 < n_thresholds; t0 += n_clusters * AT, ++turn) {
        float T[AT];
        unsigned int n[AT];
#pragma unroll
        for (int j = 0; j < AT; ++j) {
            const int t = t0 + j * n_clusters;
            T[j] = t < n_thresholds ? thresholds[t] : __int_as_float(0x7fc00000);
            n[j] = 0;
        }
        float p = 0.f, most = T[0];
#pragma unroll
        for (int j = 1; j < AT; ++j) most = fmaxf(most, T[j]);       // (a NaN threshold is no threshold)
        const auto begin = [&] { p = -INFINITY; };
        const auto stop = [&] { return !(p <= most); };              // nothing passes from here on (a row's rest was never read)
        if (cmp == FSD_CMP_LE) {
            tune_walk(rows, begin, [&](float d) {
                p = fmax_nan(p, d);                   // NaN stays and never passes
#pragma unroll
                for (int j = 0; j < AT; ++j) n[j] += p <= T[j];
            }, stop, [] {});
        } else {
            tune_walk(rows, begin, [&](float d) {
                p = fmax_nan(p, d);
#pragma unroll
                for (int j = 0; j < AT; ++j) n[j] += p < T[j];
            }, stop, [] {});
        }
#pragma unroll
        for (int j = 0; j < AT; ++j) {
            const unsigned int w = __reduce_add_sync(0xffffffffu, n[j]);
            if (lane == 0) part[warp][j] = w;
        }
        if (rows.wait.lost) lost = 1;
        __syncthreads();
        uint64_t sum = 0;
        if (tid < AT)
            for (int w = 0; w < static_cast<int>(blockDim.x >> 5); ++w) sum += part[w][tid];
        if (lost) sum = kTuneLost;
        if constexpr (CS > 1) {
            // (two buffers take turns; nobody is a turn ahead by more than one: see the barrier below)
            if (turn == 0) cg::this_cluster().barrier_wait();
            if (rank == 0 && tid == 0 && !rows.wait.lost) mbar_arrive_expect_tx(&link[turn & 1], CS * AT * 8);
            if (tid < AT && !(FSD_TUNE_SILENT && rank == CS - 1))
                st_async(cluster_addr(&got[turn & 1][rank][tid], 0), sum, cluster_addr(&link[turn & 1], 0));
            if (rank == 0 && tid < 32) {
                rows.wait(&link[turn & 1], (turn >> 1) & 1);
                if (tid < AT) {
                    bool all = !rows.wait.lost;
                    sum = 0;
                    for (int r = 0; r < CS; ++r) { sum += got[turn & 1][r][tid]; all = all && got[turn & 1][r][tid] != kTuneLost; }
                    if (!all) sum = kTuneLost;
                }
            }
            if (t0 + n_clusters * AT < n_thresholds) cg::this_cluster().sync();   // more walks than one: nobody overtakes block 0
        }
        if (rank == 0 && tid < AT && t0 + tid * n_clusters < n_thresholds) {
            const int t = t0 + tid * n_clusters;
            const float nan = __int_as_float(0x7fc00000);
            mean_len[t] = sum == kTuneLost ? nan : static_cast<float>(static_cast<double>(sum) / static_cast<double>(B));
            frac[t] = sum == kTuneLost ? nan : static_cast<float>(static_cast<double>(sum) / (static_cast<double>(B) * static_cast<double>(G)));
        }
        __syncthreads();                              // `part` is free again
    }
    tune_drain(rows);
    if constexpr (CS > 1) leave_last(rows.wait.lost);
}

// ---- calibration: one cluster (or block), radix selection over the prefix maxima ----------------
// Calls f(key, count) for every run of equal prefix maxima of this thread's rows.
template <typename F>
__device__ __forceinline__ void for_prefix_maxima(TuneRows& rows, F f) {
    float p = 0.f;
    uint32_t key = 0;
    unsigned int run = 0;
    tune_walk(rows, [&] { p = 0.f; key = 0; run = 0; },
              [&](float d) {
                  p = fmax_nan(p, d);
                  const uint32_t kn = tune_key(p);
                  if (kn != key && run > 0) { f(key, run); run = 0; }
                  key = kn;
                  ++run;
              },
              [] { return false; }, [&] { f(key, run); });
}

constexpr int kTuneList = kTuneBins / kTuneCluster;                        // candidates of a block that are ranked directly
struct CalibrateShared {
    uint64_t bar[2];                                  // tiles
    uint64_t link[3][3];                              // [digit][parts of the histogram | sums | the digit found]
    uint64_t list_link;
    unsigned int hist[kTuneBins];
    unsigned int recv[kTuneCluster][kTuneBins / kTuneCluster];   // this block's part of the peers' histograms; later, in block 0,
                                                      // everybody's candidates (sent when all have the first digit, so when all have read)
    uint64_t sums[kTuneCluster];
    uint64_t found[2];                                // digit | keys equal to it << 32, keys below it | most of a block's equal to it << 32
    uint32_t list[kTuneList];                         // this block's candidates
    unsigned int warp_sum[kTuneThreads / 32];
    unsigned int n_list, count;
    int lost;                                         // block 0's: a wait of some thread of the cluster has run out
};

// A row's prefix maxima never fall, so a thread adds once per distinct value (two or three a row of
// eight).  Per digit: every block pushes the eighth of its histogram that block r is to add up to
// block r, then its sum over that eighth to everybody, and the block whose eighth holds the wanted
// rank pushes the digit to everybody.  If no block has more than kTuneList keys that share the first digit, they are
// pushed to block 0, which goes on with them by itself, two more histograms (9 and 10 bits) of at most eight keys a thread: a digit
// of the whole cluster's is a walk over all rows and three exchanges, 3 us.  us on a B200 by one block and four 8-bit digits / by the cluster's digits
// where more than 512 keys in all share the first (some 800 of 4096 x 8 do) / now:
//   4096 x 8 57 / 12.2 / 9.8    8192 x 10 - / 16.3 / 13.1    32768 x 20 821 / 73.8 / 73.9 (the walks' shared-memory atomics are the larger part)
template <int CS>
__global__ void __launch_bounds__(kTuneThreads) fsd_calibrate_kernel(const float* __restrict__ D, int B, int G, float target,
                                                                     int cmp, float* __restrict__ T_out,
                                                                     float* __restrict__ achieved_out, int silent) {
    extern __shared__ __align__(16) float tune_buf[];
    __shared__ __align__(16) CalibrateShared sh;
    const int rank = CS == 1 ? 0 : static_cast<int>(cg::this_cluster().block_rank());
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) {
        for (int k = 0; k < 2; ++k) mbar_init(&sh.bar[k], 1);
        for (int k = 0; k < 9; ++k) mbar_init(&sh.link[0][0] + k, 1);
        mbar_init(&sh.list_link, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        sh.count = 0; sh.n_list = 0; sh.lost = 0;
    }
    for (int i = tid; i < kTuneBins / 4; i += kTuneThreads) reinterpret_cast<uint4*>(sh.hist)[i] = make_uint4(0, 0, 0, 0);
    for (int i = tid; i < kTuneList; i += kTuneThreads) sh.list[i] = 0xffffffffu;
    __syncthreads();
    if constexpr (CS > 1) cg::this_cluster().barrier_arrive();   // "this block's barriers are ready": waited for before the first push
    launch_in_turn();
    TuneRows rows = tune_rows(D, B, G, rank, CS, tune_buf, sh.bar, FSD_TUNE_SILENT);
    TuneWait& tune_wait = rows.wait;

    // positions that must be accepted: ceil(target * B), within [0, B * G]  (the host refuses negative and NaN targets)
    const double want = ceil(static_cast<double>(target) * static_cast<double>(B));
    const double most = static_cast<double>(B) * static_cast<double>(G);
    const unsigned int need = want <= 0.0 ? 0u : static_cast<unsigned int>(want < most ? want : most);

    uint32_t prefix = 0;
    unsigned int left = need, below = 0, equal = 0;   // rank still to be found; keys below / equal to the prefix found
    bool found = need > 0, ranked = false;
    if constexpr (CS > 1) { if (need == 0) cg::this_cluster().barrier_wait(); }
    if (need > 0) {
#pragma unroll 1
        for (int digit = 0; digit < 3; ++digit) {
            const int shift = digit == 0 ? 19 : digit == 1 ? 9 : 0;
            const uint32_t mask = digit == 0 ? 0u : digit == 1 ? 0xfff80000u : 0xfffffe00u;   // the digits before this one
            const uint32_t width = digit == 0 ? 4095u : digit == 1 ? 1023u : 511u;
            const int part = digit == 0 ? kTuneBins / CS : 1024 / CS;      // bins a block adds up
            if (digit > 0) {
                for (int i = tid; i < 1024 / 4; i += kTuneThreads) reinterpret_cast<uint4*>(sh.hist)[i] = make_uint4(0, 0, 0, 0);
                __syncthreads();
            }
            for_prefix_maxima(rows, [&](uint32_t key, unsigned int count) {
                if (key <= kKeyInf && (key & mask) == prefix) atomicAdd(&sh.hist[(key >> shift) & width], count);
            });
            const unsigned int (*mine)[kTuneBins / kTuneCluster] = sh.recv;
            if constexpr (CS > 1) {
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                if (tid == 0) mbar_arrive_expect_tx(&sh.link[digit][0], static_cast<uint32_t>(part) * 4 * CS);
                if (tid == 1) mbar_arrive_expect_tx(&sh.link[digit][1], 8 * CS);
                if (tid == 2) mbar_arrive_expect_tx(&sh.link[digit][2], 16);
                __syncthreads();
                if (digit == 0) cg::this_cluster().barrier_wait();
                if (tid < CS) bulk_push(cluster_addr(&sh.recv[rank][0], tid), sh.hist + tid * part, static_cast<uint32_t>(part) * 4, cluster_addr(&sh.link[digit][0], tid));
                tune_wait(&sh.link[digit][0], 0);
            } else {
                __syncthreads();
            }
            // this block's part: its bins (8 a thread when a block has them all, else at most one) and their running sum
            constexpr int kMost = CS > 1 ? 1 : kTuneBins / kTuneThreads;
            unsigned int c[kMost], sum = 0;
            const int per = CS > 1 ? 1 : part / kTuneThreads;
#pragma unroll
            for (int q = 0; q < kMost; ++q) {
                c[q] = 0;
                if (CS > 1) {
                    if (tid < part) {
#pragma unroll
                        for (int r = 0; r < CS; ++r) c[q] += mine[r][tid];
                    }
                } else if (q < per) {
                    c[q] = sh.hist[per * tid + q];
                }
                sum += c[q];
            }
            unsigned int incl = sum;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const unsigned int up = __shfl_up_sync(0xffffffffu, incl, d);
                if (lane >= d) incl += up;
            }
            if (lane == 31) sh.warp_sum[warp] = incl;
            __syncthreads();
            unsigned int before = 0, all = 0;
#pragma unroll
            for (int w = 0; w < kTuneThreads / 32; ++w) { const unsigned int ws = sh.warp_sum[w]; if (w < warp) before += ws; all += ws; }
            if constexpr (CS > 1) {
                if (tid < CS && !(FSD_TUNE_SILENT && rank == CS - 1)) st_async(cluster_addr(&sh.sums[rank], tid), all, cluster_addr(&sh.link[digit][1], tid));
                tune_wait(&sh.link[digit][1], 0);
                if (__syncthreads_or(tune_wait.lost)) { found = false; break; }      // (the same for the block: what follows has barriers)
                all = 0;
                for (int r = 0; r < CS; ++r) { const unsigned int v = static_cast<unsigned int>(sh.sums[r]); if (r < rank) before += v; all += v; }
            }
            if (all < left) { found = false; break; } // fewer acceptable positions than needed (the same for all)
            unsigned int run = before + incl - sum;
            if (left > run && left <= run + sum) {    // one thread of the cluster
#pragma unroll
                for (int q = 0; q < kMost; ++q) {
                    if (left > run && left <= run + c[q]) {
                        unsigned int worst = c[q];
                        if constexpr (CS > 1) {
                            worst = 0;
#pragma unroll
                            for (int r = 0; r < CS; ++r) worst = max(worst, mine[r][tid]);
                        }
                        const uint64_t w0 = static_cast<uint32_t>((CS > 1 ? rank * part : 0) + per * tid + q) | static_cast<uint64_t>(c[q]) << 32, w1 = run | static_cast<uint64_t>(worst) << 32;
                        if constexpr (CS > 1) {
                            for (int r = 0; r < CS; ++r) {
                                st_async(cluster_addr(&sh.found[0], r), w0, cluster_addr(&sh.link[digit][2], r));
                                st_async(cluster_addr(&sh.found[1], r), w1, cluster_addr(&sh.link[digit][2], r));
                            }
                        } else {
                            sh.found[0] = w0; sh.found[1] = w1;
                        }
                        run = left;                   // (found: no other bin)
                    }
                    run += c[q];
                }
            }
            if constexpr (CS > 1) tune_wait(&sh.link[digit][2], 0); else __syncthreads();
            const uint64_t w0 = sh.found[0];
            prefix |= static_cast<uint32_t>(w0) << shift;
            equal = static_cast<unsigned int>(w0 >> 32);
            const unsigned int lower = static_cast<unsigned int>(sh.found[1]);
            below += lower; left -= lower;
            if (__syncthreads_or(tune_wait.lost)) { found = false; break; }
            // everybody has read: the histogram and the rest may be written again
            if (digit == 0 && (sh.found[1] >> 32) <= kTuneList) { ranked = true; break; }
        }
    }
    if (ranked) {
        // the keys that share the first digit, from all blocks to block 0
        for_prefix_maxima(rows, [&](uint32_t key, unsigned int count) {
            if ((key & 0xfff80000u) != prefix || key > kKeyInf) return;
            const unsigned int at = atomicAdd(&sh.n_list, count);
            for (unsigned int q = 0; q < count && at + q < kTuneList; ++q) sh.list[at + q] = key;       // (at most kTuneList of a block's, unless a wait ran out)
        });
        if constexpr (CS > 1) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            if (rank == 0 && tid == 0) mbar_arrive_expect_tx(&sh.list_link, CS * kTuneList * 4);
            __syncthreads();
            if (tid == 0) bulk_push(cluster_addr(&sh.recv[rank][0], 0), sh.list, kTuneList * 4, cluster_addr(&sh.list_link, 0));
            if (rank == 0) tune_wait(&sh.list_link, 0);
        }
        __syncthreads();
        if (rank == 0) {
            // (where there is nothing, the lists hold 0xffffffff: no key, its upper bits are no prefix)
            const uint32_t* const keys = CS > 1 ? reinterpret_cast<const uint32_t*>(&sh.recv[0][0]) : sh.list;
#pragma unroll 1
            for (int digit = 1; digit < 3; ++digit) {
                const int shift = digit == 1 ? 10 : 0;
                const uint32_t mask = digit == 1 ? 0xfff80000u : 0xfffffc00u, width = digit == 1 ? 511u : 1023u;
                reinterpret_cast<uint2*>(sh.hist)[tid] = make_uint2(0, 0);      // 1024 bins, two a thread
                __syncthreads();
#pragma unroll
                for (int q = 0; q < (CS > 1 ? CS * kTuneList / kTuneThreads : 1); ++q) {
                    const uint32_t key = keys[tid + q * kTuneThreads];
                    if ((key & mask) == prefix) atomicAdd(&sh.hist[(key >> shift) & width], 1u);
                }
                __syncthreads();
                const uint2 c = reinterpret_cast<const uint2*>(sh.hist)[tid];
                unsigned int incl = c.x + c.y;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const unsigned int up = __shfl_up_sync(0xffffffffu, incl, d);
                    if (lane >= d) incl += up;
                }
                if (lane == 31) sh.warp_sum[warp] = incl;
                __syncthreads();
                unsigned int run = incl - c.x - c.y;
#pragma unroll
                for (int w = 0; w < kTuneThreads / 32; ++w) if (w < warp) run += sh.warp_sum[w];
                if (left > run && left <= run + c.x + c.y) {                     // one thread
                    const bool second = left > run + c.x;
                    sh.found[0] = static_cast<uint32_t>(2 * tid + (second ? 1 : 0)) | static_cast<uint64_t>(second ? c.y : c.x) << 32;
                    sh.found[1] = second ? run + c.x : run;
                }
                __syncthreads();
                prefix |= static_cast<uint32_t>(sh.found[0]) << shift;
                equal = static_cast<unsigned int>(sh.found[0] >> 32);
                below += static_cast<unsigned int>(sh.found[1]);
                left -= static_cast<unsigned int>(sh.found[1]);
                __syncthreads();                      // (found and the histogram may be written again)
            }
        }
    }

    // the threshold, then the mean accepted length it gives: known from the counts, or (no selection, or +inf) one more walk
    float T;
    if (need == 0) {
        T = 0.f;
    } else if (!found) {
        T = INFINITY;
    } else {
        const float v = __uint_as_float(prefix);
        T = cmp == FSD_CMP_LE ? v : (v == INFINITY ? INFINITY : __uint_as_float(prefix + 1u));   // next float above v
    }
    const auto tell_lost = [&] {
        if (rows.wait.lost) { if constexpr (CS > 1) *cg::this_cluster().map_shared_rank(&sh.lost, 0) = 1; else sh.lost = 1; }
    };
    tell_lost();
    unsigned int total = below + equal;
    // (a first digit of +inf's holds nothing else that counts, so that every block decides alike)
    if (need == 0 || !found || (prefix & 0xfff80000u) == kKeyInf) {
        unsigned int n = 0;
        for_prefix_maxima(rows, [&](uint32_t key, unsigned int count) {
            if (key <= kKeyInf && passes(__uint_as_float(key), T, cmp)) n += count;
        });
        n = __reduce_add_sync(0xffffffffu, n);
        tell_lost();
        if (lane == 0 && n) atomicAdd(CS > 1 ? cg::this_cluster().map_shared_rank(&sh.count, 0) : &sh.count, n);
        if constexpr (CS > 1) cg::this_cluster().sync(); else __syncthreads();
        total = sh.count;                             // (block 0's is the one that is used)
    } else {
        // pushes from and to a block are through before it leaves
        if constexpr (CS > 1) cg::this_cluster().sync(); else __syncthreads();
    }
    if (rank == 0 && tid == 0) {
        const float nan = __int_as_float(0x7fc00000);
        *T_out = sh.lost ? nan : T;
        *achieved_out = sh.lost ? nan : static_cast<float>(static_cast<double>(total) / static_cast<double>(B));
    }
    tune_drain(rows);
}

// ---- labels: each position on its own ---------------------------------------------------------
__global__ void fsd_accept_labels_kernel(const float* __restrict__ D, size_t n, float T, int cmp, uint8_t* __restrict__ labels) {
    launch_in_turn();
    const size_t stride = static_cast<size_t>(gridDim.x) * blockDim.x;
    for (size_t i = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += stride)
        labels[i] = passes(D[i], T, cmp) ? 1 : 0;
}
#undef FSD_TUNE_SILENT

}  // namespace fsd
