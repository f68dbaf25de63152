// C ABI of the verification library: argument checks, workspace layout, kernel launches.
// See include/fsd_verify.h for the contract of every entry point.
#include <climits>
#include <cstdint>
#include <cuda_runtime.h>
#include <atomic>
#include <ctime>
#include <mutex>
#include <unistd.h>

#include "fsd_verify.h"
#include "fsd_device.cuh"
#include "fsd_finish.cuh"
#include "fsd_pair_generic.cuh"
#include "fsd_pair_stream.cuh"
#include "fsd_row.cuh"
#include "fsd_tuning.cuh"

namespace {

using namespace fsd;

constexpr size_t kAlign = 256;
constexpr int kMaxBlocks = 256;                                        // of the streaming kernel (one per SM)
constexpr size_t kExchangeBytes = 2 * kMaxBlocks * sizeof(GroupMsg);
inline size_t align_up(size_t x) { return (x + kAlign - 1) / kAlign * kAlign; }
inline bool aligned(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

struct Workspace {
    int32_t* item_bits;
    int32_t* item_status;
    CallFlags* flags;
    GroupMsg* exchange;        // the streaming kernel's statistics exchange
    PairRecord* records;       // per-pair totals of the streaming kernel
    size_t bytes;
};

Workspace carve(void* base, int B, int G) {
    Workspace w;
    const size_t items = static_cast<size_t>(B) * G;
    char* p = static_cast<char*>(base);
    w.item_bits = reinterpret_cast<int32_t*>(p);
    p += align_up(items * sizeof(int32_t));
    w.item_status = reinterpret_cast<int32_t*>(p);
    p += align_up(items * sizeof(int32_t));
    w.flags = reinterpret_cast<CallFlags*>(p);
    p += kAlign;
    w.exchange = reinterpret_cast<GroupMsg*>(p);
    p += kExchangeBytes;
    w.records = reinterpret_cast<PairRecord*>(p);
    p += align_up(items * sizeof(PairRecord));
    w.bytes = static_cast<size_t>(p - static_cast<char*>(base));
    return w;
}

int check_opts(const fsd_opts* o) {
    if (o == nullptr) return FSD_ERR_NULL;
    if (o->struct_size != sizeof(fsd_opts)) return FSD_ERR_ENUM;
    if (o->divergence < FSD_DIV_JS || o->divergence > FSD_DIV_TV) return FSD_ERR_ENUM;
    if (o->mode < FSD_MODE_FSD || o->mode > FSD_MODE_RFSD) return FSD_ERR_ENUM;
    if (o->compare < FSD_CMP_LT || o->compare > FSD_CMP_LE) return FSD_ERR_ENUM;
    if (o->sample < FSD_SAMPLE_INVCDF || o->sample > FSD_SAMPLE_GREEDY) return FSD_ERR_ENUM;
    if (o->logit_dtype < FSD_F32 || o->logit_dtype > FSD_BF16) return FSD_ERR_ENUM;
    if (o->threshold != o->threshold) return FSD_ERR_ENUM;   // NaN threshold
    return FSD_OK;
}

int check_shape(int B, int G, int V) {
    if (B < 1 || G < 1 || V < 1) return FSD_ERR_SHAPE;
    if (static_cast<long long>(B) * (static_cast<long long>(G) + 1) > INT_MAX) return FSD_ERR_SHAPE;
    return FSD_OK;
}

// CTAs per row of the finish kernel: one or two vectors of logits a thread and a warp for every pair to be
// judged, at most the portable cluster size, and no more CTAs than one wave of two per SM (148 SMs) when the
// batch is large.
int finish_cluster_size(int B, int G, int V) {
    int cs = 1;
    while (cs < kPortableCluster && (static_cast<long long>(cs) * kFinishThreads * 8 < V || cs * kFinishWarps < G) &&
           static_cast<long long>(B) * cs * 2 <= 2 * 148)
        cs <<= 1;
    return cs;
}

std::atomic<void*> g_stage_event{nullptr};   // see fsd_set_stage_event
std::atomic<int> g_mark_timeout{0};          // see fsd_set_timeout_injection
std::atomic<int> g_group_size{0};            // see fsd_set_group_size

// A number no other launch is given, of which a call's number is made (see CallFlags).  The counter's values are spread
// over 64 bits by an invertible mixing (the finalizer of splitmix64), from a start that differs from process to process:
// the time in nanoseconds, the process and where its stack is.  (std::random_device may throw, and this is behind a C entry.)
uint64_t spread(uint64_t x) {
    x = (x ^ (x >> 30)) * 0xbf58476d1ce4e5b9ull;
    x = (x ^ (x >> 27)) * 0x94d049bb133111ebull;
    return x ^ (x >> 31);
}
uint64_t nonce_start() {
    timespec t = {};
    clock_gettime(CLOCK_REALTIME, &t);
    return spread(static_cast<uint64_t>(t.tv_sec) * 1000000000ull + static_cast<uint64_t>(t.tv_nsec)) ^
           spread(static_cast<uint64_t>(getpid()) << 32) ^ spread(reinterpret_cast<uintptr_t>(&t));
}
uint64_t next_nonce() {
    static std::atomic<uint64_t> counter{nonce_start()};
    return spread(counter.fetch_add(0x9e3779b97f4a7c15ull));
}

// ---- streaming kernel launch -----------------------------------------------------------
constexpr int kMaxDev = 64;

// Attributes of a kernel that takes all of an SM's shared memory, and how many clusters of each size from 1 to kMaxClusterSize the
// device holds at once (0: none).  Puts nothing on a stream.
template <typename K>
bool prepare_clusters(K kernel, int threads, size_t smem, int* most) {
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem)) != cudaSuccess) return false;
    const bool wide = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
    for (int cs = 1; cs <= kMaxClusterSize; ++cs) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(static_cast<unsigned>(256 * cs), 1, 1);
        cfg.blockDim = dim3(static_cast<unsigned>(threads), 1, 1);
        cfg.dynamicSmemBytes = smem;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = static_cast<unsigned>(cs); attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int n = 0;
        if ((cs <= kPortableCluster || wide) && cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) n = 0;
        most[cs - 1] = n;
    }
    cudaGetLastError();                                                // (a size the device refuses is no error of this call's)
    return true;
}
// How a kernel is launched in clusters, and set up while the kernel in front drains: it waits for that one's end itself.
// (A kernel that stores into the shared memory of its cluster's blocks needs the attribute also where a cluster is one block:
// without it the store is an illegal instruction.)  cs 0: no clusters, single blocks (with the attribute the streaming kernel
// takes 0.3 us more).
struct ClusterLaunch {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    ClusterLaunch(int clusters, int cs, int threads, size_t smem, cudaStream_t s) {
        cfg.gridDim = dim3(static_cast<unsigned>(cs > 0 ? clusters * cs : clusters), 1, 1);
        cfg.blockDim = dim3(static_cast<unsigned>(threads), 1, 1);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = s;
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = static_cast<unsigned>(cs > 0 ? cs : 1); attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = cs > 0 ? 2 : 1;
    }
};

// One block per SM.  Puts nothing on a stream.
template <int DT, int DIV, bool RAGGED>
int prepare_stream(int dev) {
    static bool ready[kMaxDev] = {};
    static std::mutex mu;
    auto kernel = fsd_pair_stream_kernel<DT, DIV, RAGGED>;
    if (dev < 0 || dev >= kMaxDev) return FSD_ERR_CUDA;
    std::lock_guard<std::mutex> lock(mu);
    if (!ready[dev]) {
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kStreamSmemBytes)) != cudaSuccess)
            return FSD_ERR_CUDA;
        int per = 0;                                 // one block must fit an SM
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, kStreamThreads, kStreamSmemBytes) != cudaSuccess || per < 1)
            return FSD_ERR_CUDA;
        ready[dev] = true;
    }
    return FSD_OK;
}

template <int DT, int DIV, bool RAGGED>
int launch_stream(const StreamParams& gp, int nsm, cudaStream_t s) {
    // as many blocks as give every pair a group, at most one per SM and what the exchange buffer holds
    const long long want = static_cast<long long>(gp.n_items) * gp.C;
    int grid = nsm < kMaxBlocks ? nsm : kMaxBlocks;
    if (want < grid) grid = static_cast<int>(want);
    if (grid < gp.C) return FSD_ERR_CUDA;
    const ClusterLaunch l(grid, 0, kStreamThreads, kStreamSmemBytes, s);
    return cudaLaunchKernelEx(&l.cfg, fsd_pair_stream_kernel<DT, DIV, RAGGED>, gp) == cudaSuccess ? FSD_OK : FSD_ERR_CUDA;
}

using PrepareFn = int (*)(int);
using LaunchFn = int (*)(const StreamParams&, int, cudaStream_t);
struct StreamKernel { PrepareFn prepare; LaunchFn launch; };
template <int DT, int DIV> StreamKernel stream_kernel(bool ragged) {
    return ragged ? StreamKernel{prepare_stream<DT, DIV, true>, launch_stream<DT, DIV, true>} : StreamKernel{prepare_stream<DT, DIV, false>, launch_stream<DT, DIV, false>};
}
template <int DT> StreamKernel stream_kernel(int div, bool ragged) {
    return div == FSD_DIV_JS ? stream_kernel<DT, FSD_DIV_JS>(ragged) : div == FSD_DIV_KL ? stream_kernel<DT, FSD_DIV_KL>(ragged) : stream_kernel<DT, FSD_DIV_TV>(ragged);
}

// Blocks per pair for the streaming kernel; 0 if the row is too long for the largest group (the
// generic kernel takes it).  Between the fewest whose slice fits on chip and kMaxGroupSize it is the
// size with the lowest estimated time -- rounds * (fixed cost of a round + cost of a step * steps a
// warp has), or half a round and half an exchange where that is longer (the totals are needed two
// rounds on).  The constants (microseconds) are measured on a B200.
template <int DT>
int group_size(int nvec_row, int items, int nsm) {
    using S = StreamShape<DT>;
    const int cmin = (nvec_row + S::kBlockVecs - 1) / S::kBlockVecs;
    const int forced = g_group_size.load();
    const int blocks = nsm < kMaxBlocks ? nsm : kMaxBlocks;
    if (forced >= cmin && forced <= kMaxGroupSize && forced <= blocks) return forced;
    int best = 0;
    double best_cost = 0.0;
    for (int C = cmin; C <= kMaxGroupSize && C <= blocks; ++C) {
        const int groups = blocks / C;
        const int rounds = (items + groups - 1) / groups;
        const int slice = (nvec_row + C - 1) / C;
        const int block_steps = (slice + (32 * S::kVecPerStep) - 1) / (32 * S::kVecPerStep);
        double round = 0.3 + 0.4 * block_steps / kComputeWarps;
        if (round < 0.5 * (round + 1.6)) round = 0.5 * (round + 1.6);
        const double cost = rounds * round;
        if (best == 0 || cost < best_cost) { best = C; best_cost = cost; }
    }
    return best;
}

// ---- row kernel launch -----------------------------------------------------------------
// Attributes, and how many clusters of each size the device holds at once.  Puts nothing on a stream.
template <int DT, int KIND, bool RAGGED>
const int* prepare_row(int dev) {
    static int most[kMaxDev][kMaxClusterSize] = {};
    static bool ready[kMaxDev] = {};
    static std::mutex mu;
    if (dev < 0 || dev >= kMaxDev) return nullptr;
    std::lock_guard<std::mutex> lock(mu);
    if (!ready[dev]) {
        if (!prepare_clusters(fsd_row_kernel<DT, KIND, RAGGED>, kFinishThreads, kRowSmemBytes, most[dev])) return nullptr;
        ready[dev] = true;
    }
    return most[dev];
}
// Blocks per batch row: the largest cluster of which the GPU holds one for every row at once (a second wave would take as long
// as the first), whose blocks have room for the row's logits and what is parked of them.  us on a B200 by the streaming and
// finish kernels / in clusters of half the size / of the size taken:
//   1 x 4 x 32000 fp32 11.5 / 11.2 / 9.6 (12)    16 x 5 x 32000 16.0 / - / 12.5 (6)    8 x 5 x 50257 16.6 / - / 13.5 (10)
//   10 x 4 x 24000 12.5 / 10.9 / 9.8 (10)    28 x 5 x 8192 12.8 / 11.7 / 10.8 (4)    4 x 16 x 8000 11.4 / 11.7 / 10.2 (12)
// (The largest is not always the fastest, 4 x 16 x 2000 9.34 in 12 and 9.40 in 8, 1 x 12 x 4000 10.7 in 12 and 10.4 in 6; over 700 random
// shapes the fastest of up to twelve would be 1 % faster.)
// At most twelve: a cluster's SMs are of one GPC, so the larger it is the sooner it waits for other kernels to end.  Beside a
// kernel that has a block on 60 (74, 90, 100, 110, 120, 132) of the SMs for 1 ms, 1 x 4 x 32000 fp32 waits for its end in clusters of 16 (14, 12, 10,
// 8 with 120, 6 with 132); the general path with 132.  Alone it takes 9.24 us in 16, 9.63 in 12, 10.1 in 8, 11.5 by the general path: twelve leave
// a call its time beside kernels that hold half of the GPU.
// A call whose clusters have less than half of the SMs is spread over more of them by the streaming kernel, and there the row kernel gains
// only while a warp has little to do: at most five items, or four where there is no second sweep whose exchange it would save (KL), or one where
// an argmax, the shortest draw, follows the sweeps of more than nine positions.  us on a B200 by the streaming and finish kernels / by this one:
//   3 x 14 x 20352 KL greedy (7 items a warp) 8.2 / 9.0    4 x 15 x 21202 KL greedy (7) 9.3 / 10.5    1 x 14 x 19328 JS (7) 11.6 / 12.2
//   2 x 11 x 10420 fp32 TV greedy (3) 9.5 / 10.2    5 x 10 x 5565 KL greedy (2) 8.4 / 8.7    but 10 x 16 x 8000 KL (4; 100 SMs) 11.3 / 9.5
// (2000 random calls: 36 were slower by more than 1.5 % without these limits, 6 with them, of which 5 by less than 6 %; the mean gain 1.24 in both.)
// One more: the argmax of a residual whose rows are not whole vectors is two passes entry by entry, which the finish kernel shares out over two
// blocks where a row has more than 4096 entries (80 x 1 x 15580 TV rFSD greedy 35.7 / 45.8 in clusters of one).
struct RowPlan { int cs, span; };                                      // cs 0: not by the row kernel
template <int DT, int KIND, bool RAGGED>
RowPlan row_plan(const FinishParams& fp, int nsm, size_t nvec_row, const int* most) {
    constexpr int step = 32 * StreamShape<DT>::kVecPerStep;
    const int B = fp.B, G = fp.G;
    const bool greedy = fp.sample == FSD_SAMPLE_GREEDY;
    const RowPlan none = {0, 0};
    if (G > kRowMaxPairs || nvec_row > static_cast<size_t>(kMaxClusterSize) * kRowMaxItems * step) return none;
    for (int cs = kMaxClusterSize; cs >= 1; --cs) {
        // (A GPU that by the occupancy calculation holds 45 clusters of three, or 26 of five, does so where their places work out: 43 to
        // 45 of three were 1.03, 1.24 and 1.38 times as long as clusters of two, 25 and 26 of five 1.19 and 1.37 times as long as clusters
        // of four, as in a second wave; 42 and 24 were faster, and other sizes up to the last cluster.  25 x 8 x 16000 KL 11.2 -> 11.5 us in 25 of five.)
        const int room = cs == 3 || cs == 5 ? most[cs - 1] * 15 / 16 : most[cs - 1];
        if (room < B) continue;
        const int span = (static_cast<int>((nvec_row + cs - 1) / cs) + step - 1) / step * step, steps = span / step;
        if (steps * G > kRowMaxItems || row_bytes_of(G, span, RAGGED) > row_smem_left<DT, KIND>()) continue;
        const int per_warp = (steps * G + kFinishWarps - 1) / kFinishWarps;
        if (2 * B * cs < nsm && per_warp > (greedy && G > 9 ? 1 : fp.div == FSD_DIV_KL ? 4 : 5)) return none;
        if (KIND == kDrawResidual && RAGGED && greedy && cs == 1 && fp.V > 8 * kFinishThreads) return none;
        return {cs, span};
    }
    return none;
}
template <int DT, int KIND, bool RAGGED>
int launch_row(const FinishParams& fp, int cs, int span, size_t nvec_row, uint64_t nonce, int injection, cudaStream_t s) {
    RowParams rp;
    rp.fin = fp;
    rp.nvec_row = static_cast<int>(nvec_row); rp.span = span; rp.nonce = nonce;
    rp.silent = injection == 2 || injection == 4;
    rp.limit_ns = rp.silent ? kInjectedWaitNs : kWaitNs;
    rp.raise = injection == 1;
    const ClusterLaunch l(fp.B, cs, kFinishThreads, kRowSmemBytes, s);
    return cudaLaunchKernelEx(&l.cfg, fsd_row_kernel<DT, KIND, RAGGED>, rp) == cudaSuccess ? FSD_OK : FSD_ERR_CUDA;
}
// One launch if the row kernel takes the call; `taken` says so.
template <int DT, int KIND, bool RAGGED>
int try_row(const FinishParams& fp, int nsm, size_t nvec_row, int dev, uint64_t nonce, int injection, cudaStream_t s, bool& taken) {
    const int* most = prepare_row<DT, KIND, RAGGED>(dev);
    if (most == nullptr) return FSD_ERR_CUDA;
    const RowPlan plan = row_plan<DT, KIND, RAGGED>(fp, nsm, nvec_row, most);
    taken = plan.cs > 0;                                               // (a row kernel is ready for a later call all the same)
    return taken ? launch_row<DT, KIND, RAGGED>(fp, plan.cs, plan.span, nvec_row, nonce, injection, s) : FSD_OK;
}
template <int DT, int KIND>
int try_row(const FinishParams& fp, int nsm, bool vec, size_t nvec_row, int dev, uint64_t nonce, int injection, cudaStream_t s, bool& taken) {
    return vec ? try_row<DT, KIND, false>(fp, nsm, nvec_row, dev, nonce, injection, s, taken) : try_row<DT, KIND, true>(fp, nsm, nvec_row, dev, nonce, injection, s, taken);
}

template <int DT>
int launch_all(PairParams pp, FinishParams fp, bool vec, CallFlags* flags, GroupMsg* exchange, PairRecord* records, cudaStream_t s) {
    const int items = pp.B * pp.G;
    int dev = 0, nsm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || nsm < 1)
        return FSD_ERR_CUDA;
    const size_t row_bytes = static_cast<size_t>(pp.V) * Logit<DT>::kBytes;
    // an unaligned row covers at most as many 16-byte granules as one that starts at a granule's last element
    const size_t nvec_row = vec ? row_bytes / 16 : (row_bytes + 16 - Logit<DT>::kBytes + 15) / 16;
    const int C = nvec_row <= static_cast<size_t>(kMaxGroupSize) * StreamShape<DT>::kBlockVecs ? group_size<DT>(static_cast<int>(nvec_row), items, nsm) : 0;
    pp.nonce = next_nonce(); pp.flags = flags;
    fp.flags = flags;
    const int injection = g_mark_timeout.load();
    fp.silent = injection == 4 ? 1 : injection == 6 ? 2 : 0;
    // everything that can fail without a launch (attributes, the occupancy queries) comes before the first thing put on the
    // stream, of the streaming kernel also where this call does not need it: a later one, under capture, may
    const StreamKernel kernel = stream_kernel<DT>(pp.div, !vec);
    if (C > 0) {
        const int rc = kernel.prepare(dev);
        if (rc != FSD_OK) return rc;
    }
#ifdef FSD_DEBUG_CHECKS
    if (cudaMemsetAsync(&flags->debug, 0, sizeof(int), s) != cudaSuccess) return FSD_ERR_CUDA;   // the debug word starts at zero
#endif
    // What fits on chip goes by the row kernel, unless a test or measurement aid asks for the streaming kernel.
    bool row = g_group_size.load() == 0 && g_stage_event.load() == nullptr;
    if (row) {
        fp.records = records;
        const int rc = fp.mode != FSD_MODE_FSD ? try_row<DT, kDrawResidual>(fp, nsm, vec, nvec_row, dev, pp.nonce, injection, s, row)
                       : fp.sample == FSD_SAMPLE_GREEDY ? try_row<DT, kDrawGreedy>(fp, nsm, vec, nvec_row, dev, pp.nonce, injection, s, row)
                                                        : try_row<DT, kDrawPt>(fp, nsm, vec, nvec_row, dev, pp.nonce, injection, s, row);
        if (rc != FSD_OK || row) return rc;
    }
    if (C > 0) {
        StreamParams sp;
        sp.target = pp.target; sp.draft = pp.draft; sp.parent = pp.parent; sp.G = pp.G;
        sp.nvec_row = static_cast<int>(nvec_row); sp.row_bytes = row_bytes; sp.n_items = items; sp.records = records;
        sp.nonce = pp.nonce; sp.flags = flags;
        sp.C = C; sp.exchange = exchange;
        const int slice = static_cast<int>((nvec_row + C - 1) / C);
        sp.slot_row_bytes = slot_row_bytes<DT>(slice); sp.slot_bytes = slot_bytes<DT>(slice, !vec);
        sp.ring = kRingBytes / sp.slot_bytes < kMaxRing ? kRingBytes / sp.slot_bytes : kMaxRing;
        // item / G by a multiplication: with 2^(l-1) < G <= 2^l, ceil(2^(31+l) / G) is exact for items below 2^31
        int l = 0;
        while ((1ll << l) < pp.G) ++l;
        sp.g_magic = l == 0 ? 0u : static_cast<uint32_t>(((1ull << (31 + l)) + pp.G - 1) / pp.G);
        sp.g_shift = l == 0 ? 0u : static_cast<uint32_t>(l - 1);
        // test aid: one block keeps its first message to itself, so that its group's exchange
        // runs out (after a shorter limit: about a tenth of a second) and the kernel's own give-up path runs;
        // mode 3: so that the others sum its slice themselves
        const bool silent = injection == 2 || injection == 3;
        sp.poll_limit = silent ? (1u << 17) : kSpinLimit;
        // fetches, somewhat below a microsecond each (beside kernels that held 140 of 148 SMs for 3 ms, with 1024 of them:
        // 64 x 8 x 152064 ended after 20 ms instead of 3.2)
        sp.help_after = injection == 2 ? 0xffffffffu : injection == 3 ? 1024 : 16384;
        sp.silent_rank = silent ? C - 1 : -1;
        sp.raise = injection == 1;                    // behave as if a bounded wait had run out
        const int rc = kernel.launch(sp, nsm, s);
        if (rc != FSD_OK) return rc;
        fp.records = records;
    } else {
        if (vec) fsd_pair_generic_kernel<DT, true><<<items, 512, 0, s>>>(pp);
        else     fsd_pair_generic_kernel<DT, false><<<items, 512, 0, s>>>(pp);
        if (cudaGetLastError() != cudaSuccess) return FSD_ERR_CUDA;
        fp.records = nullptr;
    }

    if (void* ev = g_stage_event.load()) {
        if (cudaEventRecord(static_cast<cudaEvent_t>(ev), s) != cudaSuccess) return FSD_ERR_CUDA;
    }
    const int cs = finish_cluster_size(fp.B, fp.G, fp.V);
    // The finish kernel may be set up while the pair kernel drains: its CTAs take the SMs the
    // pair kernel's CTAs leave, build their tables, and wait (griddepcontrol.wait) for the pair
    // kernel to complete before they read anything it wrote.
    const ClusterLaunch l(fp.B, cs, kFinishThreads, 0, s);
    const auto finish = fp.mode != FSD_MODE_FSD ? fsd_finish_kernel<DT, kDrawResidual>
                        : fp.sample == FSD_SAMPLE_GREEDY ? fsd_finish_kernel<DT, kDrawGreedy> : fsd_finish_kernel<DT, kDrawPt>;
    return cudaLaunchKernelEx(&l.cfg, finish, fp) == cudaSuccess ? FSD_OK : FSD_ERR_CUDA;
}

int verify_common(const void* target, const void* draft, const int32_t* tokens, const float* u_accept,
                  const float* u_sample, const int32_t* parent, int B, int G, int V, int max_depth,
                  const fsd_opts* o, int32_t* accept_len, int32_t* path, int32_t* next_token,
                  float* divergence, int32_t* row_status, void* workspace, size_t workspace_bytes,
                  void* stream) {
    const size_t es = o->logit_dtype == FSD_BF16 ? 2 : 4;
    if (!aligned(target, es) || !aligned(draft, es) || !aligned(u_sample, 4) || !aligned(accept_len, 4) ||
        !aligned(next_token, 4) || !aligned(divergence, 4) || !aligned(row_status, 4) ||
        !aligned(tokens, 4) || !aligned(u_accept, 4) || !aligned(parent, 4) || !aligned(path, 4) ||
        !aligned(workspace, kAlign))
        return FSD_ERR_ALIGN;
    Workspace ws = carve(workspace, B, G);
    if (workspace_bytes < ws.bytes) return FSD_ERR_WORKSPACE;

    PairParams pp;
    pp.target = target; pp.draft = draft; pp.tokens = tokens; pp.u_accept = u_accept; pp.parent = parent;
    pp.B = B; pp.G = G; pp.V = V;
    pp.div = o->divergence; pp.mode = o->mode; pp.cmp = o->compare; pp.T = o->threshold;
    pp.divergence = divergence; pp.item_bits = ws.item_bits; pp.item_status = ws.item_status;

    FinishParams fp;
    fp.target = target; fp.draft = draft; fp.parent = parent; fp.u_sample = u_sample;
    fp.B = B; fp.G = G; fp.V = V;
    fp.tokens = tokens; fp.u_accept = u_accept;
    fp.div = o->divergence; fp.mode = o->mode; fp.cmp = o->compare; fp.sample = o->sample; fp.max_depth = max_depth;
    fp.T = o->threshold; fp.records = nullptr; fp.divergence = divergence;
    fp.item_bits = ws.item_bits; fp.item_status = ws.item_status;
    fp.accept_len = accept_len; fp.path = path; fp.next_token = next_token; fp.row_status = row_status;

    const bool vec = (static_cast<size_t>(V) * es) % 16 == 0 && aligned(target, 16) && aligned(draft, 16);
    fp.vec = vec ? 1 : 0;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    return o->logit_dtype == FSD_BF16 ? launch_all<FSD_BF16>(pp, fp, vec, ws.flags, ws.exchange, ws.records, s)
                                       : launch_all<FSD_F32>(pp, fp, vec, ws.flags, ws.exchange, ws.records, s);
}

struct HostStaging {
    char *target, *draft, *tokens, *u_accept, *u_sample, *accept_len, *next_token, *divergence, *row_status, *ws;
    size_t n_target, n_draft, n_items4, n_rows4, n_ws, bytes;
};

HostStaging carve_staging(void* base, int B, int G, int V, size_t es) {
    HostStaging h;
    h.n_target = static_cast<size_t>(B) * (G + 1) * V * es;
    h.n_draft = static_cast<size_t>(B) * G * V * es;
    h.n_items4 = static_cast<size_t>(B) * G * 4;
    h.n_rows4 = static_cast<size_t>(B) * 4;
    h.n_ws = carve(nullptr, B, G).bytes;
    char* p = static_cast<char*>(base);
    auto take = [&](size_t n) { char* q = p; p += align_up(n); return q; };
    h.target = take(h.n_target); h.draft = take(h.n_draft);
    h.tokens = take(h.n_items4); h.u_accept = take(h.n_items4); h.u_sample = take(h.n_rows4);
    h.accept_len = take(h.n_rows4); h.next_token = take(h.n_rows4);
    h.divergence = take(h.n_items4); h.row_status = take(h.n_rows4);
    h.ws = take(h.n_ws);
    h.bytes = static_cast<size_t>(p - static_cast<char*>(base));
    return h;
}

// The address at which kernels of the current device reach n bytes of pinned host memory; null where they may not use
// them in place: pageable memory, memory that is pinned in part (pages are pinned one by one, so each is looked at; arrays of
// more pages than a few are better copied), an address off an element's boundary.
void* mapped_pointer(const void* host, size_t n) {
    constexpr size_t kPage = 4096, kMostPages = 16;
    if (!aligned(host, 4) || n > kMostPages * kPage) return nullptr;
    char* first = nullptr;
    for (size_t at = 0;; at = at + kPage < n ? at + kPage : n - 1) {
        cudaPointerAttributes a;
        if (cudaPointerGetAttributes(&a, static_cast<const char*>(host) + at) != cudaSuccess) { cudaGetLastError(); return nullptr; }
        if (a.type != cudaMemoryTypeHost || a.devicePointer == nullptr) return nullptr;
        if (at == 0) first = static_cast<char*>(a.devicePointer);
        else if (static_cast<char*>(a.devicePointer) != first + at) return nullptr;
        if (at == n - 1) return first;
    }
}
bool overlap(const void* a, size_t na, const void* b, size_t nb) {
    const uintptr_t x = reinterpret_cast<uintptr_t>(a), y = reinterpret_cast<uintptr_t>(b);
    return x < y + nb && y < x + na;
}

// Built-in scratch of fsd_verify_chain_static.  In host code this name is only a handle for
// cudaGetSymbolAddress; the kernels get the device address that call returns.
static __device__ __align__(256) unsigned char g_static_scratch[FSD_STATIC_SCRATCH_BYTES];

constexpr int kMaxDevices = 64;
std::mutex g_static_mutex;
void* g_static_ptr[kMaxDevices] = {};

// Device address of g_static_scratch on the current device (looked up once per device).
int static_scratch(void** out) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return FSD_ERR_CUDA;
    std::lock_guard<std::mutex> lock(g_static_mutex);
    if (g_static_ptr[dev] == nullptr) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_static_scratch) != cudaSuccess || p == nullptr) return FSD_ERR_CUDA;
        g_static_ptr[dev] = p;
    }
    *out = g_static_ptr[dev];
    return FSD_OK;
}

// A block on its own where a walk gives no thread more than one row: there the cluster's start and its
// pushes cost more than they share out (300 x 6 on a B200: calibration 6.2 us in one block, 8.7 us in a
// cluster; 4096 x 8: 34 and 11).
bool tuning_in_one_block(int B) { return B <= kTuneThreads; }
// A tuning kernel on `clusters` clusters; shared memory for as many of a block's rows as there are, up to what is staged.
template <typename... KArgs, typename... Args>
int launch_tuning(void (*kernel)(KArgs...), int threads, int cs, int clusters, int B, int G, void* stream, Args... args) {
    // two tiles, or as much as the block's rows take (rounded out to 16 bytes at both ends)
    const long long rows = ((B + 3ll) / 4 + cs - 1) / cs * 4, want = rows * G * 4 + 32;
    const size_t bytes = static_cast<size_t>(want <= kTuneTileBytes - 16 ? want : 2 * kTuneTileBytes);
    // (the calibration has 35 KB of its own; 48 KB in all need no attribute)
    if (bytes > 12 * 1024 && cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * kTuneTileBytes) != cudaSuccess) return FSD_ERR_CUDA;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(clusters) * cs, 1, 1);
    cfg.blockDim = dim3(static_cast<unsigned>(threads), 1, 1);
    cfg.dynamicSmemBytes = bytes;
    cfg.stream = static_cast<cudaStream_t>(stream);
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cs; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cs > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...) == cudaSuccess ? FSD_OK : FSD_ERR_CUDA;
}

}  // namespace

extern "C" {

void fsd_default_opts(fsd_opts* opts) {
    if (opts == nullptr) return;
    opts->struct_size = sizeof(fsd_opts);
    opts->divergence = FSD_DIV_JS;
    opts->mode = FSD_MODE_FSD;
    opts->compare = FSD_CMP_LT;
    opts->sample = FSD_SAMPLE_INVCDF;
    opts->logit_dtype = FSD_BF16;
    opts->threshold = 0.0f;
}

int fsd_workspace_bytes(int B, int positions, int V, const fsd_opts* opts, size_t* bytes_out) {
    if (bytes_out == nullptr) return FSD_ERR_NULL;
    int rc = check_opts(opts);
    if (rc != FSD_OK) return rc;
    rc = check_shape(B, positions, V);
    if (rc != FSD_OK) return rc;
    *bytes_out = carve(nullptr, B, positions).bytes;
    return FSD_OK;
}

int fsd_verify_chain(const void* target_logits, const void* draft_logits, const int32_t* draft_tokens,
                     const float* u_accept, const float* u_sample, int B, int gamma, int V,
                     const fsd_opts* opts, int32_t* accept_len, int32_t* next_token, float* divergence,
                     int32_t* row_status, void* workspace, size_t workspace_bytes, void* stream) {
    int rc = check_opts(opts);
    if (rc != FSD_OK) return rc;
    if (!target_logits || !draft_logits || !u_sample || !accept_len || !next_token || !divergence ||
        !row_status || !workspace)
        return FSD_ERR_NULL;
    if (opts->mode != FSD_MODE_FSD && (!draft_tokens || !u_accept)) return FSD_ERR_NULL;
    rc = check_shape(B, gamma, V);
    if (rc != FSD_OK) return rc;
    return verify_common(target_logits, draft_logits, draft_tokens, u_accept, u_sample, nullptr, B, gamma, V, 0,
                         opts, accept_len, nullptr, next_token, divergence, row_status, workspace,
                         workspace_bytes, stream);
}

int fsd_verify_tree(const void* target_logits, const void* draft_logits, const int32_t* parent,
                    const float* u_sample, int B, int N, int V, int max_depth, const fsd_opts* opts,
                    int32_t* accept_len, int32_t* path, int32_t* next_token, float* divergence,
                    int32_t* row_status, void* workspace, size_t workspace_bytes, void* stream) {
    int rc = check_opts(opts);
    if (rc != FSD_OK) return rc;
    if (!target_logits || !draft_logits || !parent || !u_sample || !accept_len || !path || !next_token ||
        !divergence || !row_status || !workspace)
        return FSD_ERR_NULL;
    if (opts->mode != FSD_MODE_FSD) return FSD_ERR_UNSUPPORTED;
    rc = check_shape(B, N, V);
    if (rc != FSD_OK) return rc;
    if (max_depth < 1 || N > kMaxTreeNodes) return FSD_ERR_SHAPE;
    return verify_common(target_logits, draft_logits, nullptr, nullptr, u_sample, parent, B, N, V, max_depth,
                         opts, accept_len, path, next_token, divergence, row_status, workspace,
                         workspace_bytes, stream);
}

int fsd_host_staging_bytes(int B, int gamma, int V, const fsd_opts* opts, size_t* bytes_out) {
    if (bytes_out == nullptr) return FSD_ERR_NULL;
    int rc = check_opts(opts);
    if (rc != FSD_OK) return rc;
    rc = check_shape(B, gamma, V);
    if (rc != FSD_OK) return rc;
    *bytes_out = carve_staging(nullptr, B, gamma, V, opts->logit_dtype == FSD_BF16 ? 2 : 4).bytes;
    return FSD_OK;
}

int fsd_verify_chain_host(const void* h_target_logits, const void* h_draft_logits, const int32_t* h_draft_tokens,
                          const float* h_u_accept, const float* h_u_sample, int B, int gamma, int V,
                          const fsd_opts* opts, int32_t* h_accept_len, int32_t* h_next_token,
                          float* h_divergence, int32_t* h_row_status, void* staging, size_t staging_bytes,
                          void* stream) {
    int rc = check_opts(opts);
    if (rc != FSD_OK) return rc;
    if (!h_target_logits || !h_draft_logits || !h_u_sample || !h_accept_len || !h_next_token || !h_divergence ||
        !h_row_status || !staging)
        return FSD_ERR_NULL;
    if (opts->mode != FSD_MODE_FSD && (!h_draft_tokens || !h_u_accept)) return FSD_ERR_NULL;
    rc = check_shape(B, gamma, V);
    if (rc != FSD_OK) return rc;
    if (!aligned(staging, kAlign)) return FSD_ERR_ALIGN;
    HostStaging h = carve_staging(staging, B, gamma, V, opts->logit_dtype == FSD_BF16 ? 2 : 4);
    if (staging_bytes < h.bytes) return FSD_ERR_WORKSPACE;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    // The logits are copied.  The small arrays are not, where the kernels can reach them where they are (pinned
    // memory): a copy of a few hundred bytes takes its 2 us on the stream all the same, and there were seven.
    // 8 x 5 x 32000 bf16, pinned: 165 us a call with the copies, of which 100 are the logits on PCIe.
    bool ok = cudaMemcpyAsync(h.target, h_target_logits, h.n_target, cudaMemcpyHostToDevice, s) == cudaSuccess;
    ok = ok && cudaMemcpyAsync(h.draft, h_draft_logits, h.n_draft, cudaMemcpyHostToDevice, s) == cudaSuccess;
    struct Array { const void* host; char* staged; size_t n; void* used; };
    Array ins[3] = {{h_draft_tokens, h.tokens, h.n_items4, nullptr}, {h_u_accept, h.u_accept, h.n_items4, nullptr}, {h_u_sample, h.u_sample, h.n_rows4, nullptr}};
    Array outs[4] = {{h_accept_len, h.accept_len, h.n_rows4, nullptr}, {h_next_token, h.next_token, h.n_rows4, nullptr},
                     {h_divergence, h.divergence, h.n_items4, nullptr}, {h_row_status, h.row_status, h.n_rows4, nullptr}};
    // outputs that share memory with an input or with one another are written when all is read, one after another
    bool apart = true;
    for (int k = 0; k < 4; ++k) {
        for (const Array& in : ins) apart = apart && (in.host == nullptr || !overlap(outs[k].host, outs[k].n, in.host, in.n));
        for (int q = 0; q < k; ++q) apart = apart && !overlap(outs[k].host, outs[k].n, outs[q].host, outs[q].n);
    }
    for (Array& a : ins) {
        if (a.host == nullptr) continue;
        a.used = mapped_pointer(a.host, a.n);
        if (a.used == nullptr) {
            a.used = a.staged;
            ok = ok && cudaMemcpyAsync(a.staged, a.host, a.n, cudaMemcpyHostToDevice, s) == cudaSuccess;
        }
    }
    if (!ok) return FSD_ERR_CUDA;
    for (Array& a : outs) {
        a.used = apart ? mapped_pointer(a.host, a.n) : nullptr;
        if (a.used == nullptr) a.used = a.staged;
    }
    rc = fsd_verify_chain(h.target, h.draft, static_cast<const int32_t*>(ins[0].used), static_cast<const float*>(ins[1].used),
                          static_cast<const float*>(ins[2].used), B, gamma, V, opts, static_cast<int32_t*>(outs[0].used),
                          static_cast<int32_t*>(outs[1].used), static_cast<float*>(outs[2].used), static_cast<int32_t*>(outs[3].used),
                          h.ws, h.n_ws, stream);
    if (rc != FSD_OK) return rc;
    for (const Array& a : outs)
        if (a.used == a.staged) ok = ok && cudaMemcpyAsync(const_cast<void*>(a.host), a.staged, a.n, cudaMemcpyDeviceToHost, s) == cudaSuccess;
    ok = ok && cudaStreamSynchronize(s) == cudaSuccess;
    return ok ? FSD_OK : FSD_ERR_CUDA;
}

int fsd_verify_chain_static(const void* target_logits, const void* draft_logits, const int32_t* draft_tokens,
                            const float* u_accept, const float* u_sample, int B, int gamma, int V,
                            const fsd_opts* opts, int32_t* accept_len, int32_t* next_token, float* divergence,
                            int32_t* row_status, void* stream) {
    int rc = check_opts(opts);
    if (rc != FSD_OK) return rc;
    if (!target_logits || !draft_logits || !u_sample || !accept_len || !next_token || !divergence || !row_status)
        return FSD_ERR_NULL;
    if (opts->mode != FSD_MODE_FSD && (!draft_tokens || !u_accept)) return FSD_ERR_NULL;
    rc = check_shape(B, gamma, V);
    if (rc != FSD_OK) return rc;
    if (static_cast<long long>(B) * gamma > FSD_STATIC_MAX_POSITIONS ||
        carve(nullptr, B, gamma).bytes > FSD_STATIC_SCRATCH_BYTES)
        return FSD_ERR_TOO_LARGE;
    void* scratch = nullptr;
    rc = static_scratch(&scratch);
    if (rc != FSD_OK) return rc;
    return verify_common(target_logits, draft_logits, draft_tokens, u_accept, u_sample, nullptr, B, gamma, V, 0,
                         opts, accept_len, nullptr, next_token, divergence, row_status, scratch,
                         FSD_STATIC_SCRATCH_BYTES, stream);
}

const char* fsd_status_string(int status) {
    switch (status) {
        case FSD_OK: return "FSD_OK";
        case FSD_ERR_NULL: return "FSD_ERR_NULL: a required pointer is NULL";
        case FSD_ERR_SHAPE: return "FSD_ERR_SHAPE: a dimension is out of range";
        case FSD_ERR_ALIGN: return "FSD_ERR_ALIGN: a pointer is misaligned";
        case FSD_ERR_ENUM: return "FSD_ERR_ENUM: an option is out of range";
        case FSD_ERR_WORKSPACE: return "FSD_ERR_WORKSPACE: workspace too small";
        case FSD_ERR_UNSUPPORTED: return "FSD_ERR_UNSUPPORTED: combination not defined";
        case FSD_ERR_CUDA: return "FSD_ERR_CUDA: the CUDA runtime refused a launch";
        case FSD_ERR_TOO_LARGE: return "FSD_ERR_TOO_LARGE: B * gamma exceeds FSD_STATIC_MAX_POSITIONS";
        default: return "unknown fsd status";
    }
}

int fsd_version(void) { return 100; }

int fsd_set_stage_event(void* event) {
    g_stage_event.store(event);
    return FSD_OK;
}

int fsd_debug_checks(int B, int positions, size_t* word_offset) {
    if (word_offset != nullptr && B >= 1 && positions >= 1) {
        const Workspace w = carve(nullptr, B, positions);
        *word_offset = static_cast<size_t>(reinterpret_cast<char*>(&w.flags->debug) - static_cast<char*>(nullptr));
    }
#ifdef FSD_DEBUG_CHECKS
    return 1;
#else
    return 0;
#endif
}

int fsd_set_timeout_injection(int mode) {
#ifdef FSD_DEBUG_CHECKS
    const bool known = (mode >= 0 && mode <= 4) || mode == 6;
#else
    const bool known = mode >= 0 && mode <= 2;
#endif
    if (!known) return FSD_ERR_ENUM;
    g_mark_timeout.store(mode);
    return FSD_OK;
}

int fsd_set_group_size(int group_size) {
    if (group_size < 0 || group_size > 16) return FSD_ERR_SHAPE;
    g_group_size.store(group_size);
    return FSD_OK;
}

int fsd_threshold_sweep(const float* divergence, int B, int positions, const float* thresholds, int n_thresholds,
                        int compare, float* mean_accept_len, float* accept_fraction, void* stream) {
    if (divergence == nullptr || thresholds == nullptr || mean_accept_len == nullptr || accept_fraction == nullptr)
        return FSD_ERR_NULL;
    if (B < 1 || positions < 1 || n_thresholds < 1) return FSD_ERR_SHAPE;
    if (static_cast<long long>(B) * positions > INT_MAX) return FSD_ERR_SHAPE;      // the kernels count in 32 bits
    if (compare != FSD_CMP_LT && compare != FSD_CMP_LE) return FSD_ERR_ENUM;
    // a cluster per group of thresholds, as many as the GPU holds at once, and as few thresholds each as that gives
    const bool one = tuning_in_one_block(B);
    const int cs = one ? 1 : kTuneCluster, most = 148 / cs, rows = (B + cs - 1) / cs;
    const int threads = rows >= kTuneThreads ? kTuneThreads : (rows + 31) / 32 * 32 < 64 ? 64 : (rows + 31) / 32 * 32;
    const int clusters = n_thresholds < most ? n_thresholds : most;
    // (4096 x 8, 2000 thresholds: 72 us with four of them a walk)
    const bool many = n_thresholds > 8ll * clusters;
    const auto kernel = one ? (many ? fsd_threshold_sweep_kernel<1, kSweepMany> : fsd_threshold_sweep_kernel<1, kSweepFew>)
                            : (many ? fsd_threshold_sweep_kernel<kTuneCluster, kSweepMany> : fsd_threshold_sweep_kernel<kTuneCluster, kSweepFew>);
    return launch_tuning(kernel, threads, cs, clusters, B, positions, stream, divergence, B, positions, thresholds, n_thresholds,
                         compare, mean_accept_len, accept_fraction, g_mark_timeout.load() == 4 ? 1 : 0);
}

int fsd_calibrate_threshold(const float* divergence, int B, int positions, float target_mean_accept_len, int compare,
                            float* threshold_out, float* achieved_out, void* stream) {
    if (divergence == nullptr || threshold_out == nullptr || achieved_out == nullptr) return FSD_ERR_NULL;
    if (B < 1 || positions < 1 || !(target_mean_accept_len >= 0.f)) return FSD_ERR_SHAPE;   // NaN target included
    if (static_cast<long long>(B) * positions > INT_MAX) return FSD_ERR_SHAPE;      // the kernels count in 32 bits
    if (compare != FSD_CMP_LT && compare != FSD_CMP_LE) return FSD_ERR_ENUM;
    const bool one = tuning_in_one_block(B);
    return launch_tuning(one ? fsd_calibrate_kernel<1> : fsd_calibrate_kernel<kTuneCluster>, kTuneThreads, one ? 1 : kTuneCluster, 1, B, positions, stream, divergence, B, positions, target_mean_accept_len, compare,
                         threshold_out, achieved_out, g_mark_timeout.load() == 4 ? 1 : 0);
}

int fsd_accept_labels(const float* divergence, int B, int positions, float threshold, int compare, uint8_t* labels,
                      void* stream) {
    if (divergence == nullptr || labels == nullptr) return FSD_ERR_NULL;
    if (B < 1 || positions < 1) return FSD_ERR_SHAPE;
    if (compare != FSD_CMP_LT && compare != FSD_CMP_LE) return FSD_ERR_ENUM;
    const size_t n = static_cast<size_t>(B) * positions;
    const unsigned blocks = static_cast<unsigned>(n / 256 + 1 < 1184 ? n / 256 + 1 : 1184);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks, 1, 1);
    cfg.blockDim = dim3(256, 1, 1);
    cfg.stream = static_cast<cudaStream_t>(stream);
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, fsd_accept_labels_kernel, divergence, n, threshold, compare, labels) == cudaSuccess ? FSD_OK : FSD_ERR_CUDA;
}

}  // extern "C"
