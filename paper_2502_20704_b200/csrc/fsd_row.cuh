// Row kernel: a whole verify call of a few batch rows in one launch, a thread-block cluster per row.
//
// Where the logits of a row -- gamma + 1 target rows, gamma draft rows -- fit the shared memory of a cluster, and the
// call's clusters the GPU at once, nothing of it has to pass through global memory: every block copies its
// share of all rows at the start, the blocks tell one another their sums by remote stores, and the row the token is drawn
// from is in shared memory already.  The streaming kernel and the finish kernel behind it (the general path) cost such a
// call two launches, an exchange between blocks through L2 of 1.6 us, a hand-over from kernel to kernel, and trips to L2
// for the records and the row.
//
// A block's share of a row is `span` granules of 16 bytes.  Its sweeps are dealt out in items, a step (8 entries a lane) of a
// pair each, pair by pair: a sixteenth of them, in one run, to every warp, so that a warp has to do with one or two pairs.
//   1. First sweep of a warp's items of a pair, as in the streaming kernel: e = 2^(logit * log2e - k),
//      Z, S (or the KL sum), "rows differ"; e parked in tensor memory.  The references k come from the maxima of the first item; a warp that
//      finds they were not near enough does its sweep over with those of all its items.  The warp that
//      is the last of a pair's folds what the pair's warps have posted and pushes the sums to all blocks of the cluster.
//   2. A warp per pair folds what the blocks sent into 1/Z_a, 1/Z_b for its block.
//   3. Second sweep of the items over the parked e, in the same order: JS sum (p+q) log2(p+q), TV sum |p - q|; folded and pushed
//      likewise (KL has none).
//   4. Every block judges all pairs from the sums of all blocks, in double precision, and draws as in the finish kernel.
// A tree's nodes are pairs like any others, each against the target row of its parent.
// The sums of a pair are added up in an order that follows from its position and the call's shape, and from nothing that other pairs hold.
// What bounds it: latency.  16 x 5 x 32000 bf16 (16 clusters of 6), cycles from where the inputs may be read: first rows landed
// 1560, first sweep 7720 (special functions 3400 of them), totals 9460, second sweep 12890 (1700), judged 15940, token 20040: 10.4 us of
// 12.5 a call among others; 15.4 by the streaming and finish kernels.  1 x 4 x 32000 fp32 11.0 -> 9.7 us, 8 x 5 x 50257 16.1 -> 13.5.
// A residual draw: 12 x 6 x 32000 (clusters of 9), relaxed rule, judged 18100, token 30770 (the other rule 14890, 19030).
// All waits are for copies of the block's own or for pushes of its cluster's blocks, which run together by
// the launch's terms; they are bounded all the same.  A block that has lost one leaves when its copies have landed, and last.
#pragma once

#include "fsd_finish.cuh"

namespace fsd {

constexpr int kRowMaxPairs = kFinishWarps;            // positions of a batch row: a warp judges one (3 x 20 x 16000 with two a warp: 14.9 us, the general path 12.9)
constexpr int kRowItemsPerWarp = 7;                   // at most; a warp's 128 columns of tensor memory would park eight (26 x 5 x 31000: 19.3 us, the general path 17.4)
constexpr int kRowMaxItems = kFinishWarps * kRowItemsPerWarp;
static_assert(kRowMaxPairs < 32 && kRowMaxPairs <= kPairRefs && kRowItemsPerWarp * kParkCols <= 128, "a lane and a reference per pair, columns");

struct alignas(16) RowPost {                          // a warp's sums of a pair
    float z[4];                // za, zb, s0, sb
    float ka, kb;
    float x;                   // second-sweep sum
    uint32_t diff;
};
static_assert(sizeof(RowPost) == 32, "16-byte accesses");

struct RowExchange {
    uint64_t landed[kRowMaxPairs + 1];                // a pair's rows; the bonus row
    uint64_t sums_in[kRowMaxPairs];                   // all blocks' sums of a pair (of the first: and the call's number)
    uint64_t ready[kRowMaxPairs];                     // its totals
    uint64_t x_in;                                    // all blocks' second-sweep sums of all pairs
    uint64_t number;                                  // the call's, as the cluster's first block read it
    alignas(16) float4 zsums[kRowMaxPairs][kMaxClusterSize];      // ka, Za, kb, Zb of each block
    float4 rest[kRowMaxPairs][kMaxClusterSize];       // its s0, sb, "rows differ"
    uint64_t x[kRowMaxPairs][kMaxClusterSize];        // (a float's bits)
    float4 tot[kRowMaxPairs];                         // Ka, 1/Za, Kb, 1/Zb
    RowPost post[kFinishWarps + kRowMaxPairs];        // warp w's of pair p at w + p: the warps' runs of items follow one another
    int first_done[kRowMaxPairs], second_done[kRowMaxPairs];
    uint32_t tmem_base;
};
template <int DT, int KIND> struct RowShared {
    RowExchange ex;
    FinishShared sh;
    ResidualShared rs;
    ExpTable<DT> bt;
};
template <int DT> struct RowShared<DT, kDrawPt> { RowExchange ex; FinishShared sh; TreeShared tr; };
template <int DT> struct RowShared<DT, kDrawGreedy> { RowExchange ex; FinishShared sh; TreeShared tr; };
// Shared memory of a block: all there is, so that no other block is on its SM (a block of another cluster that waits for
// tensor memory there while its own cluster waits for it could wait for good).
constexpr int kRowSmemBytes = 227 * 1024;
template <int DT, int KIND> __host__ __device__ constexpr int row_smem_left() { return kRowSmemBytes - static_cast<int>((sizeof(RowShared<DT, KIND>) + 127) / 128 * 128) - 128; }
// bytes of the logits of a row with G pairs in a block
__host__ __device__ constexpr int row_bytes_of(int G, int span, bool ragged) { return (2 * G + 1) * span * 16 + (ragged ? G * 32 : 0); }

struct RowParams {
    FinishParams fin;          // (records: not null, not read)
    int nvec_row;              // granules of a row, at most
    int span;                  // of which a block takes so many: whole steps
    uint64_t nonce;
    uint64_t limit_ns;         // of a wait
    int silent;                // test aid: the last block of each cluster keeps its first sums to itself
    int raise;                 // test aid: every row is marked
};

// ---- a step of the first sweep: eight entries a lane and row ---------------------------------
struct Sums { uint64_t za2, zb2, sa2, sb2; float kk; uint32_t diff; };     // packed (even, odd) partial sums
constexpr float kClampAt = -1.0e30f;
template <int DT> constexpr uint32_t kFillBits = DT == FSD_BF16 ? 0xF149F149u : 0xF149F2CAu;      // its bits, as entries of a vector
template <int DT> __device__ __forceinline__ uint4 fill_vector() { return make_uint4(kFillBits<DT>, kFillBits<DT>, kFillBits<DT>, kFillBits<DT>); }
// CLAMP (JS): -inf becomes -1e30: 2^y = 0 and 0 * y = 0 stay finite (NaN passes through); no other bit changes by it
template <int DT, int DIV, bool CLAMP>
__device__ __forceinline__ void first_step(uint4 (&wa)[StreamShape<DT>::kVecPerStep], uint4 (&wb)[StreamShape<DT>::kVecPerStep], float ca, float cb, Sums& t, float (&e)[kParkCols]) {
    constexpr int EPV = Logit<DT>::kPerVec;
    const uint64_t l2 = pack2(kLog2e, kLog2e), ca2 = pack2(ca, ca), cb2 = pack2(cb, cb);
#pragma unroll
    for (int v = 0; v < StreamShape<DT>::kVecPerStep; ++v) {
        uint4 a = wa[v], b = wb[v];
        if constexpr (CLAMP && DIV == FSD_DIV_JS && DT == FSD_BF16) {
            constexpr uint32_t c = kFillBits<DT>;
            a.x = bf16x2_max_nan(a.x, c); a.y = bf16x2_max_nan(a.y, c); a.z = bf16x2_max_nan(a.z, c); a.w = bf16x2_max_nan(a.w, c);
            b.x = bf16x2_max_nan(b.x, c); b.y = bf16x2_max_nan(b.y, c); b.z = bf16x2_max_nan(b.z, c); b.w = bf16x2_max_nan(b.w, c);
        }
        if constexpr (DIV != FSD_DIV_TV) t.diff |= (a.x ^ b.x) | (a.y ^ b.y) | (a.z ^ b.z) | (a.w ^ b.w);
        float xa[EPV], xb[EPV];
        unpack_vec<DT>(a, xa);
        unpack_vec<DT>(b, xb);
#pragma unroll
        for (int j = 0; j < EPV; j += 2) {
            float a0 = xa[j], a1 = xa[j + 1], b0 = xb[j], b1 = xb[j + 1];
            if constexpr (CLAMP && DIV == FSD_DIV_JS && DT == FSD_F32) {
                a0 = fmax_nan(a0, kClampAt); a1 = fmax_nan(a1, kClampAt); b0 = fmax_nan(b0, kClampAt); b1 = fmax_nan(b1, kClampAt);
            }
            const uint64_t ya2 = fma2(pack2(a0, a1), l2, ca2), yb2 = fma2(pack2(b0, b1), l2, cb2);
            float ya0, ya1, yb0, yb1;
            unpack2(ya2, ya0, ya1);
            unpack2(yb2, yb0, yb1);
            const float ea0 = ex2(ya0), ea1 = ex2(ya1), eb0 = ex2(yb0), eb1 = ex2(yb1);
            const uint64_t ea2 = pack2(ea0, ea1), eb2 = pack2(eb0, eb1);
            t.za2 = add2(t.za2, ea2);
            t.zb2 = add2(t.zb2, eb2);
            if constexpr (DIV == FSD_DIV_JS) {
                t.sa2 = fma2(ea2, ya2, t.sa2);
                t.sb2 = fma2(eb2, yb2, t.sb2);
            }
            if constexpr (DIV == FSD_DIV_KL) {       // (q = 0 < p, a draft logit of -inf, gives +inf)
                if (ea0 > 0.f) t.kk = fmaf(ea0, ya0 - yb0, t.kk);
                if (ea1 > 0.f) t.kk = fmaf(ea1, ya1 - yb1, t.kk);
            }
            e[v * EPV + j] = ea0; e[v * EPV + j + 1] = ea1;
            e[kStepEntries + v * EPV + j] = eb0; e[kStepEntries + v * EPV + j + 1] = eb1;
        }
    }
}
// A step of the second sweep, from parked values; ia, ib bring them to p and q
template <int DIV>
__device__ __forceinline__ void second_step(const float (&e)[kParkCols], float ia, float ib, uint64_t& x2) {
    const uint64_t ia2 = pack2(ia, ia), ib2 = pack2(ib, ib);
    // s = p + q + 1e-37 keeps lg2 finite where both terms vanish; the shift is below one ulp of any s that matters
    const uint64_t tiny2 = pack2(1e-37f, 1e-37f);
#pragma unroll
    for (int j = 0; j < kStepEntries; j += 2) {
        const uint64_t ea2 = pack2(e[j], e[j + 1]), eb2 = pack2(e[kStepEntries + j], e[kStepEntries + j + 1]);
        if constexpr (DIV == FSD_DIV_JS) {
            const uint64_t s2 = fma2(eb2, ib2, fma2(ea2, ia2, tiny2));
            float s0, s1;
            unpack2(s2, s0, s1);
            x2 = fma2(s2, pack2(lg2(s0), lg2(s1)), x2);
        } else {
            // separately rounded products: a fused p - q would make TV(p, p) != 0
            const uint64_t d2 = fma2(mul2(eb2, ib2), pack2(-1.f, -1.f), mul2(ea2, ia2));
            float d0, d1;
            unpack2(d2, d0, d1);
            x2 = add2(x2, pack2(fabsf(d0), fabsf(d1)));
        }
    }
}
// Four values summed over the warp: lanes 8 q to 8 q + 7 return the q-th sum.
__device__ __forceinline__ float fold_four(float v0, float v1, float v2, float v3, int lane) {
    const bool hi = (lane & 16) != 0, up = (lane & 8) != 0;
    const float k0 = (hi ? v2 : v0) + __shfl_xor_sync(0xffffffffu, hi ? v0 : v2, 16);
    const float k1 = (hi ? v3 : v1) + __shfl_xor_sync(0xffffffffu, hi ? v1 : v3, 16);
    float k = (up ? k1 : k0) + __shfl_xor_sync(0xffffffffu, up ? k0 : k1, 8);
#pragma unroll
    for (int m = 4; m > 0; m >>= 1) k += __shfl_xor_sync(0xffffffffu, k, m);
    return k;
}
// 1/Z to the last bit or so; 0 where the row is not a valid distribution (NaN included)
__device__ __forceinline__ float reciprocal_total(float z) {
    if (!(z > 1.0e-30f && z < 1.0e30f)) return 0.f;
    const float r = rcp(z);
    return fmaf(r, fmaf(-z, r, 1.f), r);
}
// Totals of a pair from its blocks' sums {ka, Za, kb, Zb}, a lane each (lanes 0 to 15 the target row's, 16 to 31 the draft row's):
// every lane returns the largest reference and 1/Z of its half's row.
__device__ __forceinline__ float2 pair_totals(const float4* sums, int cs, int lane) {
    const bool b_side = lane >= 16;
    float k = -INFINITY, z = 0.f;
    if ((lane & 15) < cs) {
        const float2 m = reinterpret_cast<const float2*>(sums + (lane & 15))[b_side];
        k = m.x; z = m.y;
    }
    const float Ka = warp_redux_max_nan(b_side ? -INFINITY : k), Kb = warp_redux_max_nan(b_side ? k : -INFINITY);
    const float K = b_side ? Kb : Ka;
    z *= pow2_ref(k, K);
#pragma unroll
    for (int m = 8; m > 0; m >>= 1) z += __shfl_xor_sync(0xffffffffu, z, m);
    return make_float2(K, reciprocal_total(z));
}

// Bounded wait of a thread; `lost` remembers that one has run out and ends further waits.
__device__ __noinline__ bool row_wait_slow(uint64_t* bar, uint64_t limit_ns) {
    const uint64_t t0 = global_ns();
#pragma unroll 1
    for (uint32_t i = 0; i < kSpinLimit; ++i) {
#pragma unroll 1
        for (int k = 0; k < 16; ++k) if (mbar_try_wait(bar, 0)) return true;
        if (global_ns() - t0 > limit_ns) break;
    }
    return false;
}
__device__ __forceinline__ void row_wait(uint64_t* bar, uint64_t limit_ns, bool& lost) {
    if (!lost && !mbar_try_wait(bar, 0) && !row_wait_slow(bar, limit_ns)) lost = true;
    __syncwarp();
}

template <int DT, int KIND, bool RAGGED>
__global__ void __launch_bounds__(kFinishThreads, 1) fsd_row_kernel(const __grid_constant__ RowParams P) {
    constexpr int EPV = Logit<DT>::kPerVec, VPS = StreamShape<DT>::kVecPerStep, SV = 32 * VPS;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127));
    RowShared<DT, KIND>& all = *reinterpret_cast<RowShared<DT, KIND>*>(smem);
    RowExchange& ex = all.ex;
    FinishShared& sh = all.sh;
    ResidualShared* rs = nullptr;
    ExpTable<DT>* bt = nullptr;
    if constexpr (KIND == kDrawResidual) { rs = &all.rs; bt = &all.bt; }
    const FinishParams& F = P.fin;
    cg::cluster_group cluster = cg::this_cluster();
    const int cs = static_cast<int>(cluster.num_blocks()), rank = static_cast<int>(cluster.block_rank());
    const int b = static_cast<int>(blockIdx.x) / cs;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int G = F.G, V = F.V, span = P.span;
    const size_t rb = static_cast<size_t>(V) * Logit<DT>::kBytes;
    const char* t_base = static_cast<const char*>(F.target) + static_cast<size_t>(b) * (G + 1) * rb;
    const char* d_base = static_cast<const char*>(F.draft) + static_cast<size_t>(b) * G * rb;
    const bool second = F.div != FSD_DIV_KL;
    // this block's granules of every row; items of a pair (one, empty, where it has none)
    const int vbeg = min(rank * span, P.nvec_row), vcnt = min(span, P.nvec_row - vbeg);
    const int steps = max(1, (vcnt + SV - 1) / SV), n_items = steps * G;
    const int workers = min(kFinishWarps, n_items);       // (each has an item)
    const int q0 = min(warp, workers) * n_items / workers, q1 = min(warp + 1, workers) * n_items / workers;      // this warp's items
    const auto warp_of = [&](int item) { return (workers * (item + 1) - 1) / n_items; };         // and whose an item is
    // the rows in shared memory: target rows, then draft rows (unaligned ones with a granule more at both ends)
    const uint32_t row_stride = static_cast<uint32_t>(span) * 16, d_stride = row_stride + (RAGGED ? 32 : 0);
    const uint32_t t_smem = smem_u32(smem) + static_cast<uint32_t>((sizeof(RowShared<DT, KIND>) + 127) / 128 * 128);
    const uint32_t d_smem = t_smem + (G + 1) * row_stride;
    FSD_CHECK(&F.flags->debug, G <= kRowMaxPairs && n_items <= kRowMaxItems && span % SV == 0, kChkSlice);
    FSD_CHECK(&F.flags->debug, row_bytes_of(G, span, RAGGED) <= (row_smem_left<DT, KIND>()), kChkStage);

    if (tid == 0) {
        for (int p = 0; p < G; ++p) { mbar_init(&ex.landed[p], 1); mbar_init(&ex.sums_in[p], 1); mbar_init(&ex.ready[p], 1); }
        mbar_init(&ex.landed[G], 1); mbar_init(&ex.x_in, 1);
        mbar_init(&sh.link[0], 1); mbar_init(&sh.link[1], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        for (int p = 0; p < G; ++p) mbar_arrive_expect_tx(&ex.sums_in[p], static_cast<uint32_t>(cs) * 32 + (p == 0 ? 8 : 0));
        mbar_arrive_expect_tx(&ex.x_in, second ? static_cast<uint32_t>(cs * G) * 8 : 0);
        sh.cand = -1; sh.last_pos = -1; sh.n_acc = G; sh.bad = 0; sh.row_sel = 0; sh.amb = 0; sh.n_close = 0; sh.next = 0; sh.far = 0;
    }
    if (tid < kRowMaxPairs) { ex.first_done[tid] = 0; ex.second_done[tid] = 0; }
    if (warp == 1 && second) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&ex.tmem_base)), "n"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if constexpr (KIND == kDrawResidual) residual_tables(*rs, tid);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");     // "this block's barriers are ready": waited for before the first push
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");                        // from here on global memory is touched

    // ---- copies: a warp those of pair p, or (p = G) the bonus row's: one warp for all of them took 2000 cycles ----
#pragma unroll 1
    for (int p = warp; p <= G; p += kFinishWarps) {
        if (lane != 0) continue;
        const char* arow = t_base + static_cast<size_t>(p) * rb;
        const uint32_t t_dst = t_smem + p * row_stride;
        uint32_t ba = static_cast<uint32_t>(vcnt) * 16, bb = p < G ? ba : 0, d_dst = d_smem + p * d_stride;
        const char* asrc = arow + static_cast<size_t>(vbeg) * 16;
        const char* bsrc = d_base + static_cast<size_t>(p) * rb + static_cast<size_t>(vbeg) * 16;
        if constexpr (RAGGED) {
            // the granules that cover the rows, from each row's rounded-down start
            const char* brow = d_base + static_cast<size_t>(p) * rb;
            const int oa = static_cast<int>(reinterpret_cast<uintptr_t>(arow) & 15), ob = static_cast<int>(reinterpret_cast<uintptr_t>(brow) & 15);
            const int na = static_cast<int>((oa + rb + 15) >> 4), nb = static_cast<int>((ob + rb + 15) >> 4);
            const int a1 = min(vbeg + vcnt, na), b0 = max(vbeg - 1, 0), b1 = min(vbeg + vcnt + 1, nb);
            ba = a1 > vbeg ? static_cast<uint32_t>(a1 - vbeg) * 16 : 0;
            bb = p < G && vcnt > 0 && b1 > b0 ? static_cast<uint32_t>(b1 - b0) * 16 : 0;
            asrc = arow - oa + static_cast<size_t>(vbeg) * 16;
            bsrc = brow - ob + static_cast<size_t>(b0) * 16;
            d_dst += static_cast<uint32_t>(b0 - (vbeg - 1)) * 16;
        }
        mbar_arrive_expect_tx(&ex.landed[p], ba + bb);
        if (ba != 0) bulk_g2s(t_dst, asrc, ba, &ex.landed[p]);
        if (bb != 0) bulk_g2s(d_dst, bsrc, bb, &ex.landed[p]);
    }
    // what the judgement wants from global memory, on its way meanwhile
    Candidate cand = {-1, 0.f, 0.f, 0.f};
    if constexpr (KIND == kDrawResidual) {
        if (warp < G) cand = candidate<DT, KIND>(F, b * G + warp, t_base + static_cast<size_t>(warp) * rb, d_base + static_cast<size_t>(warp) * rb);
        if constexpr (DT == FSD_BF16) {                   // (longer than the copies take: 12 x 6 x 32000, the warps are through 2500 to 5000 cycles after the start, the first rows land after 1270)
            for (int i = tid; i < kBf16Count; i += kFinishThreads) bf16_table_entry(*bt, *rs, i);
        }
    }
    // lane p: the target row pair p is judged against (a tree: its parent's; an invalid one moves ignored data)
    int my_row = lane;
    bool my_bad = false;
    if constexpr (KIND != kDrawResidual) {
        if (F.parent != nullptr) {
            const int parent = lane < G ? __ldg(F.parent + static_cast<size_t>(b) * G + lane) : -1;
            my_bad = lane < G && (parent < -1 || parent >= lane);
            my_row = my_bad ? 0 : parent + 1;
        }
    }
    uint64_t number = 0;
    if (tid == 0) {
        sh.u = F.u_sample[b];
        if (rank == 0) number = call_number(F.flags, P.nonce);
    }
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");       // every block of the cluster runs and its barriers are ready

    bool lost = false;
    const uint32_t taddr = second ? ex.tmem_base + (static_cast<uint32_t>(32 * (warp & 3)) << 16) + static_cast<uint32_t>(128 * (warp >> 2)) : 0;
    // What a block raises where a wait of the draw's runs out is the number the first block of its cluster looks for: that block's
    // own reading, to all of them.  (A row 0 that ends meanwhile moves the epoch on, and two blocks could read two numbers.
    // Told in front of the first sweep, 16 x 5 x 32000 took 0.04 us more: the reading is a trip to L2.)
    const auto tell_number = [&] {
        if (rank == 0 && warp == 0) {
            const uint64_t n = __shfl_sync(0xffffffffu, number, 0);
            if (lane < cs) st_async(cluster_addr(&ex.number, lane), n, cluster_addr(&ex.sums_in[0], lane));
        }
    };
    const auto sweeps = [&](auto div_tag) {
        constexpr int DIV = decltype(div_tag)::value;
        // A vector of item (p, step)'s rows, target row `tr`
        const auto fetch = [&](int p, int tr, int step, int v, uint4& wa, uint4& wb) {
            const int g = step * SV + v * 32 + lane;      // granule of the block's share
            wa = fill_vector<DT>(); wb = wa;              // (where there is nothing: 2^y = 0)
            if (g >= vcnt) return;
            wa = ld_shared16(t_smem + tr * row_stride + g * 16);
            if constexpr (!RAGGED) {
                wb = ld_shared16(d_smem + p * d_stride + g * 16);
            } else {                                      // the draft row's entries moved onto the target row's
                const int oa = static_cast<int>((reinterpret_cast<uintptr_t>(t_base) + tr * rb) & 15), ob = static_cast<int>((reinterpret_cast<uintptr_t>(d_base) + p * rb) & 15);
                const uint32_t at = d_smem + p * d_stride + (g + (ob < oa ? 0 : 1)) * 16, shift = static_cast<uint32_t>(ob - oa) & 15u;
                wb = ld_shared16(at);
                if (shift != 0) wb = shifted<DT>(wb, ld_shared16(at + 16), shift);
                if (vbeg + g == 0 || vbeg + g >= P.nvec_row - 2) {
                    const int k0 = (vbeg + g) * EPV - oa / Logit<DT>::kBytes;
                    wa = masked_vector<DT>(wa, k0, V);
                    wb = masked_vector<DT>(wb, k0, V);
                }
            }
        };
        // ---- 1. first sweep: this warp's items of one pair after another ----
#pragma unroll 1
        for (int q = q0, j = 0, p = q0 / steps; q < q1; ++p) {
            const int s0 = q - p * steps, n = min(q1 - q, steps - s0);       // its steps s0 to s0 + n - 1 of the pair
            const int tr = __shfl_sync(0xffffffffu, my_row, p);
            row_wait(&ex.landed[p], P.limit_ns, lost);
            if (tr != p) row_wait(&ex.landed[tr], P.limit_ns, lost);
            // The references come from the maxima of the first step, or of all of them where that has no finite logit: near enough for
            // ordinary logits (see kNearZ), otherwise the sweep is done over with exact maxima.
            float ka, kb;
            const auto look = [&](int items) {
                float ma = -INFINITY, mb = -INFINITY;
#pragma unroll 1
                for (int v = 0; v < items * VPS; ++v) {
                    uint4 wa, wb;
                    fetch(p, tr, s0 + v / VPS, v % VPS, wa, wb);
                    ma = fmax_nan(ma, vector_max<DT>(wa)); mb = fmax_nan(mb, vector_max<DT>(wb));
                }
                __syncwarp();
                ka = reference(warp_redux_max_nan(ma)); kb = reference(warp_redux_max_nan(mb));
            };
            look(1);
            if (n > 1 && (ka == -INFINITY || kb == -INFINITY)) look(n);
            Sums t;
            float za, zb;
#pragma unroll 1
            for (bool again = false;; again = true) {
                const float ca = ka == -INFINITY ? 0.f : -ka, cb = kb == -INFINITY ? 0.f : -kb;
                t = Sums{0, 0, 0, 0, 0.f, 0};
#pragma unroll 2
                for (int i = 0; i < n; ++i) {
                    uint4 wa[VPS], wb[VPS];
                    float e[kParkCols];
#pragma unroll
                    for (int v = 0; v < VPS; ++v) fetch(p, tr, s0 + i, v, wa[v], wb[v]);
                    first_step<DT, DIV, true>(wa, wb, ca, cb, t, e);
                    if constexpr (DIV != FSD_DIV_KL) {
                        FSD_CHECK(&F.flags->debug, j + i < kRowItemsPerWarp, kChkTmem);
                        __syncwarp();
                        tmem_st16(taddr + (j + i) * kParkCols, e);
                    }
                }
                za = sum2(t.za2); zb = sum2(t.zb2);
                if (again || n == 1 || __all_sync(0xffffffffu, za + zb < kNearZ)) break;
                look(n);
                if constexpr (DIV != FSD_DIV_KL) tmem_wait_st();     // what was stored goes to the same columns: it has to be there first
            }
            q += n; j += n;
            // folded over the lanes, posted; the last of the pair's posts are folded, a lane each, and pushed
            const float k = fold_four(za, zb, DIV == FSD_DIV_KL ? t.kk : sum2(t.sa2), sum2(t.sb2), lane);
            const bool differ = DIV == FSD_DIV_TV || __any_sync(0xffffffffu, t.diff != 0);
            RowPost& post = ex.post[warp + p];
            if ((lane & 7) == 0) post.z[lane >> 3] = k;
            if (lane == 4) *reinterpret_cast<float4*>(&post.ka) = make_float4(ka, kb, 0.f, __uint_as_float(differ ? 1u : 0u));
            __syncwarp();
            const int w0 = warp_of(p * steps), posts = warp_of((p + 1) * steps - 1) - w0 + 1;
            int done = 0;                                 // (what a warp that has lost posts is nobody's: its block sends nothing then, and its cluster's waits run out)
            if (lane == 0 && !lost) { __threadfence_block(); done = atomicAdd(&ex.first_done[p], 1) + 1; }
            if (__shfl_sync(0xffffffffu, done, 0) == posts) {
                __threadfence_block();
                const RowPost w = lane < posts ? ex.post[w0 + p + lane] : RowPost{{0.f, 0.f, 0.f, 0.f}, -INFINITY, -INFINITY, 0.f, 0u};
                const float Ka = warp_redux_max_nan(w.ka), Kb = warp_redux_max_nan(w.kb);
                const float fa = pow2_ref(w.ka, Ka), fb = pow2_ref(w.kb, Kb);
                const float da = w.ka == -INFINITY ? 0.f : w.ka - Ka, db = w.kb == -INFINITY ? 0.f : w.kb - Kb;
                const float v2 = DIV == FSD_DIV_KL ? scale_kl(fa, fmaf(da - db, w.z[0], w.z[2])) : fa * fmaf(da, w.z[0], w.z[2]);
                const float v3 = DIV == FSD_DIV_KL ? 0.f : fb * fmaf(db, w.z[1], w.z[3]);
                const float sum = fold_four(__fmul_rn(w.z[0], fa), __fmul_rn(w.z[1], fb), v2, v3, lane);
                const uint32_t any = __any_sync(0xffffffffu, w.diff != 0) ? 1u : 0u;
                const float Za = __shfl_sync(0xffffffffu, sum, 0), Zb = __shfl_sync(0xffffffffu, sum, 8), sa = __shfl_sync(0xffffffffu, sum, 16), sb = __shfl_sync(0xffffffffu, sum, 24);
                if (!(P.silent && rank == cs - 1 && p == 0)) {
                    for (int i = lane; i < 4 * cs; i += 32) {
                        const int peer = i >> 2, k4 = i & 3;
                        const uint64_t word = k4 == 0 ? pack2(Ka, Za) : k4 == 1 ? pack2(Kb, Zb) : k4 == 2 ? pack2(sa, sb) : any;
                        st_async(cluster_addr(k4 < 2 ? &ex.zsums[p][rank] : &ex.rest[p][rank], peer) + (k4 & 1) * 8, word, cluster_addr(&ex.sums_in[p], peer));
                    }
                }
            }
        }
        tell_number();
        if constexpr (DIV != FSD_DIV_KL) {
            __syncwarp();
            tmem_wait_st();
            // ---- 2. totals, a warp per pair ----
            if (warp < G) {
                const int p = warp;
                row_wait(&ex.sums_in[p], P.limit_ns, lost);
                const float2 tot = pair_totals(ex.zsums[p], cs, lane);
                if ((lane & 15) == 0) reinterpret_cast<float2*>(&ex.tot[p])[lane >> 4] = tot;
                __syncwarp();
                if (lane == 0 && !lost) mbar_arrive(&ex.ready[p]);
            }
            // ---- 3. second sweep ----
#pragma unroll 1
            for (int q = q0, j = 0, p = q0 / steps; q < q1; ++p) {
                const int n = min(q1 - q, (p + 1) * steps - q);
                row_wait(&ex.ready[p], P.limit_ns, lost);
                const float4 t = ex.tot[p];
                RowPost& post = ex.post[warp + p];
                const float ia = pow2_ref(post.ka, t.x) * t.y, ib = pow2_ref(post.kb, t.z) * t.w;
                uint64_t x2 = 0;
                __syncwarp();
#pragma unroll 2
                for (int i = 0; i < n; ++i) {
                    float e[kParkCols];
                    tmem_ld16(taddr + (j + i) * kParkCols, e);
                    tmem_wait_ld();
                    second_step<DIV>(e, ia, ib, x2);
                }
                q += n; j += n;
                float x = sum2(x2);
#pragma unroll
                for (int m = 16; m > 0; m >>= 1) x += __shfl_xor_sync(0xffffffffu, x, m);
                const int w0 = warp_of(p * steps), posts = warp_of((p + 1) * steps - 1) - w0 + 1;
                int done = 0;
                if (lane == 0 && !lost) { post.x = x; __threadfence_block(); done = atomicAdd(&ex.second_done[p], 1) + 1; }
                if (__shfl_sync(0xffffffffu, done, 0) == posts) {
                    __threadfence_block();
                    float v = lane < posts ? *const_cast<volatile float*>(&ex.post[w0 + p + lane].x) : 0.f;
#pragma unroll
                    for (int m = 8; m > 0; m >>= 1) v += __shfl_xor_sync(0xffffffffu, v, m);
                    v = __shfl_sync(0xffffffffu, v, 0);
                    if (lane < cs) st_async(cluster_addr(&ex.x[p][rank], lane), __float_as_uint(v), cluster_addr(&ex.x_in, lane));
                }
            }
        }
    };
    if (F.div == FSD_DIV_JS) sweeps(std::integral_constant<int, FSD_DIV_JS>{});
    else if (F.div == FSD_DIV_KL) sweeps(std::integral_constant<int, FSD_DIV_KL>{});
    else sweeps(std::integral_constant<int, FSD_DIV_TV>{});

    // ---- 4. divergences, accept bits, status: a pair per warp; what does not need the second sweep's sums comes before they do ----
    int st = 0, first = G;
    if (warp < G) {
        const int i = warp;
        row_wait(&ex.sums_in[i], P.limit_ns, lost);
        Stats c = no_stats();
        if (lane < cs) {
            const float4 z = ex.zsums[i][lane], r = ex.rest[i][lane];
            c.ka = z.x; c.za = z.y; c.kb = z.z; c.zb = z.w; c.s0 = r.x; c.sb = r.y; c.diff = __float_as_uint(r.z);
        }
        PairTotals tot = fold_parts(c, 0.f, __shfl_sync(0xffffffffu, my_bad, i) ? kRecordBadTree : kRecordStats, F.div);
        const Judged early = judge_pair_early<KIND>(F, rs, tot, i, cand, lane);
        if (second) {
            row_wait(&ex.x_in, P.limit_ns, lost);
            tot.X = warp_sum(lane < cs ? static_cast<double>(__uint_as_float(static_cast<uint32_t>(ex.x[i][lane]))) : 0.0);
        }
        if (lane == 0) {
            float D;
            int bit, s;
            judge_late(F, tot, early, D, bit, s);
            if (rank == 0) F.divergence[b * G + i] = D;
            st |= s;
            bool tree = false;
            if constexpr (KIND != kDrawResidual) { tree = F.parent != nullptr; if (tree) all.tr.bit[i] = static_cast<int8_t>(bit); }
            if (!tree && !bit && i < first) first = i;
        }
    }
    if (lane == 0) {
        if (st) atomicOr(&sh.bad, st);
        if (first < G) atomicMin(&sh.n_acc, first);
    }
    if (warp == kFinishWarps - 1) row_wait(&ex.landed[G], P.limit_ns, lost);      // (every pair's copies have been waited for by somebody; without them nobody has got here)
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    Link link = {0, __syncthreads_or(lost) != 0, &ex.number};
    if (link.lost && tid <= G) thread_wait(&ex.landed[tid], 0, 0);             // no copy may still be on its way into a block that leaves
    if (second) {                                         // the second sweep is through with tensor memory
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(ex.tmem_base), "n"(kTmemCols) : "memory");
    }

    // ---- 5. accepted prefix or path, token ----
    int n = sh.n_acc, row_sel = n;
    if constexpr (KIND != kDrawResidual) {
        if (F.parent != nullptr && !link.lost) {
            tree_select(F.parent + static_cast<size_t>(b) * G, G, F.max_depth, rank == 0 ? F.path + static_cast<size_t>(b) * F.max_depth : nullptr, sh, all.tr);
            __syncthreads();
            n = sh.n_acc; row_sel = sh.row_sel;
            FSD_CHECK(&F.flags->debug, n >= 0 && n <= F.max_depth, kChkPath);
        }
    }
    int status = sh.bad;
    FSD_CHECK(&F.flags->debug, link.lost || (n >= 0 && row_sel >= 0 && row_sel <= G), kChkRow);
    if (link.lost) {
        n = 0;                                            // (nothing of the row is valid but its status)
    } else if (status & FSD_ROW_BADTREE) {
        n = 0;
        if (rank == 0 && tid == 0) F.next_token[b] = -1;
    } else {
        const bool rejected = KIND == kDrawResidual && n < G;
        Draw d;
        d.a_row = t_base + static_cast<size_t>(row_sel) * rb;
        d.b_row = d_base + static_cast<size_t>(rejected ? n : 0) * rb;
        d.b = b; d.n = n; d.V = V; d.cs = cs; d.rank = rank; d.shared_out = false; d.vec = F.vec != 0; d.u = static_cast<double>(sh.u);
        d.span = span; d.local = t_smem + row_sel * row_stride - static_cast<uint32_t>(vbeg) * 16;
        draw_token<DT, KIND, true>(F, sh, rs, bt, d, link, status, rejected);
    }
    if (rank == 0 && tid == 0) {
        F.accept_len[b] = n;
        F.row_status[b] = status | (link.lost || P.raise || timed_out(F.flags, number) ? FSD_ROW_TIMEOUT : 0);
        // (The rows need nothing of one another, and a row is marked where a wait of its own cluster ran out: a block that has lost one before the draw sends
        // nothing there, so that this block's own wait runs out; one that loses one in the draw has raised the flag, see cluster_exchange.  A cluster that starts
        // after row 0's has ended, other kernels in its place until then, has another number, which is raised and looked for by itself alone.)
        if (b == 0) { F.flags->number = number; atomicAdd(reinterpret_cast<unsigned long long*>(&F.flags->epoch), 1ull); }
    }
    leave_last(link.lost);
}

}  // namespace fsd
