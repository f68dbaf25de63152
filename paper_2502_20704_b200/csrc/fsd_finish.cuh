// Finish kernel: one thread-block cluster per batch row.
//   1. Turns the per-pair totals left by the streaming kernel into divergences and accept
//      bits (or takes the bits the generic kernel already wrote).
//   2. Finds the accepted prefix (chain) or the deepest accepted path (tree).
//   3. Draws the replacement / bonus token from one target row (and, for the SD residual, one
//      draft row) by an inverse CDF in vocabulary order.
//
// The kernel is serial by nature -- judge, choose the row, read it, total it, find the crossing -- and takes
// 6 us on a small batch, most of them trips to L2 and instructions that run once.  So each kind of
// draw is an instantiation of its own, the cluster's CTAs tell one another what they must by remote
// stores that count themselves in (no cluster barrier in the path), and a row is read once.
//
// Drawing from P_T (the FSD rule, and every bonus token): each warp owns a contiguous run of the
// vocabulary, each thread a reference exponent of its own, the largest logit it has met so far (moved by
// exact powers of two); the weights are single-precision exponentials (one MUFU ex2 each, relative error
// at most a few 1e-7) summed in double precision.  The sums, brought to one scale, are combined in a fixed
// order (thread -> warp -> CTA -> cluster), and the CTA that owns the warp in whose run the total passes
// u * total re-walks that run with the same weights, an iteration of it per warp.  The cumulative sums
// therefore differ from exact ones by less than 1e-6 of the total: the token is the exact one whenever
// u * total lies further than that from both ends of its interval, and a neighbour otherwise.
// Drawing from the SD residual max(0, P_T - P_D) (Eq. 3) subtracts nearly equal numbers, so there the
// exponentials are double precision and the sums agree with a sequential double sum to rounding.
// bf16 logits have few values: e^x comes from a table of all bf16 numbers between 2^-13 and 64 of either
// sign (built while the streaming kernel drains), which leaves two shared-memory reads and four
// double-precision instructions an entry.  fp32 logits take a 256-entry table times a degree-4
// polynomial (about forty instructions).  Usually one pass over the two rows suffices: which
// entries carry residual weight depends on the ratio of the two normalisers only, the rejected pair's
// record gives that ratio closely enough to class every entry that is not within a margin of the
// boundary, and the sums follow from the classed sums once the exact normalisers are known; entries
// inside the margin are settled afterwards, and a row with too many of them in one thread takes a
// second pass.
#pragma once

#include <climits>

#include "fsd_device.cuh"
#include "fsd_pair_generic.cuh"
#include "fsd_pair_stream.cuh"

namespace fsd {

constexpr int kFinishThreads = 512;
constexpr int kFinishWarps = kFinishThreads / 32;
constexpr int kMaxTreeNodes = 1024;

struct FinishParams {
    const void* target;        // [B, G+1, V]
    const void* draft;         // [B, G,   V]
    const int32_t* parent;     // tree only
    const int32_t* tokens;     // [B, G] or null
    const float* u_accept;     // [B, G] or null
    const float* u_sample;     // [B]
    int B, G, V;
    int div, mode, cmp, sample, max_depth;
    int vec;                   // rows are 16-byte aligned and a whole number of vectors
    float T;
    const PairRecord* records; // per-pair totals of the streaming kernel, or null (generic kernel ran)
    int32_t* item_bits;        // [B, G] read when records == null
    int32_t* item_status;      // [B, G] read when records == null
    CallFlags* flags;
    int silent;                // debug build, test aid: the last CTA of each cluster keeps its first exchange's values to itself (1) or sends them late (2)
    float* divergence;         // [B, G] written here when records != null
    int32_t* accept_len;       // [B]
    int32_t* path;             // [B, max_depth] (tree) or null
    int32_t* next_token;       // [B]
    int32_t* row_status;       // [B]
};

constexpr int kExchangeDoubles = 7;      // most values a CTA tells its cluster at once
// With more pairs than a CTA has warps, the cluster's CTAs share the judging (CTA r takes pairs r, r + cs, ...)
// and tell one another the accept bits: up to 64 * kJudgeWords of them each.
constexpr int kJudgeWords = 4;
constexpr int kExpTable = 256;
// e^x of the bf16 numbers with 2^-13 <= |x| < 64, both signs
constexpr int kBf16Lowest = 114 << 7, kBf16Count = 19 << 7;
// what a kernel draws: from P_T, its argmax, or (after a rejection) from the SD residual
enum : int { kDrawPt = 0, kDrawGreedy = 1, kDrawResidual = 2 };

struct FinishShared {
    uint64_t link[2];              // barriers of the cluster's exchanges
    double got[2][kMaxClusterSize][kExchangeDoubles];   // what the CTAs of the cluster sent (see cluster_exchange)
    double sc[kMaxClusterSize];
    double red_d[32 * 2];
    float red_f[32 * 2];
    double warp_tot[kFinishWarps];
    double seg_tot[kFinishWarps];  // of the iterations find_crossing looks at
    float warp_k[kFinishWarps];    // draw from P_T: the warps' largest references
    unsigned long long bits[kJudgeWords];   // accept bits of the pairs this CTA judged for its cluster
    float u;                   // the row's uniform
    int far;                   // draw from P_T: some thread's reference is out of a double's range; argmax: an invalid logit
    int amb;                   // residual draw: some thread needs the second pass
    int n_close;               // how many threads have close calls; two where one has some of two kinds
    int next;                  // part of the table to be built next
    int cand;                  // find_crossing: highest index with a positive weight
    int last_pos;              // highest index with a positive weight in this CTA
    int row_sel;               // target row the token is drawn from
    int n_acc;
    int bad;
    int best_key;              // depth * 2048 + (2047 - node) of the chosen tree node, or -1
};

struct TreeShared {
    int16_t parent[kMaxTreeNodes];
    int16_t jump[kMaxTreeNodes];
    int16_t depth[kMaxTreeNodes];
    int8_t ok[kMaxTreeNodes];
    int8_t bit[kMaxTreeNodes];
};
struct NoTree {};                  // (a residual draw is never a tree's)

// 2^y in double precision (relative error about 2e-16) for -1000 < y < 1000; 0 below, NaN for NaN.
// y = (k + r) / 256 with integer k and |r| <= 1/2: 2^y = 2^(k >> 8) * table[k & 255] * 2^(r/256),
// the last factor by a degree-4 polynomial in r (|r ln2 / 256| <= 1.4e-3, remainder < 5e-17).
__device__ __forceinline__ double exp2_table(double y, const double* table) {
    if (!(y > -1000.0)) return y != y ? y : 0.0;
    const double kMagic = 6755399441055744.0;                      // 1.5 * 2^52: the sum's low word is round(256 y)
    const double t = fma(y, 256.0, kMagic);
    const int k = __double2loint(t);
    const double r = fma(y, 256.0, kMagic - t);                    // 256 y - k, exact: |r| <= 1/2
    // coefficients (ln2 / 256)^i / i!
    double p = fma(r, 2.239395190875157e-12, 3.308302680541371e-09);
    p = fma(p, r, 3.665565596910106e-06);
    p = fma(p, r, 2.7076061740622863e-03);
    p = fma(p, r, 1.0);
    const double m = table[k & (kExpTable - 1)] * p;               // in [1, 2.0001)
    const int hi = __double2hiint(m) + ((k >> 8) << 20);           // scale by 2^(k >> 8): stays normal for |y| < 1000
    return __hiloint2double(hi, __double2loint(m));
}

// The same function, value for value above y = -990 and exactly 0 below about there, for the tight
// loops of the residual draw: no branch (callers clamp y and say when the result is to be 0; they
// have excluded NaN), and the constants
// come as arguments so that a loop keeps them in registers instead of rebuilding each 64-bit
// immediate at every use.
struct Exp2Consts { double magic, scale, c4, c3, c2, c1; };
__device__ __forceinline__ Exp2Consts exp2_consts(const double* opaque) {
    // read through shared memory: the compiler cannot turn them back into immediates
    return Exp2Consts{opaque[0], opaque[1], opaque[2], opaque[3], opaque[4], opaque[5]};
}
__device__ __forceinline__ double exp2_table_fast(double y, bool below, const double* table, const Exp2Consts& c) {
    const double t = fma(y, c.scale, c.magic);
    const int k = __double2loint(t);
    const double r = fma(y, c.scale, c.magic - t);
    double p = fma(r, c.c4, c.c3);
    p = fma(p, r, c.c2);
    p = fma(p, r, c.c1);
    p = fma(p, r, 1.0);
    const double m = table[k & (kExpTable - 1)] * p;
    const int hi = __double2hiint(m) + ((k >> 8) << 20);
    return below ? 0.0 : __hiloint2double(hi, __double2loint(m));     // a select, not a branch
}
// y = x * log2e - k for the tight loops: x is clamped in single precision at the logit below which
// y would pass -1000 (`xmin`, with a margin), and `below` tells exp2_table_fast to return exactly 0
__device__ __forceinline__ double exp2_of_logit(float x, float xmin, double nk, const double* table, const Exp2Consts& c) {
    const bool below = !(x > xmin);
    return exp2_table_fast(fma(static_cast<double>(fmaxf(x, xmin)), kLog2eD, nk), below, table, c);
}

// What the CTAs of a cluster tell one another: every CTA pushes a few doubles into every CTA's shared
// memory (its own included) and waits for all of its own to arrive.  No cluster barrier, no fence: the
// barrier.cluster form took twice as long.  Two barriers and buffers alternate, which is
// enough: nobody can be two exchanges ahead of a CTA whose values it still lacks.  The peers must be
// known to run (an arrive at kernel entry that is waited for before the first exchange); a CTA that
// has had its last exchange may leave.  Called by all threads with the same values, and with a barrier
// of the CTA between two calls; returns the buffer: got[rank][k].
// Where some thread's wait runs out, all of the CTA's give up: the call's flag is raised, `lost` is set and the caller
// has to return.  Such a CTA sends nothing any more (a peer that has what it needs may have left) and leaves last
// (others may send still).  The first CTA looks at the flag when it writes the row's status, at its end: a CTA that
// gave up waiting for somebody's values has raised it before they were sent, and the first has them all by then.
struct Link {
    int turn;                  // exchanges so far
    bool lost;                 // (the same for all of the CTA's threads)
    const uint64_t* number;    // where the call's number is: what the first CTA of the cluster looks for in the flag
};
template <int N>
__device__ __forceinline__ const double (*cluster_exchange(const FinishParams& P, FinishShared& sh, int cs, int rank, Link& link, const double (&v)[N]))[kExchangeDoubles] {
    static_assert(N <= kExchangeDoubles, "width of the exchange buffer");
    const int buf = link.turn & 1;
    if (threadIdx.x == 0) mbar_arrive_expect_tx(&sh.link[buf], static_cast<uint32_t>(cs) * N * 8);
    bool send = threadIdx.x < cs;
#ifdef FSD_DEBUG_CHECKS
    if (P.silent == 1 && link.turn == 0 && rank == cs - 1 && threadIdx.x != rank) send = false;
    if (P.silent == 2 && link.turn == 0 && rank == cs - 1) {
        const uint64_t t0 = global_ns();
        for (int i = 0; i < 100000 && global_ns() - t0 < 3 * kInjectedWaitNs; ++i) __nanosleep(1000);
    }
    const uint64_t limit_ns = P.silent == 1 || (P.silent == 2 && rank == 1) ? kInjectedWaitNs : P.silent == 2 ? 10 * kInjectedWaitNs : 0;
#else
    constexpr uint64_t limit_ns = 0;
#endif
    if (send) {
        const uint32_t dst = cluster_addr(&sh.got[buf][rank][0], threadIdx.x), bar = cluster_addr(&sh.link[buf], threadIdx.x);
#pragma unroll
        for (int k = 0; k < N; ++k) st_async(dst + 8 * k, static_cast<uint64_t>(__double_as_longlong(v[k])), bar);
    }
    link.lost = __syncthreads_or(!thread_wait(&sh.link[buf], (link.turn >> 1) & 1, limit_ns)) != 0;
    if (link.lost && threadIdx.x == 0) raise_flag(P.flags, *const_cast<const volatile uint64_t*>(link.number));
    ++link.turn;
    return sh.got[buf];
}

// Divergence, accept bit and status of one pair from the streaming kernel's totals.
// A pair's totals from the parts its record holds (one per block of the streaming group), in
// double: Z = sum 2^y, S = sum 2^y * y, K = sum 2^ya (ya - yb), all relative to the largest
// part reference (the parts' references are integers, so the factors are exact powers of two).
struct PairTotals {
    double Za, Zb, Sa, Sb, K, X;
    float ka, kb;
    uint32_t differ;
    uint32_t state;            // the record's state word
};
// 2^d for an integer-valued d <= 0, exact; 0 below the normal range
__device__ __forceinline__ double pow2_int_d(double d) {
    return d < -1022.0 ? 0.0 : __hiloint2double((1023 + static_cast<int>(d)) << 20, 0);
}
__device__ __forceinline__ Stats no_stats() {
    Stats c;
    c.ka = -INFINITY; c.kb = -INFINITY; c.za = 0.f; c.zb = 0.f; c.s0 = 0.f; c.sb = 0.f; c.x = 0.f; c.diff = 0;
    return c;
}
// Called by all 32 lanes, with a part of the pair each (no_stats() where there is none) and its second-sweep sum;
// every lane returns the totals.
__device__ __forceinline__ PairTotals fold_parts(const Stats& c, float x, uint32_t state, int div) {
    PairTotals t;
    t.state = state;
    const float ka = warp_redux_max_nan(c.ka), kb = warp_redux_max_nan(c.kb);      // NaN references win
    t.ka = ka; t.kb = kb;
    const double da = c.ka == -INFINITY ? 0.0 : static_cast<double>(c.ka) - ka;
    const double db = c.kb == -INFINITY ? 0.0 : static_cast<double>(c.kb) - kb;
    const double fa = (c.ka == -INFINITY || da != da) ? 0.0 : pow2_int_d(da);
    const double fb = (c.kb == -INFINITY || db != db) ? 0.0 : pow2_int_d(db);
    t.Za = warp_sum(fa * c.za); t.Zb = warp_sum(fb * c.zb);
    t.Sa = 0.0; t.Sb = 0.0; t.K = 0.0;
    if (div == FSD_DIV_KL) {
        const bool inf = c.s0 == INFINITY;
        const double k = inf ? 0.0 : fa * (static_cast<double>(c.s0) + (da - db) * c.za);
        t.K = warp_sum(k);
        if (__any_sync(0xffffffffu, inf)) t.K = static_cast<double>(INFINITY);
    } else {
        t.Sa = warp_sum(fa * (static_cast<double>(c.s0) + da * c.za));
        t.Sb = warp_sum(fb * (static_cast<double>(c.sb) + db * c.zb));
    }
    t.X = warp_sum(static_cast<double>(x));
    t.differ = __any_sync(0xffffffffu, c.diff != 0) ? 1u : 0u;
    return t;
}
// Lane r folds part r of the record.
__device__ inline PairTotals fold_record(const PairRecord* rec, int div) {
    static_assert(kMaxGroupSize <= 32, "one lane per part");
    const int r = threadIdx.x & 31;
    Stats c = no_stats();
    float x = 0.f;
    // every lane fetches its part at once with the count (one trip to L2); parts beyond the count are stale
    const int rr = r < kMaxGroupSize ? r : 0;
    const Stats cr = rec->part[rr];
    const float xr = rec->x[rr];
    const uint32_t state = rec->state;
    if (r < static_cast<int>(rec->ncta) && r < kMaxGroupSize) { c = cr; x = xr; }
    return fold_parts(c, x, state, div);
}

// A candidate's token, logits and uniform, for the ratio test (residual draws alone)
struct Candidate { int x; float ax, bx, ua; };
// What of a pair's judgement does not need the second sweep's sum
struct Judged {
    bool bad_tree, finite, ratio_ok;
    double base;               // KL: the divergence; JS: its part without the mixture's entropy
};
__device__ __forceinline__ Judged judge_early(const FinishParams& P, const PairTotals& r, double lnZa, double lnZb, const Candidate& c) {
    Judged j;
    j.bad_tree = (r.state & kRecordBadTree) != 0;
    j.finite = isfinite(r.ka) && isfinite(r.kb) && r.Za > 0.0 && r.Zb > 0.0 && isfinite(r.Za) && isfinite(r.Zb);
    j.base = divergence_base(P.div, r.Za, r.Zb, lnZa, lnZb, r.Sa, r.Sb, r.K);
    j.ratio_ok = false;
    if (P.mode != FSD_MODE_FSD && j.finite && c.x >= 0 && c.x < P.V) {
        double pacc;                                                    // Eq. 1
        if (c.bx == -INFINITY) {
            pacc = (c.ax != -INFINITY) ? 1.0 : 0.0;
        } else {
            // ln P(x) = (x*log2e - k) ln2 - ln Z with the same float log2e the sums were built with
            const double la = (static_cast<double>(c.ax) * static_cast<double>(kLog2e) - r.ka) * kLn2D - lnZa;
            const double lb = (static_cast<double>(c.bx) * static_cast<double>(kLog2e) - r.kb) * kLn2D - lnZb;
            pacc = exp(la - lb);
            pacc = pacc < 1.0 ? pacc : 1.0;
        }
        j.ratio_ok = static_cast<double>(c.ua) < pacc;                 // Eq. 2
    }
    return j;
}
__device__ __forceinline__ void judge_late(const FinishParams& P, const PairTotals& r, const Judged& j, float& D_out, int& bit_out, int& st_out) {
    if (j.bad_tree) {
        D_out = __int_as_float(0x7fc00000); bit_out = 0; st_out = FSD_ROW_BADTREE;
        return;
    }
    float D = __int_as_float(0x7fc00000);
    if (j.finite) D = r.differ ? static_cast<float>(divergence_of(P.div, j.base, r.X)) : 0.0f;
    const bool div_ok = j.finite && passes(D, P.T, P.cmp);
    D_out = D;
    bit_out = P.mode == FSD_MODE_FSD ? div_ok : P.mode == FSD_MODE_SD ? j.ratio_ok : (div_ok || j.ratio_ok);          // Eq. 6
    st_out = j.finite ? 0 : FSD_ROW_NONFINITE;
}

// ---- how a row is shared out for the draw -------------------------------------------------------
// In units, a 16-byte vector of the row (rows off a 16-byte boundary: the aligned granules that cover it), or one
// entry.  A warp of the cluster owns `iters` times 32 consecutive units, its lanes read neighbours: consecutive
// threads on consecutive addresses.  (With a run of units per thread a warp's load touched 32 lines, which were
// gone from L1 when the next one wanted the rest of them.)
struct Draw {
    const char* a_row;
    const char* b_row;
    int b, n, V, cs, rank;
    bool shared_out;           // the cluster's CTAs have shared the judging: no pair's reference is at hand
    bool vec;                  // both rows are whole vectors on 16-byte boundaries
    double u;
    int span;                  // LOCAL draws: granules of the target row that a CTA of the cluster holds in its shared memory ...
    uint32_t local;            // ... and the address there at which granule 0 of the row would lie
};
struct Share { int units, iters, first; };            // where the run's row ends, iterations of a warp, the warp's first unit
template <bool ANY_SIZE = false>                      // of the cluster; else a power of two
__device__ __forceinline__ Share row_share(int units, int cs, int rank, int warp) {
    Share s;
    s.units = units;
    if constexpr (ANY_SIZE) {
        const uint32_t all = static_cast<uint32_t>(cs) * kFinishThreads;
        s.iters = static_cast<int>((static_cast<uint32_t>(units) + all - 1) / all);
    } else {
        const int shift = 9 + 31 - __clz(cs);         // log2(cs * kFinishWarps * 32)
        s.iters = static_cast<int>((static_cast<uint32_t>(units) + (1u << shift) - 1) >> shift);
    }
    const long long first = static_cast<long long>(rank * kFinishWarps + warp) * s.iters * 32;
    s.first = first < units ? static_cast<int>(first) : units;
    return s;
}
// The same for the granules of the target row, of which a CTA takes what it has at hand (LOCAL: a row in shared memory).
template <bool LOCAL>
__device__ __forceinline__ Share granule_share(const Draw& d, int granules, int warp) {
    if constexpr (!LOCAL) return row_share(granules, d.cs, d.rank, warp);
    Share s;
    s.units = min(granules, (d.rank + 1) * d.span);
    s.iters = (d.span + kFinishThreads - 1) / kFinishThreads;
    s.first = min(d.rank * d.span + warp * s.iters * 32, s.units);
    return s;
}
// The target row as granules: the granule that holds entry 0 starts `off` entries in front of it.
template <int DT, bool LOCAL> struct Granules {
    const void* base;
    uint32_t local;
    int off, count, V;
    __device__ __forceinline__ explicit Granules(const Draw& d) : local(d.local), V(d.V) {
        const char* const row = d.a_row;
        const int v = d.V;
        const int bytes = static_cast<int>(reinterpret_cast<uintptr_t>(row) & 15);
        base = row - bytes;
        off = bytes / Logit<DT>::kBytes;
        count = (off + v + Logit<DT>::kPerVec - 1) / Logit<DT>::kPerVec;
    }
    __device__ __forceinline__ uint4 fetch(int g, int end) const {       // -inf where there is no entry, and from granule `end` on
        constexpr uint32_t kNone = DT == FSD_BF16 ? 0xff80ff80u : 0xff800000u;
        if (g >= end) return make_uint4(kNone, kNone, kNone, kNone);
        if constexpr (LOCAL) return ld_shared16(local + static_cast<uint32_t>(g) * 16); else return ldg_vec(base, g);
    }
    __device__ __forceinline__ uint4 cut(uint4 v, int g) const {         // the first and last granule's entries that are not the row's
        const int k0 = g * Logit<DT>::kPerVec - off;
        return g < count && (k0 < 0 || k0 + Logit<DT>::kPerVec > V) ? masked_vector<DT>(v, k0, V, true) : v;
    }
};
// Calls f(k, a_k, b_k) for this warp's entries, unit by unit: vectors where `vec`, else single entries.
template <int DT, bool ANY_SIZE, typename F>
__device__ __forceinline__ void for_units(const Draw& d, int warp, int lane, bool with_b, F f) {
    constexpr int EPV = Logit<DT>::kPerVec;
    const Share s = row_share<ANY_SIZE>(d.vec ? d.V / EPV : d.V, d.cs, d.rank, warp);
    for (int it = 0; it < s.iters; ++it) {
        const int u = s.first + it * 32 + lane;
        if (u >= s.units) break;
        if (d.vec) {
            float xa[EPV], xb[EPV];
            unpack_vec<DT>(ldg_vec(d.a_row, u), xa);
            if (with_b) {
                unpack_vec<DT>(ldg_vec(d.b_row, u), xb);
            } else {
#pragma unroll
                for (int j = 0; j < EPV; ++j) xb[j] = 0.f;
            }
#pragma unroll
            for (int j = 0; j < EPV; ++j) f(u * EPV + j, xa[j], xb[j]);
        } else {
            f(u, load_logit<DT>(d.a_row, u), with_b ? load_logit<DT>(d.b_row, u) : 0.f);
        }
    }
}
// One inclusive scan over a warp
__device__ __forceinline__ double warp_scan(double v, int lane) {
#pragma unroll
    for (int q = 1; q < 32; q <<= 1) {
        const double o = __shfl_up_sync(0xffffffffu, v, q);
        if (lane >= q) v += o;
    }
    return v;
}
// Sixteen values, one a warp of the CTA, scanned by every warp for itself: lane w has warp w's.
struct Prefix {
    double v, upto, total;
    __device__ __forceinline__ Prefix(double value, int lane) {
        v = lane < kFinishWarps ? value : 0.0;
        upto = warp_scan(v, lane);
        total = __shfl_sync(0xffffffffu, upto, kFinishWarps - 1);
    }
    // the first whose running total (on top of `base`) passes t, or -1; and the total in front of it
    __device__ __forceinline__ int passes(double base, double t, double& before) const {
        const unsigned over = __ballot_sync(0xffffffffu, v > 0.0 && base + upto > t);
        const int w = over != 0 ? __ffs(over) - 1 : -1;
        before = base + __shfl_sync(0xffffffffu, upto - v, w < 0 ? 0 : w);
        return w;
    }
    // the same, but the last with weight where rounding has lost the crossing
    __device__ __forceinline__ int crossing(double t, double& before) const {
        int w = passes(0.0, t, before);
        if (w < 0) {
            w = 31 - __clz(__ballot_sync(0xffffffffu, v > 0.0) | 1u);
            before = __shfl_sync(0xffffffffu, upto - v, w);
        }
        return w;
    }
};
// Finds the entry at which the running sum over a warp's share passes `target`: all warps of the CTA take an
// iteration of that share each.  weights(unit, w[]) fills in the weights of a unit's EPU entries (0 where there is
// none), first_entry(unit) is the index of its first.  The last entry with weight where rounding loses the crossing.
template <int EPU, typename W, typename E>
__device__ __forceinline__ void find_crossing(const FinishParams& P, FinishShared& sh, const Draw& d, const Share& share, double target, W weights, E first_entry) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    double base = 0.0;
    int last = -1;                                    // highest index with weight this thread has seen
#pragma unroll 1
    for (int r0 = 0; r0 < share.iters; r0 += kFinishWarps) {
        const int u = share.first + (r0 + warp) * 32 + lane;
        double w[EPU], usum = 0.0;
        int ulast = -1;
#pragma unroll
        for (int j = 0; j < EPU; ++j) w[j] = 0.0;
        if (r0 + warp < share.iters && u < share.units) {
            weights(u, w);
#pragma unroll
            for (int j = 0; j < EPU; ++j) { usum += w[j]; if (w[j] > 0.0) ulast = first_entry(u) + j; }
        }
        last = max(last, ulast);
        const double upto = warp_scan(usum, lane);
        if (lane == 31) sh.seg_tot[warp] = upto;
        __syncthreads();
        double before;
        const Prefix seg(sh.seg_tot[lane & (kFinishWarps - 1)], lane);
        const int found = seg.passes(base, target, before);
        if (found >= 0) {                             // the same for all threads
            if (warp != found) return;
            const unsigned over = __ballot_sync(0xffffffffu, usum > 0.0 && before + upto > target), some = __ballot_sync(0xffffffffu, usum > 0.0);
            const int src = over != 0 ? __ffs(over) - 1 : 31 - __clz(some);
            if (lane == src) {
                double run = before + upto - usum;
                int tok = -1;
#pragma unroll
                for (int j = 0; j < EPU; ++j) {
                    run += w[j];
                    if (tok < 0 && w[j] > 0.0 && run > target) tok = first_entry(u) + j;
                }
                if (tok < 0) tok = ulast;             // lost to the order of the additions
                FSD_CHECK(&P.flags->debug, tok >= 0 && tok < d.V, kChkToken);
                P.next_token[d.b] = tok;
            }
            return;
        }
        base += seg.total;
        __syncthreads();                              // seg_tot is free again
    }
    last = __reduce_max_sync(0xffffffffu, last);
    if (lane == 0 && last >= 0) atomicMax(&sh.cand, last);
    __syncthreads();
    if (tid == 0) P.next_token[d.b] = sh.cand;
}

// Tree: the deepest node whose whole path passes (ties: lowest index), its depth and path.
// Called by all threads of the CTA; leaves sh.n_acc / sh.row_sel and writes the path if `pth` is given.
__device__ __noinline__ void tree_select(const int32_t* par, int G, int max_depth, int32_t* pth, FinishShared& sh, TreeShared& tr) {
    const int tid = threadIdx.x, lane = tid & 31;
    // Depth of every node and "all nodes from the root down to it pass", by pointer jumping:
    // every node keeps (nodes counted, all pass, next ancestor) for the stretch of its path it
    // has seen so far and doubles that stretch each round, so ceil(log2 depth) rounds do for any
    // tree shape (a serial walk takes N dependent steps for a chain-shaped tree of N nodes).
    const bool good = !(sh.bad & FSD_ROW_BADTREE);
    constexpr int kPer = (kMaxTreeNodes + kFinishThreads - 1) / kFinishThreads;
    if (tid == 0) sh.best_key = -1;
    if (good) {
        for (int j = tid; j < G; j += kFinishThreads) {
            const int16_t p = static_cast<int16_t>(par[j]);
            tr.parent[j] = p;
            tr.jump[j] = p;
            tr.depth[j] = 1;
            tr.ok[j] = tr.bit[j];
        }
        __syncthreads();
        for (int span = 1; span < G; span <<= 1) {
            int nj[kPer], nd[kPer], no[kPer];
            bool more = false;
#pragma unroll
            for (int q = 0; q < kPer; ++q) {
                const int j = tid + q * kFinishThreads;
                nj[q] = -1; nd[q] = 0; no[q] = 0;
                if (j < G) {
                    const int p = tr.jump[j];
                    nj[q] = p; nd[q] = tr.depth[j]; no[q] = tr.ok[j];
                    if (p >= 0) { nj[q] = tr.jump[p]; nd[q] += tr.depth[p]; no[q] &= tr.ok[p]; }
                    more = more || nj[q] >= 0;
                }
            }
            const bool any = __syncthreads_or(more) != 0;
#pragma unroll
            for (int q = 0; q < kPer; ++q) {
                const int j = tid + q * kFinishThreads;
                if (j < G) {
                    tr.jump[j] = static_cast<int16_t>(nj[q]);
                    tr.depth[j] = static_cast<int16_t>(nd[q]);
                    tr.ok[j] = static_cast<int8_t>(no[q]);
                }
            }
            if (!any) break;                          // every node has reached the root (what is read below, its reader wrote)
            __syncthreads();
        }
        // deepest passing node within max_depth, ties to the lowest index
        int key = -1;
        for (int j = tid; j < G; j += kFinishThreads) {
            const int d = tr.depth[j];
            if (tr.ok[j] && d <= max_depth) {
                const int k = d * 2048 + (2047 - j);
                key = k > key ? k : key;
            }
        }
        key = __reduce_max_sync(0xffffffffu, key);
        if (lane == 0 && key >= 0) atomicMax(&sh.best_key, key);
    }
    __syncthreads();
    const int key = sh.best_key;
    const int best = key < 0 ? -1 : 2047 - (key & 2047), best_depth = key < 0 ? 0 : key >> 11;
    if (tid == 0) { sh.n_acc = best_depth; sh.row_sel = best + 1; }
    if (pth != nullptr) {
        for (int d = best_depth + tid; d < max_depth; d += kFinishThreads) pth[d] = -1;
        if (tid == 0)
            for (int j = best, d = best_depth - 1; j >= 0 && d >= 0; j = tr.parent[j], --d) pth[d] = j;
    }
}

// ---- the draw from P_T ---------------------------------------------------------------------------
__device__ __forceinline__ double pow2_any(int e) { return __hiloint2double((1023 + e) << 20, 0); }      // |e| < 1000

// A weight (0 or a normal number up to 1) widened to double with integer instructions: the conversion instruction
// shares the special-function pipe with ex2 and would double the pass' time there.  0 becomes 2^-127, which is
// nothing beside the thread's largest weight, a half or more.
__device__ __forceinline__ double widen(float w) {
    const uint32_t u = __float_as_uint(w);
    return __hiloint2double(static_cast<int>((u >> 3) + 0x38000000u), static_cast<int>(u << 29));
}
template <int DT> __device__ __forceinline__ float vector_max(const uint4& v) {          // NaN if one is
    if constexpr (DT == FSD_BF16) {
        const uint32_t m2 = bf16x2_max_nan(bf16x2_max_nan(v.x, v.y), bf16x2_max_nan(v.z, v.w));
        return fmax_nan(bf16_lo(m2), bf16_hi(m2));
    } else {
        return fmax_nan(fmax_nan(__uint_as_float(v.x), __uint_as_float(v.y)), fmax_nan(__uint_as_float(v.z), __uint_as_float(v.w)));
    }
}

// Inverse CDF over P_T.  Writes the row's token, adds to its status (uniform over the cluster).
template <int DT, bool LOCAL = false>
__device__ __forceinline__ void draw_pt(const FinishParams& P, FinishShared& sh, const Draw& d, Link& link, int& status) {
    constexpr int EPV = Logit<DT>::kPerVec;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const Granules<DT, LOCAL> gr(d);
    const Share mine = granule_share<LOCAL>(d, gr.count, warp);
    FSD_CHECK(&P.flags->debug, mine.first >= 0 && mine.first <= gr.count && (LOCAL || static_cast<long long>(mine.iters) * kFinishThreads * d.cs >= gr.count), kChkChunk);
    // ---- one pass: this thread's weights 2^(logit * log2e - kr) in double, kr the largest logit's exponent so far;
    //      four vectors are asked for before the first is used ----
    constexpr int BV = 4;
    double csum = 0.0;
    float kr = -INFINITY;
    for (int it = 0; it < mine.iters; it += BV) {
        uint4 v[BV];
#pragma unroll
        for (int q = 0; q < BV; ++q) v[q] = gr.fetch(it + q < mine.iters ? mine.first + (it + q) * 32 + lane : INT_MAX, mine.units);
        float vm = -INFINITY;
#pragma unroll
        for (int q = 0; q < BV; ++q) {
            if (it + q < mine.iters) v[q] = gr.cut(v[q], mine.first + (it + q) * 32 + lane);
            vm = fmax_nan(vm, vector_max<DT>(v[q]));
        }
        if (!(vm * kLog2e <= kr)) {                   // (a NaN comes through here and stays in csum)
            const float kn = ceilf(vm * kLog2e);
            csum = kr == -INFINITY ? 0.0 : csum * pow2_int_d(static_cast<double>(kr) - kn);
            kr = kn;
        }
        const float nk = kr == -INFINITY ? 0.f : -kr;
        double part[BV];
#pragma unroll
        for (int q = 0; q < BV; ++q) {
            part[q] = 0.0;
            if (it + q < mine.iters) {
                float x[EPV];
                unpack_vec<DT>(v[q], x);
#pragma unroll
                for (int e = 0; e < EPV; ++e) part[q] += widen(ex2(fmaf(x[e], kLog2e, nk)));
            }
        }
        csum += (part[0] + part[1]) + (part[2] + part[3]);
        if (!(vm < INFINITY)) csum = vm - vm;         // (a NaN or +inf logit: `widen` takes finite weights)
    }
    const bool usable = kr > -INFINITY && kr < INFINITY;
    const bool far = usable && fabsf(kr) > 900.f;
    if (far) sh.far = 1;
    const float wk = warp_redux_max_nan(usable ? kr : -INFINITY);
    if (lane == 0) sh.warp_k[warp] = wk;

    // ---- totals of warp, CTA and cluster, in a fixed order and on one scale: 2^0, or where a reference is out of a
    //      double's reach the largest reference of the cluster ----
    double K = 0.0, W, w_v, w_upto;
    [[maybe_unused]] double blocks_v = 0.0, blocks_upto = 0.0;      // LOCAL: the CTAs' totals and running totals, a lane each
    const double (*all)[kExchangeDoubles];
#pragma unroll 1
    for (bool scaled = false;; scaled = true) {
        double val = kr == -INFINITY ? 0.0 : !usable ? csum * static_cast<double>(__int_as_float(0x7fc00000))
                     : scaled ? csum * pow2_int_d(static_cast<double>(kr) - K) : far ? 0.0 : csum * pow2_any(static_cast<int>(kr));
        val = warp_sum(val);
        if (lane == 0) sh.warp_tot[warp] = val;
        __syncthreads();
        const Prefix pre(sh.warp_tot[lane & (kFinishWarps - 1)], lane);
        w_v = pre.v; w_upto = pre.upto;
        const double mine2[2] = {pre.total, scaled ? 0.0 : static_cast<double>(sh.far)};
        all = cluster_exchange(P, sh, d.cs, d.rank, link, mine2);
        if (link.lost) return;
        if constexpr (LOCAL) {                        // (clusters of up to twelve: one scan is shorter than twelve additions in a row)
            const double (&its)[kExchangeDoubles] = all[lane < d.cs ? lane : 0];
            const Prefix blocks(lane < d.cs ? its[0] : 0.0, lane);
            blocks_v = blocks.v; blocks_upto = blocks.upto;
            W = blocks.total;
            if (!__any_sync(0xffffffffu, its[1] != 0.0)) break;
        } else {
            double any = 0.0;
            W = 0.0;
            for (int r = 0; r < d.cs; ++r) { W += all[r][0]; any += all[r][1]; }
            if (any == 0.0) break;
        }
        float m = -INFINITY;
        for (int w = 0; w < kFinishWarps; ++w) m = fmaxf(m, sh.warp_k[w]);
        __syncthreads();
        const double mk[1] = {m};
        all = cluster_exchange(P, sh, d.cs, d.rank, link, mk);
        if (link.lost) return;
        K = -INFINITY;
        for (int r = 0; r < d.cs; ++r) K = fmax(K, all[r][0]);
    }
    if (!(isfinite(W) && W > 0.0)) {                  // a NaN or +inf logit, or no finite one: uniform over the cluster
        status |= FSD_ROW_NONFINITE;
        if (d.rank == 0 && tid == 0) P.next_token[d.b] = -1;
        return;
    }
    const double t = d.u * W;
    double cpre = 0.0;
    int owner = -1;
    if constexpr (LOCAL) {
        // (with weight: the scan's lanes add in different orders, and one without may be an ulp above the one before it)
        const unsigned past = __ballot_sync(0xffffffffu, blocks_v > 0.0 && blocks_upto > t);
        owner = past != 0 ? __ffs(past) - 1 : -1;
        const double before_it = __shfl_sync(0xffffffffu, blocks_upto, owner > 0 ? owner - 1 : 0);
        cpre = owner > 0 ? before_it : 0.0;
    } else {
        double run = 0.0;
        for (int r = 0; r < d.cs && owner < 0; ++r) {
            cpre = run;
            run += all[r][0];
            if (run > t) owner = r;
        }
    }
    if (owner < 0) {                                  // t >= W after rounding (uniform): the last token that has weight
        int lastp = -1;
        const float nk = kr == -INFINITY ? 0.f : -kr;
        for (int it = 0; it < mine.iters; ++it) {
            const int g = mine.first + it * 32 + lane;
            if (g >= mine.units) break;
            float x[EPV];
            unpack_vec<DT>(gr.cut(gr.fetch(g, mine.units), g), x);
#pragma unroll
            for (int e = 0; e < EPV; ++e) if (ex2(fmaf(x[e], kLog2e, nk)) > 0.f) lastp = g * EPV - gr.off + e;
        }
        lastp = __reduce_max_sync(0xffffffffu, lastp);
        if (lane == 0 && lastp >= 0) atomicMax(&sh.last_pos, lastp);
        __syncthreads();
        const double mine1[1] = {static_cast<double>(sh.last_pos)};
        all = cluster_exchange(P, sh, d.cs, d.rank, link, mine1);
        if (link.lost) return;
        int best = -1;
        for (int r = 0; r < d.cs; ++r) best = max(best, static_cast<int>(all[r][0]));
        if (d.rank == 0 && tid == 0) P.next_token[d.b] = best;
        return;
    }
    if (owner != d.rank) return;
    // the warp in whose share the total passes the target, and the target on that warp's own scale
    Prefix pre(0.0, lane);
    pre.v = w_v; pre.upto = w_upto;
    double before;
    const int cw = pre.crossing(t - cpre, before);
    const float ck = sh.warp_k[cw];
    const double up = pow2_int_d(-fabs(static_cast<double>(ck) - K)), rest = t - cpre - before;
    const double target = static_cast<double>(ck) > K ? rest * up : rest / up;
    const float nk = -ck;
    const Share crossing = granule_share<LOCAL>(d, gr.count, cw);
    find_crossing<EPV>(P, sh, d, crossing, target,
        [&](int g, double (&w)[EPV]) {
            float x[EPV];
            unpack_vec<DT>(gr.cut(gr.fetch(g, crossing.units), g), x);
#pragma unroll
            for (int e = 0; e < EPV; ++e) w[e] = static_cast<double>(ex2(fmaf(x[e], kLog2e, nk)));
        },
        [&](int g) { return g * EPV - gr.off; });
}

// argmax of P_T == argmax of the logits, ties to the lowest index.  One pass: the largest logit, its index, and
// whether the row is a valid distribution (no NaN, no +inf, something finite).
template <int DT, bool LOCAL = false>
__device__ __forceinline__ void draw_argmax(const FinishParams& P, FinishShared& sh, const Draw& d, Link& link, int& status) {
    constexpr int EPV = Logit<DT>::kPerVec;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const Granules<DT, LOCAL> gr(d);
    const Share mine = granule_share<LOCAL>(d, gr.count, warp);
    float best = -INFINITY;
    int idx = 0x7fffffff;
    bool bad = false;
#pragma unroll 4
    for (int it = 0; it < mine.iters; ++it) {
        const int g = mine.first + it * 32 + lane;
        const uint4 v = gr.cut(gr.fetch(g, mine.units), g);
        const float vm = vector_max<DT>(v);
        bad = bad || !(vm < INFINITY);
        if (vm > best) {
            best = vm;
            float x[EPV];
            unpack_vec<DT>(v, x);
#pragma unroll
            for (int j = EPV - 1; j >= 0; --j) if (x[j] == vm) idx = g * EPV - gr.off + j;
        }
    }
    const float wb = warp_redux_max_nan(best);                            // (best is never NaN)
    const int wi = __reduce_min_sync(0xffffffffu, best == wb ? idx : 0x7fffffff);
    const bool wbad = __any_sync(0xffffffffu, bad);
    if (lane == 0) { sh.red_f[warp] = wb; sh.red_d[warp] = wi; if (wbad) sh.far = 1; }
    __syncthreads();
    const float lb = lane < kFinishWarps ? sh.red_f[lane] : -INFINITY;
    const int li = lane < kFinishWarps ? static_cast<int>(sh.red_d[lane]) : 0x7fffffff;
    const float cb = warp_redux_max_nan(lb);
    const int ci = __reduce_min_sync(0xffffffffu, lb == cb ? li : 0x7fffffff);
    const double mine3[3] = {cb, static_cast<double>(ci), static_cast<double>(sh.far)};
    const double (*all)[kExchangeDoubles] = cluster_exchange(P, sh, d.cs, d.rank, link, mine3);
    if (link.lost) return;
    if (d.rank == 0 && threadIdx.x == 0) {
        double gb = all[0][0], gi = all[0][1], gbad = all[0][2];
        for (int r = 1; r < d.cs; ++r) {
            if (all[r][0] > gb || (all[r][0] == gb && all[r][1] < gi)) { gb = all[r][0]; gi = all[r][1]; }
            gbad += all[r][2];
        }
        const bool ok = gbad == 0.0 && gb > -INFINITY;
        P.next_token[d.b] = ok ? static_cast<int>(gi) : -1;
        if (!ok) status |= FSD_ROW_NONFINITE;         // (this thread writes it)
    }
}

// ---- the draw from the SD residual -----------------------------------------------------------------
constexpr int kPairRefs = 32;                         // (a pair beyond these has its record folded again)
struct PairRef { double za, zb, ln_rho; float ka, kb; };      // normalisers relative to 2^ka, 2^kb, log of their ratio; ka NaN: not usable
struct ResidualShared {
    double exp_table[kExpTable];                      // 2^(j/256)
    double exp_consts[8];                             // the constants of exp2_table (see exp2_consts)
    PairRef ref[kPairRefs];                           // of the pairs this CTA has judged
    double wsum[kFinishWarps][4];                     // the warps' za, zb, sa, sb
    double cq[2];                                     // the close calls' e_a, e_b where one thread of the CTA has some, of one kind
    int cq_warp;
};
template <int DT> struct ExpTable {};                // (fp32 logits have no table of their own)
// e^x of the bf16 numbers from 2^-13 to 64, at [sign * kBf16Count + magnitude's bits - kBf16Lowest].  (From 2^-9 on, every
// fourth warp of the pass met a smaller logit in a step, and its lane's sixteen entries one by one took as long as all others.)
template <> struct ExpTable<FSD_BF16> {
    double e[2 * kBf16Count];
};
// e^x of a bf16 number, to double precision, whatever it is
__device__ __noinline__ double exp_bf16(float x, const ExpTable<FSD_BF16>& t) {
    const uint32_t bits = __float_as_uint(x) >> 16, m = (bits & 0x7fffu) - kBf16Lowest;
    if (m < static_cast<uint32_t>(kBf16Count)) return t.e[(bits >> 15) * kBf16Count + m];
    if (static_cast<int>(m) < 0) {                    // |x| < 2^-13: the series' next term is below 2^-71
        const double y = x;
        return fma(fma(fma(fma(y, 1.0 / 24, 1.0 / 6), y, 0.5), y, 1.0), y, 1.0);
    }
    if (x < -700.f) return 0.0;                       // (-inf among them)
    return exp(static_cast<double>(x));
}
// All sixteen entries of two vectors within the table
__device__ __forceinline__ bool in_table(const uint4& a, const uint4& b) {
    constexpr uint32_t kMag = 0x7fff7fffu;
    const uint32_t w[8] = {a.x & kMag, a.y & kMag, a.z & kMag, a.w & kMag, b.x & kMag, b.y & kMag, b.z & kMag, b.w & kMag};
    uint32_t lo = w[0], hi = w[0];
#pragma unroll
    for (int i = 1; i < 8; ++i) { lo = __vminu2(lo, w[i]); hi = __vmaxu2(hi, w[i]); }
    return (lo & 0xffffu) >= kBf16Lowest && (lo >> 16) >= kBf16Lowest && (hi & 0xffffu) < kBf16Lowest + kBf16Count && (hi >> 16) < kBf16Lowest + kBf16Count;
}
// e^x of both entries of a packed pair there; `table` is its shared-memory address
__device__ __forceinline__ void table_exp2(uint32_t pair, uint32_t table, double& e0, double& e1) {
    const uint32_t m = pair - kBf16Lowest * 0x10001u;                       // (no borrow between the halves)
    const uint32_t idx = (m & 0x0fff0fffu) + (m >> 15 & 0x00010001u) * kBf16Count;
    asm("ld.shared.f64 %0, [%1];" : "=d"(e0) : "r"(table + (idx & 0xffffu) * 8));
    asm("ld.shared.f64 %0, [%1];" : "=d"(e1) : "r"(table + (idx >> 16) * 8));
}
// What a pass over a thread's entries leaves: normalisers; sums over the entries clearly above the ratio; sums over the
// first kind of close call (entries whose logits differ by qd); the other close calls.  An entry is above where its
// logits differ by more than ln rho: `hi` and `lo` are ln rho_est plus and minus the margin.
struct Classed {
    double za, zb, sa, sb, qa, qb;
    float qd;                                         // NaN: none yet
    int close, k0, k1;                                // number and indices of the other close calls
    __device__ __forceinline__ void close_call(int k, float d, double pa, double pb) {
        if (qd != qd) qd = d;
        if (d == qd) { qa += pa; qb += pb; return; }
        if (close == 0) k0 = k; else k1 = k;
        ++close;
    }
    __device__ __forceinline__ void entry(int k, float xa, float xb, double pa, double pb, float hi, float lo) {
        const float d = xa - xb;                      // (both -inf: NaN, no weight)
        za += pa;
        zb += pb;
        if (d > hi) { sa += pa; sb += pb; }
        else if (d >= lo) close_call(k, d, pa, pb);
    }
};
// e^x on a pass' scale by the 256-entry table and the polynomial, whatever x is but NaN (0 below xmin); with k = 0, bit for bit
// what the table of bf16 exponentials holds
struct RowExp {
    double nk;
    float xmin;
    __device__ __forceinline__ RowExp(double k) : nk(-k), xmin(static_cast<float>((k - 990.0) * kLn2D)) {}
    __device__ __forceinline__ double operator()(float x, const double* table, const Exp2Consts& c) const { return exp2_of_logit(x, xmin, nk, table, c); }
};
// The pass over bf16 vectors, by the table.  A function of its own: the registers of everything around it would
// otherwise be spilled inside its loop.  About twenty instructions an entry (two of them shared-memory reads, four
// double-precision).
__device__ __noinline__ void classed_pass_bf16(const void* a_row, const void* b_row, const Share share, float hi, float lo,
                                               const ExpTable<FSD_BF16>& bt, Classed& out) {
    const uint32_t table = smem_u32(bt.e);
    const int u0 = share.first + (threadIdx.x & 31), u1 = min(share.first + share.iters * 32, share.units);
    Classed c = out;
    uint4 na = make_uint4(0, 0, 0, 0), nb = na;       // the vectors after these, on their way
    if (u0 < u1) { na = ldg_vec(a_row, u0); nb = ldg_vec(b_row, u0); }
#pragma unroll 1
    for (int u = u0; u < u1; u += 32) {
        const uint4 va = na, vb = nb;
        if (u + 32 < u1) { na = ldg_vec(a_row, u + 32); nb = ldg_vec(b_row, u + 32); }
        const int k = u * 8;
        if (!in_table(va, vb)) {                      // an entry of the vectors is small, large or -inf
#pragma unroll 1
            for (int e = 0; e < 8; ++e) {
                const float xa = load_logit<FSD_BF16>(a_row, k + e), xb = load_logit<FSD_BF16>(b_row, k + e);
                c.entry(k + e, xa, xb, exp_bf16(xa, bt), exp_bf16(xb, bt), hi, lo);
            }
            continue;
        }
        const uint32_t wa[4] = {va.x, va.y, va.z, va.w}, wb[4] = {vb.x, vb.y, vb.z, vb.w};
        bool close = false;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            double pa[2], pb[2];
            table_exp2(wa[q], table, pa[0], pa[1]);
            table_exp2(wb[q], table, pb[0], pb[1]);
            const float d[2] = {bf16_lo(wa[q]) - bf16_lo(wb[q]), bf16_hi(wa[q]) - bf16_hi(wb[q])};
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const double one = __hiloint2double(d[e] > hi ? 0x3ff00000 : 0, 0);
                c.za += pa[e];
                c.zb += pb[e];
                c.sa = fma(pa[e], one, c.sa);
                c.sb = fma(pb[e], one, c.sb);
                close = close || (d[e] >= lo && !(d[e] > hi));         // (as in Classed::entry: between the bounds, both included)
            }
        }
        if (close) {
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const float xa = (e & 1) ? bf16_hi(wa[e >> 1]) : bf16_lo(wa[e >> 1]), xb = (e & 1) ? bf16_hi(wb[e >> 1]) : bf16_lo(wb[e >> 1]);
                const float d = xa - xb;
                if (d >= lo && !(d > hi)) c.close_call(k + e, d, exp_bf16(xa, bt), exp_bf16(xb, bt));
            }
        }
    }
    out = c;
}
// The same for rows whose logits lie so far off 0 that most are outside the table, or that they need a reference: every
// exponential by the small table and the polynomial, in straight-line code (in the loop above, for the lanes that meet an entry
// outside the table, it cost the other rows 9 %: 64 x 8 x 152064, strict rule, 133 -> 145 us).  It is called from two kernels, so that the
// compiler has to be told that the table is in shared memory (64 x 8 x 152064 100 below 0, strict rule: 146 us by generic loads, now 142).
__device__ __noinline__ void classed_pass_far(const void* a_row, const void* b_row, const Share share, float hi, float lo,
                                              const RowExp ea, const RowExp eb, const ResidualShared& rs, Classed& out) {
    __builtin_assume(__isShared(&rs));
    const int u0 = share.first + (threadIdx.x & 31), u1 = min(share.first + share.iters * 32, share.units);
    Classed c = out;
    uint4 na = make_uint4(0, 0, 0, 0), nb = na;       // the vectors after these, on their way
    if (u0 < u1) { na = ldg_vec(a_row, u0); nb = ldg_vec(b_row, u0); }
#pragma unroll 1
    for (int u = u0; u < u1; u += 32) {
        const uint4 va = na, vb = nb;
        if (u + 32 < u1) { na = ldg_vec(a_row, u + 32); nb = ldg_vec(b_row, u + 32); }
        const int k = u * 8;
        const uint32_t wa[4] = {va.x, va.y, va.z, va.w}, wb[4] = {vb.x, vb.y, vb.z, vb.w};
        const Exp2Consts ec = exp2_consts(rs.exp_consts);
        bool close = false;
        const auto add = [&](float xa, float xb) {
            const double pa = ea(xa, rs.exp_table, ec), pb = eb(xb, rs.exp_table, ec);
            const float d = xa - xb;                  // (both -inf: NaN, no weight)
            const double one = __hiloint2double(d > hi ? 0x3ff00000 : 0, 0);
            c.za += pa;
            c.zb += pb;
            c.sa = fma(pa, one, c.sa);
            c.sb = fma(pb, one, c.sb);
            close = close || (d >= lo && !(d > hi));  // (as in Classed::entry: between the bounds, both included)
        };
#pragma unroll
        for (int q = 0; q < 4; ++q) { add(bf16_lo(wa[q]), bf16_lo(wb[q])); add(bf16_hi(wa[q]), bf16_hi(wb[q])); }
        if (close) {
#pragma unroll 1
            for (int e = 0; e < 8; ++e) {
                const float xa = load_logit<FSD_BF16>(a_row, k + e), xb = load_logit<FSD_BF16>(b_row, k + e), d = xa - xb;
                if (d >= lo && !(d > hi)) c.close_call(k + e, d, ea(xa, rs.exp_table, ec), eb(xb, rs.exp_table, ec));
            }
        }
    }
    out = c;
}
// Four values summed over the warp: lanes 8 q to 8 q + 7 return the q-th sum.
__device__ __forceinline__ double fold_four(double v0, double v1, double v2, double v3, int lane) {
    const bool hi = (lane & 16) != 0, up = (lane & 8) != 0;
    const double k0 = (hi ? v2 : v0) + shfl_xor_d(hi ? v0 : v2, 16);
    const double k1 = (hi ? v3 : v1) + shfl_xor_d(hi ? v1 : v3, 16);
    double k = (up ? k1 : k0) + shfl_xor_d(up ? k0 : k1, 8);
#pragma unroll
    for (int m = 4; m > 0; m >>= 1) k += shfl_xor_d(k, m);
    return k;
}
// How far from ln rho_est an entry's difference has to be to be classed in the pass.  The record's ratio is good to about
// 2e-7 (measured), and the difference and the bounds, numbers of about ln rho, are rounded to single precision (6e-8 of
// them each): half the margin covers the one (checked afterwards), half the other.  With 2e-5 throughout, four rows in ten
// of 32000 fp32 entries, and nearly all of 152064, had close calls (16 x 6 x 64000 fp32 36.5 us, now 35.1).
__device__ __forceinline__ float residual_margin(double ln_rho) { return fabs(ln_rho) < 8.0 ? 2e-6f : 2e-5f; }
constexpr double kMostLnRho = 80.0;

template <int DT, bool ANY_SIZE>
__device__ __forceinline__ void draw_residual(const FinishParams& P, FinishShared& sh, ResidualShared& rs, const ExpTable<DT>& bt,
                                              const Draw& d, Link& link, int& status, bool greedy) {
    constexpr int EPV = Logit<DT>::kPerVec;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int b = d.b, n = d.n, cs = d.cs, rank = d.rank, G = P.G;
    const char *a_row = d.a_row, *b_row = d.b_row;
    const double* tab = rs.exp_table;
    double* const sc = sh.sc;
    // ---- references.  The rejected pair's record has references (log2 domain) for both rows, near their maxima and
    //      common to the cluster; without a record one pass for the CTA-local maxima (exact) ----
    double kra = 0.0, krb = 0.0;
    double zea = 0.0, zeb = 0.0, ln_rho = 0.0;
    bool common = false, tabled = false;
    if (P.records != nullptr) {
        PairRef ref;
        ref.za = 0.0; ref.zb = 0.0; ref.ln_rho = 0.0; ref.ka = __int_as_float(0x7fc00000); ref.kb = ref.ka;
        if (n < kPairRefs && !d.shared_out) {
            ref = rs.ref[n];
        } else {
            const PairTotals t = fold_record(P.records + (static_cast<size_t>(b) * G + n), P.div);
            if (t.state & kRecordStats) { ref.za = t.Za; ref.zb = t.Zb; ref.ln_rho = log(t.Za) - log(t.Zb); ref.ka = t.ka; ref.kb = t.kb; }
        }
        if (isfinite(ref.ka) && isfinite(ref.kb)) {
            kra = ref.ka; krb = ref.kb; zea = ref.za; zeb = ref.zb;
            ln_rho = ref.ln_rho + (kra - krb) * kLn2D;
            common = true;
            // bf16: plain e^x (no reference), by the table, as long as it does not overflow and most entries are in the table: largest
            // logits of about -44 (rows reach some 20 below) to 64 (a record's reference can be 2^30 below its row's largest entry,
            // no more).  16 x 5 x 50264, strict rule, logits 60 below 0: 48 us by the table
            tabled = DT == FSD_BF16 && fminf(ref.ka, ref.kb) >= -64.f && fmaxf(ref.ka, ref.kb) <= 92.f;
            if (tabled) { zea *= pow2_any(static_cast<int>(ref.ka)); zeb *= pow2_any(static_cast<int>(ref.kb)); kra = 0.0; krb = 0.0; }
        }
    }
    float mx[2] = {-INFINITY, -INFINITY};
    if (!common) {
        for_units<DT, ANY_SIZE>(d, warp, lane, true, [&](int, float xa, float xb) {
            mx[0] = fmaxf(mx[0], xa);
            mx[1] = fmaxf(mx[1], xb);
        });
        block_max<2>(mx, sh.red_f);
    }
    const double Ra = common ? 0.0 : mx[0], Rb = common ? 0.0 : mx[1];   // this CTA's references (logit domain)

    // common references: y = x * log2e - k; logits below xmin give 2^y < 2^-990 and count as 0
    const Exp2Consts ec = exp2_consts(rs.exp_consts);
    const RowExp ea(kra), eb(krb);
    auto exp_a = [&](float x) -> double { if constexpr (DT == FSD_BF16) { if (tabled) return exp_bf16(x, bt); } return ea(x, tab, ec); };
    auto exp_b = [&](float x) -> double { if constexpr (DT == FSD_BF16) { if (tabled) return exp_bf16(x, bt); } return eb(x, tab, ec); };

    // ---- global normalisers of both rows (double) ----
    double Ma, Mb, iZa = 0.0, iZb = 0.0;
    bool residual = true;
    // One pass instead of two, where it can be shown to give the same sums.  An entry has residual
    // weight iff e_a / Z_a > e_b / Z_b, i.e. e_a > rho * e_b with rho = Z_a / Z_b, which is known
    // only after the pass -- but the record gives rho to about 2e-7.  Entries are classed against
    // rho_est * (1 +- margin): for those clearly above, e_a and e_b are summed separately, and their
    // residual weight is then sum e_a / Z_a - sum e_b / Z_b with the exact normalisers.
    // The few entries between the two bounds are settled with the exact normalisers afterwards: bf16 logits
    // differ by multiples of a step, so where ln rho falls next to one (0 above all, two rows with the same
    // normaliser) hundreds of entries do, but they all have the same difference, hence the same ratio and
    // the same answer: the first such difference a thread meets has sums of its own.  Two entries of another
    // difference are remembered; a thread with more of them, or an estimate that turns out further off than
    // half the margin, sends the whole row through the second pass instead.
    Classed c = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, __int_as_float(0x7fc00000), 0, -1, -1};
    bool one_pass = false;
    float margin = 0.f;
    double Za = 0.0, Zb = 0.0, flags = 1.0;               // flags, cluster-wide: 0 no CTA has close calls of two threads or kinds, 2 some has, 1 a second pass is needed
    const double (*all)[kExchangeDoubles];
    if (common) {
        // the usual case (a rejected pair with a record): both rows, two independent exponentials an entry
        const bool classify = !greedy && zea > 0.0 && zeb > 0.0 && isfinite(zea) && isfinite(zeb) && fabs(ln_rho) < kMostLnRho;
        margin = residual_margin(ln_rho);
        const float hi = static_cast<float>(ln_rho + margin), lo = static_cast<float>(ln_rho - margin);
        bool done = false;
        if constexpr (DT == FSD_BF16) {
            const Share share = row_share<ANY_SIZE>(d.V / 8, cs, rank, warp);
            if (d.vec && tabled) classed_pass_bf16(a_row, b_row, share, hi, lo, bt, c);
            else if (d.vec) classed_pass_far(a_row, b_row, share, hi, lo, ea, eb, rs, c);
            done = d.vec;
        }
        if constexpr (DT == FSD_BF16) {               // (a loop of its own: with the choice inside it, 8 x 5 x 50257 28.7 -> 31.0 us)
            if (!done && tabled) { for_units<DT, ANY_SIZE>(d, warp, lane, true, [&](int k, float xa, float xb) { c.entry(k, xa, xb, exp_bf16(xa, bt), exp_bf16(xb, bt), hi, lo); }); done = true; }
        }
        if (!done) for_units<DT, ANY_SIZE>(d, warp, lane, true, [&](int k, float xa, float xb) { c.entry(k, xa, xb, ea(xa, tab, ec), eb(xb, tab, ec), hi, lo); });
        if (!classify || c.close > 2) {
            atomicOr(&sh.amb, 1);
        } else if (c.qd == c.qd) {
            if (atomicAdd(&sh.n_close, c.close > 0 ? 2 : 1) == 0) { rs.cq[0] = c.qa; rs.cq[1] = c.qb; rs.cq_warp = warp; }
        }
        {
            const double k = fold_four(c.za, c.zb, c.sa, c.sb, lane);
            if ((lane & 7) == 0) rs.wsum[warp][lane >> 3] = k;
        }
        __syncthreads();
        double mine[7] = {};                              // (the first warp sends)
        if (warp == 0) {
            static_assert(kFinishWarps == 16, "two warps' sums a lane");
            double k = rs.wsum[lane & 7][lane >> 3] + rs.wsum[8 + (lane & 7)][lane >> 3];
#pragma unroll
            for (int m = 4; m > 0; m >>= 1) k += shfl_xor_d(k, m);
#pragma unroll
            for (int q = 0; q < 4; ++q) mine[q] = __shfl_sync(0xffffffffu, k, 8 * q);
            const bool one = sh.n_close == 1;
            mine[4] = sh.amb ? 1.0 : sh.n_close > 1 ? 2.0 : 0.0;
            mine[5] = one ? rs.cq[0] : 0.0;
            mine[6] = one ? rs.cq[1] : 0.0;
        }
        all = cluster_exchange(P, sh, cs, rank, link, mine);
        if (link.lost) return;
        Ma = 0.0; Mb = 0.0; flags = 0.0;
        // (a CTA a lane, here and below: sums over eight of them in a row are a third of a microsecond each)
        const double (&its)[kExchangeDoubles] = all[lane < cs ? lane : 0];
        Za = lane < cs ? its[0] : 0.0; Zb = lane < cs ? its[1] : 0.0;
#pragma unroll
        for (int m = 8; m > 0; m >>= 1) { Za += shfl_xor_d(Za, m); Zb += shfl_xor_d(Zb, m); }
        Za = __shfl_sync(0xffffffffu, Za, 0); Zb = __shfl_sync(0xffffffffu, Zb, 0);
        flags = __any_sync(0xffffffffu, its[4] == 1.0) ? 1.0 : __any_sync(0xffffffffu, its[4] == 2.0) ? 2.0 : 0.0;
    } else {
        double z[2] = {0.0, 0.0};
        for_units<DT, ANY_SIZE>(d, warp, lane, true, [&](int, float xa, float xb) {
            if (Ra > -INFINITY) z[0] += exp2_table((static_cast<double>(xa) - Ra) * kLog2eD, tab);
            if (Rb > -INFINITY) z[1] += exp2_table((static_cast<double>(xb) - Rb) * kLog2eD, tab);
        });
        block_sum<2>(z, sh.red_d);
        const double mine[4] = {Ra, Rb, z[0], z[1]};
        all = cluster_exchange(P, sh, cs, rank, link, mine);
        if (link.lost) return;
        Ma = -INFINITY; Mb = -INFINITY;
        for (int r = 0; r < cs; ++r) { Ma = fmax(Ma, all[r][0]); Mb = fmax(Mb, all[r][1]); }
        for (int r = 0; r < cs; ++r) {
            if (all[r][0] > -INFINITY) Za += all[r][2] * exp2_table((all[r][0] - Ma) * kLog2eD, tab);
            if (all[r][1] > -INFINITY) Zb += all[r][3] * exp2_table((all[r][1] - Mb) * kLog2eD, tab);
        }
    }
    {
        const bool a_ok = isfinite(Ma) && isfinite(Za) && Za > 0.0, b_ok = isfinite(Mb) && isfinite(Zb) && Zb > 0.0;
        if (!a_ok) {                                      // uniform over the cluster
            status |= FSD_ROW_NONFINITE;
            if (rank == 0 && tid == 0) P.next_token[b] = -1;
            return;
        }
        if (!b_ok) { residual = false; status |= FSD_ROW_NONFINITE; }
        else { iZa = 1.0 / Za; iZb = 1.0 / Zb; }
        one_pass = b_ok && flags != 1.0 && fabs(zea * Zb - zeb * Za) <= 0.5 * margin * zeb * Za;
    }

    // the residual weights of a unit of vectors (the usual case)
    auto vector_weights = [&](int u, double (&w)[EPV]) {
        if constexpr (DT == FSD_BF16) {
            const uint4 va = ldg_vec(a_row, u), vb = ldg_vec(b_row, u);
            if (tabled && in_table(va, vb)) {
                const uint32_t wa[4] = {va.x, va.y, va.z, va.w}, wb[4] = {vb.x, vb.y, vb.z, vb.w}, table = smem_u32(bt.e);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    double a0, a1, b0, b1;
                    table_exp2(wa[q], table, a0, a1);
                    table_exp2(wb[q], table, b0, b1);
                    w[2 * q] = fmax(a0 * iZa - b0 * iZb, 0.0);
                    w[2 * q + 1] = fmax(a1 * iZa - b1 * iZb, 0.0);
                }
                return;
            }
        }
#pragma unroll 1
        for (int e = 0; e < EPV; ++e) {
            const double v = fmax(exp_a(load_logit<DT>(a_row, u * EPV + e)) * iZa - exp_b(load_logit<DT>(b_row, u * EPV + e)) * iZb, 0.0);
#pragma unroll
            for (int q = 0; q < EPV; ++q) if (q == e) w[q] = v;
        }
    };
    // No close call in the whole row, or those of one thread a CTA (the usual case): the classed sums, already exchanged,
    // are all there is to know.
    const auto residual_of = [&](double sa, double sb, double qa, double qb) { return fmax(sa * iZa - sb * iZb, 0.0) + fmax(qa * iZa - qb * iZb, 0.0); };
    if (one_pass && flags == 0.0 && d.vec) {
        // (With the sums of all CTAs taken one after another: 16 x 6 x 64000 fp32, strict rule, 32.1 us, now 30.0; 2 x 4 x 152064 22.9,
        // now 21.8; 12 x 6 x 32000, relaxed rule, 20.5, now 18.6.)
        const double (&its)[kExchangeDoubles] = all[lane < cs ? lane : 0];
        const Prefix blocks(lane < cs ? residual_of(its[2], its[3], its[5], its[6]) : 0.0, lane);
        const double t = d.u * blocks.total;
        const unsigned past = __ballot_sync(0xffffffffu, blocks.v > 0.0 && blocks.upto > t);     // (with weight, as in draw_pt)
        const int owner = past != 0 ? __ffs(past) - 1 : -1;
        const double before_it = __shfl_sync(0xffffffffu, blocks.upto, owner > 0 ? owner - 1 : 0), cpre = owner > 0 ? before_it : 0.0;
        if (owner >= 0) {                                 // (no mass, or lost to rounding at the very end: the general way)
            if (owner != rank) return;
            asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
            const int w = lane & (kFinishWarps - 1);
            const bool one = sh.n_close == 1 && rs.cq_warp == w;
            double before;
            const int cw = Prefix(residual_of(rs.wsum[w][2], rs.wsum[w][3], one ? rs.cq[0] : 0.0, one ? rs.cq[1] : 0.0), lane).crossing(t - cpre, before);
            find_crossing<EPV>(P, sh, d, row_share<ANY_SIZE>(d.V / EPV, cs, rank, cw), t - cpre - before, vector_weights, [&](int u) { return u * EPV; });
            return;
        }
    }

    for (int attempt = 0; attempt < 2; ++attempt) {
        // weight of one vocabulary entry: the SD residual, or (no residual mass) P_T on the pass' scale
        auto weight = [&](float xa, float xb) -> double {
            if (common) {
                const double pa = exp_a(xa);
                if (!residual) return pa;
                const double r = pa * iZa - exp_b(xb) * iZb;
                return r > 0.0 ? r : 0.0;
            }
            if (!residual) return Ra > -INFINITY ? exp2_table((static_cast<double>(xa) - Ra) * kLog2eD, tab) : 0.0;
            const double r = exp2_table((static_cast<double>(xa) - Ma) * kLog2eD, tab) * iZa -
                             exp2_table((static_cast<double>(xb) - Mb) * kLog2eD, tab) * iZb;
            return r > 0.0 ? r : 0.0;
        };
        double csum = 0.0, wbest = 0.0;
        int kbest = 0x7fffffff;
        if (attempt == 0 && one_pass && residual) {
            csum = c.sa * iZa - c.sb * iZb;
            if (!(csum > 0.0)) csum = 0.0;
            const double q = c.qa * iZa - c.qb * iZb;
            if (q > 0.0) csum += q;
            for (int j = 0; j < c.close; ++j) {           // the entries that were too close to call, now with the exact normalisers
                const int k = j == 0 ? c.k0 : c.k1;
                const double r = exp_a(load_logit<DT>(a_row, k)) * iZa - exp_b(load_logit<DT>(b_row, k)) * iZb;
                if (r > 0.0) csum += r;
            }
        } else if (d.vec && common && residual) {
            const Share share = row_share<ANY_SIZE>(d.V / EPV, cs, rank, warp);
#pragma unroll 1
            for (int u = share.first + lane; u < min(share.first + share.iters * 32, share.units); u += 32) {
                double w[EPV];
                vector_weights(u, w);
#pragma unroll
                for (int e = 0; e < EPV; ++e) {
                    csum += w[e];
                    if (greedy && w[e] > wbest) { wbest = w[e]; kbest = u * EPV + e; }
                }
            }
        } else {
            for_units<DT, ANY_SIZE>(d, warp, lane, residual, [&](int k, float xa, float xb) {
                const double w = weight(xa, xb);
                csum += w;
                if (greedy && w > wbest) { wbest = w; kbest = k; }
            });
        }
        // totals of warp and CTA, in a fixed order
        csum = warp_sum(csum);
        if (lane == 0) sh.warp_tot[warp] = csum;
        if (greedy) {                                     // arg-max of the warp, ties to the lowest index
#pragma unroll
            for (int m = 16; m > 0; m >>= 1) {
                const double ob = shfl_xor_d(wbest, m);
                const int oi = __shfl_xor_sync(0xffffffffu, kbest, m);
                if (ob > wbest || (ob == wbest && oi < kbest)) { wbest = ob; kbest = oi; }
            }
            if (lane == 0) { sh.red_d[warp * 2] = wbest; sh.red_d[warp * 2 + 1] = kbest; }
        }
        __syncthreads();
        const Prefix pre(sh.warp_tot[lane & (kFinishWarps - 1)], lane);
        if (greedy) {
            wbest = sh.red_d[0]; kbest = static_cast<int>(sh.red_d[1]);
            for (int w = 1; w < kFinishWarps; ++w) {
                const double ob = sh.red_d[w * 2];
                const int oi = static_cast<int>(sh.red_d[w * 2 + 1]);
                if (ob > wbest || (ob == wbest && oi < kbest)) { wbest = ob; kbest = oi; }
            }
        }
        const double mine[4] = {pre.total, Ra, wbest, static_cast<double>(kbest)};
        all = cluster_exchange(P, sh, cs, rank, link, mine);
        if (link.lost) return;

        // cluster totals on a common reference
        double M = -INFINITY;
        for (int r = 0; r < cs; ++r) M = fmax(M, all[r][1]);
        double W = 0.0;
        __syncthreads();                                  // everybody is done with the last attempt's factors
        if (tid < cs) sc[tid] = residual || common ? 1.0 : (all[tid][1] > -INFINITY ? exp2_table((all[tid][1] - M) * kLog2eD, tab) : 0.0);
        __syncthreads();
        for (int r = 0; r < cs; ++r) W += all[r][0] * sc[r];
        if (residual && !(W > 0.0)) {                     // no residual mass: draw from P_T (uniform decision)
            residual = false;
            continue;
        }
        if (!residual && !(isfinite(M) && isfinite(W) && W > 0.0)) {     // uniform over the cluster
            status |= FSD_ROW_NONFINITE;
            if (rank == 0 && tid == 0) P.next_token[b] = -1;
            return;
        }
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

        if (greedy) {                                     // arg-max over the cluster
            double gb = all[0][2] * sc[0];
            int gi = static_cast<int>(all[0][3]);
            for (int r = 1; r < cs; ++r) {
                const double rb = all[r][2] * sc[r];
                if (rb > gb || (rb == gb && static_cast<int>(all[r][3]) < gi)) { gb = rb; gi = static_cast<int>(all[r][3]); }
            }
            if (rank == 0 && tid == 0) P.next_token[b] = gi;
            return;
        }

        const double t = d.u * W;
        double cpre = 0.0, run = 0.0;
        int owner = -1;
        for (int r = 0; r < cs && owner < 0; ++r) {
            cpre = run;
            run += all[r][0] * sc[r];
            if (run > t) owner = r;
        }
        if (owner < 0) {                                  // t >= W after rounding (uniform): the last token that has weight
            int lastp = -1;
            for_units<DT, ANY_SIZE>(d, warp, lane, residual, [&](int k, float xa, float xb) { if (weight(xa, xb) > 0.0) lastp = k; });
            lastp = __reduce_max_sync(0xffffffffu, lastp);
            if (lane == 0 && lastp >= 0) atomicMax(&sh.last_pos, lastp);
            __syncthreads();
            const double mine1[1] = {static_cast<double>(sh.last_pos)};
            all = cluster_exchange(P, sh, cs, rank, link, mine1);
            if (link.lost) return;
            int best = -1;
            for (int r = 0; r < cs; ++r) best = max(best, static_cast<int>(all[r][0]));
            if (rank == 0 && tid == 0) P.next_token[b] = best;
            return;
        }
        if (owner != rank) return;
        const double t_local = (t - cpre) / sc[owner];    // the target on this CTA's own scale
        double before;
        const int cw = pre.crossing(t_local, before);
        const double target = t_local - before;
        if (d.vec && common && residual) {
            find_crossing<EPV>(P, sh, d, row_share<ANY_SIZE>(d.V / EPV, cs, rank, cw), target, vector_weights, [&](int u) { return u * EPV; });
        } else if (d.vec) {
            find_crossing<EPV>(P, sh, d, row_share<ANY_SIZE>(d.V / EPV, cs, rank, cw), target,
                [&](int u, double (&w)[EPV]) {
#pragma unroll 1
                    for (int e = 0; e < EPV; ++e) {
                        const double v = weight(load_logit<DT>(a_row, u * EPV + e), residual ? load_logit<DT>(b_row, u * EPV + e) : 0.f);
#pragma unroll
                        for (int q = 0; q < EPV; ++q) if (q == e) w[q] = v;
                    }
                },
                [&](int u) { return u * EPV; });
        } else {
            find_crossing<1>(P, sh, d, row_share<ANY_SIZE>(d.V, cs, rank, cw), target,
                [&](int u, double (&w)[1]) { w[0] = weight(load_logit<DT>(a_row, u), residual ? load_logit<DT>(b_row, u) : 0.f); },
                [&](int u) { return u; });
        }
        return;
    }
}

// ---- what the finish kernel and the row kernel share -------------------------------------------
template <int DT, int KIND>
__device__ __forceinline__ Candidate candidate(const FinishParams& P, int item, const char* a_row, const char* b_row) {
    Candidate c = {-1, 0.f, 0.f, 0.f};
    if constexpr (KIND == kDrawResidual) {
        c.x = P.tokens[item];
        if (c.x >= 0 && c.x < P.V) { c.ax = load_logit<DT>(a_row, c.x); c.bx = load_logit<DT>(b_row, c.x); }
        c.ua = P.u_accept[item];
    }
    return c;
}
// (`rs` and `bt` below: of residual draws alone, else null.)
// Position i of a row judged by a warp, as far as that goes without the second sweep's sum (its first lane returns that).
template <int KIND>
__device__ __forceinline__ Judged judge_pair_early(const FinishParams& P, ResidualShared* rs, const PairTotals& tot, int i, const Candidate& c, int lane) {
    // the two logarithms the judgement needs, by two lanes at once
    const double lz = log(lane == 1 ? tot.Zb : tot.Za);
    const double lnZa = lz, lnZb = __shfl_down_sync(0xffffffffu, lz, 1);
    Judged j = {false, false, false, 0.0};
    if (lane == 0) {
        j = judge_early(P, tot, lnZa, lnZb, c);
        if constexpr (KIND == kDrawResidual) {
            if (i < kPairRefs) {
                PairRef ref;
                ref.za = tot.Za; ref.zb = tot.Zb; ref.ln_rho = lnZa - lnZb; ref.ka = (tot.state & kRecordStats) ? tot.ka : __int_as_float(0x7fc00000); ref.kb = tot.kb;
                rs->ref[i] = ref;
            }
        }
    }
    return j;
}
// What a residual draw's tables start from, by the block's first threads; a barrier before they are read.
__device__ __forceinline__ void residual_tables(ResidualShared& rs, int tid) {
    if (tid < kExpTable) rs.exp_table[tid] = exp2(static_cast<double>(tid) * (1.0 / kExpTable));
    if (tid == 0) {
        rs.exp_consts[0] = 6755399441055744.0; rs.exp_consts[1] = 256.0;
        rs.exp_consts[2] = 2.239395190875157e-12; rs.exp_consts[3] = 3.308302680541371e-09;
        rs.exp_consts[4] = 3.665565596910106e-06; rs.exp_consts[5] = 2.7076061740622863e-03;
    }
}
// Entry i of the table of bf16 exponentials, of either sign
__device__ __forceinline__ void bf16_table_entry(ExpTable<FSD_BF16>& bt, const ResidualShared& rs, int i) {
    const double x = __uint_as_float(static_cast<uint32_t>(kBf16Lowest + i) << 16);
    bt.e[i] = exp2_table(x * kLog2eD, rs.exp_table);
    bt.e[kBf16Count + i] = exp2_table(-x * kLog2eD, rs.exp_table);
}
// The row's token.  `rejected`: drawn from the residual where the kind is.
template <int DT, int KIND, bool LOCAL>
__device__ __forceinline__ void draw_token(const FinishParams& P, FinishShared& sh, ResidualShared* rs, const ExpTable<DT>* bt, const Draw& d, Link& link, int& status, bool rejected) {
    if constexpr (KIND == kDrawPt) {
        draw_pt<DT, LOCAL>(P, sh, d, link, status);
    } else if constexpr (KIND == kDrawGreedy) {
        draw_argmax<DT, LOCAL>(P, sh, d, link, status);
    } else {
        const bool greedy = P.sample == FSD_SAMPLE_GREEDY;
        if (!rejected) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        if (rejected) draw_residual<DT, LOCAL>(P, sh, *rs, *bt, d, link, status, greedy);
        else if (greedy) draw_argmax<DT, LOCAL>(P, sh, d, link, status);
        else draw_pt<DT, LOCAL>(P, sh, d, link, status);
    }
}

template <int DT, int KIND>
__global__ void __launch_bounds__(kFinishThreads, 2) fsd_finish_kernel(const __grid_constant__ FinishParams P) {
    __shared__ FinishShared sh;
    __shared__ ResidualShared rs;                        // (used by the residual's instantiation alone)
    __shared__ ExpTable<DT> bt;
    __shared__ std::conditional_t<KIND == kDrawResidual, NoTree, TreeShared> tr;
    cg::cluster_group cluster = cg::this_cluster();
    const int cs = static_cast<int>(cluster.num_blocks());
    const int rank = static_cast<int>(cluster.block_rank());
    const int b = static_cast<int>(blockIdx.x) / cs;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int G = P.G, V = P.V;
    const size_t rb = static_cast<size_t>(V) * Logit<DT>::kBytes;
    const char* t_base = static_cast<const char*>(P.target) + static_cast<size_t>(b) * (G + 1) * rb;
    const char* d_base = static_cast<const char*>(P.draft) + static_cast<size_t>(b) * G * rb;
    const bool tree = KIND != kDrawResidual && P.parent != nullptr;

    if (tid == 0) {
        mbar_init(&sh.link[0], 1); mbar_init(&sh.link[1], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");     // "this CTA has started": waited for below
    if (tid == 0) { sh.cand = -1; sh.last_pos = -1; sh.n_acc = G; sh.bad = 0; sh.row_sel = 0; sh.amb = 0; sh.n_close = 0; sh.next = 0; sh.far = 0; }
    if (tid < kJudgeWords) sh.bits[tid] = 0;
    if constexpr (KIND == kDrawResidual) {
        residual_tables(rs, tid);
    }
    __syncthreads();
    // What comes behind this kernel may be set up while it runs.  (A residual draw allows that when its pass is through:
    // earlier, the next call's blocks are spread over the SMs as its rows end, 64 x 8 x 152064 136.5 -> 140 us.)
    if constexpr (KIND != kDrawResidual) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // everything above touched no global memory; what follows reads what the pair kernel wrote
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");       // every CTA of the cluster runs: its shared memory may be written
    Link link = {0, false, &P.flags->number};
    if (blockIdx.x == 0 && tid == 0) atomicAdd(reinterpret_cast<unsigned long long*>(&P.flags->epoch), 1ull);     // (nothing here reads it)

    // ---- 1. divergences, accept bits, status of this row's pairs ----
    // (asked for now, needed later: each is a trip to L2 or HBM of its own)
    float u_mine = 0.f;                               // (one load: the array may be in host memory)
    if (tid == 0) u_mine = P.u_sample[b];
    int st = 0, first = G;
    if (tid == 0 && timed_out(P.flags, *reinterpret_cast<const volatile uint64_t*>(&P.flags->number))) st |= FSD_ROW_TIMEOUT;
    const bool shared_out = P.records != nullptr && cs > 1 && G > kFinishWarps && G <= 64 * kJudgeWords * cs;
    if (P.records != nullptr) {
        // a pair per warp: its lanes fold the parts of the pair's record, the first of them judges it
        const int step = shared_out ? cs : 1, i0 = shared_out ? rank : 0;
        for (int i = warp * step + i0; i < G; i += kFinishWarps * step) {
            const int item = b * G + i;
            // (the candidate's logits are on their way while the record is folded)
            const Candidate c = candidate<DT, KIND>(P, item, t_base + static_cast<size_t>(i) * rb, d_base + static_cast<size_t>(i) * rb);
            const PairTotals tot = fold_record(P.records + item, P.div);
            float D = 0.f;
            int bit = 0, s = 0;
            const Judged j = judge_pair_early<KIND>(P, &rs, tot, i, c, lane);
            if (lane == 0) {
                judge_late(P, tot, j, D, bit, s);
                if (shared_out || rank == 0) P.divergence[item] = D;
                st |= s;
                if (tree) {
                    if constexpr (KIND != kDrawResidual) {
                        if (!shared_out) tr.bit[i] = static_cast<int8_t>(bit);
                        else if (bit) atomicOr(&sh.bits[i / cs >> 6], 1ull << (i / cs & 63));
                    }
                } else if (!bit && i < first) {
                    first = i;
                }
            }
        }
    } else {
        for (int i = tid; i < G; i += kFinishThreads) {
            const int item = b * G + i;
            const int bit = P.item_bits[item];
            st |= P.item_status[item];
            if constexpr (KIND != kDrawResidual) { if (tree) tr.bit[i] = static_cast<int8_t>(bit); }
            if (!tree && !bit && i < first) first = i;
        }
    }
    if constexpr (KIND == kDrawResidual && DT == FSD_BF16) {
        // The table, by whichever warps have no pair to judge (left), a warp's worth at a time: judging is trips to L2 and
        // chains of double-precision latencies, the table 1.2 us of instruction issue.
        for (;;) {
            int part = 0;
            if (lane == 0) part = atomicAdd(&sh.next, 1);
            part = __shfl_sync(0xffffffffu, part, 0);
            if (part >= kBf16Count / 32) break;
            bf16_table_entry(bt, rs, part * 32 + lane);
        }
    }
    if (tid == 0) sh.u = u_mine;
    st = __reduce_or_sync(0xffffffffu, st);
    first = __reduce_min_sync(0xffffffffu, first);
    if (lane == 0) {
        if (st) atomicOr(&sh.bad, st);
        if (!tree) atomicMin(&sh.n_acc, first);
    }
    __syncthreads();
    if (shared_out) {
        // (the bits travel as what a double's bits are; nothing computes with them)
        double mine[1 + kJudgeWords];
        mine[0] = __longlong_as_double(static_cast<long long>(sh.bad) << 32 | sh.n_acc);
#pragma unroll
        for (int k = 0; k < kJudgeWords; ++k) mine[1 + k] = __longlong_as_double(static_cast<long long>(sh.bits[k]));
        const double (*all)[kExchangeDoubles] = cluster_exchange(P, sh, cs, rank, link, mine);
        int bad = 0, prefix = G;
        for (int r = 0; r < cs; ++r) {
            const long long w = __double_as_longlong(all[r][0]);
            bad |= static_cast<int>(w >> 32);
            prefix = min(prefix, static_cast<int>(w & 0xffffffff));
        }
        if constexpr (KIND != kDrawResidual)
            for (int i = tree ? tid : G; i < G; i += kFinishThreads)
                tr.bit[i] = static_cast<int8_t>(__double_as_longlong(all[i % cs][1 + (i / cs >> 6)]) >> (i / cs & 63) & 1);
        __syncthreads();
        if (tid == 0 && !link.lost) { sh.bad = bad; sh.n_acc = prefix; }      // (its own are in range)
        __syncthreads();
    }

    // ---- 2. accepted prefix (chain) or deepest accepted path (tree) ----
    int n = sh.n_acc, row_sel = n;
    if constexpr (KIND != kDrawResidual) {
        if (tree && !link.lost) {                    // (lost: whether the parents are valid is not known)
            tree_select(P.parent + static_cast<size_t>(b) * G, G, P.max_depth,
                        rank == 0 ? P.path + static_cast<size_t>(b) * P.max_depth : nullptr, sh, tr);
            __syncthreads();
            n = sh.n_acc; row_sel = sh.row_sel;
            FSD_CHECK(&P.flags->debug, row_sel >= 0 && row_sel <= G && n >= 0 && n <= P.max_depth, kChkPath);
        }
    }
    FSD_CHECK(&P.flags->debug, link.lost || (row_sel >= 0 && row_sel <= G && n >= 0 && n <= (tree ? P.max_depth : G)), kChkRow);
    int status = sh.bad;

    // ---- 3. token draw ----
    const bool residual = KIND == kDrawResidual && n < G, bad_tree = (status & FSD_ROW_BADTREE) != 0;      // (uniform over the cluster)
    Draw d;
    d.a_row = t_base + static_cast<size_t>(row_sel) * rb;
    d.b_row = d_base + static_cast<size_t>(residual ? n : 0) * rb;
    d.b = b; d.n = n; d.V = V; d.cs = cs; d.rank = rank; d.shared_out = shared_out; d.vec = P.vec != 0; d.u = static_cast<double>(sh.u);
    d.span = 0; d.local = 0;
    if (link.lost) {
        n = 0;                                           // (nothing of the row is valid but its status)
    } else if (bad_tree) {
        n = 0;
        if (rank == 0 && tid == 0) P.next_token[b] = -1;
    } else {
        draw_token<DT, KIND, false>(P, sh, &rs, &bt, d, link, status, residual);
    }
    if (rank == 0 && tid == 0) {
        P.accept_len[b] = n;
        P.row_status[b] = status | (link.lost || timed_out(P.flags, *reinterpret_cast<const volatile uint64_t*>(&P.flags->number)) ? FSD_ROW_TIMEOUT : 0);
    }
    leave_last(link.lost);
}
}  // namespace fsd
