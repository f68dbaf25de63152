// Streaming per-(row, position) kernel: every logit is read from HBM once.
//
// A (row, position) pair is split along the vocabulary over a GROUP of C thread blocks (C <= 24,
// chosen by the host from what fits on chip and the number of pairs), one block of sixteen compute
// warps and one helper warp per SM.  The groups are persistent: group g takes pairs g, g + groups, ...
//
// The blocks of a group wait for one another's sums, and usually all of them run.  The launch does not promise it: a
// cooperative launch would, but it starts only when the kernel in front has ended and that end has been polled for (a
// period of 2.05 us; calls in a row took multiples of it), while a launch with programmatic stream serialization is set
// up before.  So a block that has waited for about fifteen milliseconds, or finds that a message it wants has been
// overwritten because the others went on without it, computes the missing blocks' messages itself, bit for bit, and goes on.
//
// A block's slice of a pair's two rows arrives in a ring of shared-memory slots (bulk asynchronous
// copies started by the helper warp; the ring is as deep as the slices allow, two slots at least).
// The compute warps are independent of one another: a warp owns a fixed run of the slice's 16-byte
// vectors (at most four steps of eight entries a lane), and in round n it does, step by step,
//   1. the first sweep of pair n: e = 2^(logit * log2e - k), the sums Z = sum e and S = sum e*y (or
//      the KL sum), a bitwise "rows differ" flag.  The references k (integers in the log2 domain) come
//      from the maxima of the part's first step (of all of it where that has no finite logit), looked at when the round
//      before is done.  That is near enough for any ordinary logits; a warp whose sums say it was not (a later logit
//      2^30 above it) does the sweep over with exact maxima.  Where a -inf spoils the entropy sums it does it over
//      with clamped logits, and clamps from then on: that changes no bit of a part it was not needed for, so a pair's
//      sums depend on its two rows alone;
//   2. interleaved with it, the SECOND sweep of pair n - 2 over the e values parked two rounds
//      earlier: p = e_a/Z_a, q = e_b/Z_b, JS needs sum (p+q) log2(p+q), TV sum |p - q|, KL nothing.
//      The new e values take the tensor-memory columns the old ones leave (64 values a lane and pair,
//      two pairs in flight, 128 columns a warp: all of the SM's tensor memory);
//   3. a fold of its five sums over its lanes, posted for the helper warp.
// The helper warp folds the sixteen warps' sums, leaves them as a tagged message in global memory,
// fetches the messages of the whole group (they live in L2), folds those and hands 1/Z_a, 1/Z_b to
// its block.  That exchange has a whole round's time: the totals of pair n are needed in round n + 2.
//
// What bounds it.  JS takes three special-function results per vocabulary entry (two ex2, one lg2):
// 512 pairs of 152064 entries are 50 us of that pipe on 148 SMs at 1965 MHz, and 48 us of HBM.  The
// kernel takes 92 us there (3.4 TB/s; the form in which all warps of a block waited for the group's
// totals between the two sweeps of a pair took 127 us): 40 rounds of 2.0 us, of which the sweeps are
// two thirds, the wait for data and totals a sixth, the fold a seventh, plus 3.5 us until the first
// slices have landed.  KL has no second sweep and no exchange and runs at 5 TB/s.  Of what was
// tried on it: ex2 on the FMA pipe for a part of the entries (+8 %, the extra instructions cost more
// than the special-function pipe gains), five and more pairs in flight in smaller parts (more rounds,
// the fold weighs more), reading the references from a full pass over the part (+1 %).
//
// Rows that are not whole 16-byte vectors (or start off a 16-byte boundary) are streamed as the
// aligned 16-byte granules that cover them; the draft row's granules are shifted onto the target
// row's in shared memory, in place, and the entries in front of and behind the rows become -1e30.  A granule
// that holds at least one byte of a row never crosses into another page.
#pragma once

#include <climits>
#include <cstddef>
#include <type_traits>

#include "fsd_device.cuh"

namespace fsd {

constexpr int kComputeWarps = 16;
constexpr int kStreamThreads = 32 * (kComputeWarps + 1);   // and one helper warp
constexpr int kMaxSteps = 4;                               // steps a warp parks per pair; two pairs in flight fill its 128 tensor-memory columns
constexpr int kStepEntries = 8;                            // vocabulary entries a lane handles per step
constexpr int kTmemCols = 512;                             // all of the SM's columns: warp w owns 32 lanes x 128 columns
constexpr int kParkCols = 2 * kStepEntries;                // e values a lane parks per step (both rows)
constexpr int kPortableCluster = 8;                        // most thread blocks of a cluster without asking for more (finish kernel)
constexpr int kMaxClusterSize = 12;                        // and at all (row kernel, see row_plan)
constexpr int kMaxGroupSize = 24;                          // most blocks in a group of the streaming kernel
constexpr uint32_t kSpinLimit = 1u << 24;                  // polls before a wait gives up
constexpr uint64_t kWaitNs = 4000000000ull;                // and its limit in time
constexpr uint64_t kInjectedWaitNs = 20000000ull;          // test aid: of waits made to run out (see fsd_set_timeout_injection)
constexpr uint32_t kSleepNs = 40;                          // sleep between two polls of a barrier in shared memory

// Partial statistics of one (target row, draft row) pair: of a warp, of a block, or -- in a pair's
// record -- of each block of the group that streamed the pair.
//   z = sum 2^y, s = sum 2^y * y with y = logit*log2e - k and k the integer reference (log2
//   domain) the sums are relative to.  s0 is the target row's s for JS and the KL sum
//   sum 2^ya (ya - yb) for KL.
struct alignas(16) Stats {
    float ka, kb;              // references; -inf: no finite logit seen; NaN: a NaN logit
    float za, zb;
    float s0, sb;
    float x;                   // second-sweep sum (in flight only)
    uint32_t diff;             // 0: the two rows are bitwise identical so far
};
static_assert(sizeof(Stats) == 32, "Stats travels as two 16-byte stores");

// What the streaming kernel leaves per pair for the finish kernel, which folds the parts in
// double precision (second-sweep sums: JS sum s log2 s, TV sum |p - q|).
struct alignas(16) PairRecord {
    Stats part[kMaxGroupSize];
    float x[kMaxGroupSize];    // each block's second-sweep sum of this pair
    uint32_t ncta;             // parts in use
    uint32_t state;            // kRecordStats | kRecordBadTree
    uint32_t pad[2];
};
static_assert(sizeof(PairRecord) == 880, "PairRecord layout");
constexpr uint32_t kRecordStats = 1, kRecordBadTree = 2;

// One block's statistics of a round as they cross global memory: 16-byte units, each stored whole
// and ending in 64 bits of call and round (see CallFlags), so that a reader knows a unit is this round's without any fence
// or flag (a unit of another round or call, or what the workspace held before, is fetched again).  That is why
// nothing has to be cleared in front of a call, which took a memset of 1.5 us in a call of 16.
struct alignas(16) GroupMsg {
    uint4 u[2];                // target row: {reference, Z, call number's high half, its low half + round}; draft row: the same
};
static_assert(sizeof(GroupMsg) == 32, "GroupMsg layout");

struct StreamParams {
    const void* target;        // [B, G+1, V]
    const void* draft;         // [B, G,   V]
    const int32_t* parent;     // [B, G] (tree) or null (chain)
    int G;
    uint32_t g_magic, g_shift; // item / G == umulhi(item, g_magic) >> g_shift for items below 2^31
    int nvec_row;              // 16-byte vectors (granules of an unaligned row, at most) per logit row
    size_t row_bytes;
    int slot_row_bytes, slot_bytes, ring;    // of the shared-memory ring (see slot_bytes())
    int n_items;               // B * G
    PairRecord* records;       // [B * G]
    uint64_t nonce;            // what the call's number is made of (see CallFlags)
    CallFlags* flags;
    int C;                     // blocks per group (<= kMaxGroupSize)
    uint32_t poll_limit;       // fetches of the group's messages before the exchange gives up (kSpinLimit normally)
    uint32_t help_after;       // fetches after which a block computes what it waits for by itself (0xffffffff: never)
    int silent_rank;           // test aid: this rank of group 0 keeps its first message to itself (-1: nobody)
    int raise;                 // test aid: the first block raises the timeout flag as it ends
    GroupMsg* exchange;        // [groups][2][C]
};

// ---- PTX wrappers -----------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
    return ok != 0;
}
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) { bulk_g2s(smem_u32(dst), src, bytes, bar); }

__device__ __forceinline__ uint64_t global_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ void raise_flag(CallFlags* flags, uint64_t number) {
    atomicExch(reinterpret_cast<unsigned long long*>(&flags->raised), static_cast<unsigned long long>(number));
}
// Bounded wait of a whole warp for a phase of an mbarrier: kSpinLimit polls or kWaitNs, whatever is
// first.  False (for every lane) and the flag raised if the phase never completes or somebody else's
// wait has run out already.
__device__ __noinline__ bool warp_wait_slow(uint64_t* bar, uint32_t parity, CallFlags* flags, uint64_t nonce) {
    uint64_t t0 = 0;
    const uint64_t number = call_number(flags, nonce);
#pragma unroll 1
    for (uint32_t i = 0; i < kSpinLimit / 64; ++i) {
#pragma unroll 1
        for (int k = 0; k < 64; ++k) {
            if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
            __nanosleep(kSleepNs);                   // (the warps that have work keep the issue slots)
        }
        // somebody has given up already: nothing this warp waits for is certain to come
        const uint64_t t = global_ns();
        if (t0 == 0) t0 = t;
        if (__any_sync(0xffffffffu, timed_out(flags, number) || t - t0 > kWaitNs)) break;
    }
    if ((threadIdx.x & 31) == 0) raise_flag(flags, number);
    return false;
}
// Bounded wait of a thread where nobody raises a flag meanwhile (the exchanges within a cluster, copies of its own).
// (In one loop: with a function of its own for the waits that take longer, the finish kernel's draws were 1 to 4 % slower.)
__device__ __forceinline__ bool thread_wait(uint64_t* bar, uint32_t parity, [[maybe_unused]] uint64_t limit_ns) {     // (a limit: debug build; 0: none)
#ifdef FSD_DEBUG_CHECKS
    const uint64_t t0 = global_ns();
#endif
#pragma unroll 1
    for (uint32_t i = 0; i < kSpinLimit; ++i) {
        if (mbar_try_wait(bar, parity)) return true;
#ifdef FSD_DEBUG_CHECKS
        if (limit_ns != 0 && global_ns() - t0 > limit_ns) break;
#endif
    }
    return false;
}
// A block that has not got what its cluster's others were to push to it leaves last: they may push still.
__device__ __forceinline__ void leave_last(bool lost) {
    if (lost) {
        asm volatile("barrier.cluster.arrive.release;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire;" ::: "memory");      // (blocks that have left count as arrived)
        __nanosleep(50000);                                              // (what they pushed last is there by now)
    }
}
__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity, const StreamParams& P) {
    if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
    return warp_wait_slow(bar, parity, P.flags, P.nonce);
}

// Pushes between the blocks of a cluster: the address of the same object in block `rank`, and a remote
// store that counts its eight bytes in on a barrier of the receiver.
__device__ __forceinline__ uint32_t cluster_addr(const void* p, int rank) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_u32(p)), "r"(rank));
    return r;
}
__device__ __forceinline__ void st_async(uint32_t addr, uint64_t v, uint32_t bar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(addr), "l"(v), "r"(bar) : "memory");
}

// tensor memory: 16 columns of this warp's 32 lanes, one value a lane and column
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const float (&r)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
        ::"r"(taddr), "f"(r[0]), "f"(r[1]), "f"(r[2]), "f"(r[3]), "f"(r[4]), "f"(r[5]), "f"(r[6]), "f"(r[7]),
        "f"(r[8]), "f"(r[9]), "f"(r[10]), "f"(r[11]), "f"(r[12]), "f"(r[13]), "f"(r[14]), "f"(r[15]));
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]), "=f"(r[4]), "=f"(r[5]), "=f"(r[6]), "=f"(r[7]),
          "=f"(r[8]), "=f"(r[9]), "=f"(r[10]), "=f"(r[11]), "=f"(r[12]), "=f"(r[13]), "=f"(r[14]), "=f"(r[15])
        : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// NaN-propagating maxima: a NaN logit must reach the row maximum so that the row is flagged
__device__ __forceinline__ uint32_t bf16x2_max_nan(uint32_t a, uint32_t b) {
    uint32_t d;
    asm("max.NaN.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}
__device__ __forceinline__ float fmax_nan(float a, float b) {
    float d;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
    return d;
}
// ---- packed pairs of floats (one instruction works on two values) --------------------------
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ float sum2(uint64_t v) {
    float lo, hi;
    unpack2(v, lo, hi);
    return lo + hi;
}

// 2^(k - K) for integer-valued k <= K, exact; 0 below the normal range, for k = -inf ("no reference"), and where
// either is NaN (the sums it scales are NaN then)
__device__ __forceinline__ float pow2_ref(float k, float K) {
    return __int_as_float(__float_as_int(fmaxf(k - K, -127.f) + 12583039.f) << 23);      // 1.5 * 2^23 + 127: the low bits are the exponent field
}
__device__ __forceinline__ float rcp(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// the reference a maximum gives (log2 domain); none (-inf) where no finite logit was seen
__device__ __forceinline__ float reference(float maximum) { return maximum <= -9.9e29f ? -INFINITY : ceilf(maximum * kLog2e); }
// a lane's Z_a + Z_b up to which the references were near enough: an entry may exceed 2^k by about 2^30, as the exponents'
// rounding allows
constexpr float kNearZ = 4.0e10f;
// maximum over the warp, NaN if any lane holds one
__device__ __forceinline__ float warp_redux_max_nan(float v) {
    float d;
    asm volatile("redux.sync.max.NaN.f32 %0, %1, 0xffffffff;" : "=f"(d) : "f"(v));
    return d;
}
// A KL partial sum brought to another reference: +inf (a logit with p > 0 = q) stays +inf even
// when the factor underflows to 0
__device__ __forceinline__ float scale_kl(float f, float v) { return v == INFINITY ? v : f * v; }

// One unit is stored and fetched as a single 128-bit access (the .b128 forms: one access, not four
// that happen to be adjacent), so a reader sees a unit either whole or not at all.
__device__ __forceinline__ void st_unit(uint4* p, float a, float b, float c, uint32_t tag) {
    const uint64_t lo = static_cast<uint64_t>(__float_as_uint(a)) | (static_cast<uint64_t>(__float_as_uint(b)) << 32);
    const uint64_t hi = static_cast<uint64_t>(__float_as_uint(c)) | (static_cast<uint64_t>(tag) << 32);
    asm volatile("{ .reg .b128 t; mov.b128 t, {%1, %2}; st.relaxed.gpu.global.b128 [%0], t; }" ::"l"(p), "l"(lo), "l"(hi) : "memory");
}
__device__ __forceinline__ uint4 ld_unit(const uint4* p) {
    uint64_t lo, hi;
    asm volatile("{ .reg .b128 t; ld.relaxed.gpu.global.b128 t, [%2]; mov.b128 {%0, %1}, t; }" : "=l"(lo), "=l"(hi) : "l"(p) : "memory");
    return make_uint4(static_cast<uint32_t>(lo), static_cast<uint32_t>(lo >> 32), static_cast<uint32_t>(hi), static_cast<uint32_t>(hi >> 32));
}

// 16-byte accesses of shared memory by address
__device__ __forceinline__ uint4 ld_shared16(uint32_t addr) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
    return v;
}
__device__ __forceinline__ void st_shared16(uint32_t addr, const uint4& v) {
    asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w));
}

// ---- shared-memory layout ---------------------------------------------------------------
// A ring of slots, each holding the block's slice of one pair: the target row's vectors (whole steps),
// then the draft row's.  The draft part of an unaligned row is copied warp by warp, each part one granule longer
// (its last vector straddles two), so there the parts lie a granule further apart.
template <int DT> struct StreamShape {
    static constexpr int kVecPerStep = kStepEntries / Logit<DT>::kPerVec;   // 16-byte vectors a lane handles per step and row
    static constexpr int kSteps = DT == FSD_BF16 ? 4 : 3;                   // most steps of a warp's part: 2 or 3 KB of each row
    static constexpr int kWarpVecs = 32 * kVecPerStep * kSteps;
    static constexpr int kBlockVecs = kComputeWarps * kWarpVecs;
    static constexpr int kStepVecs = 32 * kVecPerStep;
};
static_assert(StreamShape<FSD_BF16>::kSteps <= kMaxSteps && StreamShape<FSD_F32>::kSteps <= kMaxSteps, "two parts fit a warp's tensor memory");
constexpr int kRingBytes = 224 * 1024;                     // shared memory for the ring (one slot is in use, the rest in flight)
constexpr int kMaxRing = 8, kMinRing = 2;
// bytes from a slot's start to its draft part, and of a whole slot, for slices of up to `slice` vectors
template <int DT> constexpr int slot_row_bytes(int slice) {
    return (slice + StreamShape<DT>::kStepVecs - 1) / StreamShape<DT>::kStepVecs * StreamShape<DT>::kStepVecs * 16;
}
template <int DT> constexpr int slot_bytes(int slice, bool ragged) { return 2 * slot_row_bytes<DT>(slice) + (ragged ? kComputeWarps * 16 : 0); }
static_assert(kMinRing * slot_bytes<FSD_BF16>(StreamShape<FSD_BF16>::kBlockVecs, true) <= kRingBytes &&
              kMinRing * slot_bytes<FSD_F32>(StreamShape<FSD_F32>::kBlockVecs, true) <= kRingBytes, "the largest slices have two slots");

// A warp's part of the block's slice: whole steps, dealt out as evenly as they go.  The warps that share
// a scheduler with the helper warp get a step more last.
struct WarpPart { int pos, first, count, steps; };     // place in the slice's order; vectors from the slice's start; steps
__device__ __forceinline__ WarpPart warp_part(int warp, int slice, int step_vecs) {
    WarpPart p;
    const int all = (slice + step_vecs - 1) / step_vecs, sb = all / kComputeWarps, sr = all % kComputeWarps;
    p.pos = (warp & 3) == 0 ? 12 + (warp >> 2) : (warp >> 2) * 3 + (warp & 3) - 1;
    p.steps = sb + (p.pos < sr ? 1 : 0);
    p.first = (p.pos * sb + (p.pos < sr ? p.pos : sr)) * step_vecs;
    p.count = p.steps == 0 ? 0 : slice - p.first < p.steps * step_vecs ? slice - p.first : p.steps * step_vecs;
    return p;
}

struct alignas(16) WarpPost {              // what a compute warp hands the helper each round (its own lanes folded)
    float z[4];                // za, zb, s0, sb of pair n
    float ka, kb;
    float x;                   // second-sweep sum of pair n - 2
    uint32_t diff;
};
struct StreamShared {
    uint64_t full[kMaxRing];                     // a slot's slices have landed
    uint64_t posted[2];                        // all compute warps have posted round n (n & 1)
    uint64_t totals[2];                        // the helper is done with the posts of round n: totals valid, slots free
    WarpPost post[2][kComputeWarps];
    alignas(16) float4 tot[2];                             // Ka, 1/Za, Kb, 1/Zb of the round's pair (0: not a valid distribution)
    uint32_t meta[kMaxRing];                     // unaligned rows: byte offset of the target row's first granule << 8 | shift of the draft row
    uint32_t tmem_base;
};
static_assert(sizeof(WarpPost) == 32 && offsetof(WarpPost, ka) == 16 && offsetof(StreamShared, post) % 16 == 0 && offsetof(StreamShared, tot) % 16 == 0, "16-byte accesses");
static_assert(alignof(StreamShared) <= 16 && kRingBytes % 16 == 0, "16-byte copies");
constexpr size_t kStreamSmemBytes = kRingBytes + sizeof(StreamShared) + 128;
static_assert(kStreamSmemBytes <= 227 * 1024, "shared memory of an SM");

// 16 bytes starting `sh` bytes into the 32 bytes (lo, hi); sh is the same for the whole warp
template <int DT>
__device__ __forceinline__ uint4 shifted(const uint4& lo, const uint4& hi, uint32_t sh) {
    uint32_t w[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
    const bool two = (sh & 8) != 0, one = (sh & 4) != 0;
#pragma unroll
    for (int i = 0; i < 6; ++i) w[i] = two ? w[i + 2] : w[i];
#pragma unroll
    for (int i = 0; i < 5; ++i) w[i] = one ? w[i + 1] : w[i];
    if constexpr (DT == FSD_BF16) {
        const uint32_t bits = (sh & 2) * 8;
#pragma unroll
        for (int i = 0; i < 4; ++i) w[i] = __funnelshift_r(w[i], w[i + 1], bits);
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
}

// The vector's entries outside [0, V) read as -1e30 (2^y = 0), or as -inf; k0 is the index of its first entry
template <int DT>
__device__ __noinline__ uint4 masked_vector(uint4 v, int k0, int V, bool minus_inf = false) {
    constexpr int EPV = Logit<DT>::kPerVec;
    uint32_t w[4] = {v.x, v.y, v.z, v.w};
    const uint32_t fill = minus_inf ? 0xff800000u : 0xf1490000u;
#pragma unroll
    for (int j = 0; j < EPV; ++j) {
        if (k0 + j >= 0 && k0 + j < V) continue;
        if constexpr (DT == FSD_BF16) w[j >> 1] = (j & 1) ? ((w[j >> 1] & 0x0000ffffu) | fill) : ((w[j >> 1] & 0xffff0000u) | fill >> 16);
        else w[j] = minus_inf ? fill : 0xf149f2cau;
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
}

// What the compute warps of a block would post of a slice's references and Z's, by one warp from global memory: the
// same parts, lanes and order of additions, so the same bits.  Lane w returns warp w's of the target row, lane 16 + w those of
// the draft row.  `off`: entries of the first granule in front of the row (both rows': the draft's are moved onto the target's).
template <int DT>
__device__ __noinline__ float2 slice_sums(const void* arow, const void* brow, int off, int V, int vbeg, int vcnt) {
    constexpr int EPV = Logit<DT>::kPerVec, VPS = StreamShape<DT>::kVecPerStep;
    const int lane = threadIdx.x & 31;
    float2 mine = make_float2(-INFINITY, 0.f);
#pragma unroll 1
    for (int w = 0; w < kComputeWarps; ++w) {
        const WarpPart part = warp_part(w, vcnt, 32 * VPS);
        if (part.steps == 0) continue;
        const auto first_entry = [&](int v) { return v * 32 + lane < part.count ? (vbeg + part.first + v * 32 + lane) * EPV - off : V; };
        const auto entry = [&](const void* row, int k) { return k >= 0 && k < V ? load_logit<DT>(row, k) : -1.0e30f; };
        float ka, kb, za, zb;
        const auto look = [&](int vectors) {
            float ma = -INFINITY, mb = -INFINITY;
#pragma unroll 1
            for (int v = 0; v < vectors; ++v) {
                const int k = first_entry(v);
#pragma unroll
                for (int e = 0; e < EPV; ++e) { ma = fmax_nan(ma, entry(arow, k + e)); mb = fmax_nan(mb, entry(brow, k + e)); }
            }
            __syncwarp();
            ka = reference(warp_redux_max_nan(ma)); kb = reference(warp_redux_max_nan(mb));
        };
        const auto sum = [&]() {                      // false: the references were not near enough
            const float ca = ka == -INFINITY ? 0.f : -ka, cb = kb == -INFINITY ? 0.f : -kb;
            uint64_t za2 = 0, zb2 = 0;
#pragma unroll 1
            for (int v = 0; v < part.steps * VPS; ++v) {
                const int k = first_entry(v);
#pragma unroll
                for (int e = 0; e < EPV; e += 2) {
                    za2 = add2(za2, pack2(ex2(fmaf(entry(arow, k + e), kLog2e, ca)), ex2(fmaf(entry(arow, k + e + 1), kLog2e, ca))));
                    zb2 = add2(zb2, pack2(ex2(fmaf(entry(brow, k + e), kLog2e, cb)), ex2(fmaf(entry(brow, k + e + 1), kLog2e, cb))));
                }
            }
            za = sum2(za2); zb = sum2(zb2);
            return __all_sync(0xffffffffu, za + zb < kNearZ) != 0;
        };
        look(VPS);
        if (ka == -INFINITY || kb == -INFINITY) look(part.steps * VPS);
        if (!sum()) { look(part.steps * VPS); sum(); }
#pragma unroll
        for (int m = 16; m > 0; m >>= 1) { za += __shfl_xor_sync(0xffffffffu, za, m); zb += __shfl_xor_sync(0xffffffffu, zb, m); }
        if (lane == w) mine = make_float2(ka, za);
        if (lane == 16 + w) mine = make_float2(kb, zb);
    }
    __syncwarp();
    return mine;
}

// Sixteen warps' Z (a lane each; the draft row's in the upper half) brought to the largest of their references and added up.
__device__ __forceinline__ float fold_z(float k, float z, bool b_side, float& Ka, float& Kb, float& f) {
    Ka = warp_redux_max_nan(b_side ? -INFINITY : k); Kb = warp_redux_max_nan(b_side ? k : -INFINITY);
    f = pow2_ref(k, b_side ? Kb : Ka);
    float sum = __fmul_rn(z, f);
#pragma unroll
    for (int m = 8; m > 0; m >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, m);
    return sum;
}
// The messages of a pair that have not come (bit r and 16 + r of miss0: block r's, of miss1: block 16 + r's), computed by the helper
// warp; the others stay as they are.  (That the path is there at all costs TV 2 us of 86 on 64 x 8 x 152064 -- without it 82
// to 84, where its code stands makes no difference -- and JS less than half a microsecond.)
template <int DT, bool RAGGED>
__device__ __noinline__ float4 missing_messages(const StreamParams& P, int item, uint32_t miss0, uint32_t miss1, float4 t) {
    const int lane = threadIdx.x & 31, r0 = lane & 15, base = P.nvec_row / P.C, rem = P.nvec_row % P.C;
    const bool b_side = lane >= 16;
    const int b = item / P.G, V = static_cast<int>(P.row_bytes / Logit<DT>::kBytes);
    int arow = item + b;
    if (P.parent != nullptr) {
        const int pr = __ldg(P.parent + item), k = item - b * P.G;
        arow = b * (P.G + 1) + (pr >= -1 && pr < k ? pr + 1 : 0);
    }
    const char* arow_p = static_cast<const char*>(P.target) + static_cast<size_t>(arow) * P.row_bytes;
    const char* brow_p = static_cast<const char*>(P.draft) + static_cast<size_t>(item) * P.row_bytes;
    const int off = RAGGED ? static_cast<int>(reinterpret_cast<uintptr_t>(arow_p) & 15) / Logit<DT>::kBytes : 0;
#pragma unroll 1
    for (int r = 0; r < P.C; ++r) {
        if (((r < 16 ? miss0 : miss1) >> (r & 15) & 0x10001u) == 0) continue;
        const float2 m = slice_sums<DT>(arow_p, brow_p, off, V, r * base + min(r, rem), base + (r < rem ? 1 : 0));
        float Ka, Kb, f;
        const float z = fold_z(m.x, m.y, b_side, Ka, Kb, f);
        if (r0 == r) { t.x = b_side ? Kb : Ka; t.y = z; }
        if (r0 + 16 == r) { t.z = b_side ? Kb : Ka; t.w = z; }
    }
    return t;
}

template <int DT, int DIV, bool RAGGED>
__global__ void __launch_bounds__(kStreamThreads, 1) fsd_pair_stream_kernel(const __grid_constant__ StreamParams P) {
    using S = StreamShape<DT>;
    constexpr int EPV = Logit<DT>::kPerVec;          // logits per 16-byte vector
    constexpr int VPS = S::kVecPerStep;
    constexpr int SV = 32 * VPS;                     // vectors of a row a warp handles per step
    constexpr bool kSecondSweep = DIV != FSD_DIV_KL;
    [[maybe_unused]] constexpr float kClamp = -1.0e30f;
    [[maybe_unused]] constexpr uint32_t kClamp2 = 0xF149F149u;       // the same as a pair of bf16
    [[maybe_unused]] constexpr uint32_t kMinusInf2 = 0xFF80FF80u;
    constexpr uint32_t kFill = DT == FSD_BF16 ? kClamp2 : 0xF149F2CAu;      // bits of kClamp

    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127));
    StreamShared& sh = *reinterpret_cast<StreamShared*>(smem + kRingBytes);

    const int C = P.C;
    const int n_groups = static_cast<int>(gridDim.x) / C;
    const int group_id = static_cast<int>(blockIdx.x) / C, rank = static_cast<int>(blockIdx.x) - group_id * C;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // rounds of this group (the blocks left over form no group)
    const int R = group_id < n_groups && group_id < P.n_items ? (P.n_items - group_id + n_groups - 1) / n_groups : 0;

    // this block's slice of every row, in vectors, and a warp's part of it (the helper's lanes know a warp's each)
    const int base = P.nvec_row / C, rem = P.nvec_row % C;
    const int vbeg = rank * base + (rank < rem ? rank : rem), vcnt = base + (rank < rem ? 1 : 0);
    const WarpPart mine = warp_part(warp < kComputeWarps ? warp : lane & (kComputeWarps - 1), vcnt, SV);
    const int steps = mine.steps;
    FSD_CHECK(&P.flags->debug, steps <= S::kSteps && vbeg + vcnt <= P.nvec_row && mine.count >= 0 && mine.first + mine.count <= (steps == 0 ? INT_MAX : vcnt), kChkSlice);

    // ---- the helper warp starts the copies ----
    int in_slot = 0, in = 0, in_item = group_id, in_par = 0;      // the pair whose slices are asked for next: its number among the group's, its id, its parent node (trees)
    auto issue_slices = [&]() {
        if (in >= R) return;
        const int slot = in_slot;
        const int b = P.G == 1 ? in_item : static_cast<int>(__umulhi(static_cast<uint32_t>(in_item), P.g_magic) >> P.g_shift);
        FSD_CHECK(&P.flags->debug, in_item >= 0 && in_item < P.n_items && b == in_item / P.G, kChkItem);
        int arow = in_item + b;                                      // chain: b * (G + 1) + i
        if (P.parent != nullptr) {
            const int i = in_item - b * P.G;
            arow = b * (P.G + 1) + ((in_par >= -1 && in_par < i) ? in_par + 1 : 0);   // an invalid node still moves (ignored) data
        }
        FSD_CHECK(&P.flags->debug, vcnt >= 0 && vcnt <= S::kBlockVecs && arow >= 0, kChkStage);
        const char* arow_p = static_cast<const char*>(P.target) + static_cast<size_t>(arow) * P.row_bytes;
        const char* brow_p = static_cast<const char*>(P.draft) + static_cast<size_t>(in_item) * P.row_bytes;
        unsigned char* dst = smem + slot * P.slot_bytes;
        if constexpr (!RAGGED) {
            if (lane == 0) mbar_arrive_expect_tx(&sh.full[slot], static_cast<uint32_t>(vcnt) * 32);
            if (lane < 2 && vcnt > 0)
                bulk_g2s(dst + lane * P.slot_row_bytes, (lane == 0 ? arow_p : brow_p) + static_cast<size_t>(vbeg) * 16, static_cast<uint32_t>(vcnt) * 16, &sh.full[slot]);
        } else {
            // granules of 16 bytes from each row's rounded-down start; the draft row needs one more where it is shifted
            const int oa = static_cast<int>(reinterpret_cast<uintptr_t>(arow_p) & 15), ob = static_cast<int>(reinterpret_cast<uintptr_t>(brow_p) & 15);
            const int na = static_cast<int>((oa + P.row_bytes + 15) >> 4), nb = static_cast<int>((ob + P.row_bytes + 15) >> 4);
            const int d = ob - oa;
            const int ga1 = min(vbeg + vcnt, na);
            const int wv0 = vbeg + mine.first;                       // lane w: warp w's part of the draft row
            const int gb = wv0 + (d < 0 ? -1 : 0), gb0 = max(gb, 0), gb1 = min(gb + mine.count + (d != 0 ? 1 : 0), nb);
            const uint32_t ba = ga1 > vbeg ? static_cast<uint32_t>(ga1 - vbeg) * 16 : 0;
            const uint32_t bb = lane < kComputeWarps && mine.count > 0 && gb1 > gb0 ? static_cast<uint32_t>(gb1 - gb0) * 16 : 0;
            // the warps moved the slot's last draft parts in place: those writes precede the copies
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            const uint32_t sum = ba + __reduce_add_sync(0xffffffffu, bb);
            if (lane == 0) {
                sh.meta[slot] = static_cast<uint32_t>(oa) << 8 | static_cast<uint32_t>(d & 15);
                mbar_arrive_expect_tx(&sh.full[slot], sum);
            }
            __syncwarp();
            if (lane == 0 && ba != 0) bulk_g2s(dst, arow_p - oa + static_cast<size_t>(vbeg) * 16, ba, &sh.full[slot]);
            if (bb != 0) bulk_g2s(dst + P.slot_row_bytes + (mine.first + mine.pos + gb0 - gb) * 16, brow_p - ob + static_cast<size_t>(gb0) * 16, bb, &sh.full[slot]);
        }
        __syncwarp();
        ++in; in_item += n_groups;
        if (++in_slot == P.ring) in_slot = 0;
        if (P.parent != nullptr && in < R) in_par = __ldg(P.parent + in_item);
    };
    if (warp == kComputeWarps) {
        if (lane == 0) {
            for (int k = 0; k < P.ring; ++k) mbar_init(&sh.full[k], 1);
            for (int k = 0; k < 2; ++k) { mbar_init(&sh.posted[k], kComputeWarps); mbar_init(&sh.totals[k], 1); }
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        __syncwarp();
        // This warp alone touches global memory.  What is in front of the kernel in its stream has to be done first: it may
        // have been launched before (programmatic stream serialization).
        asm volatile("griddepcontrol.wait;" ::: "memory");
        if (P.parent != nullptr && R > 0) in_par = __ldg(P.parent + in_item);
        for (int q = 0; q < P.ring; ++q) issue_slices();
    } else {
        if (kSecondSweep && warp == 0) {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sh.tmem_base)), "n"(kTmemCols) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        }
        // lanes without a vector in the slice's last step read "-inf" there: no copy ever writes behind the slice
        // (an unaligned draft row's vectors there are masked)
        const int end = (vcnt + SV - 1) / SV * SV;
        for (int v = vcnt + static_cast<int>(threadIdx.x); v < end; v += 32 * kComputeWarps) {
            for (int q = 0; q < P.ring; ++q) {
                *reinterpret_cast<uint4*>(smem + q * P.slot_bytes + v * 16) = make_uint4(kFill, kFill, kFill, kFill);
                if constexpr (!RAGGED) *reinterpret_cast<uint4*>(smem + q * P.slot_bytes + P.slot_row_bytes + v * 16) = make_uint4(kFill, kFill, kFill, kFill);
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");

    // second sweep and totals lag two rounds behind; KL has neither
    const int n_end = R == 0 ? 0 : (kSecondSweep ? R + 2 : R);

    if (warp < kComputeWarps) {
        const uint32_t taddr = kSecondSweep ? sh.tmem_base + (static_cast<uint32_t>(32 * (warp & 3)) << 16) + static_cast<uint32_t>(128 * (warp >> 2)) : 0;
        const uint64_t l2 = pack2(kLog2e, kLog2e);
        bool dead = false;
        float ka1 = -INFINITY, kb1 = -INFINITY, ka2 = -INFINITY, kb2 = -INFINITY;     // references of pairs n - 1 and n - 2
        // shared-memory addresses of this lane's first vectors in slot 0
        const uint32_t my_a = smem_u32(smem) + static_cast<uint32_t>(mine.first + lane) * 16;
        const uint32_t my_b = smem_u32(smem) + static_cast<uint32_t>(P.slot_row_bytes) + static_cast<uint32_t>(mine.first + (RAGGED ? mine.pos : 0) + lane) * 16;
        // Running maxima of the next pair's parts.  They fix its references, ceil(max * log2e).  Usually only the part's
        // first step is looked at: the reference need not be the maximum, only near enough (see `near`).
        float ma = -INFINITY, mb = -INFINITY;
        uint32_t pa = kMinusInf2, pb = kMinusInf2;
        auto maxima = [&](const uint4& wa, const uint4& wb) {
            if constexpr (DT == FSD_BF16) {
                pa = bf16x2_max_nan(pa, bf16x2_max_nan(bf16x2_max_nan(wa.x, wa.y), bf16x2_max_nan(wa.z, wa.w)));
                pb = bf16x2_max_nan(pb, bf16x2_max_nan(bf16x2_max_nan(wb.x, wb.y), bf16x2_max_nan(wb.z, wb.w)));
            } else {
                ma = fmax_nan(ma, fmax_nan(fmax_nan(__uint_as_float(wa.x), __uint_as_float(wa.y)), fmax_nan(__uint_as_float(wa.z), __uint_as_float(wa.w))));
                mb = fmax_nan(mb, fmax_nan(fmax_nan(__uint_as_float(wb.x), __uint_as_float(wb.y)), fmax_nan(__uint_as_float(wb.z), __uint_as_float(wb.w))));
            }
        };
        // Vector v of an unaligned row's part in the slot at byte offset `o`: the draft's vector moves onto the target's
        // entries, what lies outside the rows becomes -1e30, in place.
        auto align_vector = [&](uint32_t o, uint32_t meta, int v) {
            const uint32_t shift = meta & 255u;
            uint4 wb = ld_shared16(my_b + o + v * 512);
            if (shift != 0) wb = shifted<DT>(wb, ld_shared16(my_b + o + v * 512 + 16), shift);
            const int g = vbeg + mine.first + v * 32 + lane;
            if (g == 0 || g >= P.nvec_row - 2 || v * 32 + lane >= mine.count) {
                const int V = static_cast<int>(P.row_bytes / Logit<DT>::kBytes);
                const int k0 = v * 32 + lane < mine.count ? g * EPV - static_cast<int>(meta >> 8) / Logit<DT>::kBytes : V;
                wb = masked_vector<DT>(wb, k0, V);
                st_shared16(my_a + o + v * 512, masked_vector<DT>(ld_shared16(my_a + o + v * 512), k0, V));
            }
            __syncwarp();                            // the neighbours have read what is overwritten now
            st_shared16(my_b + o + v * 512, wb);
        };
        // the references the maxima give; none (-inf) where no finite logit was seen
        auto references = [&](float& ka, float& kb) {
            if constexpr (DT == FSD_BF16) { ma = fmax_nan(bf16_lo(pa), bf16_hi(pa)); mb = fmax_nan(bf16_lo(pb), bf16_hi(pb)); pa = kMinusInf2; pb = kMinusInf2; }
            __syncwarp();
            const float ra = warp_redux_max_nan(ma), rb = warp_redux_max_nan(mb);
            ma = -INFINITY; mb = -INFINITY;
            ka = reference(ra);
            kb = reference(rb);
        };

        // ---- first sweep of step s of the pair in the slot at byte offset `o` ----
        struct Sums { uint64_t za2, zb2, sa2, sb2; float kk; uint32_t diff; };     // packed (even, odd) partial sums
        const auto zero_sums = [] { return Sums{0, 0, 0, 0, 0.f, 0}; };
        auto first_sweep = [&](auto clamp_tag, int s, uint32_t o, uint64_t ca2, uint64_t cb2, Sums& t, float (&e)[kParkCols]) {
            constexpr bool CLAMP = decltype(clamp_tag)::value;
#pragma unroll
            for (int v = 0; v < VPS; ++v) {
                uint4 wa = ld_shared16(my_a + o + (s * VPS + v) * 512);
                uint4 wb = ld_shared16(my_b + o + (s * VPS + v) * 512);
                if constexpr (CLAMP && DIV == FSD_DIV_JS && DT == FSD_BF16) {
                    // -inf becomes -1e30: 2^y = 0 and 0 * y = 0 stay finite (NaN passes through)
                    wa.x = bf16x2_max_nan(wa.x, kClamp2); wa.y = bf16x2_max_nan(wa.y, kClamp2);
                    wa.z = bf16x2_max_nan(wa.z, kClamp2); wa.w = bf16x2_max_nan(wa.w, kClamp2);
                    wb.x = bf16x2_max_nan(wb.x, kClamp2); wb.y = bf16x2_max_nan(wb.y, kClamp2);
                    wb.z = bf16x2_max_nan(wb.z, kClamp2); wb.w = bf16x2_max_nan(wb.w, kClamp2);
                }
                if constexpr (DIV != FSD_DIV_TV) t.diff |= (wa.x ^ wb.x) | (wa.y ^ wb.y) | (wa.z ^ wb.z) | (wa.w ^ wb.w);
                float xa[EPV], xb[EPV];
                unpack_vec<DT>(wa, xa);
                unpack_vec<DT>(wb, xb);
#pragma unroll
                for (int j = 0; j < EPV; j += 2) {
                    float a0 = xa[j], a1 = xa[j + 1], b0 = xb[j], b1 = xb[j + 1];
                    if constexpr (CLAMP && DIV == FSD_DIV_JS && DT == FSD_F32) {
                        a0 = fmax_nan(a0, kClamp); a1 = fmax_nan(a1, kClamp); b0 = fmax_nan(b0, kClamp); b1 = fmax_nan(b1, kClamp);
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
        };

        float ka = -INFINITY, kb = -INFINITY;        // references of pair n
        int slot = 0;
        uint32_t so = 0;                             // its slot, and the slot's byte offset
        uint32_t phase = 0;                          // of its slot
        bool clamp = false;                          // this warp has met a -inf: the entropy sums (JS) take clamped logits
        const auto look_at_all = [&](uint32_t o, float& ra, float& rb) {
#pragma unroll 1
            for (int v = 0; v < steps * VPS; ++v) maxima(ld_shared16(my_a + o + v * 512), ld_shared16(my_b + o + v * 512));
            references(ra, rb);
        };
        // A pair's part, in slot `s` at byte offset `o`: aligned (an unaligned row's), its first step looked at for the
        // references.  Done for the next pair at the end of a round, so that two slots suffice.
        auto look = [&](int s, uint32_t o, float& ra, float& rb) {
            if constexpr (RAGGED) {
                const uint32_t meta = sh.meta[s];
#pragma unroll 1
                for (int v = 0; v < steps * VPS; ++v) align_vector(o, meta, v);
                __syncwarp();
            }
            if (steps > 0) {
#pragma unroll
                for (int v = 0; v < VPS; ++v) maxima(ld_shared16(my_a + o + v * 512), ld_shared16(my_b + o + v * 512));
            }
            references(ra, rb);
            if (steps > 1 && (ra == -INFINITY || rb == -INFINITY)) look_at_all(o, ra, rb);
        };
        // Both sweeps of a round, step by step.  FULL: a pair in both (this one's first sweep, the second sweep of n - 2), so
        // that a step is one run of straight-line code whose two strands cover one another's latencies; otherwise (the first
        // and last rounds) each strand is looked at.
        auto sweeps = [&](auto full_tag, auto clamp_tag, const int n, const bool first, const float ia, const float ib, Sums& t, uint64_t& x2) {
            constexpr bool FULL = decltype(full_tag)::value;
            const bool live = FULL || first;
            [[maybe_unused]] const bool old = FULL || n >= 2;
            {
                const float ca = ka == -INFINITY ? 0.f : -ka, cb = kb == -INFINITY ? 0.f : -kb;
                const uint64_t ca2 = pack2(ca, ca), cb2 = pack2(cb, cb);
                const uint64_t ia2 = pack2(ia, ia), ib2 = pack2(ib, ib);
                // s = p + q + 1e-37 keeps lg2 finite where both terms vanish; the shift is below one ulp of any s that matters
                const uint64_t tiny2 = pack2(1e-37f, 1e-37f);
                __syncwarp();                        // converged from here to the fold
                [[maybe_unused]] const uint32_t tslot = taddr + static_cast<uint32_t>((n & 1) * (kMaxSteps * kParkCols));
#pragma unroll
                for (int s = 0; s < S::kSteps; ++s) {
                    if (s < steps) {
                        [[maybe_unused]] float eo[kParkCols], e[kParkCols];
                        if constexpr (kSecondSweep) {
                            if (old) tmem_ld16(tslot + s * kParkCols, eo);
                        }
                        if (live) first_sweep(clamp_tag, s, so, ca2, cb2, t, e);
                        if constexpr (kSecondSweep) {
                            if (old) tmem_wait_ld();
                            if (live) {
                                FSD_CHECK(&P.flags->debug, (s + 1) * kParkCols <= 64, kChkTmem);
                                tmem_st16(tslot + s * kParkCols, e);
                            }
                            if (old) {
#pragma unroll
                                for (int j = 0; j < kStepEntries; j += 2) {
                                    const uint64_t ea2 = pack2(eo[j], eo[j + 1]), eb2 = pack2(eo[kStepEntries + j], eo[kStepEntries + j + 1]);
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
                        }
                    }
                }
            }
        };

        if (R > 0) {
            dead = !warp_wait(&sh.full[0], 0, P);
            if (!dead) look(0, 0, ka, kb);
        }
#pragma unroll 1
        for (int n = 0; n < n_end && !dead; ++n) {
            const bool live = n < R;
            // ---- the totals of pair n - 2 ----
            float ia = 0.f, ib = 0.f;
            if (n >= 2) {
                if (!warp_wait(&sh.totals[n & 1], ((n - 2) >> 1) & 1, P)) { dead = true; break; }
                if constexpr (kSecondSweep) {
                    const float4 t = sh.tot[n & 1];
                    ia = pow2_ref(ka2, t.x) * t.y;
                    ib = pow2_ref(kb2, t.z) * t.w;
                }
            }
            Sums t = zero_sums();
            uint64_t x2 = 0;
            const bool full = n >= 2 && live;
            if (full && (DIV != FSD_DIV_JS || !clamp)) {
                sweeps(std::true_type{}, std::false_type{}, n, true, ia, ib, t, x2);
            } else if (full) {
                sweeps(std::true_type{}, std::true_type{}, n, true, ia, ib, t, x2);
            } else {
                sweeps(std::false_type{}, std::true_type{}, n, live, ia, ib, t, x2);
            }
            // Were the references near enough (see kNearZ)?  If not, the first sweep is done over with exact maxima.  Has a
            // -inf spoilt the entropy sums (-inf * 0)?  Then it is done over with clamped logits, and clamped at once from now on.
            if (live) {
                const float z = sum2(t.za2) + sum2(t.zb2);
                bool near = z < kNearZ;
                if constexpr (DIV == FSD_DIV_JS) near = near && fabsf(sum2(t.sa2)) + fabsf(sum2(t.sb2)) < 1.0e15f;
                if (__any_sync(0xffffffffu, !near)) {
                    if (DIV != FSD_DIV_JS || __any_sync(0xffffffffu, !(z < kNearZ))) look_at_all(so, ka, kb); else clamp = true;
                    const float ca = ka == -INFINITY ? 0.f : -ka, cb = kb == -INFINITY ? 0.f : -kb;
                    t = zero_sums();
                    __syncwarp();
                    if constexpr (kSecondSweep) tmem_wait_st();      // the quick form's values go to the same columns: they have to be there first
#pragma unroll 1
                    for (int s = 0; s < steps; ++s) {
                        float e[kParkCols];
                        first_sweep(std::true_type{}, s, so, pack2(ca, ca), pack2(cb, cb), t, e);
                        if constexpr (kSecondSweep) tmem_st16(taddr + static_cast<uint32_t>((n & 1) * (kMaxSteps * kParkCols) + s * kParkCols), e);
                    }
                }
            }
            // ---- fold over the lanes: sums by halving, the second-sweep sum joins where the four have become one ----
            {
                const float v0 = sum2(t.za2), v1 = sum2(t.zb2), v2 = DIV == FSD_DIV_KL ? t.kk : sum2(t.sa2), v3 = sum2(t.sb2);
                const bool hi = (lane & 16) != 0, up = (lane & 8) != 0;
                float k0 = (hi ? v2 : v0) + __shfl_xor_sync(0xffffffffu, hi ? v0 : v2, 16);
                float k1 = (hi ? v3 : v1) + __shfl_xor_sync(0xffffffffu, hi ? v1 : v3, 16);
                float k = (up ? k1 : k0) + __shfl_xor_sync(0xffffffffu, up ? k0 : k1, 8);
                if constexpr (kSecondSweep) {
                    float x = sum2(x2);
                    x += __shfl_xor_sync(0xffffffffu, x, 16);
                    x += __shfl_xor_sync(0xffffffffu, x, 8);
                    const bool odd = (lane & 4) != 0;                    // from here on, these lanes carry x
                    k = (odd ? x : k) + __shfl_xor_sync(0xffffffffu, odd ? k : x, 4);
                    k += __shfl_xor_sync(0xffffffffu, k, 2);
                    k += __shfl_xor_sync(0xffffffffu, k, 1);
                } else {
#pragma unroll
                    for (int m = 4; m > 0; m >>= 1) k += __shfl_xor_sync(0xffffffffu, k, m);
                }
                const bool differ = DIV == FSD_DIV_TV || __any_sync(0xffffffffu, t.diff != 0);
                WarpPost& w = sh.post[n & 1][warp];
                if ((lane & 7) == 0) w.z[lane >> 3] = k;
                if (lane == 4) *reinterpret_cast<float4*>(&w.ka) = make_float4(ka, kb, k, __uint_as_float(differ ? 1u : 0u));
                __syncwarp();                        // (every lane is through with the slot, too: it takes the pair after the next two)
                if (lane == 0) mbar_arrive(&sh.posted[n & 1]);
            }
            ka2 = ka1; kb2 = kb1; ka1 = ka; kb1 = kb;
            if constexpr (kSecondSweep) {
                __syncwarp();                        // tensor-memory instructions want the warp converged
                tmem_wait_st();
            }
            // ---- the next pair: its slot, its references ----
            if (++slot == P.ring) { slot = 0; so = 0; phase ^= 1; } else { so += P.slot_bytes; }
            ka = -INFINITY; kb = -INFINITY;
            if (n + 1 < R) {
                if (!warp_wait(&sh.full[slot], phase, P)) { dead = true; break; }
                look(slot, so, ka, kb);
            }
        }
    } else {
        // ---- helper warp: fold the warps' posts, exchange with the group, hand out the totals ----
        // where this group exchanges its statistics: [parity][rank] messages
        GroupMsg* const xg = P.exchange + static_cast<size_t>(group_id < n_groups ? group_id : 0) * 2 * C;
        int item = group_id;
        uint32_t help_after = P.help_after;
        int n = 0;
        const uint64_t number = call_number(P.flags, P.nonce);     // (asked for in front of the block's barrier: small calls +0.3 us)
#pragma unroll 1
        for (; n < n_end; ++n, item += n_groups) {
            const int par = n & 1;
            const uint32_t tag = static_cast<uint32_t>(number) + static_cast<uint32_t>(n), high = static_cast<uint32_t>(number >> 32);   // what this round's messages carry
            bool bad = false;
            if (n < R && rank == 0 && P.parent != nullptr) {
                const int pr = __ldg(P.parent + item);
                bad = pr < -1 || pr >= item % P.G;
            }
            if (!warp_wait(&sh.posted[par], (n >> 1) & 1, P)) break;
            FSD_CHECK(&P.flags->debug, n >= R || (item >= 0 && item < P.n_items && rank < kMaxGroupSize), kChkRecord);
            // What the compute warps wait for comes first: Z and the references.  Lanes 0..15 take the
            // target row's of one warp each, lanes 16..31 the draft row's.
            __syncwarp();
            const WarpPost& w = sh.post[par][lane & 15];
            const bool b_side = lane >= 16;
            const float wk = b_side ? w.kb : w.ka, wz = b_side ? w.z[1] : w.z[0];
            float s = b_side ? w.z[3] : w.z[2], x = b_side ? 0.f : w.x;         // (read now: the slot is free once the totals are out)
            const bool differ = __any_sync(0xffffffffu, w.diff != 0);
            float Ka = -INFINITY, Kb = -INFINITY, f = 0.f;
            if (n < R) {
                const float z = fold_z(wk, wz, b_side, Ka, Kb, f);
                if constexpr (kSecondSweep) {
                    // lanes 0 and 16 each store one 16-byte unit of this block's message; every unit ends in the round's tag
                    if ((lane & 15) == 0 && !(n == 0 && group_id == 0 && rank == P.silent_rank))
                        st_unit(&xg[par * C + rank].u[b_side], b_side ? Kb : Ka, z, __uint_as_float(high), tag);
                    // (while it travels: the slot all warps are through with takes the pair after the next two)
                    __syncwarp();
                    issue_slices();
                    // group totals for the second sweep (float is enough there): lane r fetches the target
                    // row's unit of block r, lane 16 + r the draft row's; a second fetch where C > 16
                    const int r0 = lane & 15;
                    float tk0 = -INFINITY, tz0 = 0.f, tk1 = -INFINITY, tz1 = 0.f;
                    bool got = false;
                    uint32_t miss0 = 0, miss1 = 0;    // messages to be computed here
#pragma unroll 1
                    for (uint32_t i = 0; i < P.poll_limit; ++i) {
                        bool ok0 = true, ok1 = true;
                        uint4 u0 = make_uint4(0, 0, ~high, 0), u1 = u0;
                        if (r0 < C) {
                            u0 = ld_unit(&xg[par * C + r0].u[b_side]);
                            ok0 = u0.w == tag && u0.z == high;
                            tk0 = __uint_as_float(u0.x); tz0 = __uint_as_float(u0.y);
                        }
                        if (r0 + 16 < C) {
                            u1 = ld_unit(&xg[par * C + r0 + 16].u[b_side]);
                            ok1 = u1.w == tag && u1.z == high;
                            tk1 = __uint_as_float(u1.x); tz1 = __uint_as_float(u1.y);
                        }
                        if (__all_sync(0xffffffffu, ok0 && ok1)) { got = true; break; }
                        // A block of the group that has sent nothing for this long may not be running at all: nothing makes the
                        // blocks of this launch resident together, another stream's kernels may hold SMs.  Its message is computed
                        // here then, so no block ever needs another one in order to finish.  (From then on the others' rounds
                        // and this block's are apart: it does not wait as long again, and the late block finds the others' messages
                        // overwritten by those of later rounds, and does not wait at all.  Waiting is cheap and computing is not, 5 us
                        // and more a slice, so a block waits for about as long as it may take to catch up.)
                        const auto overwritten = [&](const uint4& u) { return u.z == high && u.w - tag - 1u < static_cast<uint32_t>(R); };
                        if (i >= help_after || __any_sync(0xffffffffu, overwritten(u0) || overwritten(u1))) {
                            if (i >= help_after) help_after = 32;
                            miss0 = __ballot_sync(0xffffffffu, !ok0); miss1 = __ballot_sync(0xffffffffu, !ok1);
                            break;
                        }
                        // has anybody's wait run out?  (then nothing this warp waits for is certain to come)
                        if ((i & 255u) == 255u && __any_sync(0xffffffffu, timed_out(P.flags, number))) break;
                    }
                    if (!got) {
                        if ((miss0 | miss1) == 0) {
                            if (lane == 0) raise_flag(P.flags, number);
                            break;
                        }
                        const float4 m = missing_messages<DT, RAGGED>(P, item, miss0, miss1, make_float4(tk0, tz0, tk1, tz1));
                        tk0 = m.x; tz0 = m.y; tk1 = m.z; tz1 = m.w;
                    }
                    const float tk = fmax_nan(tk0, tk1);
                    const float Ga = warp_redux_max_nan(b_side ? -INFINITY : tk), Gb = warp_redux_max_nan(b_side ? tk : -INFINITY);
                    const float G = b_side ? Gb : Ga;
                    float tz = tz0 * pow2_ref(tk0, G);
                    if (C > 16) tz = fmaf(tz1, pow2_ref(tk1, G), tz);
#pragma unroll
                    for (int m = 8; m > 0; m >>= 1) tz += __shfl_xor_sync(0xffffffffu, tz, m);
                    // 1 / Z to the last bit or so; 0 where the row is not a valid distribution (NaN included)
                    float iz = 0.f;
                    if (tz > 1.0e-30f && tz < 1.0e30f) { const float r = rcp(tz); iz = fmaf(r, fmaf(-tz, r, 1.f), r); }
                    if ((lane & 15) == 0) *reinterpret_cast<float2*>(reinterpret_cast<float*>(&sh.tot[par]) + 2 * b_side) = make_float2(G, iz);
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&sh.totals[par]);
                }
                // ---- what only the record needs ----
                const float d = wk == -INFINITY ? 0.f : wk - (b_side ? Kb : Ka);
                if constexpr (DIV == FSD_DIV_KL) {
                    const float d_b = __shfl_down_sync(0xffffffffu, d, 16);
                    s = b_side ? 0.f : scale_kl(f, fmaf(d - d_b, wz, s));
                } else {
                    s = f * fmaf(d, wz, s);
                }
#pragma unroll
                for (int m = 8; m > 0; m >>= 1) s += __shfl_xor_sync(0xffffffffu, s, m);
                const float z_b = __shfl_down_sync(0xffffffffu, z, 16), s_b = __shfl_down_sync(0xffffffffu, s, 16);
                if (lane == 0) {
                    PairRecord* r = P.records + item;
                    Stats c;
                    c.ka = Ka; c.kb = Kb; c.za = z; c.zb = z_b; c.s0 = s; c.sb = s_b; c.x = 0.f; c.diff = differ ? 1u : 0u;
                    r->part[rank] = c;
                    if (rank == 0) { r->ncta = static_cast<uint32_t>(C); r->state = bad ? kRecordBadTree : kRecordStats; }
                    if (n == 0 && blockIdx.x == 0) P.flags->number = number;
                }
            }
            if constexpr (kSecondSweep) {
                if (n >= 2) {
#pragma unroll
                    for (int m = 8; m > 0; m >>= 1) x += __shfl_xor_sync(0xffffffffu, x, m);
                    if (lane == 0) P.records[item - 2 * n_groups].x[rank] = x;
                }
            } else {
                __syncwarp();
                if (lane == 0) mbar_arrive(&sh.totals[par]);
                issue_slices();
            }
        }
        if (blockIdx.x == 0 && lane == 0) {
            if (n == 0) P.flags->number = number;     // (a wait of the first round ran out)
            if (P.raise) raise_flag(P.flags, number);
        }
        // Every copy started has landed before the block may leave: normally the rounds consumed them all;
        // after a wait that ran out some may still be on their way (a copy, once started, always completes).
        for (int k = in > P.ring ? in - P.ring : 0; k < in; ++k) {
#pragma unroll 1
            for (uint32_t i = 0; i < kSpinLimit; ++i)
                if (__all_sync(0xffffffffu, mbar_try_wait(&sh.full[k % P.ring], (k / P.ring) & 1))) break;
        }
    }

    if constexpr (kSecondSweep) {
        // ---- release tensor memory ----
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        __syncwarp();
        if (warp == 0)
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(sh.tmem_base), "n"(kTmemCols) : "memory");
    }
}

}  // namespace fsd
