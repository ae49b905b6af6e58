// Pieces shared by the decode kernels: launch arguments, mbarrier / bulk-copy PTX wrappers, the
// division of the step line among CTAs, the producer warp, and the merge of partial softmax states.
//
// Execution shape (both kernels): a persistent grid of one CTA per SM.  Every (sequence, KV head) unit
// is cut into steps of `pps` pages (16 or 32 tokens); the steps of all units form one line that is
// divided among the CTAs.  Inside a CTA one producer warp streams pages into a shared-memory ring with
// bulk asynchronous copies that signal mbarriers; NW consumer warps each take a contiguous run of steps and keep
// an online-softmax state (running max m in the log2 domain, running sum l, unnormalised output) per unit.
// At the end of an epoch the warps' states are merged by log-sum-exp; if several CTAs share a unit each
// writes a partial and the last to arrive (an atomic ticket, no waiting) merges them.
#pragma once

#include "spark_common.cuh"

namespace spark {

constexpr int kMaxSlots = 32;
constexpr unsigned long long kWaitLimitNs = 1000000000ull;   // every device-side wait gives up after one second
constexpr unsigned kClockEvery = 256;                        // polls between two looks at the clock
constexpr unsigned kFull = 0xffffffffu;
constexpr int kRec = kHeadDim + 4;           // floats per head record: 128 outputs, running max, running sum, pad
constexpr int kMaxCap = 8;                    // units per epoch, at most (see Epoch)
constexpr float kLn2 = 0.6931471805599453f;

// Division of 0 <= x < 2^31 by a divisor the host knows: a multiply and a correction (an integer division is some
// 130 cycles, and seven of them stood in a row between the plan and a CTA's first page copy).
struct FastDiv {
    unsigned d, m;
    static FastDiv of(unsigned d) { FastDiv f; f.d = d; f.m = d > 1 ? static_cast<unsigned>((1ull << 32) / d) : 0xffffffffu; return f; }
    __device__ __forceinline__ int div(int x) const
    {
        unsigned q = __umulhi(static_cast<unsigned>(x), m);          // the quotient or one less
        if (static_cast<unsigned>(x) - q * d >= d) ++q;
        return static_cast<int>(q);
    }
};

// Units per epoch that a launch may use, and what each number leaves for the ring.  An epoch's units take shared memory
// (operand tables, records) from the ring, so the number is chosen with the plan, from the lengths: few where CTAs' runs are
// long and a unit boundary (3 us) is a small part of them, many where a CTA meets many units, one where it meets one.
// (Chosen from the cache's capacity instead, eight sequences of 150..4000 tokens took 19.6 us in a cache for 4016 tokens,
// 27.0 in one for 16 K and 35.6 in one for 128 K; 32 x 2048 41.6 and, in a cache for 32 K, 49.3.)
struct EpochCaps {
    unsigned long long slots;                // ring slots with 1 .. kMaxCap units (a byte each)
    int tail_base, tail_step;                // bytes of the record area with one unit, and more for each further one
    int shortest, middle, even, longest;     // units for runs of up to kRunShort, kRunMiddle, kRunLong steps and above
    int by_units;                            // CUDA-core kernel: by the units that a CTA may meet (see choose_cap)
};
constexpr int kRunShort = 160, kRunMiddle = 512, kRunLong = 1024;

struct DecodeArgs {
    const void* q;
    const unsigned char* pages;
    const int32_t* block_table;
    int max_blocks;
    const int32_t* lens;
    const float* qnorm;
    float* out;
    float* lse;
    const float* other_out;                  // attention over further tokens of the same sequences (a dense tail), merged
    const float* other_lse;                  // into the published result; null: none
    int B, Hq, Hkv;
    int64_t n_pool_pages;
    PageLayout L;
    float scale_log2e;
    int* status;
    int* tickets;
    float* partials;
    int slot_stride;
    int pps;                                 // pages per step (= per ring slot): 1 or 2
    unsigned one;                            // 1, which the compiler does not know (see expand_nibble)
    FastDiv by_grid, by_hkv;                 // CTAs of the grid; KV heads
    int per_unit, extra;                     // aligned mode (see Plan): CTAs per unit; units with one more
    FastDiv by_q, by_q1;                     // per_unit and per_unit + 1
    EpochCaps caps;                          // units per epoch, chosen with the plan
    int slack, ragged_slack;                 // steps that the longest share may be above the even one (see Plan)
    float ragged_from;                       // unequal units in whole CTAs from this many shortest units per even share
    int whole_steps;                         // a step per consumer warp; units up to this are not split (see Plan)
    int prefix_off;                          // shared-memory offset of the steps-per-sequence prefix and the lengths
    int ring_off;                            // shared-memory offset of the ring (behind the prefix); records and tables follow it
    int late_wait;                           // the kernel before waited at its top, released after that and writes only other_out /
                                             // other_lse: wait where they are read (a successor may be released before that)
    int overlap;                             // the page stream need not wait for the kernel before (SPARK_FLAG_OVERLAP_PREVIOUS)
    unsigned seed;                           // sampled recovery: seed of the per-entry draws
    const int* page_rows;                    // ragged pages: slot rows in use per pool page (else null: whole pages)
    int q_by_value;                          // host side only: q is a HOST pointer whose bytes travel as a launch parameter
};

// largest query (bytes) that may travel as a launch parameter (kernel parameters are limited to 32764 bytes)
constexpr int kMaxQueryByValueBytes = 24 * 1024;

// control block at the start of dynamic shared memory
constexpr int kCtrlBytes = 1024;                                 // full[32], empty[32], flags, plan, epoch units
// the steps-per-sequence prefix and the lengths sit between a kernel's fixed shared-memory areas and the ring and
// are as large as the batch needs, so small batches leave their room to the ring
inline int prefix_bytes(int batch) { return ((2 * batch + 1) * 4 + 127) / 128 * 128; }

// Shared merge area: `nw + cap - 1` states of `g` heads ([record][head][kRec] floats: 128 outputs, m, l).
__host__ __device__ constexpr int merge_step(int g) { return (g * kRec * 4 + 127) / 128 * 128; }
__host__ __device__ constexpr int merge_base(int nw, int g) { return (nw * g * kRec * 4 + 127) / 128 * 128; }

// ---- PTX helpers ----------------------------------------------------------------------------------
__device__ __forceinline__ unsigned smem_u32(const void* p)
{
    return static_cast<unsigned>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, unsigned bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, unsigned parity)
{
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// Expiry test of a polling loop: looks at the nanosecond clock every kClockEvery polls (the first look
// only records the start), so a wait is bounded by wall time, not by how fast the poll happens to spin.
struct WaitClock {
    unsigned it = 0;
    unsigned long long t0 = 0;
    __device__ __forceinline__ bool expired()
    {
        if ((++it & (kClockEvery - 1)) != 0) return false;
        const unsigned long long now = global_ns();
        if (t0 == 0) { t0 = now; return false; }
        return now - t0 > kWaitLimitNs;
    }
};
// Wait with a time limit.  On expiry (or if another thread already gave up) the CTA-wide abort
// flag is set, the status word records the timeout and the caller carries on without the data; the
// kernel then finishes structurally (same barriers) and returns.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, unsigned parity, volatile int* abort_flag, int* status)
{
    WaitClock wc;
    while (!wc.expired()) {
        if (mbar_try_wait(bar, parity)) return true;
        if (*abort_flag) return false;
    }
    *abort_flag = 1;
    record_error(status, SPARK_ERR_DEVICE_TIMEOUT);
    return false;
}
// Bulk copy global -> shared that signals `bar`; `policy` is an L2 eviction policy (pages are read once
// per step, so they are streamed evict-first and leave the L2 to the small tables and the partials).
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, unsigned bytes, uint64_t* bar, uint64_t policy)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;"
        ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar)), "l"(policy)
        : "memory");
}
__device__ __forceinline__ uint64_t policy_evict_first()
{
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}
// Consumer side of a ring slot: wait until the data of revolution `round` has landed in `slot`.
// A parity wait alone cannot tell "revolution r has not been armed yet" from "revolution r is
// complete" (consumers of different revolutions of one slot are different warps), so the slot's
// revolution counter, written by the producer when it arms the barrier, is checked first.
__device__ __forceinline__ bool slot_wait(uint64_t* full, volatile int* seq, int slot, int round,
                                          volatile int* abort_flag, int* status)
{
    WaitClock wc;
    while (seq[slot] != round + 1) {
        if (wc.expired() || *abort_flag) {
            if (!*abort_flag) { *abort_flag = 1; record_error(status, SPARK_ERR_DEVICE_TIMEOUT); }
            return false;
        }
    }
    return mbar_wait(&full[slot], round & 1, abort_flag, status);
}
template <int NT> __device__ __forceinline__ void consumer_sync()
{
    asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory");
}

__device__ __forceinline__ int steps_of(int len, int pps)
{
    return ((len + kPageTokens - 1) / kPageTokens + pps - 1) / pps;
}

__device__ __forceinline__ int clamp_len(int len, int max_tokens)
{
    return len < 0 ? 0 : (len > max_tokens ? max_tokens : len);
}

// A (sequence, KV head) unit on the step line.
struct UnitRef {
    int b, h;
    int start;               // line position of its first step
    int steps;
};

// The unit that holds line position g (must be < total).
__device__ __forceinline__ UnitRef locate_unit(const int* prefix, int B, int Hkv, int g)
{
    int lo = 0, hi = B;                                   // first b' in (lo, hi] with Hkv*prefix[b'] > g
#pragma unroll 1
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (static_cast<int64_t>(Hkv) * prefix[mid] > g) hi = mid; else lo = mid;
    }
    UnitRef u;
    u.b = lo;
    u.steps = prefix[lo + 1] - prefix[lo];
    const int r = g - Hkv * prefix[lo];
    u.h = r / u.steps;
    u.start = Hkv * prefix[lo] + u.h * u.steps;
    return u;
}
// The next non-empty unit (the caller knows that there is one).
__device__ __forceinline__ void next_unit(const int* prefix, int Hkv, UnitRef& u)
{
    u.start += u.steps;
    if (++u.h < Hkv) return;
    u.h = 0;
    do { ++u.b; u.steps = prefix[u.b + 1] - prefix[u.b]; } while (u.steps == 0);
}

// A CTA works through its run of steps in EPOCHS of up to `cap` units.  Inside an epoch of N steps the
// consumer warps take CONTIGUOUS runs (N / NW steps each, the first N % NW warps one more), so a warp
// meets a unit boundary only where one falls into its own run: it then writes its state to a record, loads the
// next unit's operands and goes on, without any CTA-wide barrier.  A run cut by the unit boundaries gives at
// most NW + cap - 1 records; the part of epoch-unit e that warp w holds is record w + e.  The ring is filled in the
// order in which the warps consume: ring step n of the epoch is step n / NW of warp n % NW.
//   Why: with a barrier, a merge and a table build per unit, every unit after a CTA's first cost 3.8 us (as
//   much as 26 pages at the HBM rate).  Before -> after: append + decode of 8 sequences of 150..4000 tokens
//   40.9 -> 30.1 us, 32 sequences of 2048 tokens (256 units on 148 SMs) 46.1 -> 44.1 us, 4 of 128K 265 -> 258 us.
struct Epoch {
    int e0, e1;              // line positions
    int n_units;
    UnitRef first;
};
__device__ __forceinline__ Epoch make_epoch(const int* prefix, int Hkv, int cap, const UnitRef& first, int g, int c1)
{
    Epoch ep;
    ep.e0 = g;
    ep.first = first;
    UnitRef u = first;
    ep.n_units = 1;
    int end = u.start + u.steps;
#pragma unroll 1
    while (ep.n_units < cap && end < c1) {
        next_unit(prefix, Hkv, u);
        end += u.steps;
        ++ep.n_units;
    }
    ep.e1 = min(end, c1);
    return ep;
}
// What the merge needs to know about an epoch's units (kept in shared memory).
struct EpochUnit {
    int b, h;
    int rec0, n_rec;         // its records in the merge area
    int first_cta, n_parts;  // CTAs that hold a part of the unit
};

// How the step line is divided among the CTAs.
//   stream mode : CTA c owns steps [c*chunk, (c+1)*chunk) of the whole line; a CTA may cross unit
//                 boundaries (exact balance; used when sequences differ in length or units are many).
//   aligned mode: every unit gets whole CTAs and is split evenly among them, so no CTA crosses a unit boundary and every CTA
//                 publishes exactly once: a boundary inside a CTA's run costs it a second table and merge, and all wait for it.
//                 Equally long units: q or q+1 CTAs each.  Unequal ones: as many as keep every share at or below the smallest bound for
//                 which the grid suffices.  Taken where the longest share is at most 4 % (and, up to kShortShare steps, kSplitSlack or
//                 kRaggedSlack steps) above the even one.  us, stream mode -> aligned: 1 x 2048 tokens 14.0 -> 9.6, 1 x 4096 15.0 -> 11.0,
//                 2 x 2048 12.6 -> 10.9, 8 x 700 13.9 -> 12.1.  With the slack at any share 4 x 10000 29.2 -> 29.7, 4 x 4000..20000 33.4 -> 34.3.
//                 Unequal units (ragged_from): with up to six heads a group from two shortest units per even share, where runs of the
//                 line would meet several units; with seven or eight, whose tables and merges take longest, always; with one or two
//                 never.  8 / 8 and 16 / 8 heads: 8 x 150..4000 17.1 -> 18.6 and 17.4 -> 18.9, 4 x 100..6000 15.1 -> 15.7 and 15.1 -> 15.8;
//                 32 / 8: 8 x 150..4000 19.3 -> 18.7, 6 x 60..4000 23.3 -> 16.3, 6 x 300..6000 20.1 -> 19.4, but below two 5 x 700..6000 17.1 ->
//                 18.0, 4 x 2000..9000 19.6 -> 20.3; 40 / 8: 8 x 500..2500 16.2 -> 17.3; 28 / 4: 2 x 600..6000 14.0 -> 13.1, 12 x 300..3000 18.6 -> 16.1;
//                 64 / 8: 2 x 600..6000 18.6 -> 14.6.  A slack of 10 or 30 steps in place of 20 gives the same within 0.1 in 26 sizes of shares
//                 of 5 to 110 steps, but for 8 x 150..4000 with 32 / 8 heads, where one of 10 does not find a division (19.8).
//                 kShortShare 50 / 100 / 200, 31 sizes with shares of 30 to 260 steps: 4 x 4000 16.7 / 17.2 / 17.1, 4 x 100..8000 21.4 / 17.9 / 17.8,
//                 8 x 1000..12000 with 28 / 4 heads 26.4 / 24.0 / 24.0, 8 x 200..7000 27.5 / 27.4 / 27.8, 11 x 6000 with 16 / 4 24.7 / 24.7 / 25.3,
//                 4 x 300..16000 27.7 / 27.0 / 25.6, 4 x 1000..14000 with 64 / 8 29.7 / 29.7 / 26.6; the others within 0.5.
//   whole units : CTA u owns unit u.  For units of at most a step per warp, where a split saves nothing and adds a
//                 partial, a ticket and the last arriver's merge (240 tokens: 8.4 us against 9.1; with two steps per warp
//                 9.7 against 9.2), and for units of up to three steps per warp where they fill most of the grid anyway
//                 (16 sequences of 60..700 tokens, 128 units: 12.7 us against 18.7).
constexpr int kSplitSlack = 10, kRaggedSlack = 20, kShortShare = 100;
struct Plan {
    int total;        // steps on the line
    int chunk;        // stream mode: steps per CTA
    int aligned;      // 0: stream, 1: aligned mode, 2: whole units
    int first_cta;    // aligned: first CTA of this CTA's unit
    int share;        // aligned: steps per CTA of the unit
    int cap, nslots;  // units per epoch and the ring slots that they leave
    int merge_off, tab_off;      // shared-memory offsets of the records and of the operand tables (behind the ring)
};

// A CTA's run of steps [c0, c1) on the line and the unit of its first step.
struct CtaRun {
    int c0, c1;
    UnitRef first;           // meaningful when c0 < c1
};

struct Ctrl {
    uint64_t* full;
    uint64_t* empty;
    volatile int* abort_flag;
    volatile int* seq;        // [32] revolution + 1 for which each slot was last armed
    Plan* plan;
    volatile int* epoch;      // [2] the epoch's end and its number of units
    EpochUnit* units;         // [kMaxCap]
    CtaRun* run;
    int* prefix;              // [B + 1] steps before each sequence (of one KV head)
    int* lens;                // [B] clamped lengths
};

__device__ __forceinline__ Ctrl make_ctrl(unsigned char* smem, int prefix_off, int B)
{
    Ctrl c;
    c.full = reinterpret_cast<uint64_t*>(smem);
    c.empty = c.full + kMaxSlots;
    c.abort_flag = reinterpret_cast<volatile int*>(smem + 512);
    c.plan = reinterpret_cast<Plan*>(smem + 528);
    c.epoch = reinterpret_cast<volatile int*>(smem + 608);
    static_assert(528 + sizeof(Plan) <= 608, "control block");
    c.seq = reinterpret_cast<volatile int*>(smem + 640);
    c.units = reinterpret_cast<EpochUnit*>(smem + 768);
    c.run = reinterpret_cast<CtaRun*>(smem + 960);
    static_assert(768 + kMaxCap * sizeof(EpochUnit) <= 960 && 960 + sizeof(CtaRun) <= kCtrlBytes, "control block");
    c.prefix = reinterpret_cast<int*>(smem + prefix_off);
    c.lens = c.prefix + B + 1;
    return c;
}

// Start of the kernel.  The PRODUCER warp alone reads packed_lens, builds the steps-per-sequence prefix and
// the plan, initialises the ring barriers, and then arrives (without waiting) on hardware barrier 2; it
// goes straight on to its first page copies.  The consumer warps wait on barrier 2 for the plan.  So the
// chain from launch to the first bytes in flight is: packed_lens (one global round trip) -> plan -> page
// ids -> bulk copies, with no CTA-wide barrier in between.
//
// All threads first ask the L2 to fetch the block table (when there is one): the producer's page-id
// loads then find their lines on the way instead of starting a second cold DRAM round trip behind
// packed_lens.  (A hint: it may run before the kernel ahead has completed.)
constexpr int kPlanBarrier = 2;
constexpr int64_t kTablePrefetchMax = 8 << 20;             // bytes of block table asked for at most

__device__ __forceinline__ void prefetch_block_table(const DecodeArgs& A, int tid, int n_threads)
{
    if (!A.block_table) return;
    int64_t bytes = static_cast<int64_t>(A.B) * A.Hkv * A.max_blocks * 4;
    if (bytes > kTablePrefetchMax) bytes = kTablePrefetchMax;
    const char* base = reinterpret_cast<const char*>(A.block_table);
#pragma unroll 1
    for (int64_t o = (static_cast<int64_t>(blockIdx.x) * n_threads + tid) * 128; o < bytes;
         o += static_cast<int64_t>(gridDim.x) * n_threads * 128)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(base + o));
}

// Units per epoch for this plan, never more than a CTA can meet.  `least` = steps of the shortest non-empty sequence.
//   Tensor-core kernel: by the length of a CTA's run.  us with 1, 2, 3, 5, 6, 8 units: runs of 100 steps (8 x 150..4000
//   tokens) 35, 27, 22.5, 22.6, 19.6, 19.6; 221 (32 x 2048, three met) 49.3, 45.3, 41.0; 344 (12 x 1000..16000) 77, 66, 64, 64,
//   62, 63; 459 (32 x 1000..16000, 28 / 4 heads, T = 38) 100, 90, 85, 83, 84, 90; 919 (32 x 1000..16000) 171, 157, 151, 151, 148,
//   151; 1900 steps (16 x 8K..128K, seven heads per group) 338 with one and 26 slots, 343 with two and 24.
//   CUDA-core kernel: it is bound by its warps, and a warp needs a slot: eight at most, of which the tables of a second unit
//   take one.  So a CTA that meets two units keeps one per epoch where slots are short (16 x 2000 tokens, fp32, T = 89: 112 us
//   with seven slots, 121 with six), and one that may meet more takes them together (8 x 150..4000 tokens: 79 us with one, 66
//   with three to six).
__device__ __forceinline__ int choose_cap(const EpochCaps& E, const Plan& pl, int least)
{
    if (pl.aligned) return 1;
    const int meets = static_cast<int>(__fdividef(static_cast<float>(pl.chunk), static_cast<float>(least))) + 2;       // at most
    if (E.by_units) return meets <= 2 ? E.even : min(meets, E.shortest);
    return min(meets, pl.chunk <= kRunShort ? E.shortest : (pl.chunk <= kRunMiddle ? E.middle : (pl.chunk <= kRunLong ? E.even : E.longest)));
}

// ceil(x / c) for 0 <= x < 2^22 and a quotient below 2^21; rc = 1 / c
__device__ __forceinline__ int ceil_div(int x, int c, float rc)
{
    int q = static_cast<int>(static_cast<float>(x + c - 1) * rc);
    const int r = x + c - 1 - q * c;
    q += r >= c ? 1 : (r < 0 ? -1 : 0);
    return q;
}
__device__ __forceinline__ int ceil_div(int x, int c) { return ceil_div(x, c, __fdividef(1.f, static_cast<float>(c))); }

// Unequal units, whole CTAs: the smallest of 32 bounds on a CTA's share, between the even share and the longest one that is
// worth it, for which the grid suffices, and this CTA's unit and its share of it under that bound; false: none.  The producer
// warp: a lane holds a sequence to see whether any bound does, then tries one, then holds a sequence again to find the CTA's.
// (Out of line: the start of a step runs cold, and most divisions do without.  The result is left in the control block.)
static __device__ __noinline__ bool ragged_run(const int* prefix, int B, int Hkv, int even, int extra, int cta, int nct, int lane, CtaRun* run, Plan* pl)
{
    int ctas = 0;
#pragma unroll 1
    for (int b = lane; b < B; b += 32) ctas += ceil_div(prefix[b + 1] - prefix[b], even + extra);
    if (__reduce_add_sync(kFull, ctas) * Hkv > nct) return false;
    const int tried = even + (extra * lane + 30) / 31;
    const float rc = __fdividef(1.f, static_cast<float>(tried));
    ctas = 0;
#pragma unroll 4
    for (int b = 0; b < B; ++b) ctas += ceil_div(prefix[b + 1] - prefix[b], tried, rc);
    const int bound = __shfl_sync(kFull, tried, __ffs(__ballot_sync(kFull, ctas * Hkv <= nct)) - 1);
    CtaRun r;
    r.c0 = r.c1 = r.first.b = r.first.h = r.first.start = r.first.steps = 0;       // (a CTA too many has nothing to do)
    int first_cta = 0, share = 1;
    int before = 0;                                        // CTAs of the sequences before
#pragma unroll 1
    for (int b0 = 0; b0 < B; b0 += 32) {
        const int b = b0 + lane, st = b < B ? prefix[b + 1] - prefix[b] : 0, n = ceil_div(st, bound), x = n * Hkv;
        int inc = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int up = __shfl_up_sync(kFull, inc, o);
            if (lane >= o) inc += up;
        }
        const unsigned past = __ballot_sync(kFull, before + inc > cta);
        if (past) {
            const int src = __ffs(past) - 1, n_u = __shfl_sync(kFull, n, src), steps = __shfl_sync(kFull, st, src);
            const int place = cta - before - __shfl_sync(kFull, inc - x, src);
            const int h = ceil_div(place + 1, n_u) - 1, k = place - h * n_u;
            share = ceil_div(steps, n_u);
            first_cta = cta - k;
            r.first.b = b0 + src; r.first.h = h; r.first.steps = steps;
            r.first.start = Hkv * prefix[b0 + src] + h * steps;
            r.c0 = r.first.start + min(steps, k * share);
            r.c1 = r.first.start + min(steps, (k + 1) * share);
            break;
        }
        before += __shfl_sync(kFull, inc, 31);
    }
    if (lane == 0) { *run = r; pl->first_cta = first_cta; pl->share = share; }
    __syncwarp();
    return true;
}

__device__ __forceinline__ CtaRun producer_prologue(const DecodeArgs& A, const Ctrl& C, int lane, int n_threads, Plan& pl)
{
    const int max_tokens = A.max_blocks * kPageTokens;
    mbar_init(&C.full[lane], 1);                           // (all kMaxSlots = 32; the plan says how many are used)
    mbar_init(&C.empty[lane], 1);
    C.seq[lane] = 0;
    if (lane == 0) { *C.abort_flag = 0; C.prefix[0] = 0; }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    // what does not depend on the lengths, before the wait: this CTA's unit in whole-unit mode (wb, wh), and its unit, its
    // place k among the unit's n CTAs in aligned mode
    const int cta = static_cast<int>(blockIdx.x), nct = static_cast<int>(gridDim.x), units = A.B * A.Hkv;
    const int wb = A.by_hkv.div(cta), wh = cta - wb * A.Hkv;
    int u = 0, k = 0, n = 1, ub = 0;
    if (A.per_unit > 0) {
        const int big = A.extra * (A.per_unit + 1);                 // CTAs that belong to units with q + 1 CTAs
        if (cta < big) { u = A.by_q1.div(cta); k = cta - u * (A.per_unit + 1); n = A.per_unit + 1; }
        else { const int v = A.by_q.div(cta - big); u = A.extra + v; k = cta - big - v * A.per_unit; n = A.per_unit; }
        ub = A.by_hkv.div(u);
    }
    if (!A.overlap) grid_wait();                           // with the flag the page stream does not depend on the kernel before
    if (!A.overlap || A.late_wait) grid_release();         // (otherwise the consumers release, see consumer_wait_previous)
    int running = 0, smin = 0x7fffffff, smax = 0, least = 0x7fffffff;
#pragma unroll 1
    for (int b0 = 0; b0 < A.B; b0 += 32) {
        const int b = b0 + lane;
        int st = 0;
        if (b < A.B) {
            const int len = A.lens[b];
            if (len < 0 || len > max_tokens) record_error(A.status, SPARK_ERR_DEVICE_BOUNDS);
            C.lens[b] = clamp_len(len, max_tokens);
            st = steps_of(clamp_len(len, max_tokens), A.pps);
            smin = min(smin, st);
            smax = max(smax, st);
            if (st > 0) least = min(least, st);
        }
        int inc = st;
        if (A.B > 1)
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int x = __shfl_up_sync(kFull, inc, o);
                if (lane >= o) inc += x;
            }
        if (b < A.B) C.prefix[b + 1] = running + inc;
        running += __shfl_sync(kFull, inc, A.B > 1 ? 31 : 0);
    }
    smin = __reduce_min_sync(kFull, smin);
    smax = __reduce_max_sync(kFull, smax);
    least = __reduce_min_sync(kFull, least);
    __syncwarp();                                          // the prefix is written
    pl.total = A.Hkv * running;
    pl.chunk = A.by_grid.div(pl.total + nct - 1);
    pl.aligned = 0; pl.first_cta = 0; pl.share = 1;
    // ragged units in whole CTAs: a unit wastes half a share on average, so where a third each would not fit it is not tried
    const int extra = pl.chunk / 25 + (pl.chunk <= kShortShare ? A.ragged_slack : 0);
    CtaRun run;
    run.first.b = run.first.h = run.first.start = run.first.steps = 0;
    if (units <= nct && (smax <= A.whole_steps || (2 * units > nct && smax <= 3 * A.whole_steps))) {
        pl.aligned = 2;
        run.first.b = wb; run.first.h = wh;
        run.first.steps = wb < A.B ? C.prefix[wb + 1] - C.prefix[wb] : 0;
        run.first.start = wb < A.B ? A.Hkv * C.prefix[wb] + wh * run.first.steps : 0;
        run.c0 = run.first.start;
        run.c1 = run.c0 + run.first.steps;
    } else if (smin == smax && smax > 0 && A.per_unit >= 1 && A.by_q.div(smax + A.per_unit - 1) * 25 <= pl.chunk * 26 + (pl.chunk <= kShortShare ? A.slack * 25 : 0)) {
        pl.aligned = 1;
        const int per = (n == A.per_unit ? A.by_q : A.by_q1).div(smax + n - 1);
        run.first.b = ub; run.first.h = u - ub * A.Hkv; run.first.steps = smax; run.first.start = u * smax;
        run.c0 = run.first.start + min(smax, k * per);
        run.c1 = run.first.start + min(smax, (k + 1) * per);
        pl.first_cta = cta - k; pl.share = per;
    } else if (units <= nct && smin != smax && smax < (1 << 22) && static_cast<float>(pl.chunk) >= A.ragged_from * static_cast<float>(least) && 3.f * static_cast<float>(pl.total) <= (3 * nct - units) * static_cast<float>(pl.chunk + extra) &&
               ragged_run(C.prefix, A.B, A.Hkv, pl.chunk, extra, cta, nct, lane, C.run, C.plan)) {
        pl.aligned = 1;
        pl.first_cta = C.plan->first_cta; pl.share = C.plan->share;
        run = *C.run;
        __syncwarp();
    } else {
        run.c0 = min(pl.total, cta * pl.chunk);
        run.c1 = min(pl.total, run.c0 + pl.chunk);
        if (run.c0 < run.c1) run.first = locate_unit(C.prefix, A.B, A.Hkv, run.c0);
    }
    pl.cap = choose_cap(A.caps, pl, least);
    pl.nslots = static_cast<int>(A.caps.slots >> (8 * (pl.cap - 1))) & 255;
    pl.merge_off = A.ring_off + pl.nslots * A.slot_stride;
    pl.tab_off = pl.merge_off + A.caps.tail_base + (pl.cap - 1) * A.caps.tail_step;
    if (lane == 0) { *C.plan = pl; *C.run = run; }
    __syncwarp();
    asm volatile("bar.arrive %0, %1;" ::"n"(kPlanBarrier), "r"(n_threads) : "memory");
    return run;
}

// consumer side of the prologue: returns once the plan, the prefix and the ring barriers are in place
__device__ __forceinline__ void consumer_wait_plan(int n_threads)
{
    asm volatile("bar.sync %0, %1;" ::"n"(kPlanBarrier), "r"(n_threads) : "memory");
}

// Consumers of a step without a late wait: what the kernel before writes is complete from here on.  A step whose page
// stream started early (SPARK_FLAG_OVERLAP_PREVIOUS) releases its successor only here: released at its top, the successor
// could start, and with the flag read its own cache, while a kernel two places ahead of it (an append to that cache, itself
// released early) was still writing; the flag only promises something of the kernel just before.
__device__ __forceinline__ void consumer_wait_previous(const DecodeArgs& A)
{
    grid_wait();
    if (A.overlap) grid_release();
}

// The CTAs that hold a part of the unit starting at step `unit_start` with `unit_steps` steps.
__device__ __forceinline__ void unit_parts(const Plan& pl, int unit_start, int unit_steps, int& first_cta, int& n_parts)
{
    if (pl.aligned == 2) { first_cta = 0; n_parts = 1; return; }
    if (!pl.aligned) {
        first_cta = unit_start / pl.chunk;
        n_parts = (unit_start + unit_steps - 1) / pl.chunk - first_cta + 1;
        return;
    }
    first_cta = pl.first_cta;
    n_parts = (unit_steps + pl.share - 1) / pl.share;      // (trailing CTAs of the unit may be empty)
}

// The producer warp.  Lane i owns ring slot i: it handles this CTA's ring steps i, i + nslots, i + 2 nslots,
// ... in order.  Per revolution of the ring every lane looks up the page ids of its step (block-table
// loads of the next revolution are issued before the current one is polled, so their latency hides
// behind the wait), then the warp polls: a lane whose slot has been released by the consumers arms
// the slot's barrier and issues its page copies at once.  Polling is bounded; on expiry the CTA-wide
// abort flag is set and the lanes wait (bounded) for their own copies in flight before returning.
// bytes of page `id` to bring in: everything, or (ragged pages) up to the last slot row in use
__device__ __forceinline__ unsigned page_copy_bytes(const DecodeArgs& A, int id)
{
    if (!A.page_rows) return static_cast<unsigned>(A.L.page_bytes);
    int rows = A.page_rows[id];
    rows = rows < 0 ? 0 : (rows > A.L.keep ? A.L.keep : rows);
    return static_cast<unsigned>(A.L.vals_off + rows * kPageTokens * A.L.esize);
}

// page ids of step `i` of unit (b, h)
__device__ __forceinline__ void producer_page_ids(const DecodeArgs& A, const Ctrl& C, const UnitRef& u, int i,
                                                  int& id0, int& id1, unsigned& n0, unsigned& n1)
{
    const int64_t row = (static_cast<int64_t>(u.b) * A.Hkv + u.h) * A.max_blocks;
    const int32_t* bt = A.block_table ? A.block_table + row : nullptr;       // no table: pages of a unit are consecutive
    id1 = -1; n1 = 0;
    id0 = bt ? bt[A.pps * i] : static_cast<int>(row + A.pps * i);
    if (A.pps == 2) {                                       // second page of the step, if the sequence has one
        if (2 * i + 1 < (C.lens[u.b] + kPageTokens - 1) / kPageTokens) {
            id1 = bt ? bt[2 * i + 1] : static_cast<int>(row + 2 * i + 1);
            if (id1 < 0 || id1 >= A.n_pool_pages) { record_error(A.status, SPARK_ERR_DEVICE_BOUNDS); id1 = 0; }
            n1 = page_copy_bytes(A, id1);
        }
    }
    if (id0 < 0 || id0 >= A.n_pool_pages) { record_error(A.status, SPARK_ERR_DEVICE_BOUNDS); id0 = 0; }
    n0 = page_copy_bytes(A, id0);
}

template <int NW>
__device__ __forceinline__ void producer_loop(const DecodeArgs& A, const Ctrl& C, unsigned char* ring,
                                              const CtaRun& run, const Plan& pl, int lane)
{
    const PageLayout L = A.L;
    const int c0 = run.c0, c1 = run.c1, NS = pl.nslots, n_total = c1 - c0;
    const uint64_t policy = policy_evict_first();
    const bool owner = lane < NS;
    unsigned char* dst = ring + static_cast<size_t>(lane) * A.slot_stride;
    uint64_t* full = &C.full[owner ? lane : 0];
    uint64_t* empty = &C.empty[owner ? lane : 0];
    bool live = true;
    int last_round = -1;                                   // last revolution in which this lane issued
    int id0 = -1, id1 = -1;
    unsigned n0 = 0, n1 = 0;                               // bytes to copy of the two pages
    Epoch ep;
    ep.e1 = c0;                                            // (a CTA without steps has no first unit)
    if (n_total > 0) ep = make_epoch(C.prefix, A.Hkv, pl.cap, run.first, c0, c1);
    // this lane's ring step n -> its step of the line (epoch, warp, place in the warp's run) -> page ids
    auto lookup = [&](int n) {
        id0 = id1 = -1; n0 = n1 = 0;
        if (!owner || n >= n_total) return;
        while (c0 + n >= ep.e1)
            ep = make_epoch(C.prefix, A.Hkv, pl.cap, locate_unit(C.prefix, A.B, A.Hkv, ep.e1), ep.e1, c1);
        int g = c0 + n;
        if (pl.cap > 1) {
            const int len = ep.e1 - ep.e0, q = len / NW, r = len - q * NW;
            const int x = g - ep.e0, i = x / NW, w = x - i * NW;
            g = ep.e0 + w * q + min(w, r) + i;
        }
        UnitRef u = ep.first;
        while (g >= u.start + u.steps) next_unit(C.prefix, A.Hkv, u);
        producer_page_ids(A, C, u, g - u.start, id0, id1, n0, n1);
    };
    // Pass t of the loop looks up ids and then issues copies.  The lookup of revolution r + 1 waits for its block-table
    // loads, so it runs before revolution r is polled (hidden behind the wait for free slots), except at the start,
    // where every slot is free and the first copies go out before the second lookup: ids 0 | copies 0 | ids 1 |
    // ids 2, copies 1 | ids 3, copies 2 ...   (One loop body: this code runs cold, its size is start-up time.)
#pragma unroll 1
    for (int t = 0; t < 2 || (t - 2) * NS < n_total; ++t) {
        const int round = t == 1 ? 0 : t - 2;              // revolution whose copies go out in this pass (t = 0, 2: none)
        const int cur0 = id0, cur1 = id1;
        const unsigned b0 = n0, b1 = n1;
        if (t != 1) lookup((t == 0 ? 0 : t - 1) * NS + lane);
        if (t == 0 || t == 2) continue;
        const int n = round * NS + lane;
        bool pending = owner && n < n_total;
        WaitClock wc;
        while (__any_sync(kFull, pending)) {
            if (pending && (round == 0 || mbar_try_wait(empty, (round - 1) & 1))) {
                C.seq[lane] = round + 1;
                mbar_expect_tx(full, b0 + (cur1 >= 0 ? b1 : 0u));
                bulk_g2s(dst, A.pages + static_cast<int64_t>(cur0) * L.page_bytes, b0, full, policy);
                if (cur1 >= 0)
                    bulk_g2s(dst + L.page_bytes, A.pages + static_cast<int64_t>(cur1) * L.page_bytes, b1, full, policy);
                last_round = round;
                pending = false;
            }
            if (wc.expired() || *C.abort_flag) { live = false; break; }
        }
        if (!live) break;
    }
    if (!live) {
        if (lane == 0) { *C.abort_flag = 1; record_error(A.status, SPARK_ERR_DEVICE_TIMEOUT); }
        if (last_round >= 0) {                             // let this lane's copy in flight land
            WaitClock wc;
            while (!wc.expired())
                if (mbar_try_wait(full, last_round & 1)) break;
        }
    }
}

// zero-length sequences: out = 0, lse = -inf, or the other token set's result (consumer threads)
template <int NT>
__device__ __forceinline__ void write_empty_sequences(const DecodeArgs& A, const int* prefix, int tid)
{
#pragma unroll 1
    for (int b = blockIdx.x; b < A.B; b += gridDim.x)
        if (prefix[b + 1] == prefix[b]) {
#pragma unroll 1
            for (int i = tid; i < A.Hq * kHeadDim; i += NT)
                A.out[static_cast<int64_t>(b) * A.Hq * kHeadDim + i] =
                    A.other_out ? A.other_out[static_cast<int64_t>(b) * A.Hq * kHeadDim + i] : 0.f;
            if (A.lse)
#pragma unroll 1
                for (int i = tid; i < A.Hq; i += NT)
                    A.lse[static_cast<int64_t>(b) * A.Hq + i] = A.other_lse ? A.other_lse[static_cast<int64_t>(b) * A.Hq + i] : -INFINITY;
        }
}

// The epoch's units as the merge needs them; one warp.  Lane w stands for consumer warp w: a step belongs to the last
// warp whose run starts at or before it.
template <int NW>
__device__ __forceinline__ void describe_epoch(const DecodeArgs& A, const Ctrl& C, const Epoch& ep, int lane)
{
    const int n = ep.e1 - ep.e0, q = n / NW, r = n - q * NW;
    if (lane == 0) { C.epoch[0] = ep.e1; C.epoch[1] = ep.n_units; }
    const int run0 = ep.e0 + (lane < NW ? lane * q + min(lane, r) : n);
    if (C.plan->cap == 1) {                                // the warps that have a step hold a record each
        if (lane == 0) {
            EpochUnit d;
            d.b = ep.first.b; d.h = ep.first.h;
            d.rec0 = 0;
            d.n_rec = min(NW, n);
            unit_parts(*C.plan, ep.first.start, ep.first.steps, d.first_cta, d.n_parts);
            C.units[0] = d;
        }
        return;
    }
    UnitRef u = ep.first;
#pragma unroll 1
    for (int e = 0; e < ep.n_units; ++e) {
        if (e) next_unit(C.prefix, A.Hkv, u);
        const int w0 = __popc(__ballot_sync(kFull, run0 <= max(u.start, ep.e0))) - 1;
        const int w1 = __popc(__ballot_sync(kFull, run0 < min(u.start + u.steps, ep.e1))) - 1;
        if (lane == e) {
            EpochUnit d;
            d.b = u.b; d.h = u.h;
            d.rec0 = w0 + e;
            d.n_rec = w1 - w0 + 1;
            unit_parts(*C.plan, u.start, u.steps, d.first_cta, d.n_parts);
            C.units[e] = d;
        }
    }
}

// Factors of a row's unnormalised sum (running maximum M, running sum Ls) and of the other token set's output, and the
// row's log-sum-exp (the identity of merge_attn_kernel).
struct PublishWeights { float own, other, lse; };
__device__ __forceinline__ PublishWeights publish_weights(const DecodeArgs& A, int64_t row, float M, float Ls)
{
    PublishWeights w;
    w.own = 1.0f / Ls; w.other = 0.f; w.lse = (M + log2f(Ls)) * kLn2;
    if (A.other_lse) {
        const float lb = A.other_lse[row], m = fmaxf(w.lse, lb);
        const float ea = expf(w.lse - m), eb = expf(lb - m), inv = 1.0f / (ea + eb);
        w.own *= ea * inv;
        w.other = eb * inv;
        w.lse = m + logf(ea + eb);
    }
    return w;
}

// Merge the records of an epoch ([record][G][kRec]: 128 unnormalised outputs, m, l) unit by unit and publish the units'
// results: directly where this CTA holds the whole unit, else as a partial followed by the last-arriver merge (only the first
// and the last unit of a CTA's run can be split).  Called by all consumer threads after a consumer_sync().
//
// A warp serves a slice (all, half or a quarter of the 128 channels) of one head of one unit from the records to the result:
// it takes the log-sum-exp weights of the records itself (lane = record), adds up its channels, and where the unit is split
// leaves its slice, takes a ticket of the slice's own and, arriving last, merges the slice of all parts.  So no barrier of the
// CTA stands between the records and the result, and the slices of a unit are merged by several warps at once, of whatever
// CTAs come last.  A ticket per unit and one CTA merging all of it behind four barriers took 3.6 us from the last record to
// the result of a 32768-token step.  us before -> after: 1 x 500 tokens 9.1 -> 8.7, 32 x 2048 41.4 -> 39.5, 8 x 5000 29.7 ->
// 28.2, 8 x 2000..16000 44.1 -> 42.1, 1 x 4096 with 64 / 8 heads 13.7 -> 12.7; fp32 1 x 1024, builds in turn, 13.0 -> 12.7.
// (Three heads a group in halves: in quarters, us, 1 x 1000 tokens with 12 / 4 heads 9.2, in halves 8.9, whole 9.5; 1 x 16000 13.2, 13.0,
// 13.7; 1 x 32768 with 6 / 2 heads 14.9, 14.5, 16.4.)
__host__ __device__ constexpr int slices_of(int g, int nw) { return 4 * g <= 8 ? 4 : (2 * g <= nw ? 2 : 1); }
// Tickets of a split unit: a slice's each, at the unit's first CTA.  (No two split units have the same one: the first ends in a
// later CTA than it starts in.)  So where tickets and partials lie does not depend on the problem, and calls of any shapes may
// take turns on one workspace.
constexpr int kTickets = 16;
constexpr size_t kTicketBytes = kMaxCtas * kTickets * sizeof(int);
constexpr int kPart = kHeadDim + 8;                           // floats of a head's partial: 128 outputs and (m, l) once per slice

template <int N> __device__ __forceinline__ void load_floats(float (&x)[N], const float* p)
{
    if constexpr (N == 4) { const float4 v = *reinterpret_cast<const float4*>(p); x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w; }
    else if constexpr (N == 2) { const float2 v = *reinterpret_cast<const float2*>(p); x[0] = v.x; x[1] = v.y; }
    else x[0] = *p;
}
template <int N> __device__ __forceinline__ void store_floats(float* p, const float (&x)[N])
{
    if constexpr (N == 4) *reinterpret_cast<float4*>(p) = make_float4(x[0], x[1], x[2], x[3]);
    else if constexpr (N == 2) *reinterpret_cast<float2*>(p) = make_float2(x[0], x[1]);
    else *p = x[0];
}
// N channels of a row of the result from its unnormalised sum
template <int N>
__device__ __forceinline__ void publish(const DecodeArgs& A, int64_t row, int ch, float (&O)[N], float M, float Ls, bool lse)
{
    const PublishWeights w = publish_weights(A, row, M, Ls);
#pragma unroll
    for (int j = 0; j < N; ++j) O[j] *= w.own;
    if (A.other_out) {
        float x[N];
        load_floats<N>(x, A.other_out + row * kHeadDim + ch);
#pragma unroll
        for (int j = 0; j < N; ++j) O[j] = fmaf(w.other, x[j], O[j]);
    }
    store_floats<N>(A.out + row * kHeadDim + ch, O);
    if (lse && A.lse) A.lse[row] = w.lse;
}

// kWide: a quarter of a head is merged from two groups of 32 parts at a time.
template <int G, int NW, int NS, bool kWide>
__device__ __forceinline__ void merge_slices(const DecodeArgs& A, const EpochUnit* units, float* merge, int n_units, int warp, int lane)
{
    constexpr int kItems = G * NS;                                // slices of a unit
    constexpr int kCh = kHeadDim / NS, VE = kCh / 32;             // channels of a slice; per lane
    static_assert(NW <= 32 && kItems <= kTickets, "a lane per record; a ticket per slice");
    bool split = false;
    // ---- a slice of the unit's sum over this CTA's records ----
#pragma unroll 1
    for (int it = warp; it < n_units * kItems; it += NW) {
        const int e = it / kItems, gg = (it - e * kItems) / NS, s = (it - e * kItems) % NS;
        const EpochUnit d = units[e];
        const float* rec = merge + (d.rec0 * G + gg) * kRec;
        const float m = lane < d.n_rec ? rec[lane * (G * kRec) + kHeadDim] : -INFINITY;
        const float l = lane < d.n_rec ? rec[lane * (G * kRec) + kHeadDim + 1] : 0.f;
        const int ch = s * kCh + lane * VE;
        float v[NW][VE];
#pragma unroll
        for (int k = 0; k < NW; ++k) {                            // every load before the first use
#pragma unroll
            for (int j = 0; j < VE; ++j) v[k][j] = 0.f;
            if (k < d.n_rec) load_floats<VE>(v[k], rec + k * (G * kRec) + ch);
        }
        float M = m;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(kFull, M, o));
        const float wt = (m == -INFINITY) ? 0.f : exp2f(m - M);
        float Ls = l * wt;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) Ls += __shfl_xor_sync(kFull, Ls, o);
        float O[VE];
#pragma unroll
        for (int j = 0; j < VE; ++j) O[j] = 0.f;
#pragma unroll
        for (int k = 0; k < NW; ++k) {
            const float f = __shfl_sync(kFull, wt, k);
#pragma unroll
            for (int j = 0; j < VE; ++j) O[j] = fmaf(v[k][j], f, O[j]);
        }
        if (d.n_parts == 1) {
            if (A.late_wait) grid_wait();
            publish<VE>(A, static_cast<int64_t>(d.b) * A.Hq + d.h * G + gg, ch, O, M, Ls, s == 0 && lane == 0);
        } else {
            split = true;
            float* part = A.partials + (static_cast<int64_t>(blockIdx.x + d.b * A.Hkv + d.h) * G + gg) * kPart;
            store_floats<VE>(part + ch, O);
            if (lane == 0) *reinterpret_cast<float2*>(part + kHeadDim + 2 * s) = make_float2(M, Ls);
        }
    }
    // ---- the slices of split units: the last warp to arrive merges the parts ----
#pragma unroll 1
    for (int it = split ? warp : n_units * kItems; it < n_units * kItems; it += NW) {
        const int e = it / kItems, gg = (it - e * kItems) / NS, s = (it - e * kItems) % NS;
        const EpochUnit d = units[e];
        if (d.n_parts == 1) continue;
        const int unit = d.b * A.Hkv + d.h, n_parts = d.n_parts;
        int* ticket = A.tickets + d.first_cta * kTickets + gg * NS + s;
        // The warp barrier orders every lane's stores before lane 0's gpu-scope release; its acquire (same atomic) and the
        // barrier behind it order every lane's reads after the other parts' stores.
        __syncwarp();
        int old = 0;
        if (lane == 0) asm volatile("atom.add.acq_rel.gpu.global.s32 %0, [%1], 1;" : "=r"(old) : "l"(ticket) : "memory");
        __syncwarp();
        if (__shfl_sync(kFull, old, 0) != n_parts - 1) continue;
        constexpr int kLanes = kCh / 4, PP = 32 / kLanes;         // lanes of a part (four channels each); parts at a time
        constexpr int kSteps = 32 / PP, kBatch = 8;               // steps of 32 parts; loads in flight of one group of parts
        // groups taken at once (bf16, one unit on the whole grid, 148 parts: 1 x 32768 tokens 11.7 us with one, 11.2 with two)
        constexpr int kTwo = kSteps == kBatch && kWide ? 2 : 1;
        constexpr int kGroups = kMaxCtas / 32;                    // (m, l) pairs a lane may hold
        constexpr int64_t kStride = static_cast<int64_t>(G) * kPart;
        const float* base = A.partials + (static_cast<int64_t>(d.first_cta + unit) * G + gg) * kPart;
        const int sub = lane / kLanes, c4 = lane % kLanes;
        float2 ml[kGroups];
#pragma unroll
        for (int k = 0; k < kGroups; ++k) {
            const int p = k * 32 + lane;
            ml[k] = p < n_parts ? *reinterpret_cast<const float2*>(base + p * kStride + kHeadDim + 2 * s) : make_float2(-INFINITY, 0.f);
        }
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        float M = -INFINITY, Ls = 0.f;
#pragma unroll
        for (int k = 0; k < kGroups; k += kTwo) {
            if (k * 32 >= n_parts) break;
#pragma unroll 1
            for (int i0 = 0; i0 < kSteps && k * 32 + i0 * PP < n_parts; i0 += kBatch) {
                float4 o4[kBatch * kTwo];
#pragma unroll
                for (int i = 0; i < kBatch * kTwo; ++i) {
                    const int p = k * 32 + (i0 + i) * PP + sub;
                    o4[i] = p < n_parts ? *reinterpret_cast<const float4*>(base + p * kStride + s * kCh + 4 * c4) : make_float4(0.f, 0.f, 0.f, 0.f);
                }
                if (k == 0 && i0 == 0) {                          // the weights, under the first loads
#pragma unroll
                    for (int x = 0; x < kGroups; ++x) M = fmaxf(M, ml[x].x);
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(kFull, M, o));
#pragma unroll
                    for (int x = 0; x < kGroups; ++x) {
                        ml[x].x = ml[x].x == -INFINITY ? 0.f : exp2f(ml[x].x - M);
                        Ls = fmaf(ml[x].y, ml[x].x, Ls);
                    }
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) Ls += __shfl_xor_sync(kFull, Ls, o);
                }
#pragma unroll
                for (int i = 0; i < kBatch * kTwo; ++i) {
                    const float f = __shfl_sync(kFull, ml[k + i / kBatch].x, ((i0 + i) * PP + sub) & 31);
                    acc.x = fmaf(o4[i].x, f, acc.x); acc.y = fmaf(o4[i].y, f, acc.y);
                    acc.z = fmaf(o4[i].z, f, acc.z); acc.w = fmaf(o4[i].w, f, acc.w);
                }
            }
        }
#pragma unroll
        for (int o = kLanes; o < 32; o <<= 1) {
            acc.x += __shfl_xor_sync(kFull, acc.x, o); acc.y += __shfl_xor_sync(kFull, acc.y, o);
            acc.z += __shfl_xor_sync(kFull, acc.z, o); acc.w += __shfl_xor_sync(kFull, acc.w, o);
        }
        if (A.late_wait) grid_wait();
        if (sub == 0) {
            float O[4] = {acc.x, acc.y, acc.z, acc.w};
            publish<4>(A, static_cast<int64_t>(d.b) * A.Hq + d.h * G + gg, s * kCh + 4 * c4, O, M, Ls, s == 0 && lane == 0);
        }
        if (lane == 0) *ticket = 0;                               // ready for the next call
    }
}
// Fifteen warps: where a CTA may hold several units, a warp takes a whole head (32 x 2048 tokens, 32 / 8 heads: 42.0 us with halves,
// 39.5 so; 2 x 3000..7000 16.1 and 14.2).  Eight warps, whose one or two heads would leave most of them idle: only with more than half
// as many units as CTAs (fp32, 2 x 300..1000 tokens, 2 / 2 heads: whole 14.1, quarters 13.0; 4 x 200..1000, 2 / 1 heads 15.7 and 14.8;
// but 16 x 100..2000, 8 / 8 heads 49.6 and 51.5).
template <int G, int NW, bool kWide = true>
__device__ __forceinline__ void merge_and_publish(const DecodeArgs& A, const Ctrl& C, float* merge, int cap, int warp, int lane)
{
    constexpr int NS = slices_of(G, NW);
    const bool whole = NW > 8 ? cap > 1 : 2 * A.B * A.Hkv > static_cast<int>(gridDim.x);       // (the same in every CTA)
    if (NS == 1 || whole) merge_slices<G, NW, 1, kWide>(A, C.units, merge, C.epoch[1], warp, lane);
    else merge_slices<G, NW, NS, kWide>(A, C.units, merge, C.epoch[1], warp, lane);
}

// An even share of the line with the cache at its capacity, and 4 %.  Equal units in whole CTAs may exceed it by A.slack steps.
inline int64_t even_steps_per_cta(int64_t units, int max_blocks, int pps, int grid)
{
    const int64_t total = units * ((max_blocks + pps - 1) / pps);
    const int64_t chunk = (total + grid - 1) / grid;
    return chunk + chunk / 25 + 1;
}
// CTAs of the persistent grid: one per SM, fewer when the cache cannot hold a step for each.
inline int decode_grid(int n_sms, int64_t units, int max_blocks, int pps)
{
    const int64_t total = units * ((max_blocks + pps - 1) / pps);
    const int64_t g = total < n_sms ? total : n_sms;
    return g < 1 ? 1 : (g > kMaxCtas ? kMaxCtas : static_cast<int>(g));
}

// Ring slots for every number of units per epoch (at most `most` slots): with(n) = the largest number of units that leaves
// at least n of them, bytes(c) = the shared memory of a launch that may choose up to c units.
struct EpochRoom {
    int ns[kMaxCap];
    size_t used[kMaxCap];
    int with(int slots) const { int c = 1; while (c < kMaxCap && ns[c] >= slots) ++c; return c; }
    size_t bytes(int cap) const { size_t b = used[0]; for (int c = 1; c < cap; ++c) b = used[c] > b ? used[c] : b; return b; }
};
inline EpochRoom epoch_room(DecodeArgs& A, int nw, int g, int tab_bytes, int smem_optin, int most)
{
    EpochRoom r;
    A.caps.tail_base = merge_base(nw, g);
    A.caps.tail_step = merge_step(g);
    A.caps.slots = 0;
    for (int cap = 1; cap <= kMaxCap; ++cap) {
        const int tail = A.caps.tail_base + (cap - 1) * A.caps.tail_step + cap * tab_bytes, room = smem_optin - A.ring_off - tail;
        int n = room > 0 ? room / A.slot_stride : 0;
        n = n > kMaxSlots ? kMaxSlots : (n > most ? most : n);
        r.ns[cap - 1] = n;
        r.used[cap - 1] = A.ring_off + static_cast<size_t>(n) * A.slot_stride + tail;
        A.caps.slots |= static_cast<unsigned long long>(n) << (8 * (cap - 1));
    }
    return r;
}

inline void set_divisors(DecodeArgs& A, int64_t units, int grid)
{
    A.by_grid = FastDiv::of(grid);
    A.by_hkv = FastDiv::of(A.Hkv);
    A.per_unit = static_cast<int>(grid / units);
    A.extra = A.per_unit > 0 ? static_cast<int>(grid - A.per_unit * units) : 0;
    A.by_q = FastDiv::of(A.per_unit > 0 ? A.per_unit : 1);
    A.by_q1 = FastDiv::of(A.per_unit + 1);
}

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// per-dtype launchers (spark_decode.cu: fp32 storage, spark_decode_mma.cu: bf16 storage)
spark_status launch_decode_f32(int G, const DecodeArgs& A, int dev, const DeviceInfo& info, cudaStream_t stream);
spark_status launch_decode_bf16(int G, const DecodeArgs& A, int dev, const DeviceInfo& info, cudaStream_t stream);
spark_status launch_decode_bf16_sampled(int G, const DecodeArgs& A, int dev, const DeviceInfo& info, cudaStream_t stream);

}  // namespace spark
