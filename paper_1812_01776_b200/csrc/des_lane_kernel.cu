// Batched discrete-event simulation of the InferLine Estimator (Section 4.2),
// lane-parallel version: one LANE per (candidate, stage), the stages of a
// candidate running side by side as a pipeline inside one warp.
//
// The pipeline is a feed-forward tree with zero delay between stages, so a
// stage is a function from its arrival stream (times never decrease) to its
// completion stream, and the batch recurrence of the centralized batched queue
// (Section 3) is, per stage,
//
//     t      = max(earliest time a replica is free, arrival[head])
//     b      = min(max batch, number of arrivals from head on with time <= t)
//     finish = t + latency[stage][hw][b-1]            (Section 4.1 profile)
//
// with batches leaving in (finish, dispatch order) order.  A warp holds up to
// floor(32 / S) candidates; lane (j, s) runs the scalar chain of stage s of
// candidate j, and all 32 chains advance together, one record per iteration and
// lane:
//
//   * examine: the lane looks at ONE record of its arrival stream.  Either the
//     record joins the open batch (arrived by the batch's dispatch time and the
//     batch is not full), or the open batch is closed (finish time from the
//     table, sorted insert into the lane's ring of batches) and the record opens
//     the next batch, on a replica never used so far or else on the one that is
//     free first (the smallest key in use);
//   * hand on: ONE record of the batches that can leave goes to the child stage
//     selected by the query's branch bit or, at a leaf, to the candidate's slab
//     as a (finish, query) record.
//
// What bounds it: the serial chain of a batch (a warp that has its scheduler to
// itself) or the issue slots (several warps per scheduler); either way the number
// of instructions per iteration and the shared-memory latency on the chain.  So
// nothing on the way between two stages touches global memory:
//
//   * The stream between two stages is a ring of kX records per lane in shared
//     memory, [position][lane], so that a warp's accesses never conflict.  The
//     top bit of a record is never set, so a position whose high word is -1 is
//     empty: the consumer sees from the word itself whether its next record is
//     there, the producer whether there is room; no counters are exchanged and
//     no barrier is needed.  A producer without room holds its hand-on step;
//     simulated times do not depend on the order in which lanes take their
//     steps.  Consumers examine whatever arrives and leaves never wait, so every
//     wait ends.  How many records a stage will see is known from the branch
//     bits, so the end of a stream needs no flag either.
//   * Of a record that has been examined only the low part (query, branch bits)
//     is needed again, when its batch leaves.  It waits in a ring of nq words; the
//     last record of a batch carries a flag, so a batch is only (finish, index of
//     its first record).  A batch may leave as soon as its finish time is not
//     after the latest dispatch time of the stage (no later batch can finish
//     before that), which keeps few records waiting.  Where more than nq records
//     lie between the oldest one still needed and the one examined, the lane
//     SPILLS: it copies the words to a ring of 2^lane_ring_log2 words of its own
//     in global memory and reads those it has overwritten from there; looked at
//     once a turn (below), switched off again when the distance shrinks.  A lane
//     whose distance outgrows that ring as well gives its candidate up (marked in
//     the overflow array; the host's fallback evaluates it with the
//     warp-per-candidate kernel).
//   * The records of a group's first stage (the trace, or another part's stream, see CUT below) are copied to shared
//     memory at least one turn (below) before their use, in pairs (cp.async, all lanes of the group).
//   * The profile tables are shared by the CTA, rows padded to an odd length so
//     that rows of different lanes start in different banks.
//   * What happens once per candidate or rarely (its first and last batch, spills,
//     the iteration bound, the next candidate) is looked at once a turn of 8 to 62
//     iterations only, behind one vote.
//
// Measured on B200, 4,096 candidates x 4 stages x 50,000 queries and 4,096 x 10 x 10^6, whole calls: streams in global memory
// 15.4 / 720 ms; streams in shared memory, the loop in C++ 6.97 / 346 ms (123 instructions an iteration, 220 cycles for a warp on
// its own); the loop in PTX and twice as long turns where a CTA has its SM to itself 6.3 / 300 to 329 ms, within the noise of
// the other on the second (108 instructions, 184 cycles and the turns).  What costs there is latency between
// dependent instructions (73 of 230 cycles) and the ALU pipe (compares, selects, logic: half the issue rate).  Learned on
// the way: a bool that lives through the loop takes one of seven predicates and costs the schedule 15 % (two of them:
// 6.94 -> 8.14 ms), so what a lane has to remember are bits of one register; the same instructions with the loads of the next
// iteration behind this one's stores take 7.7 ms; one branch in the loop, never taken, 50 cycles.
#include "il_internal.h"

#include <algorithm>
#include <type_traits>

namespace il {

namespace {

constexpr int kLaneWarps = 4;                 // warps per CTA: one per scheduler even in a grid of few CTAs
constexpr uint64_t kInf = ~0ull;
constexpr uint64_t kLatest = 0x7fefffffffffffffull;      // no record or key is larger
constexpr int kX = 8;                         // records of a stream between two stages
constexpr uint32_t kLast = 0x80000000u;       // flag of a batch's last record in that ring
constexpr int kTurn = 16;                     // iterations (two less) between two looks at finished groups, spills, bounds, where a lane
                                              // keeps much; else half of what a group has before it
constexpr int kQuickTurn = 8;                 // the same while a stage is about to start or to end
constexpr uint32_t kQuickLooks = 128;         // looks at a candidate within which a stage counts as about to start

__device__ __forceinline__ uint64_t lds64(uint32_t a)
{
    uint64_t v;
    asm volatile("ld.shared.u64 %0, [%1];" : "=l"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t lds32(uint32_t a)
{
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}
// Words that two lanes share.  Stream records, and the records in a join's windows: each is complete in itself, so no
// ordering between words is needed.  A join's counts: stored behind the warp barrier that follows the records they cover.
__device__ __forceinline__ uint64_t lds64_shared(uint32_t a)
{
    uint64_t v;
    asm volatile("ld.relaxed.cta.shared.u64 %0, [%1];" : "=l"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t lds32_shared(uint32_t a)
{
    uint32_t v;
    asm volatile("ld.relaxed.cta.shared.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void sts32_shared_if(bool c, uint32_t a, uint32_t v)
{
    asm volatile("{ .reg .pred p; setp.ne.u32 p, %0, 0; @p st.relaxed.cta.shared.u32 [%1], %2; }" ::"r"((uint32_t)c), "r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void sts64(uint32_t a, uint64_t v) { asm volatile("st.shared.u64 [%0], %1;" ::"r"(a), "l"(v) : "memory"); }
__device__ __forceinline__ void sts32(uint32_t a, uint32_t v) { asm volatile("st.shared.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory"); }

// The same under a predicate: a lane's steps
// are straight-line code (a branch costs the warp more than the few instructions it would skip).
__device__ __forceinline__ void sts64_if(bool c, uint32_t a, uint64_t v)
{
    asm volatile("{ .reg .pred p; setp.ne.u32 p, %0, 0; @p st.shared.u64 [%1], %2; }" ::"r"((uint32_t)c), "r"(a), "l"(v) : "memory");
}
__device__ __forceinline__ void stg64_if(bool c, uint64_t *a, uint64_t v)
{
    asm volatile("{ .reg .pred p; setp.ne.u32 p, %0, 0; @p st.global.u64 [%1], %2; }" ::"r"((uint32_t)c), "l"(a), "l"(v) : "memory");
}
__device__ __forceinline__ void stg32_if(bool c, uint32_t *a, uint32_t v)
{
    asm volatile("{ .reg .pred p; setp.ne.u32 p, %0, 0; @p st.global.u32 [%1], %2; }" ::"r"((uint32_t)c), "l"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void ldg32_if(bool c, const uint32_t *a, uint32_t &v)      // leaves v alone otherwise
{
    asm volatile("{ .reg .pred p; setp.ne.u32 p, %1, 0; @p ld.global.ca.u32 %0, [%2]; }" : "+r"(v) : "r"((uint32_t)c), "l"(a) : "memory");
}
// 16 bytes from global to shared memory, asynchronously and past L1 (another SM may be writing next to them).  Each half is a
// record that is complete before it is asked for.
__device__ __forceinline__ void copy16(uint32_t dst, const uint64_t *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ uint64_t ldg64_shared(const uint64_t *a)
{
    uint64_t v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(a) : "memory");
    return v;
}
// Counts of a stream's records that are there: published behind a fence that follows the records, read with acquire.
__device__ __forceinline__ uint32_t ldg32_acquire(const uint32_t *a)
{
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(a) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t ldg32_shared(const uint32_t *a)
{
    uint32_t v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(a) : "memory");
    return v;
}
__device__ __forceinline__ void stg32_shared(uint32_t *a, uint32_t v)
{
    asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void copies_done() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Shared memory of a CTA: the tables ([S * H] rows of Bmax | 1 words, one word in front of them), then per warp
// the batch keys [kr][lane] (aligned to their size: a ring address is (counter & mask) | base), per warp the
// streams [kX][lane], a row of empty records (the "child" of a leaf), per warp the miss counts of the groups
// (feasibility only), per warp the words of examined records [nq][lane], and per warp and group the next `ahead` records
// of its arrival stream, 16 bytes apart so that groups start in different banks.
// Where a CTA's dynamic shared memory starts with the toolkit at hand.  The host plans for it; a launch that finds it elsewhere
// needs up to a row of batch keys more to align them and takes it from the words of examined records (more spills).
constexpr uint32_t kSmemBase = 1024;
__host__ __device__ inline uint32_t key_bytes(int kr) { return (uint32_t)kr * 256u; }
constexpr uint32_t kXBytes = kX * 256u;
__host__ __device__ inline size_t table_bytes(int rows, int Bmax) { return ((size_t)rows * (Bmax | 1) + 1) * 4; }
__host__ __device__ inline uint32_t stretch_bytes(int ahead) { return (uint32_t)ahead * 8u + 16u; }
__host__ __device__ inline size_t ring_bytes(int kr, int nq, int stretch)
{
    return (size_t)kLaneWarps * (key_bytes(kr) + nq * 128u + kXBytes + (size_t)stretch);
}
constexpr size_t kTailBytes = 256 + kLaneWarps * 128;

// ---- Cut pipelines: who does what ---------------------------------------------------------------------------------
// SMs set aside for root nodes, one warp per scheduler: 16 nodes a warp (up to 64 an SM), a third of the device at most.
__host__ __device__ inline uint32_t root_sms_for(uint32_t nodes, uint32_t num_sms)
{
    const uint32_t want = (nodes + 4u * kRootGroups - 1u) / (4u * kRootGroups), most = num_sms / 3u > 0u ? num_sms / 3u : 1u;
    return want < 1u ? 1u : want < most ? want : most;
}

constexpr unsigned kRoleNone = 0, kRoleRoots = 1, kRoleParts = 2;
constexpr uint32_t kDead = 0x80000000u;       // in place of a stream's count: no more records will come, and some are missing

// The first CTA on an SM gets a number; the first `root_sms` of them take root nodes and have the SM to themselves.  (Without
// that a root shares its scheduler with one or two warps, and everything else waits for it.)  Called by one thread of a CTA.
__device__ unsigned lane_cta_role(const LaneCut &cut, uint32_t root_sms)
{
    uint32_t *ctl = cut.ctl, sm;
    asm("mov.u32 %0, %%smid;" : "=r"(sm));
    if (cut.sms_seen) sm %= (uint32_t)cut.sms_seen;
    if (sm >= kCtlSms) return atomicAdd(ctl + kCtlOrder, 1u) < root_sms ? kRoleRoots : kRoleParts;
    if (atomicAdd(ctl + kCtlSlot + sm, 1u) == 0u) {
        const unsigned role = atomicAdd(ctl + kCtlOrder, 1u) < root_sms ? kRoleRoots : kRoleParts;
        atomicExch(ctl + kCtlRole + sm, role);
        return role;
    }
    unsigned role = 0u;
    for (int k = 0; k < (1 << 16) && role == 0u; k++) {       // (the other CTA is a few instructions away from telling)
        role = atomicAdd(ctl + kCtlRole + sm, 0u);
        if (role == 0u) __nanosleep(100);
    }
    if (role != kRoleRoots) return kRoleParts;
    // As many leave as the grid has CTAs planned beside those of root nodes.  More come where another stream's kernel holds the
    // rest of the device, and those take parts: if all of them left, CTA after CTA would come and go, and the few that came
    // first would do all the work (two SMs, 4,096 candidates of a tree of 6, 3,000 queries: 10.1 ms; 0.66 with this).
    const uint32_t beside = (gridDim.x - 1u) / (uint32_t)cut.num_sms * root_sms;
    return atomicAdd(ctl + kCtlLeft, 1u) < beside ? kRoleNone : kRoleParts;
}

// The part a warp starts with: root nodes, or by the order in which warps start, the parts in the order of the pipeline,
// each as many warps as the host has planned for it.  (A warp that finds no more of its part goes on with the next.)
__device__ int lane_first_part(const LaneCut &cut, bool for_roots)
{
    if (for_roots) return 0;
    uint32_t w = 0;
    if ((threadIdx.x & 31) == 0) w = atomicAdd(cut.ctl + kCtlTicket, 1u);
    w = __shfl_sync(0xffffffffu, w, 0);
    const int t0 = cut.shared ? 1 : 0;
    for (int t = t0; t < cut.n_part; t++) {
        if (w < (uint32_t)cut.part[t].warps) return t;
        w -= (uint32_t)cut.part[t].warps;
    }
    return t0 + (int)(w % (uint32_t)(cut.n_part - t0));
}

// The merge of a join's two incoming streams, one lane per candidate: records in time order, at equal times the first
// parent's first; a query that follows both edges passes with the later of its two records.  A record can be taken when
// what comes next on the other side is known.  A bit per query tells whether its first record has been taken.  The bits'
// words are in a small write-back cache in shared memory, `entries` per lane (where other parts keep words of examined
// records); queries come in nearly in order, so a word is new when it is first needed, and one that had to make room
// goes to global memory.  Bound by the latency of an iteration, a record each: the two heads from shared memory, their
// order, the query's word: about 260 cycles.  511 candidates of a diamond, 50,000 queries: 53 ms with the merge in the stages'
// loop, 13.1 as a part (29 with branches for the words, 23.3 with the words in global memory alone).
__device__ __noinline__ void lane_merge(const DesParams &p, const LaneCut &cut, int part, uint32_t tbw, uint32_t ahead, uint32_t cache, uint32_t entries,
                                        unsigned long long &naps, uint32_t &quit)
{
    const unsigned full = 0xffffffffu;
    const LanePart &pt = cut.part[part];
    const LaneStream &xa = cut.stream[pt.in], &xb = cut.stream[pt.in_b], &xo = cut.stream[pt.out_a];
    const int lane = threadIdx.x & 31, s = pt.stage[0], qi = p.qbits, rb = p.rec_bits;
    const uint32_t qmask = (1u << (qi + rb)) - 1u, imask = (1u << qi) - 1u;
    const uint32_t window = ahead, wmask = window - 1u, its = window / 2u;
    const uint32_t wa = tbw + (uint32_t)min(lane, pt.groups - 1) * stretch_bytes(2 * (int)ahead), wb = wa + window * 8u;
    const uint32_t na = (uint32_t)xa.len, nb = (uint32_t)xb.len;
    const bool always = p.any_bits == 0;        // no conditional edges: every query comes from both sides
    // (a lane may also wait while others of its warp have records)
    const unsigned long long limit = (p.iter_limit ? p.iter_limit : (8ull * (unsigned)p.n * (unsigned)(p.S + 1) + 4096ull) * 4ull) / its + 1ull;
    unsigned long long spent = 0;
    bool more = lane < pt.groups, has = false, dead = false;
    uint32_t c = 0, ia = 0, ib = 0, fed_a = 0, fed_b = 0, have_a = 0, have_b = 0, tail = 0, pub = 0;
    const uint64_t *src_a = nullptr, *src_b = nullptr;
    const uint32_t *count_a = nullptr, *count_b = nullptr;
    uint64_t *out = nullptr;
    uint32_t *count = nullptr, *seen = nullptr;
    uint32_t seen_new = 0;      // words from here on have not been touched
    const uint32_t row0 = cache + (uint32_t)lane * 8u, emask = entries - 1u;

    // copies what is there of a stream into its window, up to `window` records from i on
    auto feed = [&](const uint64_t *src, uint32_t w, uint32_t i, uint32_t have, uint32_t n, uint32_t &fed) {
        uint32_t to = min(i + window, have);
        if (to != n) to &= ~1u;
        if (to > fed && (to & 1u)) sts64(w + ((to - 1u) & wmask) * 8u, ldg64_shared(src + (to - 1u)));
        for (uint32_t k = fed; k + 1u < to; k += 2u) copy16(w + (k & wmask) * 8u, src + k);
        fed = max(fed, to);
    };
    for (uint32_t look = 1u;; look++) {
        copies_done();
        uint32_t in_a = fed_a, in_b = fed_b;             // what has arrived
        if (has && spent++ == limit) {
            atomicCAS(p.status, 0, IL_ERR_ITER_LIMIT);
            atomicOr(&p.counters[5], 1ull);
            dead = true;
        }
        if (has && (dead || quit != 0u || (ia == na && ib == nb))) {
            __threadfence();
            const bool ok = ia == na && ib == nb && !dead;
            if (ok && tail != (uint32_t)xo.len) { atomicCAS(p.status, 0, IL_ERR_ITER_LIMIT); atomicOr(&p.counters[5], 2ull); }
            stg32_shared(count, ok ? tail : kDead);
            has = false;
        }
        if (!has && more) {
            c = atomicAdd(cut.ctl + kCtlWork + part, 1u);
            more = c < (uint32_t)p.n_cand && quit == 0u;
            if (more) {
                const int32_t of = cut.root_of[c];
                auto row = [&](const LaneStream &x) { return x.by_node ? (uint32_t)max(of, 0) : c; };
                has = true; dead = of < 0;
                ia = 0; ib = 0; fed_a = 0; fed_b = 0; have_a = 0; have_b = 0; tail = 0; pub = 0;
                in_a = 0; in_b = 0; spent = 0; seen_new = 0;
                for (uint32_t k = 0; k < entries; k++) sts64(row0 + k * 256u, kInf);      // word number (none) << 32 | word
                src_a = xa.base + (int64_t)row(xa) * xa.stride + xa.off; count_a = xa.count + row(xa);
                src_b = xb.base + (int64_t)row(xb) * xb.stride + xb.off; count_b = xb.count + row(xb);
                out = xo.base + (int64_t)row(xo) * xo.stride + xo.off; count = xo.count + row(xo);
                seen = cut.seen + ((int64_t)c * cut.n_join + pt.join_no) * cut.seen_words;
                if (dead) { stg32_shared(count, kDead); has = false; }
            }
        }
        if (!__any_sync(full, has || more)) break;
        auto starving = [&](uint32_t i, uint32_t have, uint32_t n) { return have != n && have - i < its; };
        auto idle = [&]() { return !has || dead || starving(ia, have_a, na) || starving(ib, have_b, nb); };
        const bool nothing = __all_sync(full, idle());
        if ((look & 7u) == 0u || nothing) {
            if (has && tail != pub) { __threadfence(); stg32_shared(count, tail); pub = tail; }
        }
        if ((look & 3u) == 0u || nothing) {
            auto ask = [&](const uint32_t *from, uint32_t i, uint32_t &have, uint32_t n) {
                if (have == n || have - i >= 2u * window) return;
                const uint32_t w = ldg32_acquire(from);
                dead |= w == kDead;
                if (w != kDead) have = max(have, w);
            };
            if (has) { ask(count_a, ia, have_a, na); ask(count_b, ib, have_b, nb); }
            if (nothing && __all_sync(full, idle() && !dead)) {
                __nanosleep(500);
                if (naps-- == 0ull) { atomicCAS(p.status, 0, IL_ERR_ITER_LIMIT); atomicOr(&p.counters[5], 1ull); }
                quit = __any_sync(full, *reinterpret_cast<volatile int *>(p.status) != 0) ? 1u : 0u;
                // (a side may have less than a step's records left for good while the other has ended or waits for it)
            }
        }
        if (has && !dead) {
            feed(src_a, wa, ia, have_a, na, fed_a);
            feed(src_b, wb, ib, have_b, nb, fed_b);
        }
        const uint32_t la = has && !dead ? in_a : ia, lb = has && !dead ? in_b : ib;
        uint64_t va = lds64(wa + (ia & wmask) * 8u), vb = lds64(wb + (ib & wmask) * 8u);
        // straight-line but for words that are not simply the next ones
        auto step = [&](auto every) {
            const uint64_t ha = ia == na ? kInf : va, hb = ib == nb ? kInf : vb;
            const bool from_a = (ha | qmask) <= (hb | qmask);
            const uint64_t rec = from_a ? ha : hb;
            const uint32_t low = (uint32_t)rec & qmask, qid = low & imask, w = qid >> 5, mine = 1u << (qid & 31u), at = row0 + (w & emask) * 256u;
            uint64_t e = lds64(at);
            const uint32_t known = (ia < la || ia == na) && (ib < lb || ib == nb) && (int64_t)rec >= 0 && IL_IN_RANGE(qid, p.n, p.status) ? 1u : 0u;
            ia += from_a ? known : 0u;
            ib += from_a ? 0u : known;
            va = lds64(wa + (ia & wmask) * 8u);
            vb = lds64(wb + (ib & wmask) * 8u);
            uint32_t both = known;
            if constexpr (!decltype(every)::value) {
                const uint32_t bits = rb > 0 ? low >> qi : known ? p.bits[qid] : 0u;
                both &= (uint32_t)(p.join_both[s][bits >> 6] >> (bits & 63u)) & 1u;
            }
            const uint32_t old = (uint32_t)(e >> 32);
            const uint32_t other = both != 0u && old != w ? 1u : 0u;
            stg32_if(other != 0u && old != ~0u && IL_IN_RANGE(old, cut.seen_words, p.status), seen + old, (uint32_t)e);
            uint32_t word = other ? 0u : (uint32_t)e;
            if (other != 0u && w != seen_new) {
                if (w < seen_new && IL_IN_RANGE(w, cut.seen_words, p.status)) word = seen[w];
#pragma unroll 1
                for (; seen_new < w; seen_new++)         // passed over: it may come later
                    if (IL_IN_RANGE(seen_new, cut.seen_words, p.status)) seen[seen_new] = 0u;
            }
            seen_new = other ? max(seen_new, w + 1u) : seen_new;
            sts64_if(both != 0u, at, (uint64_t)w << 32 | (word ^ mine));
            const uint32_t passes = both != 0u ? (word >> (qid & 31u)) & 1u : known;
            stg64_if(passes != 0u && IL_IN_RANGE(tail, xo.len, p.status), out + tail, rec);
            tail += passes;
        };
        if (always) {
#pragma unroll 2
            for (uint32_t k = 0; k < its; k++) step(std::true_type{});
        } else {
#pragma unroll 1
            for (uint32_t k = 0; k < its; k++) step(std::false_type{});
        }
    }
}

// ---- One iteration of a lane, in PTX ------------------------------------------------------------------------------
// Why PTX: a warp that has its scheduler to itself is bound by the iteration's latency.  A compare here takes the condition
// before it along (setp.and), where the compiler joins finished predicates by instructions of their own, and what the next
// iteration reads (its record, the room for the record in hand, the time of the open batch, the low part to hand on) is requested as soon as
// it is known where it lies, before this iteration's stores.
// Records and keys are compared as doubles: words below 0x7ff0... order the same as the doubles of their bits, and a double takes one
// instruction on a pipe that is idle otherwise, where a 64-bit integer takes two on the ALU pipe (5 % of a launch with
// three warps per scheduler).  A word with the sign or all exponent bits set compares as false.
// The seven forms of the iteration (lane_simulation: step) are one text.  A form gives what is its own: more operands, more
// registers, how the tails of its ways out move, the way out itself, how the deeper insertion is reached, what more it hands back.
// Operands by number: 0 to 20 the state that all forms have, then what state a form adds, the inputs that all have, a form's.
#define IL_LOAD(type, name, number) ".reg ." #type " " #name "; mov." #type " " #name ", %" #number ";\n"
#define IL_STORE(type, name, number) "mov." #type " %" #number ", " #name ";\n"
#define IL_STEP_STATE(X) \
    X(b32, i, 0) X(b32, bm, 1) X(b32, lpos, 2) X(b32, lfull, 3) X(b32, tpos, 4) X(b32, at1, 5) X(b32, at2, 6) X(b64, tk, 7) \
    X(b32, prev, 8) X(b64, rec, 9) X(b32, lat, 10) X(b32, xs, 11) X(b32, epos, 12) X(b32, efull, 13) X(b32, e_on, 14) \
    X(b64, e_key, 15) X(b32, e_idx, 16) X(b32, qv, 17) X(b32, tail_a, 18) X(b32, rw, 19) X(b32, sa, 20)
#define IL_STATE_OPERANDS \
    "+r"(i), "+r"(bm), "+r"(lpos), "+r"(lfull), "+r"(tpos), "+r"(at1), "+r"(at2), "+l"(tk), "+r"(prev), "+l"(rec), "+r"(lat), \
    "+r"(xs), "+r"(epos), "+r"(efull), "+r"(e_on), "+l"(e_key), "+r"(e_idx), "+r"(qv), "+r"(tail_a), "+r"(rw), "+r"(sa)
#define IL_STEP_INPUTS(n0, n1, n2, n3, n4, n5, n6, n7, n8, n9, n10, n11, n12, n13, n14, n15, n16) \
    IL_LOAD(b32, xin, n0) IL_LOAD(b32, xin_mask, n1) IL_LOAD(b32, xin_row, n2) IL_LOAD(b32, tab, n3) IL_LOAD(b32, kfb, n4) \
    IL_LOAD(b32, kfm, n5) IL_LOAD(b32, kb, n6) IL_LOAD(b32, rm, n7) IL_LOAD(b32, mbm1, n8) IL_LOAD(b32, tick, n9) \
    IL_LOAD(b32, qmask, n10) IL_LOAD(b32, tmask, n11) IL_LOAD(b32, qb, n12) IL_LOAD(b32, nqm, n13) IL_LOAD(b32, xa, n14) \
    IL_LOAD(b32, xam, n15) IL_LOAD(b32, down, n16)
#define IL_INPUT_OPERANDS \
    "r"(xin), "r"(xin_mask), "r"(xin_row), "r"(tab), "r"(kfb), "r"(kfm), "r"(kb), "r"(rm), "r"(mbm1), "r"(tick), "r"(qmask), \
    "r"(~qmask), "r"(qb), "r"(nq - 1u), "r"(xa), "r"(xam), "r"(down)
// The record to examine: joins the open batch, or closes it and opens the next.  The record in hand: handed on where there is room.
#define IL_EXAMINE \
    "and.b32 a, epos, rm; or.b32 a, a, kb; ld.shared.b64 fk, [a];\n" \
    "and.b32 a, lpos, kfm; or.b32 a, a, kfb; ld.shared.b64 kf, [a];\n" \
    "ld.shared.b64 k1, [at1]; ld.shared.b64 k2, [at2];\n" \
    "mov.b64 td, tk; mov.b64 {rl, rh}, rec; mov.u32 xs_was, xs; mov.u32 sa_was, sa;\n" \
    "setp.ne.u32 t, tpos, efull; selp.b32 rh, rh, -1, t; mov.b64 r, {rl, rh};\n" \
    "setp.ge.s32 taken, rh, 0; setp.ge.and.u32 t, bm, mbm1, taken; setp.gt.or.f64 open, r, td, t;\n" \
    "sub.u32 y, i, bm; add.u32 y, y, -1;\n" \
    "add.u32 wa, i, -1; and.b32 wa, wa, nqm; mad.lo.u32 wa, wa, 128, qb;\n" \
    "@taken add.u32 i, i, 1; and.b32 xs, i, xin_mask; mad.lo.u32 xs, xs, xin_row, xin; ld.relaxed.cta.shared.b64 rec, [xs];\n" \
    "setp.lt.s32 hand, rw, 0; setp.ne.and.u32 hand, e_on, 0, hand; setp.ge.and.s32 hd|ho, down, 0, hand; setp.lt.and.s32 fin, qv, 0, hand;\n" \
    "and.b32 x, qv, 0x7fffffff; mov.b64 {lo, hi}, e_key; and.b32 lo, lo, tmask; or.b32 a, lo, x; mov.b64 v, {a, hi}; mov.u32 ta_was, tail_a;\n"
// (the tails have moved) what the next iteration needs of the child's stream and of the tables; the next batch to hand on, if it may
// leave; a record for the child.
#define IL_FETCH \
    "and.b32 sa, tail_a, xam; or.b32 sa, sa, xa; ld.relaxed.cta.shared.u32 rw, [sa+4];\n" \
    "mad.wide.u32 key, lat, tick, tk; mov.b64 {kl, kh}, key; and.b32 kl, kl, tmask; or.b32 kl, kl, y; mov.b64 key, {kl, kh};\n" \
    "@taken add.u32 bm, bm, 1; @open mov.u32 bm, 0; mad.lo.u32 a, bm, 4, tab; ld.shared.u32 lat, [a];\n" \
    "setp.eq.or.u32 fetch, e_on, 0, fin; setp.ne.and.u32 fetch, epos, tpos, fetch; setp.le.and.f64 fetch, fk, td, fetch;\n" \
    "mov.b64 {fl, fh}, fk;\n" \
    "@hand add.u32 e_idx, e_idx, 1; @fetch and.b32 e_idx, fl, qmask; and.b32 a, e_idx, nqm; mad.lo.u32 a, a, 128, qb; ld.shared.u32 qv, [a];\n" \
    "@hd st.relaxed.cta.shared.b64 [sa_was], v;\n"
// The closed batch goes behind the last one of the ring or just before it; the replica that is free first; the record's low part
// to the ring of examined records, its position in the stream emptied; counters.
#define IL_INSERT \
    "@fetch mov.b64 e_key, fk; @fin mov.u32 e_on, 0; @fetch mov.u32 e_on, 1; @fetch add.u32 epos, epos, 256; @fetch add.u32 efull, efull, 256;\n" \
    "and.b32 at0, tpos, rm; or.b32 at0, at0, kb;\n" \
    "setp.lt.f64 pf, kf, key; selp.b64 first, kf, key, pf;\n" \
    "setp.eq.u32 pz, tpos, lfull; setp.lt.and.f64 pz, r, first, pz; selp.b64 first, first, r, pz;\n" \
    "mov.b64 {fl, fh}, first; or.b32 fl, fl, qmask; mov.b64 first, {fl, fh}; selp.b64 tk, first, tk, open;\n" \
    "setp.lt.and.f64 ov, key, k1, open; selp.u32 sd, at1, at0, ov;\n" \
    "@open st.shared.b64 [sd], key; @ov st.shared.b64 [at0], k1;\n" \
    "setp.lt.and.f64 dp, key, k2, ov; mov.u32 pos, tpos; mov.u32 left, lpos;\n" \
    "setp.eq.and.u32 pop, tpos, lfull, open;\n" \
    "mov.u32 word, prev; @open or.b32 word, word, 0x80000000; @taken st.shared.u32 [wa], word;\n" \
    "@taken st.relaxed.cta.shared.u32 [xs_was+4], -1;\n" \
    "@open add.u32 tpos, tpos, 256; @open mov.u32 at2, at1; @open mov.u32 at1, at0;\n" \
    "@pop add.u32 lpos, lpos, 256; @pop add.u32 lfull, lfull, 256;\n" \
    "@taken and.b32 prev, rl, qmask;\n"
// A batch that goes further back, past the batches that finish later: four a round.  Each lane by itself, or (WARP) all lanes behind
// a vote: a chain of 4 takes 6.7 ms without it and 7.3 with it, but a tree of 6 feasibility only 21.3 and 20.2, and fan-out
// 17.9 and 17.6 (taken while the loop was written; a chain feasibility only has not been timed without the vote).
#define IL_DEEPER(SKIP, FIRST, WHO, AGAIN) \
    SKIP "\n" \
    "mov.u32 sd, left; sub.u32 pos, pos, 256;\n" \
    "DEEPER:\n" \
    "sub.u32 left, pos, sd;\n" \
    "and.b32 at0, pos, rm; or.b32 at0, at0, kb; sub.u32 a1, pos, 256; and.b32 a1, a1, rm; or.b32 a1, a1, kb;\n" \
    "sub.u32 a2, pos, 512; and.b32 a2, a2, rm; or.b32 a2, a2, kb; sub.u32 a3, pos, 768; and.b32 a3, a3, rm; or.b32 a3, a3, kb;\n" \
    "sub.u32 a4, pos, 1024; and.b32 a4, a4, rm; or.b32 a4, a4, kb;\n" \
    "ld.shared.b64 e1, [a1]; ld.shared.b64 e2, [a2]; ld.shared.b64 e3, [a3]; ld.shared.b64 e4, [a4];\n" \
    FIRST " setp.lt.and.f64 t, key, e1, t; setp.gt.and.u32 ov, left, 256, t; setp.lt.and.f64 ov, key, e2, ov;\n" \
    "setp.gt.and.u32 pz, left, 512, ov; setp.lt.and.f64 pz, key, e3, pz; setp.gt.and.u32 pf, left, 768, pz; setp.lt.and.f64 pf, key, e4, pf;\n" \
    "@t st.shared.b64 [at0], e1; @ov st.shared.b64 [a1], e2; @pz st.shared.b64 [a2], e3; @pf st.shared.b64 [a3], e4;\n" \
    "@t mov.u32 at0, a1; @ov mov.u32 at0, a2; @pz mov.u32 at0, a3; @pf mov.u32 at0, a4; " WHO "st.shared.b64 [at0], key;\n" \
    "sub.u32 pos, pos, 1024; " AGAIN "\n" \
    "PLACED:\n"
#define IL_DEEPER_LANE IL_DEEPER("@!dp bra PLACED;", "setp.gt.u32 t, left, 0;", "", "@pf bra DEEPER;")
#define IL_DEEPER_WARP \
    IL_DEEPER("vote.sync.any.pred pf, dp, 0xffffffff; @!pf bra.uni PLACED;", "setp.gt.and.u32 t, left, 0, dp;", "@dp ", \
              "setp.ne.and.u32 dp, pos, 1, pf; vote.sync.any.pred pf, dp, 0xffffffff; @pf bra.uni DEEPER;")
#define IL_STEP(MORE_STATE, INPUTS, REGISTERS, TAILS, OUT, DEEPER, MORE_BACK) \
    "{\n" IL_STEP_STATE(IL_LOAD) MORE_STATE INPUTS \
    ".reg .pred t, taken, open, pop, ov, dp, pz, pf, hand, hd, ho, fin, fetch;\n" \
    ".reg .u32 at0, sd, rl, rh, kl, kh, fl, fh, word, wa, x, y, lo, hi, a, xs_was, sa_was, ta_was, pos, left, a1, a2, a3, a4;\n" \
    ".reg .b64 kf, k1, k2, fk, key, td, r, first, v, e1, e2, e3, e4;\n" REGISTERS \
    IL_EXAMINE TAILS IL_FETCH OUT IL_INSERT DEEPER IL_STEP_STATE(IL_STORE) MORE_BACK "}"
// One way out: its tail; the record as it leaves the pipeline, without branch bits.
#define IL_ONE_TAIL "@hand add.u32 tail_a, tail_a, tail_step;\n"
#define IL_PLAIN_RECORD "mov.b64 w, {lo, hi}; shr.u64 w, w, rb; cvt.u64.u32 v, a; or.b64 w, w, v; "

}  // namespace

// FEAS: feasibility only (Section 4.3, "Feasible"): leaving queries are compared with the objective as
//       they leave, nothing is written to a slab, and a candidate is dropped as soon as more queries
//       have missed the objective than the P99 rule allows.
// CUT:  pipelines with branch points.  A pipeline is cut into PARTS, chains of stages without a branch between them
//       (LaneCut, built by the host), and a warp simulates one part of as many candidates as fit: L lanes each.  What
//       passes from one part to the next is a stream in global memory, written once by the last lane of a part and
//       read by the group of lanes that has the next one, which may run in any warp of the launch at the same time:
//         * The producer publishes every few turns how many records are there (a fence, then the count); a consumer
//           reads the count with acquire and copies records to shared memory as a root does with the trace.  A
//           producer never waits for a consumer (streams are whole), and parts are handed out in the order of the
//           pipeline to warps in the order in which they start, so whoever waits waits for a group that runs: every
//           wait ends, and has a bound all the same.  A warp none of whose groups has records to examine sleeps.
//         * Part 0 is the root stage alone, and (where no query leaves there) its groups are ROOT NODES, the distinct configurations of the root
//           among the candidates (some hundred at most: hardware x batch x replicas), so it is simulated once per
//           configuration and not once per candidate.  Its chain is as long as the trace and everything waits for it,
//           so its CTAs have their SM to themselves.
//         * A part that only leaves the pipeline (the rule) needs no memory for its stream: the records come in the
//           region of the candidate's slab row that they go to, and no record leaves before it was examined.
//       Against one group of lanes for the whole tree (each lane as many iterations as the root has records, whatever
//       its branch sees, and a branch step in the loop): 7,001 candidates of a tree of 6, 199,999 queries 66 -> 33 ms;
//       8,192, feasibility only, 100,000 queries 34.9 -> 19.4 ms; the covering candidates of a sweep over a tree of 8 17.4 -> 14.5
//       ms; fan-out, 2,048 candidates of 6 stages, 100,000 queries 21.7 -> 15.7 ms.  Up to a warp per scheduler the root is
//       what takes the time (250 to 265 cycles an iteration with its turns), beyond that the ALU pipe.
// FORK: fan-out (with CUT) -- a query goes down every edge whose condition holds, a copy that finds none leaves, and
//       the slab keeps per query the record of the copy that left last.  Joins: the streams of a stage's two incoming edges
//       are merged by a part of its own (lane_merge) before the part that begins with the stage.
template <bool FEAS, bool CUT, bool FORK>
__device__ __forceinline__ void lane_simulation(const DesParams &p, const LaneCut &cut, unsigned char *smem_raw)
{
    // A stream record is (time << q) | low part; the low part is the query index, below the query's
    // branch bits when the records carry them (rb > 0: no stage then looks the bits up).  Keys of batches
    // use the same q, with the index of the batch's first arrival in the low part.
    const int qi = p.qbits, rb = CUT ? p.rec_bits : 0;
    const int q = qi + rb;
    const uint32_t qmask = (1u << q) - 1u, imask = (1u << qi) - 1u;      // q <= 31
    const uint32_t tick = 1u << q;

    const unsigned full = 0xffffffffu;
    const int wid = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int kr = p.lane_slots == 16 ? 16 : 32;      // batch ring positions of a lane
    const int rowlen = p.Bmax | 1;
    uint32_t smem_bytes;
    asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(smem_bytes));
    const uint32_t smem_end = (uint32_t)__cvta_generic_to_shared(smem_raw) + smem_bytes;
    smem_raw += p.smem_skip;
    const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(smem_raw);
    const uint32_t tab0 = sbase + 4u;
    const uint32_t rings = (sbase + (uint32_t)table_bytes(p.S * p.H, p.Bmax) + key_bytes(kr) - 1u) & ~(key_bytes(kr) - 1u);
    // words of examined records a lane keeps in shared memory: half of what was planned where the rings start later than
    // planned (they are at most 8 KB late, and half of the fewest words, 64 for each of 128 lanes, are 16 KB)
    auto end_with = [&](int words) { return rings + (uint32_t)(ring_bytes(kr, words, p.lane_stretch) + kTailBytes); };
    const uint32_t nq = (uint32_t)p.lane_words >> (end_with(p.lane_words) > smem_end ? 1 : 0);
    if (end_with((int)nq) > smem_end) { atomicCAS(p.status, 0, IL_ERR_CUDA); return; }      // launched with less than planned
    const uint32_t kbw = rings + (uint32_t)wid * key_bytes(kr), kb = kbw + (uint32_t)lane * 8u;
    const uint32_t xb0 = rings + kLaneWarps * key_bytes(kr);
    const uint32_t xbw = xb0 + (uint32_t)wid * kXBytes, xb = xbw + (uint32_t)lane * 8u;
    const uint32_t nowhere = xb0 + kLaneWarps * kXBytes;
    const uint32_t qb0 = nowhere + (uint32_t)kTailBytes;
    const uint32_t qb = qb0 + (uint32_t)wid * nq * 128u + (uint32_t)lane * 4u;
    const uint32_t tbw = qb0 + kLaneWarps * nq * 128u + (uint32_t)(wid * p.lane_stretch);     // the warp's stretches of arrival streams
    const uint32_t ahead = (uint32_t)p.lane_ahead;
    unsigned *missw = reinterpret_cast<unsigned *>(smem_raw + (nowhere - sbase) + 256u + (uint32_t)wid * 128u);   // per group
    const uint32_t rm = (uint32_t)(kr - 1) << 8;      // ring counters epos, lpos, tpos count in bytes of a row

    // Cut pipelines: a CTA that is the first on its SM may take that SM for root nodes; as many others that come there as are planned leave.
    uint32_t root_warps = 1u;
    bool for_roots = false;
    (void)root_warps; (void)for_roots;
    if (CUT && cut.shared) {
        const uint32_t nodes = cut.ctl[kCtlNodes];
        const uint32_t root_sms = root_sms_for(nodes, (uint32_t)cut.num_sms);
        root_warps = root_sms * kLaneWarps;
        if (threadIdx.x == 0) missw[0] = lane_cta_role(cut, root_sms);
        __syncthreads();
        const unsigned role = *reinterpret_cast<unsigned *>(smem_raw + (nowhere - sbase) + 256u);
        __syncthreads();
        if (role == kRoleNone) return;
        for_roots = role == kRoleRoots;
    }

    for (int r = threadIdx.x; r < p.S * p.H * p.Bmax; r += kLaneWarps * 32)
        sts32(tab0 + (uint32_t)(r / p.Bmax * rowlen + r % p.Bmax) * 4u, (uint32_t)p.lat[r]);
    if (threadIdx.x < 32) sts64(nowhere + (uint32_t)lane * 8u, kInf);
    if (threadIdx.x == 0) sts32(sbase, 0u);
    __syncthreads();

    const uint32_t gmask = (uint32_t)((1ull << p.lane_ring_log2) - 1ull);
    const int64_t wslot = (int64_t)blockIdx.x * kLaneWarps + wid;
    uint32_t *spill_ring = reinterpret_cast<uint32_t *>(p.lane_ws) + ((wslot * p.lanes_per_slot + lane) << p.lane_ring_log2);
    // (cut: a group may also wait for records while others of its warp have some)
    const unsigned long long limit =
        (p.iter_limit ? p.iter_limit : (8ull * (unsigned)p.n * (unsigned)(p.S + 1) + 4096ull) * (CUT ? 4ull : 1ull)) / kTurn + 1ull;
    // a spill has to start before a record still needed is overwritten, two turns from now at the latest
    const uint32_t reach = min((uint32_t)(nq - kTurn - 2), gmask - 2u * kTurn);
    // (and a turn may not be so long that it would come too late)
    // (kept from the compiler, which schedules the loop of chains by 5 % worse when it knows where this comes from)
    uint32_t half = ahead / 2u;
    asm volatile("" : "+r"(half));
    const uint32_t long_reach = gmask > 2u * half && nq > half + 2u ? min((uint32_t)(nq - half - 2), gmask - 2u * half) : 0u;
    const int most_kept = (int)min(nq, gmask + 1u) - 4;
    const uint32_t poll = ahead > 64u ? 1u : 3u;       // cut: looks between two at the streams, less one
    (void)poll;
    unsigned long long batches = 0, alg_ops = 0, exits_seen = 0, exits_due = 0;
    unsigned early = 0;          // candidates dropped before the end of the trace (feasibility only)
    unsigned long long naps = p.iter_limit ? p.iter_limit : cut.naps;      // bound on the sleeps of a warp
    uint32_t quit = 0u;          // the launch has failed: nothing more is waited for
    (void)naps; (void)quit;

    int part = CUT ? lane_first_part(cut, for_roots) : 0;
    for (int parts_left = CUT ? cut.n_part : 1; parts_left > 0; parts_left--, part = CUT && part + 1 == cut.n_part ? 0 : part + 1) {
    const LanePart *pt = CUT ? cut.part + part : nullptr;
    if (FORK && pt->len == 0) { lane_merge(p, cut, part, tbw, ahead, qb0 + (uint32_t)wid * nq * 128u, nq / 2u, naps, quit); continue; }
    const int L = CUT ? pt->len : p.S;                // lanes of a candidate
    const bool per_node = CUT && part == 0 && cut.shared;      // the items are root nodes, not candidates
    const uint32_t n_items = per_node ? cut.ctl[kCtlNodes] : (uint32_t)p.n_cand;
    const int groups = !CUT ? p.cpw : per_node ? (int)min((uint32_t)kRootGroups, (n_items + root_warps - 1u) / root_warps) : pt->groups;
    const int j = lane / L, row = lane - j * L;
    const bool lane_used = j < groups;
    const int s = !CUT ? row : pt->stage[lane_used ? row : 0];
    const bool is_first = row == 0 && lane_used, is_last = row == L - 1 && lane_used;

    // static facts of this lane's stage
    const uint32_t n_in = lane_used ? (uint32_t)p.n_s[CUT || row < p.S ? s : 0] : 0u;
    const unsigned group_mask = lane_used ? (((L < 32 ? 1u << L : 0u) - 1u) << (j * L)) : 0u;
    const int root_lane = lane_used ? j * L : 0;
    // arrival stream: the lane's ring, for the first lane of a group its stretch of the trace or of another part's stream.
    // Copies are of aligned pairs, so a stream that starts at an odd record of its row is counted from one.
    const LaneStream *xs_in = CUT && pt->in >= 0 ? cut.stream + pt->in : nullptr;
    const uint32_t odd = CUT && xs_in ? (uint32_t)xs_in->off & 1u : 0u;
    const uint32_t n_first = (CUT ? (uint32_t)p.n_s[pt->stage[0]] : (uint32_t)p.n) + odd;       // where the group's stream ends
    const uint32_t tb = tbw + (uint32_t)(lane_used ? j : 0) * stretch_bytes((int)ahead);
    const uint32_t xin = is_first ? tb : xb, xin_mask = is_first ? ahead - 1u : kX - 1u, xin_row = is_first ? 8u : 256u;
    // the child's stream; at the last stage the row of empty records
    const bool has_child = lane_used && !is_last;
    const uint32_t xa = has_child ? xbw + (uint32_t)(lane + 1) * 8u : nowhere + (uint32_t)lane * 8u;
    const uint32_t xam = has_child ? (kX - 1) * 256u : 0u;
    const uint32_t tail_step = has_child ? 256u : 8u;
    const int down = has_child ? row : -1;            // (a register that the loop compares with zero: a predicate kept through it costs more)
    // cut: the last stage's two ways out, taken by a record where (bits & mask) == want; neither: it leaves
    const int out_kind = CUT ? pt->out_kind : FEAS ? kOutLeaf : kOutOne;
    auto bit_at = [&](int b) { return b >= 0 ? 1u << (rb > 0 ? qi + b : b) : 0u; };      // (rb = 0: bits looked up)
    const bool two = CUT && out_kind >= kOutTwo;
    const uint32_t mask_a = two && is_last ? bit_at(p.cbit_a[s]) : 0u, mask_b = two && is_last && p.child_b[s] >= 0 ? bit_at(p.cbit_b[s]) : 0u;
    const uint32_t want_a = two && is_last ? (p.cval_a[s] ? mask_a : 0u) : ~0u;
    const uint32_t want_b = two && is_last && p.child_b[s] >= 0 ? (p.cval_b[s] ? mask_b : 0u) : ~0u;
    const uint32_t looks_up = two && is_last && rb == 0 ? mask_a | mask_b : 0u;
    const uint32_t room_a = CUT ? (uint32_t)(pt->out_a >= 0 ? cut.stream[pt->out_a].len : pt->n_leave) : (uint32_t)p.n;     // records its way a holds
    const uint64_t *trace = rb > 0 ? p.ptrace_b : p.ptrace;
    // either of two streams of the same row: the second one's tail counts from the first one's start
    const uint32_t from_b = CUT && !FORK && out_kind == kOutTwo ? (uint32_t)(cut.stream[pt->out_b].off - cut.stream[pt->out_a].off) * 8u : 0u;
    (void)want_a; (void)want_b; (void)looks_up; (void)from_b; (void)room_a; (void)trace;

    // State of the lane's candidate:
    int64_t c = 0;
    uint32_t node = 0;           // cut: the candidate's root node
    // Yes or no, in one register: kept as bools these would be predicates that live through the loop, of which there are
    // seven in all (chain of 4, one warp per scheduler: 9.4 ms for 6.9).
    enum : uint32_t {
        kHas = 1,                // the group holds a candidate
        kNoMore = 2,             // the group will get no further candidate
        kLive = 4, kBad = 8,     // this lane's stage has records; the candidate's configuration is out of range
        kOver = 16,              // the candidate has been given up
        kStarted = 32,           // a first record has opened a batch
        kSpill = 64,
        kNobody = 128,           // cut: the stream's producer has given up
        kDecided = 256,          // cut, feasibility only: the candidate is decided (a root node: all of its candidates are)
        kFirst = 512, kLastStage = 1024, // first and last stage of the group (always)
    };
    uint32_t is = (lane_used ? 0u : (uint32_t)kNoMore) | (is_first ? (uint32_t)kFirst : 0u) | (is_last ? (uint32_t)kLastStage : 0u);
    uint32_t Rm1 = 0;            // replicas less one, in bytes of a ring row
    uint32_t kfb = nowhere, kfm = 0;         // where the first batch in use is looked up (one replica: kInf, which compares as later)
    uint32_t efull = 0;          // tpos with the batch ring full: epos + its size; epos until a first record has opened a batch
    uint32_t lfull = 0;          // tpos with every replica in use or about to be: lpos + replicas less one
    uint32_t mbm1 = 0;
    uint32_t tab = tab0;         // the lane's row of the tables
    uint64_t *out = nullptr;     // records of the last stage: the stream of way a, or the stage's region of the slab row (fan-out: the row)
    uint64_t *out_b = nullptr, *out_c = nullptr;     // two ways: the stream of way b; where records leave
    uint32_t *count_a = nullptr, *count_b = nullptr; // the streams' published counts
    const uint64_t *src = nullptr;           // the group's arrival stream
    const uint32_t *src_count = nullptr;     // cut: its count
    uint32_t avail = 0;          // records of it that are there
    uint32_t pub_a = 0, pub_b = 0;           // tails published
    uint32_t n_left = 0;         // two ways: queries (fan-out: copies) that have left the pipeline at this lane
    uint32_t n_cur = 0;          // records of the arrival stream; i counts those examined
    uint32_t i = 0;
    uint32_t bm = ~0u;           // size of the open batch less one (~0: none is open)
    uint64_t tk = 0;             // latest dispatch time as (t << q) | qmask
    uint32_t epos = 0, lpos = 0, tpos = 0;   // batch ring: [lpos, tpos) in use by replicas, [epos, tpos) not yet handed on
    uint32_t tpos_seen = 0;      // tpos when batches were last counted
    uint32_t prev = 0;           // low part of record i - 1, with its flag
    uint32_t e_on = 0;           // 1: a batch is being handed on:
    uint64_t e_key = 0;          //   its key
    uint32_t e_idx = 0;          //   the record to hand on next
    uint32_t tail_a = 0, tail_b = 0;         // records handed on: to the child in bytes of a ring row, out in bytes
    uint32_t at1 = kb | rm, at2 = kb | (rm - 256u);          // where the last two batches of the ring are
    uint32_t fed = 0;            // records of its stream requested for the group's first lane
    uint32_t qv = 0;             // low part of the record to hand on (where there is one)
    // No record before low_idx is needed any more once every batch up to low_key has been handed on (next_*: the
    // same for a later moment)
    uint32_t low = 0, next_idx = 0;
    uint64_t next_key = 0;
    unsigned nb = 0;
    uint32_t turns = 1, turns_hi = 0;        // iteration bound, in turns
    uint32_t look = 0;
    bool any_spill = false;
    // feasibility only: finish and deadline of a query that has just left, of every other iteration
    uint64_t late_fin[2] = {0, 0}, late_arr[2] = {kLatest, kLatest};
    uint32_t miss_local = 0;
    (void)node; (void)avail; (void)pub_a; (void)pub_b; (void)src_count; (void)look;

    __syncwarp();
    for (int k = 0; k < kX; k++) sts64(xb + (uint32_t)k * 256u, kInf);       // lanes without a stage see no record either
    sts64(at1, 0ull); sts64(at2, 0ull);
    __syncwarp();

    auto test_late = [&]() {
        for (int k = 0; k < 2; k++) {
            miss_local += late_fin[k] > late_arr[k] ? 1u : 0u;
            late_arr[k] = kLatest;
        }
    };
    // cut, feasibility only: misses seen by this lane are added to the candidate's; whoever passes the limit decides it
    auto set = [&](uint32_t bit, bool yes) { is = yes ? is | bit : is & ~bit; };
    auto count_misses = [&]() {
        const uint32_t before = atomicAdd(cut.miss + c, miss_local);
        if (before <= p.miss_allow && before + miss_local > p.miss_allow) {
            p.out_feasible[c] = 0;
            early += i < n_cur ? 1u : 0u;
        }
        if (before + miss_local > p.miss_allow) is |= kDecided;
        miss_local = 0;
    };

    for (;;) {
        // ---- every turn of 8 to 62 iterations: does a lane need more than its steps?  A stream at its start or its end, a
        // candidate that is decided, records in reach of being overwritten, the iteration bound.  (Kept short: its
        // latency is on the chain of every iteration, a kTurn-th of it.)
        if (FEAS) test_late();
        if (FEAS && !CUT && miss_local) { atomicAdd(missw + j, miss_local); miss_local = 0; }
        if (FEAS && CUT && miss_local && (look & 3u) == 0u) count_misses();
        nb += (tpos - tpos_seen) >> 8;
        tpos_seen = tpos;
        // Records before `low` are not needed any more.  Cheap and late: all batches closed when next_idx was the
        // open batch's first record have been handed on once the front of the ring is beyond the largest key of
        // that moment.
        const uint64_t fk = epos != tpos ? lds64(kb | (epos & rm)) : kInf;
        const uint64_t lk = lds64(kb | ((tpos - 256u) & rm));
        if (fk > next_key) {
            low = e_on != 0u ? min(next_idx, e_idx) : next_idx;
            next_idx = i - (bm + 1u);
            next_key = lk;
        }
        copies_done();
        __syncwarp();
        turns--;
        // A stage whose first record is late (few queries visit it, or none until late in the trace), or whose last one has
        // long passed, needs nothing until that record comes or the group's root is at the end of the trace.  (With a look at it
        // in every turn, and short turns until it had started: chain of 4 whose branch is first taken 20 queries before
        // the end of 50,000, one warp per scheduler, 11.0 ms; 8.9 now, 8.7 where half of the queries take the branch.)
        const bool waits = i != n_cur && !(is & kStarted);
        const bool starts = waits && (int)lds32_shared(xin + (i & xin_mask) * xin_row + 4u) >= 0, closes = i == n_cur && bm != ~0u;
        bool attn = !(is & kNoMore) && (starts || closes || turns == 0u || (row == 0 && i == n_cur));
        attn |= i - low > reach || (is & kSpill);
        if (FEAS && !CUT) attn |= (is & kHas) && missw[j] > p.miss_allow;
        if (CUT) attn |= (is & kHas) && ((is & kNobody) || (is & kDecided) || quit);
        if (__any_sync(full, attn)) {
        bool done = i == n_cur && bm == ~0u && epos == tpos && e_on == 0u;
        bool stop = FEAS && !CUT && (is & kHas) && missw[j] > p.miss_allow;       // this lane ends its group's candidate here
        if (CUT) stop = (is & kHas) && ((is & kNobody) || (is & kDecided) || quit);
        bool give_up = false;
        if (i - low > reach || (is & kSpill)) {
            // the oldest record still needed, exactly
            low = i - (bm + 1u);
            if (e_on) low = min(low, e_idx);
#pragma unroll 1
            for (uint32_t k = epos; k != tpos; k += 256u) low = min(low, (uint32_t)lds64(kb | (k & rm)) & qmask);
            const uint32_t span = i - low;
            if (!(is & kSpill) && span > (uint32_t)(nq - kTurn - 2)) {
#pragma unroll 1
                for (uint32_t k = low; k != i; k++)
                    if (IL_IN_RANGE(k & gmask, gmask + 1ull, p.status))
                        spill_ring[k & gmask] = lds32(qb + ((k & (nq - 1u)) << 7));
                is |= kSpill;
            } else if ((is & kSpill) && span < nq / 2u) {
                is &= ~(uint32_t)kSpill;
            }
            give_up |= p.lane_wrap && span + 2u * kTurn > gmask;
        }
        if (turns == 0u && !done) {
            turns = ~0u;
            if (turns_hi-- == 0u) {
                atomicCAS(p.status, 0, IL_ERR_ITER_LIMIT);
                atomicOr(&p.counters[5], 1ull);
                stop = true;
            }
        }
        stop = (__ballot_sync(full, stop) & group_mask) != 0u;                // the whole group
        if (FEAS && CUT) set(kDecided, (__ballot_sync(full, (is & kDecided)) & group_mask) != 0u);
        // (behind the vote: a producer also ends early because the candidate is decided, which the first lane alone has looked up)
        if (CUT) give_up = (give_up || ((is & kHas) && (is & kNobody))) && !(is & kDecided);
        if (p.lane_wrap) {
            const bool group_gives_up = (__ballot_sync(full, give_up) & group_mask) != 0u;
            if (group_gives_up && !(is & kOver)) { is |= kOver; if ((is & kHas) && !per_node) p.ovf[c] = 1; }
            stop |= group_gives_up;
        }
        if (stop) {
            n_cur = i; bm = ~0u; epos = tpos; efull = tpos; e_on = 0u; late_arr[0] = kLatest; late_arr[1] = kLatest; is &= ~(uint32_t)kStarted;
            done = true;
        }
        // The first record of a stream opens a batch on an unused replica, and the last batch is closed by the
        // end of the stream; both once per candidate, so here and not in every iteration.
        if (!done && !(is & kStarted)) {
            const uint32_t at = xin + (i & xin_mask) * xin_row;
            const uint64_t rec = lds64_shared(at);
            if ((int64_t)rec >= 0) {
                tk = rec | qmask;
                bm = 0; i++;
                prev = (uint32_t)rec & qmask;
                sts32_shared_if(true, at + 4u, ~0u);
                is |= kStarted;
                efull = epos + rm + 256u;
            }
        } else if (!done && i == n_cur && bm != ~0u && tpos != efull) {
            const uint64_t key = ((tk + (uint64_t)lds32(tab + bm * 4u) * tick) & ~(uint64_t)qmask) | (i - 1u - bm);
            uint32_t pos = tpos;
            for (; pos != lpos; pos -= 256u) {
                const uint64_t before = lds64(kb | ((pos - 256u) & rm));
                if (before <= key) break;
                sts64(kb | (pos & rm), before);
            }
            sts64(kb | (pos & rm), key);
            tpos += 256u;
            bm = ~0u;
            tk = kLatest;       // nothing more will be dispatched: every batch may leave
            prev |= kLast;
            sts32(qb + (((i - 1u) & (nq - 1u)) << 7), prev);
            if ((is & kSpill) && IL_IN_RANGE((i - 1u) & gmask, gmask + 1ull, p.status)) spill_ring[(i - 1u) & gmask] = prev;
        }
        const unsigned dm = __ballot_sync(full, done);
        const bool turn = !(is & kNoMore) && (dm & group_mask) == group_mask;
        if (__any_sync(full, turn)) {
            // wrap up the candidate the group has finished
            if (turn && (is & kHas)) {
                if (FEAS && CUT && miss_local && !stop) count_misses();
                if ((is & kLive) && !(is & kOver) && !(CUT && quit != 0u)) {
                    batches += nb;
                    alg_ops += 3ull * n_in + (unsigned long long)nb * ((Rm1 >> 8) + mbm1 + 6u);
                }
                const bool decided = FEAS && (CUT ? (is & kDecided) : missw[j] > p.miss_allow);
                // every record of a group that ran to its end must have come out of its last stage, into a stream or
                // through a leaf (checked over all groups of the warp when the kernel ends)
                if ((is & kLive) && (is & kLastStage) && !stop && !decided) {
                    exits_seen += (unsigned long long)(tail_a >> 3) + (two ? ((tail_b - from_b) >> 3) + n_left : 0u);
                    exits_due += CUT ? (unsigned long long)pt->n_out : (unsigned long long)(unsigned)p.n;
                }
                if (FEAS && !CUT && row == 0) {
                    p.out_feasible[c] = (is & kOver) ? 2 : (decided || (is & kBad) ? 0 : 1);
                    early += (decided && i < n_in) ? 1u : 0u;        // the root had not reached the end of the trace
                }
                if (CUT && (count_a || count_b)) {
                    // all that will come, or that nothing will: then who reads the stream gives up as well
                    __threadfence();
                    const bool ok = !stop && !(is & kBad);
                    if (count_a) stg32_shared(count_a, ok ? tail_a >> 3 : kDead);
                    if (count_b) stg32_shared(count_b, ok ? (tail_b - from_b) >> 3 : kDead);
                }
                if (CUT && FEAS && (is & kFirst) && xs_in && xs_in->by_node && !(is & kBad)) atomicSub(cut.refs + node, 1u);
            }
            __syncwarp();
            // the group's next candidate
            unsigned long long g = 0;
            if (turn && row == 0) g = CUT ? (unsigned long long)atomicAdd(cut.ctl + kCtlWork + part, 1u) : atomicAdd(&p.counters[0], 1ull);
            g = __shfl_sync(full, g, root_lane);
            il_stage_config cfg = {0, 1, 1, 0};
            const bool got = turn && g < n_items && !(CUT && quit != 0u);
            bool bad = false;
            if (CUT) {
                int32_t of = 0;
                if (got && !per_node) of = cut.root_of[g];
                bad = of < 0;
                if (turn) node = per_node ? (uint32_t)g : (uint32_t)max(of, 0);
                if (got && !bad) {
                    if (per_node) {
                        const uint32_t w = cut.node_cfg[g];
                        cfg.hw = (uint8_t)w; cfg.max_batch = (uint8_t)(w >> 8); cfg.replicas = (uint8_t)(w >> 16);
                    } else {
                        cfg = p.configs[g * p.S + s];
                    }
                }
            } else {
                if (got) cfg = p.configs[g * p.S + s];
                bad = got && (cfg.hw >= p.H || cfg.max_batch < 1 || cfg.max_batch > p.Bmax ||
                              cfg.replicas < 1 || cfg.replicas > IL_MAX_REPLICAS);
                bad = (__ballot_sync(full, bad) & group_mask) != 0u;
            }
            if (turn) {
                set(kHas, got);
                set(kNoMore, !got);
                c = (int64_t)g;      // g < n_items whenever the group got a candidate: rows of the slab, the
                set(kBad, bad);      // overflow array and the output exist for it
                is &= ~(uint32_t)kOver;
                if (CUT) {
                    auto row_at = [&](const LaneStream &x) { return x.base + (int64_t)(!got ? 0u : x.by_node ? node : (uint32_t)c) * x.stride + x.off; };
                    auto count_at = [&](const LaneStream &x) { return x.count + (!got ? 0u : x.by_node ? node : (uint32_t)c); };
                    uint64_t *slab = FEAS ? nullptr : reinterpret_cast<uint64_t *>(p.slab + (got && !per_node ? c : 0) * p.slab_stride);
                    out_c = FORK || FEAS ? slab : slab + pt->leave_off;
                    out = out_c;
                    if (pt->out_a >= 0) { out = row_at(cut.stream[pt->out_a]); if ((is & kLastStage)) count_a = count_at(cut.stream[pt->out_a]); }
                    if (pt->out_b >= 0) { out_b = row_at(cut.stream[pt->out_b]); if ((is & kLastStage)) count_b = count_at(cut.stream[pt->out_b]); }
                    src = xs_in ? row_at(*xs_in) - odd : rb > 0 ? p.ptrace_b : p.ptrace;
                    src_count = xs_in ? count_at(*xs_in) : nullptr;
                    avail = xs_in ? odd : n_first;
                    is &= ~(uint32_t)kNobody; is &= ~(uint32_t)kDecided; pub_a = 0; tail_b = from_b; pub_b = tail_b;
                    if (got && (is & kBad) && !FEAS && !FORK)      // (the call fails, but the percentile pass reads the row)
                        for (int k = row; k < pt->n_leave; k += L) out_c[k] = 0;
                } else {
                    uint64_t *slab = FEAS ? nullptr : reinterpret_cast<uint64_t *>(p.slab + (got ? c : 0) * p.slab_stride);
                    if (got && (is & kBad)) {
                        if (row == 0) atomicCAS(p.status, 0, IL_ERR_BAD_CONFIG);
                        if (!FEAS) for (int k = row; k < p.n; k += L) slab[k] = 0;
                    }
                    out = slab;
                    src = p.ptrace;
                    avail = n_first;
                }
                set(kLive, got && !(is & kBad) && n_in > 0);
                Rm1 = (cfg.replicas - 1u) << 8;
                kfb = Rm1 != 0u ? kb : nowhere + (uint32_t)lane * 8u;
                kfm = Rm1 != 0u ? rm : 0u;
                is &= ~(uint32_t)kStarted; efull = 0; lfull = Rm1;
                mbm1 = cfg.max_batch - 1u;
                tab = tab0 + (uint32_t)(((is & kLive) ? s * p.H + cfg.hw : 0) * rowlen) * 4u;
                n_left = 0;
                i = row == 0 ? odd : 0u;
                n_cur = (is & kLive) ? n_in + i : i;
                for (int k = 0; k < kX; k++) sts64(xb + (uint32_t)k * 256u, kInf);
                if (FEAS && !CUT && row == 0) missw[j] = 0u;
                bm = ~0u; tk = 0;
                epos = 0; lpos = 0; tpos = 0; tpos_seen = 0;
                at1 = kb | rm; at2 = kb | (rm - 256u);
                sts64(at1, 0ull); sts64(at2, 0ull);       // (no batch before the first one)
                prev = 0;
                e_on = 0u; e_idx = 0;
                tail_a = 0;
                is &= ~(uint32_t)kSpill; low = i; next_idx = i; next_key = 0;
                nb = 0;
                turns = (uint32_t)limit; turns_hi = (uint32_t)(limit >> 32);
                late_arr[0] = kLatest; late_arr[1] = kLatest; miss_local = 0;
                fed = odd;
                if (row == 0) for (uint32_t k = 0; k < ahead; k++) sts64(tb + k * 8u, kInf);
            }
            __syncwarp();     // the rings are empty before anybody looks
            if (__all_sync(full, (is & kNoMore))) break;
        }
        any_spill = __any_sync(full, (is & kSpill));
        __syncwarp();     // a root's first position is empty before another lane of the group fills it again below
        }

        uint32_t at = __shfl_sync(full, i, root_lane);      // records the group's first lane has examined
        if (CUT) {
            // ---- the streams between the parts: what has been written is published, and what others have written is
            // looked up, every fourth (second where turns are long) turn or when there is nothing to do
            const bool feeds = (is & kHas) && !(is & kBad) && !(is & kNobody) && !(is & kDecided);
            auto short_of = [&](uint32_t records) { return feeds && avail != n_first && avail - at < records; };
            // no group has a turn's records before it: nothing is lost by waiting for the next ones
            const bool idle = !__any_sync(full, (is & kFirst) && (is & kHas) && !short_of(kTurn));
            look++;
            if ((look & poll) == 0u || idle) {
                if (((look & (2u * poll + 1u)) == 0u || idle) && (is & kHas) && ((count_a && tail_a != pub_a) || (count_b && tail_b != pub_b))) {
                    __threadfence();
                    if (count_a) stg32_shared(count_a, tail_a >> 3);
                    if (count_b) stg32_shared(count_b, (tail_b - from_b) >> 3);
                    pub_a = tail_a; pub_b = tail_b;
                }
                if (__any_sync(full, short_of(2u * ahead))) {
                    uint32_t word = 0;
                    if ((is & kFirst) && short_of(2u * ahead)) word = ldg32_acquire(src_count);
                    word = __shfl_sync(full, word, root_lane);
                    __syncwarp();     // (what the first lane has acquired, the others of its group copy)
                    if (short_of(2u * ahead)) { set(kNobody, word == kDead); avail = (is & kNobody) ? avail : max(avail, word + odd); }
                }
                if (FEAS && (is & kFirst) && (is & kHas)) {
                    if (per_node) set(kDecided, ldg32_shared(cut.refs + node) == 0u);
                    else if (!(is & kBad)) if (ldg32_shared(cut.miss + c) > p.miss_allow) is |= kDecided;
                }
            }
            if (idle) {
                if (!__any_sync(full, (is & kFirst) && (is & kHas) && !short_of(kTurn))) {
                    __nanosleep(500);
                    turns++;
                    if (naps-- == 0ull) {
                        atomicCAS(p.status, 0, IL_ERR_ITER_LIMIT);
                        atomicOr(&p.counters[5], 1ull);
                    }
                    quit = __any_sync(full, *reinterpret_cast<volatile int *>(p.status) != 0) ? 1u : 0u;
                    continue;
                }
            }
        }
        // (A stage waits for the next turn to open its first batch and to close its last one.  One that has not started within
        // the first kQuickLooks looks has late records: no short turns for it.  The other lengths are two less than half of what a
        // group has before it: one record of that is missing when the first lane is at an odd one, since copies are of pairs.)
        const bool quick = (i != n_cur && !(is & kStarted) && (uint32_t)limit - turns < kQuickLooks) || (i == n_cur && bm != ~0u);
        const int turn_its = (int)__reduce_min_sync(full, quick ? kQuickTurn : i - low <= long_reach ? (int)half - 2 :
                                                    CUT ? max(kTurn - 2, min((int)half - 2, (most_kept - (int)(i - low)) & ~1)) : kTurn - 2);

        // The group's next records: requested two turns before their use where they are there, by all lanes of the group.
        {
            uint32_t to = (is & kHas) && !(is & kBad) ? min(at + ahead, avail) : 0u;
            if (to != n_first) to &= ~1u;
            // (a stream that starts or ends within a pair)
            if (CUT && (is & kFirst) && to > fed && (fed & 1u)) sts64(tb + (fed & (ahead - 1u)) * 8u, ldg64_shared(src + fed));
            if ((is & kFirst) && to > fed && (to & 1u) && !((fed & 1u) && to == fed + 1u))
                sts64(tb + ((to - 1u) & (ahead - 1u)) * 8u, ldg64_shared(src + (to - 1u)));
            // the first lane can examine turn_its records of what has arrived before; if less has, they are waited for
            const bool near = (is & kFirst) && (is & kHas) && to > fed && fed - at < (uint32_t)turn_its;
            const uint32_t by = 2u * (uint32_t)L;
            uint32_t k = ((fed + 1u) & ~1u) + 2u * (uint32_t)row;
            auto copy_pair = [&](uint32_t at) { copy16(tb + (at & (ahead - 1u)) * 8u, src + at); };
            if constexpr (CUT) {      // (a lane on its own copies sixteen pairs; four a round are independent)
#pragma unroll 1
                for (; k + 3u * by + 1u < to; k += 4u * by) { copy_pair(k); copy_pair(k + by); copy_pair(k + 2u * by); copy_pair(k + 3u * by); }
            }
#pragma unroll 1
            for (; k + 1u < to; k += by) copy_pair(k);
            if (to > fed) fed = to;
            if (__any_sync(full, near)) { copies_done(); __syncwarp(); }
        }

        // One iteration (IL_STEP), in the form that the way out of the group's last stage asks for.
        uint32_t xs = xin + (i & xin_mask) * xin_row, sa = xa | (tail_a & xam);
        uint64_t rec = lds64_shared(xs);                    // record to examine
        uint32_t rw = lds32_shared(sa + 4u);                // where the record in hand goes: empty?
        uint32_t lat = lds32(tab + bm * 4u);                // time of the open batch
        auto step = [&](auto spilling, auto kind, auto turn_of) {
            constexpr bool SPILL = decltype(spilling)::value;
            [[maybe_unused]] constexpr int TURN = decltype(turn_of)::value;
            constexpr int OUT = decltype(kind)::value;
            [[maybe_unused]] uint32_t bits = qv;
            if (OUT == kOutAny && looks_up != 0u && e_on != 0u && IL_IN_RANGE(qv & imask, p.n, p.status)) bits = p.bits[qv & imask];
            [[maybe_unused]] uint32_t leaves = 0u;
            [[maybe_unused]] const uint64_t left_rec = e_key;              // what leaves: key and low part of the record in hand
            [[maybe_unused]] const uint32_t left_low = qv & ~kLast;
            [[maybe_unused]] const uint32_t i_was = i, tpos_was = tpos, prev_was = prev;
#ifdef IL_CHECKED
            if (e_on != 0u && down < 0) {
                bool in = IL_IN_RANGE(qv & imask, p.n, p.status);
                if (OUT != kOutTwo && OUT != kOutAny) {
                    in &= IL_IN_RANGE(tail_a >> 3, room_a, p.status);
                } else {
                    if ((bits & mask_a) == want_a) in &= IL_IN_RANGE(tail_a >> 3, room_a, p.status);
                    if ((bits & mask_b) == want_b) in &= IL_IN_RANGE((tail_b - from_b) >> 3, cut.stream[pt->out_b].len, p.status);
                }
                if (!in) e_on = 0u;
            }
#endif
            if constexpr (OUT == kOutOne) {
                asm volatile(IL_STEP("", IL_STEP_INPUTS(21, 22, 23, 24, 25, 26, 27, 28, 29, 30, 31, 32, 33, 34, 35, 36, 37) IL_LOAD(b32, tail_step, 38) IL_LOAD(b64, out, 39),
                                     ".reg .b64 o;\n", IL_ONE_TAIL,
                                     "mad.wide.u32 o, ta_was, 1, out; @ho st.global.b64 [o], v;\n",
                                     IL_DEEPER_LANE, "")
                             : IL_STATE_OPERANDS
                             : IL_INPUT_OPERANDS, "r"(tail_step), "l"(out)
                             : "memory");
            } else if constexpr (OUT == kOutLeaf && FEAS) {
                // (compared with its deadline two iterations later, when that has come)
                asm volatile(IL_STEP(IL_LOAD(b64, late_arr, 22) IL_LOAD(b64, late_fin, 21) IL_LOAD(b32, nobody, 44) IL_LOAD(b32, line, 23),
                                     IL_STEP_INPUTS(24, 25, 26, 27, 28, 29, 30, 31, 32, 33, 34, 35, 36, 37, 38, 39, 40) IL_LOAD(b32, tail_step, 41) IL_LOAD(b64, trace, 42)
                                     IL_LOAD(b32, imask, 43),
                                     ".reg .pred nl; .reg .b64 o;\n", IL_ONE_TAIL,
                                     "setp.gt.f64 nl, late_fin, late_arr; @nl add.u32 line, line, 1; mov.b64 late_fin, {lo, hi};\n"
                                     "and.b32 a, x, imask; selp.b32 a, a, nobody, ho; mad.wide.u32 o, a, 8, trace; ld.global.nc.b64 late_arr, [o];\n",
                                     IL_DEEPER_WARP, IL_STORE(b64, late_fin, 21) IL_STORE(b64, late_arr, 22) IL_STORE(b32, line, 23))
                             : IL_STATE_OPERANDS, "+l"(late_fin[TURN]), "+l"(late_arr[TURN]), "+r"(miss_local)
                             : IL_INPUT_OPERANDS, "r"(tail_step), "l"(p.deadline), "r"(imask), "r"((uint32_t)p.n)
                             : "memory");
            } else if constexpr (OUT == kOutLeaf && FORK) {
                // (several copies of a query may leave: the slab keeps the last one's record)
                asm volatile(IL_STEP("", IL_STEP_INPUTS(21, 22, 23, 24, 25, 26, 27, 28, 29, 30, 31, 32, 33, 34, 35, 36, 37) IL_LOAD(b32, tail_step, 38) IL_LOAD(b64, out, 39)
                                     IL_LOAD(b32, imask, 40) IL_LOAD(b32, rb, 41),
                                     ".reg .b64 o, w;\n", IL_ONE_TAIL,
                                     "and.b32 a, x, imask; mad.wide.u32 o, a, 8, out;\n" IL_PLAIN_RECORD "@ho red.relaxed.gpu.global.max.u64 [o], w;\n",
                                     IL_DEEPER_WARP, "")
                             : IL_STATE_OPERANDS
                             : IL_INPUT_OPERANDS, "r"(tail_step), "l"(out_c), "r"(imask), "r"(rb)
                             : "memory");
            } else if constexpr (OUT == kOutLeaf) {
                asm volatile(IL_STEP("", IL_STEP_INPUTS(21, 22, 23, 24, 25, 26, 27, 28, 29, 30, 31, 32, 33, 34, 35, 36, 37) IL_LOAD(b32, tail_step, 38) IL_LOAD(b64, out, 39)
                                     IL_LOAD(b32, imask, 40) IL_LOAD(b32, rb, 41),
                                     ".reg .b64 o, w;\n", IL_ONE_TAIL,
                                     "mad.wide.u32 o, ta_was, 1, out;\n" "and.b32 a, x, imask; " IL_PLAIN_RECORD "@ho st.global.b64 [o], w;\n",
                                     IL_DEEPER_LANE, "")
                             : IL_STATE_OPERANDS
                             : IL_INPUT_OPERANDS, "r"(tail_step), "l"(out), "r"(imask), "r"(rb)
                             : "memory");
            } else if constexpr (OUT == kOutTwo && FORK) {
                // (a record goes down every way whose condition holds)
                asm volatile(IL_STEP(IL_LOAD(b32, tail_b, 21),
                                     IL_STEP_INPUTS(22, 23, 24, 25, 26, 27, 28, 29, 30, 31, 32, 33, 34, 35, 36, 37, 38) IL_LOAD(b32, mask_a, 39) IL_LOAD(b32, mask_b, 40)
                                     IL_LOAD(b32, want_a, 41) IL_LOAD(b32, want_b, 42) IL_LOAD(b64, out, 43) IL_LOAD(b64, out_b, 44),
                                     ".reg .pred ga, gb; .reg .b64 o; .reg .u32 ma, mb;\n",
                                     "and.b32 ma, qv, mask_a; and.b32 mb, qv, mask_b;\n"
                                     "setp.eq.and.u32 ga, ma, want_a, ho; setp.eq.and.u32 gb, mb, want_b, ho;\n"
                                     "@hd add.u32 tail_a, tail_a, 256; @ga add.u32 tail_a, tail_a, 8;\n",
                                     "mad.wide.u32 o, ta_was, 1, out; @ga st.global.b64 [o], v; mad.wide.u32 o, tail_b, 1, out_b; @gb st.global.b64 [o], v; @gb add.u32 tail_b, tail_b, 8;\n",
                                     IL_DEEPER_WARP, IL_STORE(b32, tail_b, 21))
                             : IL_STATE_OPERANDS, "+r"(tail_b)
                             : IL_INPUT_OPERANDS, "r"(mask_a), "r"(mask_b), "r"(want_a), "r"(want_b), "l"(out), "l"(out_b)
                             : "memory");
            } else if constexpr (OUT == kOutTwo) {
                // (either way: one store; way b's tail counts from where way a's stream starts)
                asm volatile(IL_STEP(IL_LOAD(b32, tail_b, 21),
                                     IL_STEP_INPUTS(22, 23, 24, 25, 26, 27, 28, 29, 30, 31, 32, 33, 34, 35, 36, 37, 38) IL_LOAD(b32, mask_a, 39) IL_LOAD(b32, want_a, 40)
                                     IL_LOAD(b64, out, 41),
                                     ".reg .pred ga, gb; .reg .b64 o; .reg .u32 ma, tt;\n",
                                     "and.b32 ma, qv, mask_a; setp.eq.and.u32 ga|gb, ma, want_a, ho; selp.b32 tt, tail_a, tail_b, ga;\n"
                                     "@hd add.u32 tail_a, tail_a, 256; @ga add.u32 tail_a, tail_a, 8; @gb add.u32 tail_b, tail_b, 8;\n",
                                     "mad.wide.u32 o, tt, 1, out; @ho st.global.b64 [o], v;\n",
                                     IL_DEEPER_LANE, IL_STORE(b32, tail_b, 21))
                             : IL_STATE_OPERANDS, "+r"(tail_b)
                             : IL_INPUT_OPERANDS, "r"(mask_a), "r"(want_a), "l"(out)
                             : "memory");
            } else {
                asm volatile(IL_STEP(IL_LOAD(b32, tail_b, 21) ".reg .b32 leaves;\n",
                                     IL_STEP_INPUTS(23, 24, 25, 26, 27, 28, 29, 30, 31, 32, 33, 34, 35, 36, 37, 38, 39) IL_LOAD(b32, bits, 40) IL_LOAD(b32, mask_a, 41)
                                     IL_LOAD(b32, mask_b, 42) IL_LOAD(b32, want_a, 43) IL_LOAD(b32, want_b, 44) IL_LOAD(b64, out, 45) IL_LOAD(b64, out_b, 46),
                                     ".reg .pred ga, gb, lv; .reg .b64 o; .reg .u32 ma, mb;\n",
                                     "and.b32 ma, bits, mask_a; and.b32 mb, bits, mask_b;\n"
                                     "setp.eq.and.u32 ga|lv, ma, want_a, ho; setp.eq.and.u32 gb, mb, want_b, ho; setp.ne.and.u32 lv, mb, want_b, lv;\n"
                                     "@hd add.u32 tail_a, tail_a, 256; @ga add.u32 tail_a, tail_a, 8;\n",
                                     "mad.wide.u32 o, ta_was, 1, out; @ga st.global.b64 [o], v; mad.wide.u32 o, tail_b, 1, out_b; @gb st.global.b64 [o], v;\n"
                                     "@gb add.u32 tail_b, tail_b, 8; selp.u32 leaves, 1, 0, lv;\n",
                                     IL_DEEPER_LANE, IL_STORE(b32, tail_b, 21) IL_STORE(b32, leaves, 22))
                             : IL_STATE_OPERANDS, "+r"(tail_b), "=r"(leaves)
                             : IL_INPUT_OPERANDS, "r"(bits), "r"(mask_a), "r"(mask_b), "r"(want_a), "r"(want_b), "l"(out), "l"(out_b)
                             : "memory");
                if (FEAS) test_late();
                if (pt->n_leave > 0 && leaves != 0u) {
                    // (a branch point at which some queries leave)
                    const uint32_t qid = left_low & imask;
                    const uint64_t fin = left_rec & ~(uint64_t)qmask;
                    if (FEAS) {
                        late_fin[0] = fin;
                        late_arr[0] = __ldg(p.deadline + qid);
                    } else if (FORK) {
                        atomicMax(reinterpret_cast<unsigned long long *>(out_c) + qid, (fin >> rb) | qid);
                    } else if (IL_IN_RANGE(n_left, pt->n_leave, p.status)) {
                        out_c[n_left] = (fin >> rb) | qid;
                    }
                    n_left++;
                }
            }
            if (SPILL) {
                // (the lane's own stores, so the words may come through L1: 32 of them with one miss)
                ldg32_if((is & kSpill) && i - e_idx > nq && IL_IN_RANGE(e_idx & gmask, gmask + 1ull, p.status), spill_ring + (e_idx & gmask), qv);
                stg32_if((is & kSpill) && i != i_was && IL_IN_RANGE((i_was - 1u) & gmask, gmask + 1ull, p.status),
                         spill_ring + ((i_was - 1u) & gmask), prev_was | (tpos != tpos_was ? kLast : 0u));
            }
        };
        auto run_turn = [&](auto kind) {
            if (any_spill) {
#pragma unroll 1
                for (int k = 0; k < turn_its; k++) step(std::true_type{}, kind, std::integral_constant<int, 0>{});
            } else {
#pragma unroll 1
                for (int k = 0; k < turn_its; k += 2) { step(std::false_type{}, kind, std::integral_constant<int, 0>{}); step(std::false_type{}, kind, std::integral_constant<int, 1>{}); }
            }
        };
        using One = std::integral_constant<int, kOutOne>;
        using Leaf = std::integral_constant<int, kOutLeaf>;
        using Two = std::integral_constant<int, kOutTwo>;
        using Any = std::integral_constant<int, kOutAny>;
        if (!CUT) run_turn(std::integral_constant<int, FEAS ? kOutLeaf : kOutOne>{});
        else if (out_kind == kOutOne) run_turn(One{});
        else if (out_kind == kOutLeaf) run_turn(Leaf{});
        else if (out_kind == kOutTwo) run_turn(Two{});
        else run_turn(Any{});
    }
    }

    for (int o = 16; o > 0; o >>= 1) {
        batches += __shfl_xor_sync(full, batches, o);
        alg_ops += __shfl_xor_sync(full, alg_ops, o);
        exits_seen += __shfl_xor_sync(full, exits_seen, o);
        exits_due += __shfl_xor_sync(full, exits_due, o);
    }
    if (lane == 0 && exits_seen != exits_due) { atomicCAS(p.status, 0, IL_ERR_ITER_LIMIT); atomicOr(&p.counters[5], 2ull); }
    if (lane == 0 && batches) { atomicAdd(&p.counters[1], batches); atomicAdd(&p.counters[2], alg_ops); }
    if (FEAS) {
        for (int o = 16; o > 0; o >>= 1) early += __shfl_xor_sync(full, early, o);
        if (lane == 0 && early) atomicAdd(&p.counters[6], (unsigned long long)early);
    }
}

// Pipelines that are chains: one group of lanes per candidate.
template <bool FEAS>
__global__ void __launch_bounds__(kLaneWarps * 32, 3) des_lane_kernel(const __grid_constant__ DesParams p)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    lane_simulation<FEAS, false, false>(p, LaneCut(), smem_raw);
}

// Pipelines cut at their branch points.
template <bool FEAS, bool FORK>
__global__ void __launch_bounds__(kLaneWarps * 32, 2) des_part_kernel(const __grid_constant__ DesParams p, const __grid_constant__ LaneCut cut)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    lane_simulation<FEAS, true, FORK>(p, cut, smem_raw);
}

namespace {

// Feasibility only: per query the latest record time at which it still meets the objective, compared as records are;
// behind the last one, for lanes that have nothing to compare, a time that none exceeds.
__global__ void __launch_bounds__(256) deadline_kernel(const uint64_t *trace, int n, uint64_t slo, uint32_t qmask, uint64_t *out)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i <= n; i += gridDim.x * blockDim.x)
        out[i] = i < n ? min((unsigned long long)((trace[i] | qmask) + slo), (unsigned long long)kLatest) : kLatest;
}

// Root nodes of a chunk: the distinct (hardware, batch, replicas) of stage 0 among its candidates, numbered, each with how
// many groups will read its streams; every candidate's node, -1 where a configuration is out of range.  One CTA: a bit per
// configuration in shared memory (a word per hardware and batch), a prefix sum over the words, and the numbers read back.
constexpr int kNodeThreads = 1024;
__global__ void __launch_bounds__(kNodeThreads) root_nodes_kernel(const RootNodeParams p)
{
    __shared__ uint32_t seen[IL_MAX_HW * IL_MAX_BATCH], first[IL_MAX_HW * IL_MAX_BATCH], sums[32];
    const int t = threadIdx.x, words = p.H * p.Bmax;
    for (int w = t; w < words; w += kNodeThreads) seen[w] = 0u;
    __syncthreads();
    for (int64_t c = t; c < p.n_cand; c += kNodeThreads) {
        bool ok = true;
        for (int s = 0; s < p.S; s++) {
            const il_stage_config k = p.configs[c * p.S + s];
            ok &= k.hw < p.H && k.max_batch >= 1 && k.max_batch <= p.Bmax && k.replicas >= 1 && k.replicas <= IL_MAX_REPLICAS;
        }
        const il_stage_config k = p.configs[c * p.S];
        if (ok) atomicOr(&seen[k.hw * p.Bmax + k.max_batch - 1], 1u << (k.replicas - 1));
        else atomicCAS(p.status, 0, IL_ERR_BAD_CONFIG);
        p.root_of[c] = ok ? (p.shared ? 0 : (int32_t)c) : -1;
        if (ok && !p.shared && p.out_feasible) p.refs[c] = (uint32_t)p.readers;
        if (p.out_feasible) { p.out_feasible[c] = ok ? 1 : 0; p.miss[c] = 0u; }
    }
    if (!p.shared) return;
    __syncthreads();
    // (IL_MAX_HW * IL_MAX_BATCH <= kNodeThreads: a word per thread)
    const uint32_t mine = t < words ? (uint32_t)__popc(seen[t]) : 0u;
    uint32_t upto = mine;
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_up_sync(0xffffffffu, upto, o);
        if ((t & 31) >= o) upto += v;
    }
    if ((t & 31) == 31) sums[t >> 5] = upto;
    __syncthreads();
    uint32_t base = 0, all = 0;
    for (int k = 0; k < kNodeThreads / 32; k++) { base += k < (t >> 5) ? sums[k] : 0u; all += sums[k]; }
    if (t < words) {
        first[t] = base + upto - mine;
        uint32_t at = first[t];
        for (uint32_t m = seen[t]; m != 0u; m &= m - 1u)
            p.node_cfg[at++] = (uint32_t)(t / p.Bmax) | (uint32_t)(t % p.Bmax + 1) << 8 | (uint32_t)__ffs((int)m) << 16;
    }
    if (t == 0) p.ctl[kCtlNodes] = all;
    __syncthreads();
    for (int64_t c = t; c < p.n_cand; c += kNodeThreads) {
        if (p.root_of[c] < 0) continue;
        const il_stage_config k = p.configs[c * p.S];
        const int w = k.hw * p.Bmax + k.max_batch - 1;
        const uint32_t at = first[w] + (uint32_t)__popc(seen[w] & ((1u << (k.replicas - 1)) - 1u));
        p.root_of[c] = (int32_t)at;
        if (p.out_feasible) atomicAdd(p.refs + at, (uint32_t)p.readers);
    }
}

template <typename K, typename... A>
cudaError_t launch_one(K kernel, int grid, size_t smem, size_t smem_most, cudaStream_t stream, const A &...args)
{
    cudaError_t e = allow_smem(kernel, smem_most);      // (these kernels have no static shared memory)
    if (e != cudaSuccess) return e;
    kernel<<<grid, kLaneWarps * 32, smem, stream>>>(args...);
    return cudaGetLastError();
}
}  // namespace

cudaError_t launch_deadlines(const DesParams &p, uint64_t *out, cudaStream_t stream)
{
    const int q = p.qbits + p.rec_bits, grid = std::min((p.n + 256) / 256, 592);
    deadline_kernel<<<grid, 256, 0, stream>>>(p.rec_bits > 0 ? p.ptrace_b : p.ptrace, p.n, (uint64_t)p.slo_us << q, (uint32_t)((1ull << q) - 1ull), out);
    return cudaGetLastError();
}

cudaError_t launch_root_nodes(const RootNodeParams &p, cudaStream_t stream)
{
    root_nodes_kernel<<<1, kNodeThreads, 0, stream>>>(p);
    return cudaGetLastError();
}

// Feasibility-only when p.out_feasible is set; cut: the pipeline's parts, nullptr for a chain.  (The host never combines
// fan-out with feasibility-only, nor with spill rings shorter than the longest stream.)
cudaError_t launch_des_lane(const DesParams &p, const LaneCut *cut, int grid, size_t smem, size_t smem_most, cudaStream_t stream)
{
    if (!cut)
        return p.out_feasible ? launch_one(des_lane_kernel<true>, grid, smem, smem_most, stream, p) : launch_one(des_lane_kernel<false>, grid, smem, smem_most, stream, p);
    if (p.fork) {
        if (p.lane_wrap || p.out_feasible) return cudaErrorInvalidValue;
        return launch_one(des_part_kernel<false, true>, grid, smem, smem_most, stream, p, *cut);
    }
    return p.out_feasible ? launch_one(des_part_kernel<true, false>, grid, smem, smem_most, stream, p, *cut)
                          : launch_one(des_part_kernel<false, false>, grid, smem, smem_most, stream, p, *cut);
}

int des_lane_warps_per_cta() { return kLaneWarps; }
int lane_root_sms(int64_t nodes, int num_sms) { return (int)root_sms_for((uint32_t)std::min<int64_t>(nodes, 1 << 20), (uint32_t)num_sms); }
int lane_stretch_bytes(int groups, int ahead) { return groups * (int)stretch_bytes(ahead); }

size_t des_lane_smem(int table_rows, int Bmax, int ring_slots, int ring_words, int stretch)
{
    return (kSmemBase + table_bytes(table_rows, Bmax) + key_bytes(ring_slots) - 1) / key_bytes(ring_slots) * key_bytes(ring_slots) -
           kSmemBase + ring_bytes(ring_slots, ring_words, stretch) + kTailBytes;
}

int des_lane_max_ctas_per_sm(size_t smem, size_t smem_most, bool cut)
{
    int n = 0;
    // (all instantiations of one kind are compiled for the same number of CTAs)
    auto ask = [&](auto kernel) {
        if (allow_smem(kernel, smem_most) != cudaSuccess) { cudaGetLastError(); return 0; }
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, kLaneWarps * 32, smem) == cudaSuccess ? n : 0;
    };
    return cut ? ask(des_part_kernel<true, false>) : ask(des_lane_kernel<true>);
}

}  // namespace il
