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
//   * A root's records are copied to shared memory at least one turn (below)
//     before their use (cp.async, all lanes of the group).
//   * The profile tables are shared by the CTA, rows padded to an odd length so
//     that rows of different lanes start in different banks.
//   * What happens once per candidate or rarely (its first and last batch, spills,
//     the iteration bound, the next candidate) is looked at once a turn of 8, 16 or
//     32 iterations only, behind one vote.
//
// Measured on B200 against the version whose streams lay in global memory (three
// gathers of 8 bytes per lane and iteration through L1, 208 instructions): about
// 120 instructions per iteration and 115 instead of 290 ns for a warp on its own;
// 4,096 candidates x 4 stages x 50,000 queries 15.4 -> 6.3 ms, 4,096 x 10 x 10^6
// 720 -> 330 ms.  With two or three warps per scheduler the ALU pipe (compares,
// selects and logic, half the issue rate) is what bounds it.  What took the loop
// from 155 to 120 ns: the trace copied ahead of its use by all lanes of a group
// (8 instructions less, no stall on the load), the word to hand on loaded an
// iteration early, comparisons as doubles, one counter per lane for the records
// it passes on.
#include "il_internal.h"

#include <type_traits>

namespace il {

namespace {

constexpr int kLaneWarps = 4;                 // warps per CTA: one per scheduler even in a grid of few CTAs
constexpr uint64_t kInf = ~0ull;
constexpr uint64_t kLatest = 0x7fefffffffffffffull;      // no record or key is larger
constexpr int kX = 8;                         // records of a stream between two stages
constexpr uint32_t kLast = 0x80000000u;       // flag of a batch's last record in that ring
constexpr int kAhead = 64;                    // records of the trace a root has before it: two long turns, a power of two
constexpr int kTurn = 16, kLongTurn = 32;     // iterations between two looks at finished groups, spills, bounds
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
// Order of two records or keys.  Words below 0x7ff0... order the same as the doubles of their bits, and a double
// is compared by one instruction on a pipe that is idle otherwise, where a 64-bit integer takes two on the ALU pipe
// (5 % of a launch with three warps per scheduler).  A word with the sign or all exponent bits set compares as false.
__device__ __forceinline__ bool before(uint64_t a, uint64_t b) { return __longlong_as_double((long long)a) < __longlong_as_double((long long)b); }
__device__ __forceinline__ bool not_after(uint64_t a, uint64_t b) { return __longlong_as_double((long long)a) <= __longlong_as_double((long long)b); }

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
__device__ __forceinline__ void sts64_shared_if(bool c, uint32_t a, uint64_t v)
{
    asm volatile("{ .reg .pred p; setp.ne.u32 p, %0, 0; @p st.relaxed.cta.shared.u64 [%1], %2; }" ::"r"((uint32_t)c), "r"(a), "l"(v) : "memory");
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
__device__ __forceinline__ void sts32_if(bool c, uint32_t a, uint32_t v)
{
    asm volatile("{ .reg .pred p; setp.ne.u32 p, %0, 0; @p st.shared.u32 [%1], %2; }" ::"r"((uint32_t)c), "r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void stg32_if(bool c, uint32_t *a, uint32_t v)
{
    asm volatile("{ .reg .pred p; setp.ne.u32 p, %0, 0; @p st.global.u32 [%1], %2; }" ::"r"((uint32_t)c), "l"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void ldg32_if(bool c, const uint32_t *a, uint32_t &v)      // leaves v alone otherwise
{
    asm volatile("{ .reg .pred p; setp.ne.u32 p, %1, 0; @p ld.global.ca.u32 %0, [%2]; }" : "+r"(v) : "r"((uint32_t)c), "l"(a) : "memory");
}
__device__ __forceinline__ void stg64_if(bool c, uint64_t *a, uint64_t v)
{
    asm volatile("{ .reg .pred p; setp.ne.u32 p, %0, 0; @p st.global.u64 [%1], %2; }" ::"r"((uint32_t)c), "l"(a), "l"(v) : "memory");
}
// 8 bytes from global to shared memory, asynchronously
__device__ __forceinline__ void copy8(uint32_t dst, const uint64_t *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void copies_done() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Shared memory of a CTA: the tables ([S * H] rows of Bmax | 1 words, one word in front of them), then per warp
// the batch keys [kr][lane] (aligned to their size: a ring address is (counter & mask) | base), per warp the
// streams [kX][lane], a row of empty records (the "child" of a leaf), per warp the miss counts of the groups
// (feasibility only), per warp the words of examined records [nq][lane], and per warp the next records of the trace
// [kAhead][group].
// Where a CTA's dynamic shared memory starts with the toolkit at hand.  The host plans for it; a launch that finds it elsewhere
// needs up to a row of batch keys more to align them and takes it from the words of examined records (more spills).
constexpr uint32_t kSmemBase = 1024;
__host__ __device__ inline uint32_t key_bytes(int kr) { return (uint32_t)kr * 256u; }
constexpr uint32_t kXBytes = kX * 256u;
__host__ __device__ inline size_t table_bytes(int rows, int Bmax) { return ((size_t)rows * (Bmax | 1) + 1) * 4; }
__host__ __device__ inline size_t ring_bytes(int kr, int nq, int cpw)
{
    return (size_t)kLaneWarps * (key_bytes(kr) + nq * 128u + kXBytes + (size_t)kAhead * cpw * 8);
}
constexpr size_t kTailBytes = 256 + kLaneWarps * 128;
constexpr int kSeen = 64;                     // joins: words of the queries' bits that are kept in shared memory
// joins: per warp and per (group, join) the counts and the windows of the two incoming streams, then the cached words
// of the queries' bits with their numbers, then which branch bits follow both edges (256 bits)
__host__ __device__ inline uint32_t join_lane_bytes(int window) { return 2u * (window + 1) * 8u + kSeen * 8u + 32u; }
__host__ __device__ inline size_t join_bytes(int cpw, int joins, int window) { return (size_t)kLaneWarps * cpw * joins * join_lane_bytes(window); }

}  // namespace

// BRANCHY: some stage routes by a branch bit (otherwise every stage has one way out).
// FEAS: feasibility only (Section 4.3, "Feasible"): leaving queries are compared with the objective as
//       they leave, nothing is written to a slab, and a candidate is dropped as soon as more queries
//       have missed the objective than the P99 rule allows.
// FORK: fan-out -- a query goes down every edge whose condition holds, a copy that finds none leaves, and
//       the slab keeps per query the record of the copy that left last (only with BRANCHY, without FEAS).
// JOIN: some stage has two incoming edges (with FORK: a query goes down both before it gets there).  A join has a
//       lane of its own, behind the stages' lanes: it merges the two incoming streams in time order, at equal
//       times the first parent's records first, swallows the record of an input that is not its query's last one
//       (one bit per query and join in global memory: the other input has been seen) and feeds the stage's ring.
//       The incoming streams have no back-pressure -- either parent may have to run ahead of the other by all
//       that the slower branch keeps in flight -- so they go to global memory whole, and the latest
//       64 to 512 records of each to shared memory, from where the join nearly always reads them.  511 candidates
//       of a diamond, 50,000 queries: 130 ms on the warp-per-candidate kernel, 53 ms here.
template <bool BRANCHY, bool FEAS, bool FORK, bool JOIN>
__device__ __forceinline__ void lane_simulation(const DesParams &p, unsigned char *smem_raw)
{
    // A stream record is (time << q) | low part; the low part is the query index, below the query's
    // branch bits when the records carry them (rb > 0: no stage then looks the bits up).  Keys of batches
    // use the same q, with the index of the batch's first arrival in the low part.
    const int qi = p.qbits, rb = BRANCHY ? p.rec_bits : 0;
    const int q = qi + rb;
    const uint32_t qmask = (1u << q) - 1u, imask = (1u << qi) - 1u;      // q <= 31
    const uint32_t tick = 1u << q;
    const uint64_t *trace = rb > 0 ? p.ptrace_b : p.ptrace;

    const unsigned full = 0xffffffffu;
    const int wid = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int kr = p.lane_slots == 16 ? 16 : 32;      // batch ring positions of a lane
    const int S = p.S, cpw = p.cpw, rowlen = p.Bmax | 1;
    const int L = JOIN ? S + p.n_join : S;            // lanes of a candidate
    uint32_t smem_bytes;
    asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(smem_bytes));
    const uint32_t smem_end = (uint32_t)__cvta_generic_to_shared(smem_raw) + smem_bytes;
    smem_raw += p.smem_skip;
    const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(smem_raw);
    const uint32_t tab0 = sbase + 4u;
    const uint32_t rings = (sbase + (uint32_t)table_bytes(S * p.H, p.Bmax) + key_bytes(kr) - 1u) & ~(key_bytes(kr) - 1u);
    // words of examined records a lane keeps in shared memory: half of what was planned where the rings start later than
    // planned (they are at most 8 KB late, and half of the fewest words, 64 for each of 128 lanes, are 16 KB)
    auto end_with = [&](int words) { return rings + (uint32_t)(ring_bytes(kr, words, cpw) + kTailBytes + join_bytes(cpw, p.n_join, p.join_window)); };
    const uint32_t nq = (uint32_t)p.lane_words >> (end_with(p.lane_words) > smem_end ? 1 : 0);
    if (end_with((int)nq) > smem_end) { atomicCAS(p.status, 0, IL_ERR_CUDA); return; }      // launched with less than planned
    const uint32_t kbw = rings + (uint32_t)wid * key_bytes(kr), kb = kbw + (uint32_t)lane * 8u;
    const uint32_t xb0 = rings + kLaneWarps * key_bytes(kr);
    const uint32_t xbw = xb0 + (uint32_t)wid * kXBytes, xb = xbw + (uint32_t)lane * 8u;
    const uint32_t nowhere = xb0 + kLaneWarps * kXBytes;
    const uint32_t qb0 = nowhere + (uint32_t)kTailBytes;
    const uint32_t qb = qb0 + (uint32_t)wid * nq * 128u + (uint32_t)lane * 4u;
    const uint32_t tb0 = qb0 + kLaneWarps * nq * 128u;        // per warp the next records of the trace, [kAhead][group]
    unsigned *missw = reinterpret_cast<unsigned *>(smem_raw + (nowhere - sbase) + 256u + (uint32_t)wid * 128u);   // per group
    const uint32_t rm = (uint32_t)(kr - 1) << 8;      // ring counters epos, lpos, tpos count in bytes of a row

    for (int r = threadIdx.x; r < S * p.H * p.Bmax; r += kLaneWarps * 32)
        sts32(tab0 + (uint32_t)(r / p.Bmax * rowlen + r % p.Bmax) * 4u, (uint32_t)p.lat[r]);
    if (threadIdx.x < 32) sts64(nowhere + (uint32_t)lane * 8u, kInf);
    if (threadIdx.x == 0) sts32(sbase, 0u);
    for (int k = 0; k < kX; k++) sts64(xb + (uint32_t)k * 256u, kInf);       // lanes without a stage see no record either
    __syncthreads();

    const int j = lane / L, row = lane - j * L;
    const bool lane_used = j < cpw;
    const bool is_join = JOIN && lane_used && row >= S;      // a lane that merges the incoming streams of a join
    const int s = JOIN && row >= S ? p.join_stage[row - S] : row;

    // static facts of this lane's stage
    int exit_off = 0;
    for (int u = 0; u < s; u++) {
        const int a = p.dest_a[u], b2 = p.dest_b[u];
        int kids = 0;
        if (a >= 0) kids += p.n_s[a];
        if (b2 >= 0 && b2 != a) kids += p.n_s[b2];
        exit_off += p.n_s[u] - kids;
    }
    const int da = FORK ? p.child_a[s] : p.dest_a[s], db = FORK ? p.child_b[s] : p.dest_b[s];
    // (with fan-out the branch bits are needed if one of the edges is conditional)
    const int bit = FORK ? ((p.cbit_a[s] >= 0 || p.cbit_b[s] >= 0) ? 0 : -1) : p.bit[s];
    // Routing by the bits of a record's low part: without fan-out to side b if (bits & mask_b), with fan-out down
    // either edge if (bits & mask) == want.
    auto bit_at = [&](int b) { return b >= 0 ? 1u << (rb > 0 ? qi + b : b) : 0u; };      // (rb = 0: bits looked up)
    const uint32_t mask_a = FORK && da >= 0 ? bit_at(p.cbit_a[s]) : 0u;
    const uint32_t mask_b = FORK ? (db >= 0 ? bit_at(p.cbit_b[s]) : 0u) : bit_at(p.bit[s]);
    const uint32_t want_a = da < 0 ? ~0u : (p.cval_a[s] ? mask_a : 0u), want_b = db < 0 ? ~0u : (p.cval_b[s] ? mask_b : 0u);
    const uint32_t n_in = lane_used && !is_join ? (uint32_t)p.n_s[s] : 0u;
    const unsigned group_mask = lane_used ? (((1u << L) - 1u) << (j * L)) : 0u;
    const int root_lane = lane_used ? j * L : 0;
    const bool is_root = row == 0;
    // arrival stream: the lane's ring, for a root the group's stretch of the trace
    const uint32_t tb = tb0 + (uint32_t)(wid * kAhead * cpw + (lane_used ? j : 0)) * 8u;
    const bool from_trace = is_root && lane_used;
    const uint32_t xin = from_trace ? tb : xb, xin_mask = from_trace ? kAhead - 1u : kX - 1u, xin_row = from_trace ? (uint32_t)cpw * 8u : 256u;
    // the child's stream on either side; towards the outside (or nowhere) the row of empty records
    const bool join_a = JOIN && da >= 0 && p.join_b[da >= 0 ? da : 0] >= 0, join_b = JOIN && db >= 0 && p.join_b[db >= 0 ? db : 0] >= 0;
    const bool tells_a = join_a && lane_used && !is_join, tells_b = join_b && lane_used && !is_join;     // its records' counts
    const bool has_a = lane_used && !is_join && da >= 0 && !join_a, has_b = BRANCHY && lane_used && !is_join && db >= 0 && !join_b;
    const uint32_t xa = has_a ? xbw + (uint32_t)(j * L + da) * 8u : nowhere + (uint32_t)lane * 8u;
    const uint32_t xc = has_b ? xbw + (uint32_t)(j * L + db) * 8u : nowhere + (uint32_t)lane * 8u;
    const uint32_t xam = has_a ? (kX - 1) * 256u : 0u, xcm = has_b ? (kX - 1) * 256u : 0u;
    const uint32_t tail_step = da >= 0 ? 256u : 8u;
    const uint32_t leaving = (uint32_t)p.n - (uint32_t)exit_off;      // slab entries from this stage's region on
    (void)leaving;

    const int64_t wslot = (int64_t)blockIdx.x * kLaneWarps + wid;
    // joins: where a stage's records for a join go (global stream, window and count in shared memory), and where the
    // join's lane finds them
    const uint32_t jbase = tb0 + (uint32_t)(kLaneWarps * kAhead * cpw) * 8u + (uint32_t)(wid * cpw * p.n_join) * join_lane_bytes(p.join_window);
    uint64_t *jg_a = nullptr, *jg_b = nullptr;
    uint32_t jw_a = nowhere, jw_b = nowhere, seen_cache = nowhere;      // (lanes that are no join's read there, and store nothing)
    uint32_t *seen = nullptr;
    (void)jbase;
    if (JOIN && lane_used) {
        uint64_t *streams = p.join_ws + (wslot * cpw + j) * p.join_elems;
        auto window = [&](int t, int side) {
            return jbase + (uint32_t)(j * p.n_join + p.join_no[t]) * join_lane_bytes(p.join_window) + (uint32_t)side * ((p.join_window + 1u) * 8u);
        };
        auto stream = [&](int t, int side) { return streams + (side ? p.join_lane_b[t] : p.join_lane_a[t]); };
        if (is_join) {
            jg_a = stream(s, 0); jw_a = window(s, 0);
            jg_b = stream(s, 1); jw_b = window(s, 1);
            seen_cache = jw_b + (p.join_window + 1u) * 8u;
            seen = p.join_seen + ((wslot * cpw + j) * p.n_join + (row - S)) * p.join_seen_words;
            for (int k = 0; k < 4; k++) sts64(seen_cache + kSeen * 8u + (uint32_t)k * 8u, p.join_both[s][k]);
        } else {
            if (join_a) { const int side = p.join_b[da] == s; jg_a = stream(da, side); jw_a = window(da, side); }
            if (join_b) { const int side = p.join_b[db] == s; jg_b = stream(db, side); jw_b = window(db, side); }
        }
    }
    const uint32_t join_na = is_join ? (uint32_t)p.join_na[s] << 8 : 0u, join_nb = is_join ? (uint32_t)p.join_nb[s] << 8 : 0u;
    const uint32_t seen_mask = is_join ? kSeen - 1u : 0u, seen_both = is_join ? seen_cache + kSeen * 8u : nowhere;
    const uint32_t win_mask = (p.join_window - 1u) * 8u, win_reach = (p.join_window - 1u) * 256u;     // (of a window's records, in bytes)
    const bool join_always = JOIN && !p.any_bits;     // no conditional edges: every query goes down both edges into a join
    const uint32_t xj = is_join && lane_used ? xbw + (uint32_t)(j * L + s) * 8u : nowhere + (uint32_t)lane * 8u;
    const uint32_t xjm = is_join && lane_used ? (kX - 1) * 256u : 0u;
    const uint32_t gmask = (uint32_t)((1ull << p.lane_ring_log2) - 1ull);
    uint32_t *spill_ring = reinterpret_cast<uint32_t *>(p.lane_ws) + ((wslot * (cpw * L) + lane) << p.lane_ring_log2);
    const unsigned long long n_cand = (unsigned long long)p.n_cand;
    const uint64_t slo_q = FEAS ? (uint64_t)p.slo_us << q : 0ull;   // the objective, aligned with a record's time field
    const unsigned long long limit =
        (p.iter_limit ? p.iter_limit : 8ull * (unsigned)p.n * (unsigned)(S + 1) + 4096ull) / kTurn + 1ull;
    // a spill has to start before a record still needed is overwritten, two turns from now at the latest
    const uint32_t reach = min((uint32_t)(nq - kTurn - 2), gmask - 2u * kTurn);
    // (and no long turn may start where it would come too late)
    const uint32_t long_reach = gmask > 2u * kLongTurn && nq > kLongTurn + 2u ? min((uint32_t)(nq - kLongTurn - 2), gmask - 2u * kLongTurn) : 0u;
    unsigned long long batches = 0, alg_ops = 0, exits_seen = 0, exits_due = 0;
    unsigned early = 0;          // candidates dropped before the end of the trace (feasibility only)

    // State of the lane's candidate:
    int64_t c = 0;
    bool has = false;            // the group holds a candidate
    bool exhausted = !lane_used; // the group will get no further candidate
    bool live = false, cand_bad = false, over = false;
    uint32_t Rm1 = 0;            // replicas less one, in bytes of a ring row
    uint32_t kfb = nowhere, kfm = 0;         // where the first batch in use is looked up (one replica: kInf, which compares as later)
    uint32_t efull = 0;          // tpos with the batch ring full: epos + its size; epos until a first record has opened a batch
    uint32_t lfull = 0;          // tpos with every replica in use or about to be: lpos + replicas less one
    bool started = false;        // a first record has opened a batch
    uint32_t mbm1 = 0;
    uint32_t tab = tab0;         // the lane's row of the tables
    uint64_t *out = nullptr;     // leaving records: the stage's region of the slab row (fan-out: the row)
    uint32_t n_left = 0;         // queries (fan-out: copies) that have left the pipeline at this lane
    uint32_t n_cur = 0;          // records of the arrival stream; i counts those examined
    uint32_t i = 0;
    uint32_t bm = ~0u;           // size of the open batch less one (~0: none is open)
    uint64_t tk = 0;             // latest dispatch time as (t << q) | qmask
    uint32_t epos = 0, lpos = 0, tpos = 0;   // batch ring: [lpos, tpos) in use by replicas, [epos, tpos) not yet handed on
    uint32_t tpos_seen = 0;      // tpos when batches were last counted
    uint32_t prev = 0;           // low part of record i - 1, with its flag
    bool e_act = false;          // a batch is being handed on:
    uint64_t e_key = 0;          //   its key
    uint32_t e_idx = 0;          //   the record to hand on next
    uint32_t tail_a = 0, tail_b = 0;         // records handed to the children, in bytes of a row
    uint32_t at1 = kb | rm, at2 = kb | (rm - 256u);          // where the last two batches of the ring are
    uint32_t fed = 0;            // records of the trace requested for the group's root
    uint32_t qv = 0;             // low part of the record to hand on (where there is one)
    bool spill = false;
    // No record before low_idx is needed any more once every batch up to low_key has been handed on (next_*: the
    // same for a later moment)
    uint32_t low = 0, next_idx = 0;
    uint64_t next_key = 0;
    unsigned nb = 0;
    uint32_t ja = 0, jb = 0;     // joins: records of either incoming stream consumed
    uint32_t seen_new = 0;       // joins: words of the queries' bits from here on have not been touched
    uint32_t turns = 1, turns_hi = 0;        // iteration bound, in turns
    bool any_spill = false;
    uint64_t late_fin = 0, late_arr = 0;     // feasibility only: finish and arrival record of a query that has just left
    uint32_t miss_local = 0;

    for (;;) {
        // ---- every kQuickTurn-th, kTurn-th or kLongTurn-th iteration: does a lane need more than its steps?  A stream at its start or its end, a
        // candidate that is decided, records in reach of being overwritten, the iteration bound.  (Kept short: its
        // latency is on the chain of every iteration, a kTurn-th of it.)
        if (FEAS && miss_local) { atomicAdd(missw + j, miss_local); miss_local = 0; }
        nb += (tpos - tpos_seen) >> 8;
        tpos_seen = tpos;
        // Records before `low` are not needed any more.  Cheap and late: all batches closed when next_idx was the
        // open batch's first record have been handed on once the front of the ring is beyond the largest key of
        // that moment.
        const uint64_t fk = epos != tpos ? lds64(kb | (epos & rm)) : kInf;
        const uint64_t lk = lds64(kb | ((tpos - 256u) & rm));
        if (fk > next_key) {
            low = e_act ? min(next_idx, e_idx) : next_idx;
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
        const bool waits = i != n_cur && !started;
        const bool starts = waits && (int)lds32_shared(xin + 4u) >= 0, closes = i == n_cur && bm != ~0u;
        bool attn = !exhausted && (starts || closes || turns == 0u || (is_root && i == n_cur));
        attn |= i - low > reach || spill;
        if (FEAS) attn |= has && missw[j] > p.miss_allow;
        if (__any_sync(full, attn)) {
        bool done = i == n_cur && bm == ~0u && epos == tpos && !e_act && !(FEAS && late_fin != 0ull);
        if (is_join && has && !cand_bad) done = ja == join_na && jb == join_nb;
        bool stop = FEAS && has && missw[j] > p.miss_allow;       // this lane ends its group's candidate here
        bool give_up = false;
        if (i - low > reach || spill) {
            // the oldest record still needed, exactly
            low = i - (bm + 1u);
            if (e_act) low = min(low, e_idx);
#pragma unroll 1
            for (uint32_t k = epos; k != tpos; k += 256u) low = min(low, (uint32_t)lds64(kb | (k & rm)) & qmask);
            const uint32_t span = i - low;
            if (!spill && span > (uint32_t)(nq - kTurn - 2)) {
#pragma unroll 1
                for (uint32_t k = low; k != i; k++)
                    if (IL_IN_RANGE(k & gmask, gmask + 1ull, p.status))
                        spill_ring[k & gmask] = lds32(qb + ((k & (nq - 1u)) << 7));
                spill = true;
            } else if (spill && span < nq / 2u) {
                spill = false;
            }
            give_up = p.lane_wrap && span + 2u * kTurn > gmask;
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
        if (p.lane_wrap) {
            const bool group_gives_up = (__ballot_sync(full, give_up) & group_mask) != 0u;
            if (group_gives_up && !over) { over = true; if (has) p.ovf[c] = 1; }
            stop |= group_gives_up;
        }
        if (stop) {
            n_cur = i; bm = ~0u; epos = tpos; efull = tpos; e_act = false; late_fin = 0; started = false;
            ja = join_na; jb = join_nb;
            done = true;
        }
        // The first record of a stream opens a batch on an unused replica, and the last batch is closed by the
        // end of the stream; both once per candidate, so here and not in every iteration.
        if (!done && !started && !is_join) {
            const uint64_t rec = lds64_shared(xin);
            if ((int64_t)rec >= 0) {
                tk = rec | qmask;
                bm = 0; i = 1;
                prev = (uint32_t)rec & qmask;
                sts32_shared_if(true, xin + 4u, ~0u);
                started = true;
                efull = epos + rm + 256u;
            }
        } else if (!done && !is_join && i == n_cur && bm != ~0u && tpos != efull) {
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
            if (spill && IL_IN_RANGE((i - 1u) & gmask, gmask + 1ull, p.status)) spill_ring[(i - 1u) & gmask] = prev;
        }
        const unsigned dm = __ballot_sync(full, done);
        const bool turn = !exhausted && (dm & group_mask) == group_mask;
        if (__any_sync(full, turn)) {
            // wrap up the candidate the group has finished
            if (turn && has) {
                if (live && !over) {
                    batches += nb;
                    alg_ops += 3ull * n_in + (unsigned long long)nb * ((Rm1 >> 8) + mbm1 + 6u);
                }
                const bool decided = FEAS && missw[j] > p.miss_allow;
                // every query of a candidate that ran to its end must have left through exactly one
                // leaf (checked over all candidates of the warp when the kernel ends)
                if (live && !over && !decided) exits_seen += BRANCHY ? n_left : da < 0 ? tail_a >> 3 : 0u;
                if (is_root && !cand_bad && !over && !decided)
                    exits_due += FORK ? (unsigned long long)p.total_leaving : (unsigned long long)(unsigned)p.n;
                if (FEAS && is_root) {
                    p.out_feasible[c] = over ? 2 : (decided || cand_bad ? 0 : 1);
                    early += (decided && i < n_in) ? 1u : 0u;        // the root had not reached the end of the trace
                }
            }
            __syncwarp();
            // the group's next candidate
            unsigned long long g = 0;
            if (turn && is_root) g = atomicAdd(&p.counters[0], 1ull);
            g = __shfl_sync(full, g, root_lane);
            il_stage_config cfg = {0, 1, 1, 0};
            const bool got = turn && g < n_cand;
            if (got && !is_join) cfg = p.configs[g * S + s];
            const bool bad = got && (cfg.hw >= p.H || cfg.max_batch < 1 || cfg.max_batch > p.Bmax ||
                                     cfg.replicas < 1 || cfg.replicas > IL_MAX_REPLICAS);
            const bool grp_bad = (__ballot_sync(full, bad) & group_mask) != 0u;
            if (turn) {
                has = got;
                exhausted = !got;
                c = (int64_t)g;      // g < n_cand whenever the group got a candidate: rows of the slab, the
                cand_bad = grp_bad;  // overflow array and the output exist for it
                over = false;
                uint64_t *slab = FEAS ? nullptr : reinterpret_cast<uint64_t *>(p.slab + (got ? c : 0) * p.slab_stride);
                if (got && cand_bad) {
                    if (is_root) atomicCAS(p.status, 0, IL_ERR_BAD_CONFIG);
                    if (!FEAS) for (int k = row; k < p.n; k += L) slab[k] = 0;
                }
                live = got && !cand_bad && n_in > 0;
                ja = is_join && got && !cand_bad ? 0u : join_na; jb = is_join && got && !cand_bad ? 0u : join_nb;
                seen_new = 0u;
                if (is_join) {
                    sts32(jw_a, 0u); sts32(jw_b, 0u);
                    for (int k = 0; k < kSeen; k++) sts64(seen_cache + (uint32_t)k * 8u, kInf);
                }
                Rm1 = (cfg.replicas - 1u) << 8;
                kfb = Rm1 != 0u ? kb : nowhere + (uint32_t)lane * 8u;
                kfm = Rm1 != 0u ? rm : 0u;
                started = false; efull = 0; lfull = Rm1;
                mbm1 = cfg.max_batch - 1u;
                tab = tab0 + (uint32_t)((live ? s * p.H + cfg.hw : 0) * rowlen) * 4u;
                out = FORK ? slab : slab + exit_off;
                n_left = 0;
                n_cur = live ? n_in : 0u;
                for (int k = 0; k < kX; k++) sts64(xb + (uint32_t)k * 256u, kInf);
                if (FEAS && is_root) missw[j] = 0u;
                i = 0; bm = ~0u; tk = 0;
                epos = 0; lpos = 0; tpos = 0; tpos_seen = 0;
                at1 = kb | rm; at2 = kb | (rm - 256u);
                sts64(at1, 0ull); sts64(at2, 0ull);       // (no batch before the first one)
                prev = 0;
                e_act = false; e_idx = 0;
                tail_a = 0; tail_b = 0;
                spill = false; low = 0; next_idx = 0; next_key = 0;
                nb = 0;
                turns = (uint32_t)limit; turns_hi = (uint32_t)(limit >> 32);
                late_fin = 0;
                fed = 0u;
                if (is_root) for (int k = 0; k < kAhead; k++) sts64(tb + (uint32_t)(k * cpw) * 8u, kInf);
            }
            __syncwarp();     // the rings are empty before anybody looks
            if (__all_sync(full, exhausted)) break;
        }
        any_spill = __any_sync(full, spill);
        __syncwarp();     // a root's first position is empty before another lane of the group fills it again below
        }
        // (A stage waits for the next turn to open its first batch and to close its last one.  One that has not started within
        // the first kQuickLooks looks has late records: no short turns for it.)
        const bool quick = !JOIN && ((i != n_cur && !started && (uint32_t)limit - turns < kQuickLooks) || (i == n_cur && bm != ~0u));
        const int turn_its = (int)__reduce_min_sync(full, quick ? kQuickTurn : i - low > long_reach ? kTurn : kLongTurn);

        // The root's next records: requested two turns before their use, by all lanes of the group.
        {
            const uint32_t at = __shfl_sync(full, i, root_lane);
            const uint32_t to = has && !cand_bad ? min(at + (uint32_t)kAhead, (uint32_t)p.n) : 0u;
#pragma unroll 1
            for (uint32_t k = fed + (uint32_t)row; k < to; k += (uint32_t)L) copy8(tb + (k & (kAhead - 1u)) * (uint32_t)cpw * 8u, trace + k);
            fed = max(fed, to);
        }

        // joins: a record for a join.  Records of its two streams are counted in bytes of a row, as tails are.  The
        // count is told to the join's lane at the top of the NEXT iteration, behind the barrier at the end of this one: whoever
        // reads a count also sees the records it covers, in the window and in the global stream.
        auto deliver = [&](bool c, uint64_t *stream, uint32_t win, uint32_t tail, uint64_t rec) {
            stg64_if(c && IL_IN_RANGE(stream + (tail >> 8) - p.join_ws, p.join_size, p.status), stream + (tail >> 8), rec);
            sts64_shared_if(c, win + 8u + ((tail >> 5) & win_mask), rec);
        };
        // joins: one step of a join's lane takes up to two records of its two incoming streams (every query can come from
        // both sides), as long as what comes next on both sides is known.  The loads stand at the top of the
        // iteration and the rest among the stages' work, so that the two hide each other's latency: one after the other,
        // with the second record's loads behind the first one's stores, an iteration took 0.6 us.
        // Whether the other input of a record's query has been seen already: the queries' bits are kept in a small
        // write-back cache; queries come in nearly in order, so a word is new when it is first needed.
        auto new_word = [&](uint64_t &e, uint32_t w) {
            const uint32_t old = (uint32_t)(e >> 32);
            if (old != ~0u && IL_IN_RANGE(old, p.join_seen_words, p.status)) seen[old] = (uint32_t)e;
            e = (uint64_t)w << 32;
            if (w < seen_new && IL_IN_RANGE(w, p.join_seen_words, p.status)) e |= seen[w];
#pragma unroll 1
            for (; seen_new < w; seen_new++)         // passed over: it may come later
                if (IL_IN_RANGE(seen_new, p.join_seen_words, p.status)) seen[seen_new] = 0u;
            seen_new = max(seen_new, w + 1u);
        };
        // joins: whether the query of a record goes down both edges into the join
        auto goes_both = [&](bool known, uint32_t low) {
            if (join_always) return known;
            const uint32_t qid = low & imask;
            uint32_t bits = rb > 0 ? low >> qi : 0u;
            if (rb == 0 && known && IL_IN_RANGE(qid, p.n, p.status)) bits = p.bits[qid];
            return known && ((lds32(seen_both + (bits >> 5) * 4u) >> (bits & 31u)) & 1u) != 0u;
        };
        auto step = [&](auto spilling) {
            constexpr bool SPILL = decltype(spilling)::value;
            // ---- joins: what has come in, the next two records of either side, room for two
            // (A parent may add one record to what have_a / have_b say before the barrier at the end; its place in the
            // window is that of a record already taken, or of one that the count does not cover and whose value is not used.)
            uint32_t have_a = 0, have_b = 0, slot0 = 0, slot1 = 0;
            uint64_t va0 = 0, va1 = 0, vb0 = 0, vb1 = 0;
            bool room0 = false, room1 = false;
            if (JOIN) {
                sts32_shared_if(tells_a, jw_a, tail_a);
                sts32_shared_if(tells_b, jw_b, tail_b);
                have_a = lds32_shared(jw_a); have_b = lds32_shared(jw_b);
                va0 = lds64_shared(jw_a + 8u + ((ja >> 5) & win_mask)); va1 = lds64_shared(jw_a + 8u + (((ja + 256u) >> 5) & win_mask));
                vb0 = lds64_shared(jw_b + 8u + ((jb >> 5) & win_mask)); vb1 = lds64_shared(jw_b + 8u + (((jb + 256u) >> 5) & win_mask));
                slot0 = xj | (tail_a & xjm); slot1 = xj | ((tail_a + 256u) & xjm);
                room0 = is_join && (int)lds32_shared(slot0 + 4u) < 0;
                room1 = (int)lds32_shared(slot1 + 4u) < 0;
            }
            // ---- everything the iteration needs from shared memory
            const uint32_t xs = xin + (i & xin_mask) * xin_row;
            const uint64_t rec = lds64_shared(xs);                    // record to examine
            const uint32_t lat = lds32(tab + bm * 4u);                // time of the open batch
            const uint64_t kf = lds64(kfb | (lpos & kfm));            // first batch in use (one replica: kInf)
            const uint64_t k1 = lds64(at1), k2 = lds64(at2);    // the last two batches
            const uint64_t fkey = lds64(kb | (epos & rm));            // first batch not handed on (if there is one)
            const uint32_t sa = xa | (tail_a & xam), sc = xc | (tail_b & xcm);
            // where the record in hand goes, and whether there is room: towards the outside always
            uint32_t bits = 0;
            if (BRANCHY && rb == 0 && e_act && bit >= 0 && IL_IN_RANGE(qv & imask, p.n, p.status)) bits = p.bits[qv & imask];
            else if (BRANCHY) bits = qv;
            const bool to_b = BRANCHY && !FORK && (bits & mask_b) != 0u;
            const bool go_a = FORK && (bits & mask_a) == want_a, go_b = FORK && (bits & mask_b) == want_b;
            const uint32_t sd = to_b ? sc : sa;
            const bool free_d = (int)lds32_shared(sd + 4u) < 0;
            const bool free_b = FORK && (int)lds32_shared(sc + 4u) < 0;
            const bool f_ok = epos != tpos && not_after(fkey, tk);

            // ---- joins: the one or two records to take
            uint64_t jrec0 = 0, jrec1 = 0, je0 = 0, je1 = 0;
            uint32_t jat0 = 0, jat1 = 0;
            bool known0 = false, known1 = false, from_a0 = false, from_a1 = false;
            if (JOIN) {
                const bool end_a = ja == join_na, end_b = jb == join_nb;
                const bool far_a = is_join && !end_a && have_a - ja > win_reach, far_b = is_join && !end_b && have_b - jb > win_reach;
                if (far_a || far_b) {
                    // (the lines from here on are complete, so they may come through L1)
                    if (far_a && IL_IN_RANGE(jg_a + (ja >> 8) - p.join_ws, p.join_size, p.status)) va0 = jg_a[ja >> 8];
                    if (far_a && (ja & 0xf00u) == 0u) asm volatile("prefetch.global.L1 [%0];" ::"l"(jg_a + (ja >> 8) + 32u));
                    if (far_b && IL_IN_RANGE(jg_b + (jb >> 8) - p.join_ws, p.join_size, p.status)) vb0 = jg_b[jb >> 8];
                    if (far_b && (jb & 0xf00u) == 0u) asm volatile("prefetch.global.L1 [%0];" ::"l"(jg_b + (jb >> 8) + 32u));
                }
                known0 = room0 && (end_a || have_a != ja) && (end_b || have_b != jb) && !(end_a && end_b);
                va0 = end_a ? kInf : va0;
                vb0 = end_b ? kInf : vb0;
                from_a0 = (va0 | qmask) <= (vb0 | qmask);
                jrec0 = from_a0 ? va0 : vb0;
                // behind it: on its side the record after it, on the other side the same one as before
                const uint32_t ja1 = ja + (from_a0 ? 256u : 0u), jb1 = jb + (from_a0 ? 0u : 256u);
                const bool end_a1 = ja1 == join_na, end_b1 = jb1 == join_nb;
                known1 = known0 && room1 && !far_a && !far_b && (end_a1 || have_a != ja1) && (end_b1 || have_b != jb1) && !(end_a1 && end_b1);
                const uint64_t va = end_a1 ? kInf : from_a0 ? va1 : va0, vb = end_b1 ? kInf : from_a0 ? vb0 : vb1;
                from_a1 = (va | qmask) <= (vb | qmask);
                jrec1 = from_a1 ? va : vb;
                jat0 = seen_cache + ((((uint32_t)jrec0 & imask) >> 5) & seen_mask) * 8u;
                jat1 = seen_cache + ((((uint32_t)jrec1 & imask) >> 5) & seen_mask) * 8u;
                je0 = lds64(jat0);                       // number of the word << 32 | word
                je1 = lds64(jat1);
            }

            // ---- examine record i, if it is there: it joins the open batch, or the open batch is closed and it
            // opens the next one
            const bool taken = (int64_t)rec >= 0 && tpos != efull;
            const bool joins = bm < mbm1 && not_after(rec, tk);
            const bool join = taken && joins, open = taken && !joins;
            const uint64_t key = ((tk + (uint64_t)lat * tick) & ~(uint64_t)qmask) | (i - 1u - bm);
            // the next batch goes to a replica never used so far (free from time 0), else to the one that is
            // free first -- maybe the one whose batch is closed just now
            const bool pop = tpos == lfull;
            const uint64_t first = before(kf, key) ? kf : key;
            // its place in the ring: behind the last one, nearly always, or just before it (a batch that finishes
            // before one dispatched earlier); further ahead is rare enough for a loop
            const uint32_t at0 = kb | (tpos & rm);
            const bool overtakes = before(key, k1);
            sts64_if(open, overtakes ? at1 : at0, key);
            sts64_if(open && overtakes, at0, k1);
            if (open && overtakes && before(key, k2)) {
                uint32_t pos = tpos - 256u;
                for (;;) {       // four at a time: the loads overlap, and most of the time one round does it
                    const uint32_t left = pos - lpos;
                    const uint32_t a0 = kb | (pos & rm), a1 = kb | ((pos - 256u) & rm), a2 = kb | ((pos - 512u) & rm),
                                   a3 = kb | ((pos - 768u) & rm), a4 = kb | ((pos - 1024u) & rm);
                    const uint64_t e1 = lds64(a1), e2 = lds64(a2), e3 = lds64(a3), e4 = lds64(a4);
                    const bool m1 = left > 0u && e1 > key, m2 = m1 && left > 256u && e2 > key,
                               m3 = m2 && left > 512u && e3 > key, m4 = m3 && left > 768u && e4 > key;
                    sts64_if(m1, a0, e1); sts64_if(m2, a1, e2); sts64_if(m3, a2, e3); sts64_if(m4, a3, e4);
                    sts64(m4 ? a4 : m3 ? a3 : m2 ? a2 : m1 ? a1 : a0, key);
                    if (!m4) break;
                    pos -= 1024u;
                }
            }
            // dispatch time: the record's, or later the time the replica is free
            const uint64_t start = ((pop && before(rec, first)) ? first : rec) | qmask;
            tk = open ? start : tk;
            tpos += open ? 256u : 0u;
            at2 = open ? at1 : at2;
            at1 = open ? at0 : at1;
            lpos += (open && pop) ? 256u : 0u;
            lfull += (open && pop) ? 256u : 0u;
            bm += join ? 1u : 0u;
            bm = open ? 0u : bm;
            // the word of record i - 1 is final now: the last one of its batch or not
            const uint32_t word = prev | (open ? kLast : 0u);
            sts32_if(taken, qb + (((i - 1u) & (nq - 1u)) << 7), word);
            sts32_shared_if(taken, xs + 4u, ~0u);
            if (SPILL) {
                stg32_if(spill && taken && IL_IN_RANGE((i - 1u) & gmask, gmask + 1ull, p.status), spill_ring + ((i - 1u) & gmask), word);
            }
            prev = taken ? (uint32_t)rec & qmask : prev;
            i += taken ? 1u : 0u;

            // ---- joins: the records are counted, and the last input of a query goes to the join's stage
            if (JOIN) {
                const uint32_t low0 = (uint32_t)jrec0 & qmask, low1 = (uint32_t)jrec1 & qmask;
                const uint32_t w0 = (low0 & imask) >> 5, w1 = (low1 & imask) >> 5, mine0 = 1u << (low0 & 31u), mine1 = 1u << (low1 & 31u);
                const bool both0 = goes_both(known0, low0);
                bool both1 = goes_both(known1, low1);
                const bool fresh = both0 && (uint32_t)(je0 >> 32) != w0;
                if (fresh) new_word(je0, w0);
                if (fresh || (both1 && (uint32_t)(je1 >> 32) != w1)) { known1 = false; both1 = false; }     // (next time)
                sts64_if(both0, jat0, je0 ^ mine0);
                if (both0 && jat0 == jat1) je1 ^= mine0;
                sts64_if(both1, jat1, je1 ^ mine1);
                const bool last0 = known0 && (!both0 || ((uint32_t)je0 & mine0) != 0u);
                const bool last1 = known1 && (!both1 || ((uint32_t)je1 & mine1) != 0u);
                sts64_shared_if(last0, slot0, jrec0);
                sts64_shared_if(last1, last0 ? slot1 : slot0, jrec1);
                ja += (known0 && from_a0 ? 256u : 0u) + (known1 && from_a1 ? 256u : 0u);
                jb += (known0 && !from_a0 ? 256u : 0u) + (known1 && !from_a1 ? 256u : 0u);
                tail_a += (last0 ? 256u : 0u) + (last1 ? 256u : 0u);
            }

            // ---- hand on
            if (FEAS) miss_local += (late_fin > late_arr + slo_q) ? 1u : 0u;
            const bool last = (int)qv < 0;
            const uint64_t e_base = e_key & ~(uint64_t)qmask;         // finish << q
            qv &= ~kLast;
            const uint32_t qid = BRANCHY ? qv & imask : qv;
            bool hand;
            if (BRANCHY) {
                if (FORK) {
                    hand = e_act && (!go_a || free_d) && (!go_b || free_b);
                    sts64_shared_if(hand && go_a && !join_a, sa, e_base | qv);
                    sts64_shared_if(hand && go_b && !join_b, sc, e_base | qv);
                    if (JOIN) {
                        deliver(hand && go_a && join_a, jg_a, jw_a, tail_a, e_base | qv);
                        deliver(hand && go_b && join_b, jg_b, jw_b, tail_b, e_base | qv);
                    }
                    tail_a += (hand && go_a) ? 256u : 0u;
                    tail_b += (hand && go_b) ? 256u : 0u;
                    // this copy leaves: the query's slab entry keeps the latest of its copies
                    if (hand && !go_a && !go_b) {
                        if (IL_IN_RANGE(qid, p.n, p.status))
                            atomicMax(reinterpret_cast<unsigned long long *>(out) + qid, (e_base >> rb) | qid);
                        n_left++;
                    }
                } else {
                    const bool leaves = to_b ? db < 0 : da < 0;
                    hand = e_act && free_d;
                    sts64_shared_if(hand && !leaves, sd, e_base | qv);
                    // (slab records are plain (finish, query) records whatever the streams carry)
                    if (!FEAS) stg64_if(hand && leaves && IL_IN_RANGE(n_left, leaving, p.status), out + n_left, (e_base >> rb) | qid);
                    if (FEAS) {
                        late_fin = (hand && leaves) ? e_base : 0ull;
                        late_arr = __ldg(trace + (hand && leaves && IL_IN_RANGE(qid, p.n, p.status) ? qid : 0u));
                    }
                    tail_a += (hand && !to_b) ? 256u : 0u;
                    tail_b += (hand && to_b) ? 256u : 0u;
                    n_left += (hand && leaves) ? 1u : 0u;
                }
            } else {
                hand = e_act && free_d;
                sts64_shared_if(hand && da >= 0, sa, e_base | qv);
                // (one counter: bytes of ring rows towards the child, of the slab on a leaf)
                if (!FEAS) stg64_if(hand && da < 0 && IL_IN_RANGE(tail_a >> 3, leaving, p.status),
                                    reinterpret_cast<uint64_t *>(reinterpret_cast<char *>(out) + tail_a), e_base | qv);
                tail_a += hand ? tail_step : 0u;
                if (FEAS) {
                    late_fin = (hand && da < 0) ? e_base : 0ull;
                    late_arr = __ldg(trace + (hand && da < 0 && IL_IN_RANGE(qid, p.n, p.status) ? qid : 0u));
                }
            }
            // the next record to hand on: of the batch in hand, or the first one of the next batch
            const bool goes_on = e_act && !(hand && last);
            const bool fetch = f_ok && !goes_on;
            e_idx += hand ? 1u : 0u;
            e_idx = fetch ? (uint32_t)fkey & qmask : e_idx;
            e_key = fetch ? fkey : e_key;
            epos += fetch ? 256u : 0u;
            efull += fetch ? 256u : 0u;
            e_act = goes_on || fetch;
            qv = lds32(qb + ((e_idx & (nq - 1u)) << 7));
            // (the lane's own stores, so the words may come through L1: 32 of them with one miss)
            if (SPILL) ldg32_if(spill && i - e_idx > nq && IL_IN_RANGE(e_idx & gmask, gmask + 1ull, p.status), spill_ring + (e_idx & gmask), qv);
            if (JOIN) __syncwarp();      // what was delivered is there for the joins' lanes
        };
        if (any_spill) {
#pragma unroll 1
            for (int k = 0; k < turn_its; k++) step(std::true_type{});
        } else {
#pragma unroll 1
            for (int k = 0; k < turn_its; k += 2) { step(std::false_type{}); step(std::false_type{}); }
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

// Pipelines with joins.  (il_kernel_name reports "des_kernel" for them, as for the form in des_kernel.cu that takes over
// where times do not fit a record.)
__global__ void __launch_bounds__(kLaneWarps * 32) des_join_lane_kernel(const __grid_constant__ DesParams p)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    lane_simulation<true, false, true, true>(p, smem_raw);
}

cudaError_t launch_des_join_lane(const DesParams &p, int grid, size_t smem, cudaStream_t stream)
{
    if (p.lane_wrap || p.out_feasible) return cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute(des_join_lane_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    des_join_lane_kernel<<<grid, kLaneWarps * 32, smem, stream>>>(p);
    return cudaGetLastError();
}

size_t des_join_lane_smem(int table_rows, int Bmax, int ring_slots, int ring_words, int cpw, int joins, int window)
{
    return (kSmemBase + table_bytes(table_rows, Bmax) + key_bytes(ring_slots) - 1) / key_bytes(ring_slots) * key_bytes(ring_slots) -
           kSmemBase + ring_bytes(ring_slots, ring_words, cpw) + kTailBytes + join_bytes(cpw, joins, window);
}

int des_join_lane_max_ctas_per_sm(size_t smem)
{
    int n = 0;
    if (cudaFuncSetAttribute(des_join_lane_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, des_join_lane_kernel, kLaneWarps * 32, smem);
    return e == cudaSuccess ? n : 0;
}

}  // namespace il
