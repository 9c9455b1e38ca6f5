// The persistent, degree-aware walk engine (FlowWalker Sections 4-5,
// re-designed for sm_103a without block-wide barriers).
//
// Scheduling (Section 5's sampler-centric model and two-level task pools):
//   * Every warp is an independent sampler with a walk slot of its own (more
//     if the caller asks) in shared memory: its share of the CTA's local task
//     pool P_L.  It
//     claims queries from one global atomic cursor over the callers' request
//     arrays (the global task pool P_G: nothing extra in global memory) and
//     runs one step at a time on whichever of its walks is ready.
//   * A step whose current row holds at most d_t entries is sampled by the
//     warp alone (the warp sampler).  A longer row becomes a CTA hub task:
//     it is cut into segments and every warp of the CTA that has a free
//     moment takes segments through shared-memory atomics (the block
//     sampler, without __syncthreads: warps join and leave freely).  The
//     warp that finishes the last segment merges the result and commits the
//     move; the walk then returns to its owner warp.  So a walk moves between
//     the warp and the block sampler at every step, by the degree of the
//     vertex it stands on, and never leaves its CTA.
//
// Selection (Section 4; no O(d) buffer in global memory), fast mode: one pass
// of weighted reservoir sampling in exponential-race form: the warp keeps one
// Efraimidis-Spirakis reservoir with exponential jumps per row segment (a
// warp sum per 256-entry stage against the remaining jump budget; random
// draws only where a record falls, about ln d per row), and segments are
// merged by an arg-min over race times (a 64-bit atomicMin of packed (time,
// index) across the warps of a hub task).
//
// Exact mode: W = the sum of integer weights, r = floor(x * W / 2^64) from the
// step's 64-bit Philox draw, pick = smallest i with inclusive prefix > r
// (inverse transform sampling).  The scan keeps the totals of up to 64 runs of
// 512-entry pairs in shared memory and only the run holding the crossing is
// scanned again (a row of one pair is picked from at once).  Measured on the
// R-MAT-20 node2vec batch of 2^15 walks: 69.8 ms with per-128-entry sums, rows
// above 8,184 entries as hub tasks and 136 KB of code (the warps waited for
// instructions 55 % of their time), 10.1 ms on this engine (4.2 ms at copy
// bandwidth; it is bound by instruction issue in the membership test).
//
// First-order rules (weighted, MetaPath, PPR) need a row's weights (and
// labels) and the one picked column, so only those are read: 4 (5) bytes per
// entry.  A lane takes four 16-byte quads of 512 entries straight into
// registers: with 32 warps per SM (64 registers) the loads in flight cover the
// latency, and the kernel is bound by instruction issue (3.1 of 4 per cycle and
// SM).  Measured on R-MAT-22 (250,007 ragged weighted walks, 5.75e6 steps):
// 37.9 ms with columns and weights through a TMA ring on 16 warps per SM,
// 22.6 ms with the weights alone through the ring on 32, 21.5 ms by direct
// loads (180 -> 75 instructions per 512 entries: no barrier waits, refills and
// shared round trip), 19.5 ms with the per-step code cut down, 14.1 ms with all
// weights in registers, one walk per warp and records through shared memory.
// 12.9 ms is what the weights take at copy bandwidth.
#pragma once

#include "fw_device.cuh"

namespace fw {
namespace {

constexpr int NHUB = 4;           // hub tasks open at once per CTA
constexpr int NSEG_MAX = 64;      // segments per hub task
constexpr int kSums = 64;         // exact mode: run totals per scan
// A row is cut into segments of kSegQuads quads (16384 entries, counted from
// its first aligned 16-entry group), or more for rows past NSEG_MAX such
// segments.  In fast mode segment j draws from random stream j and the step
// takes the smallest race time over the segments, whichever sampler (a warp
// alone, or a CTA hub task) scans the row: the pick depends on the row, not
// on the threshold d_t or the launch shape.
constexpr int kSegQuads = 4096;
constexpr int STAGE = 256;             // entries per reservoir stage: two 128-entry halves, a quad of each per lane
constexpr int PAIR = 2 * STAGE;        // entries of one scan iteration
constexpr int CHUNK = 1024;            // node2vec: columns staged (and tested) at a time
// node2vec: a chunk of n entries whose window holds more than kDenseRatio n +
// kDenseMin further values of N(prev) is searched from its own side.  Measured
// (R-MAT-20 / R-MAT-25 batches, ms): 1 n + 128: 39.8 / 203; 2 n + 256: 39.2 /
// 202; 3 n + 512: 37.8 / 198.6; 4 n + 1024: 37.2 / 198.3.
constexpr int kDenseRatio = 4, kDenseMin = 1024;
constexpr int NSPL = 128;              // node2vec: splitters of a dense window
constexpr int kSplCap = 154;           // their search reads up to here
constexpr int ST_EMPTY = 0, ST_READY = 1, ST_HUB = 2, ST_FINISH = 3;
// hub task control word: state << 24 | segments << 16 | next segment to hand out
constexpr unsigned H_FREE = 0u, H_SETUP = 1u << 24, H_ACTIVE = 2u << 24, H_STATE = 0xFFu << 24;
__device__ __forceinline__ int hub_nseg(unsigned ctl) { return (int)(ctl >> 16 & 0xFFu); }
__device__ __forceinline__ int hub_next(unsigned ctl) { return (int)(ctl & 0xFFFFu); }

// A CTA hub task: one step of one walk whose row is longer than d_t.  The
// step itself is what the owner's slot says (it does not change until the
// task is done).
struct HubTask {
    unsigned ctl;     // one atomic claims a segment and tells whether the task
                      // was live and how many segments it has
    int slot;         // owner slot (index into the CTA's slots)
    int done_seg;
    unsigned long long best;  // (race-time bits << 32) | row index
};

struct __align__(16) Slot {
    ReqDev rq;          // the walk's request, copied in when the walk starts
    long long q;        // local query index inside its request
    long long pbeg;     // row of prev (node2vec)
    long long row[2];   // offsets of cur's row
    int req, cur, prev, t, lim, k, pdeg, state;
};

struct CtaHead {
    HubTask hub[NHUB];
    int hub_open;       // hub tasks with segments left to hand out (a hint: claims decide)
    int working;        // warps that may still hold walks
    int abort_flag;
};

// Per-warp shared memory.
struct __align__(16) WarpHead {
    float rec[16];                  // a lane's eight running sums and weights (stage_records)
    unsigned long long cnt[C_NUM];
    unsigned long long idle_since;  // when the warp ran out of work (0: it has some)
    unsigned nap;                   // idle back-off (ns)
    int exhausted;                  // no query is left to claim
    int done;                       // no walk is left either (not counted in CtaHead::working)
};
constexpr int kHeadBytes = (sizeof(CtaHead) + 127) & ~127;
constexpr int kWarpHeadBytes = (sizeof(WarpHead) + 63) & ~63;

// Offsets inside a warp's area.  node2vec: a chunk's columns (and one word
// that equals no vertex id), its membership bytes, the splitters of a dense
// window, the barrier of the columns' copies.
template <bool N2V>
struct Area {
    static constexpr int COL = 0;
    static constexpr int MASK = COL + (N2V ? CHUNK * 4 + 16 : 0);
    static constexpr int SPL = MASK + (N2V ? CHUNK : 0);
    static constexpr int BAR = SPL + (N2V ? kSplCap * 4 : 0);
    static constexpr int HEAD = (BAR + (N2V ? 8 : 0) + 63) & ~63;
    static constexpr int BYTES = HEAD + kWarpHeadBytes;
};

// After the warps' areas and the slots, exact mode keeps the run totals of each
// warp's scan and the segment totals of the hub tasks.
template <bool EXACT, bool N2V>
constexpr size_t cta_smem(int warps, int sw) {
    return (size_t)kHeadBytes + (size_t)warps * ((size_t)sw * sizeof(Slot) + Area<N2V>::BYTES) +
           (EXACT ? (size_t)(warps * kSums + NHUB * NSEG_MAX) * 8 : 0);
}

// A warp's weighted reservoir (exponential race with exponential jumps), run
// over a row segment's entries 256 at a time.  tau = the current minimum race
// time E_i / w_i (E_i ~ Exp(1)) and sel its entry; X = Xh + Xl (an
// unevaluated FP32 sum, so that subtracting many stage totals does not
// drift) = the weight still to pass before some entry beats tau.  An entry of
// weight w beats the minimum with probability 1 - exp(-w tau), so the weight
// skipped before the next record is Exp(1) / tau; the record's own time is
// the race time conditioned to lie below tau.  Every lane holds the same
// state.
//
// Record i uses words (i & 1 ? z, w : x, y) of random block i / 2 of the
// segment's stream.  Lane l holds the draws of record have - 32 + l, handed
// out by shuffles: one Philox evaluation and one logarithm of the warp per 32
// records (a segment of d entries makes about ln d).
struct Res {
    float tau;
    int sel;
    float Xh, Xl;
    int i, have;    // records so far; draws evaluated so far
    float u1, nl2;  // this lane's draws: u1 and -log u2

    __device__ __forceinline__ void init() {
        tau = __int_as_float(0x7f800000);  // +inf
        sel = -1;
        Xh = 0.0f;
        Xl = 0.0f;
        i = 0;
        have = 0;
    }
};

// The order in which segment results compete: the smaller race time wins,
// the smaller row index breaks a tie (race times are positive, so their FP32
// bit patterns order as the values do).
__device__ __forceinline__ unsigned long long race_key(const Res& r) {
    return ((unsigned long long)__float_as_uint(r.tau) << 32) | (unsigned)r.sel;
}

// Entries per segment of a row of d entries whose first aligned 16-entry group
// starts at row index r_a: seg_q quads (kSegQuads in fast mode, whose random
// streams are the segments'), or more for rows of more than NSEG_MAX such
// segments; a multiple of 32 quads (one quad per lane).
__device__ __forceinline__ int seg_entries(int r_a, int d, int seg_q) {
    const unsigned nq = ((unsigned)(d - r_a) + 3) >> 2;
    const unsigned sq = max((unsigned)seg_q, (nq + NSEG_MAX - 1) / NSEG_MAX);
    return (int)(((sq + 31) & ~31u) << 2);
}

// Find every record inside a stage, in visiting order (lane by lane, j
// ascending: any fixed order gives the same law), and leave R with the skip
// budget past the stage.  The stage starts at row index e0; w: this lane's
// entries (0: outside the row or excluded), row indices e0 + 4 lane + j
// (j < 4) and e0 + 4 lane + 124 + j (j >= 4); own: their sum.
template <bool N2V>
__device__ __forceinline__ void stage_records(Res& R, const float (&w)[8], float own, int e0, int lane,
                                              float* __restrict__ rec, const Slot& sl, int stream) {
    float incl = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const float n = __shfl_up_sync(FULL, incl, o);
        if (lane >= o) incl += n;
    }
    const float tot = __shfl_sync(FULL, incl, 31);
    // running sums in visiting order (non-decreasing: no weight is negative)
    float cum[8];
    cum[0] = (incl - own) + w[0];
#pragma unroll
    for (int j = 1; j < 8; ++j) cum[j] = cum[j - 1] + w[j];
    float target = R.Xh + R.Xl;  // a record falls on the first entry whose cumulative weight reaches target
    unsigned live = 0;           // N2V: entries that a record may still fall on
    int last = -1, from = 0;     // else: visiting position of the last record, first lane that may hold the next
    if (N2V) {
#pragma unroll
        for (int j = 0; j < 8; ++j)
            if (w[j] > 0.0f) live |= 1u << j;
    }
#pragma unroll 1
    for (;;) {
        int L, jj;
        float wr, cr;  // the record's weight and running sum
        if (N2V) {
            // this lane's first entry that reaches target: a binary search of cum
            int j = cum[3] < target ? 4 : 0;
            j += (j ? cum[5] : cum[1]) < target ? 2 : 0;
            j += (j & 4 ? (j & 2 ? cum[6] : cum[4]) : (j & 2 ? cum[2] : cum[0])) < target ? 1 : 0;
            // (j = 7 stands for 7 and for none)
            unsigned hit = live >> j << j;
            if (cum[7] < target) hit = 0u;
            const unsigned m = __ballot_sync(FULL, hit != 0u);
            if (!m) break;
            L = __ffs(m) - 1;
            jj = __shfl_sync(FULL, __ffs(hit) - 1, L);
            const bool b0 = jj & 1, b1 = jj & 2, b2 = jj & 4;
            wr = b2 ? (b1 ? (b0 ? w[7] : w[6]) : (b0 ? w[5] : w[4])) : (b1 ? (b0 ? w[3] : w[2]) : (b0 ? w[1] : w[0]));
            cr = b2 ? (b1 ? (b0 ? cum[7] : cum[6]) : (b0 ? cum[5] : cum[4]))
                    : (b1 ? (b0 ? cum[3] : cum[2]) : (b0 ? cum[1] : cum[0]));
            wr = __shfl_sync(FULL, wr, L);
            cr = __shfl_sync(FULL, cr, L);
            // later records lie beyond this one
            if (lane < L) live = 0u;
            if (lane == L) live = live >> (jj + 1) << (jj + 1);
        } else {
            // The first lane whose entries reach target hands them out through
            // shared memory and eight lanes look at one each: fewer
            // instructions than the search and the selects above (weighted
            // R-MAT-22 14.8 -> 14.5 ms).  In the node2vec build it measured
            // slower (R-MAT-25 182 -> 191 ms: the barrier keeps the compiler
            // from moving loads ahead).
            const unsigned m = from > 31 ? 0u : __ballot_sync(FULL, cum[7] >= target && own > 0.0f) >> from << from;
            if (!m) break;
            L = __ffs(m) - 1;
            if (lane == L) {
                reinterpret_cast<float4*>(rec)[0] = make_float4(cum[0], cum[1], cum[2], cum[3]);
                reinterpret_cast<float4*>(rec)[1] = make_float4(cum[4], cum[5], cum[6], cum[7]);
                reinterpret_cast<float4*>(rec)[2] = make_float4(w[0], w[1], w[2], w[3]);
                reinterpret_cast<float4*>(rec)[3] = make_float4(w[4], w[5], w[6], w[7]);
            }
            __syncwarp();
            const float c = rec[lane & 7], x = rec[8 + (lane & 7)];
            const unsigned in = __ballot_sync(FULL, c >= target && x > 0.0f && 8 * L + (lane & 7) > last) & 0xFFu;
            if (!in) {  // (only where the last record's own entry still reaches target)
                from = L + 1;
                continue;
            }
            jj = __ffs(in) - 1;
            wr = __shfl_sync(FULL, x, jj);
            cr = __shfl_sync(FULL, c, jj);
            last = 8 * L + jj;
            from = L;
        }
        R.sel = e0 + 4 * L + jj + (jj >= 4 ? 124 : 0);
        if (R.i == R.have) {
            const uint4 o = lane_block(sl.rq.seed, (uint64_t)(sl.rq.q_id0 + sl.q), (uint32_t)sl.t, (uint32_t)stream,
                                       (uint32_t)(R.i + lane) >> 1);
            R.u1 = unit_open(lane & 1 ? o.z : o.x);
            R.nl2 = -__logf(unit_open(lane & 1 ? o.w : o.y));
            R.have += 32;
        }
        const float u1 = __shfl_sync(FULL, R.u1, R.i);
        const float nl = __shfl_sync(FULL, R.nl2, R.i);
        ++R.i;
        // -log u by the fast intrinsic (u is at least 2^-24, well inside its
        // accurate range); the conditioned draw keeps log1pf/expm1f, whose
        // arguments are tiny once many entries have been seen
        float e;
        if (isinf(R.tau)) e = -__logf(u1);
        else e = -log1pf(u1 * expm1f(-wr * R.tau));
        R.tau = __fdividef(e, wr);
        R.Xh = __fdividef(nl, R.tau);
        target = cr + R.Xh;
    }
    R.Xh = target - tot;
    R.Xl = 0.0f;
}

// Offer a pair of stages: w[8 h + j] = this lane's entries of stage h, ordered
// as stage_records takes them; two: the second stage has entries of the row.
// A stage's total is the xor butterfly sum of its lanes' sums (the same in
// every lane, as a + b = b + a in IEEE arithmetic); the two butterflies share
// their last four steps, one stage in each half of the warp.
template <bool N2V>
__device__ __forceinline__ void offer_pair(Res& R, float (&w)[16], bool two, int e0, int lane,
                                           float* __restrict__ rec, const Slot& sl, int stream) {
    const float own0 = ((w[0] + w[1]) + (w[2] + w[3])) + ((w[4] + w[5]) + (w[6] + w[7]));
    const float own1 = ((w[8] + w[9]) + (w[10] + w[11])) + ((w[12] + w[13]) + (w[14] + w[15]));
    const bool up = lane & 16;
    float v = up ? own1 : own0;
    v += __shfl_xor_sync(FULL, up ? own0 : own1, 16);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
    const float t0 = __shfl_sync(FULL, v, 0), t1 = __shfl_sync(FULL, v, 16);
    // no record in either stage (the common case): X -= t0, X -= t1 with the
    // rounding errors kept (Fast2Sum: Xh is the larger)
    const float a = R.Xh - t0;
    const bool ok0 = a + R.Xl > 0.0f;
    const float al = R.Xl + ((R.Xh - a) - t0);
    const float b = a - t1;
    const bool ok1 = b + al > 0.0f;
    if (ok0 && (ok1 || !two)) {
        R.Xh = b;
        R.Xl = al + ((a - b) - t1);
        return;
    }
    float tot = t0, own = own0;
#pragma unroll 1
    for (;;) {
        if (R.Xh - tot + R.Xl > 0.0f) {
            const float s = R.Xh - tot;
            R.Xl += (R.Xh - s) - tot;
            R.Xh = s;
        } else {
            const float ws[8] = {w[0], w[1], w[2], w[3], w[4], w[5], w[6], w[7]};
            stage_records<N2V>(R, ws, own, e0, lane, rec, sl, stream);
        }
        if (!two) return;
        two = false;
        // the second stage takes the first one's place (moved, not indexed:
        // an index would put w in local memory)
#pragma unroll
        for (int j = 0; j < 8; ++j) w[j] = w[8 + j];
        e0 += STAGE;
        tot = t1;
        own = own1;
    }
}

// Exact mode: W = the sum of the integer weights, r = floor(x W / 2^64) from
// the step's 64-bit Philox draw x, the pick = the first entry whose inclusive
// prefix exceeds r.  A scan keeps the totals of up to kSums runs of `div` pairs
// in shared memory; the run that r falls into is scanned again, until it is
// one pair, which is picked from.  A row of one pair is picked from at once.
struct ExactScan {
    unsigned long long W;      // sum of the weights scanned
    unsigned long long x;      // the step's draw
    unsigned long long r;      // r less the prefix before the range (once known)
    unsigned long long* sums;  // kSums run totals (shared memory)
    int div, np;               // pairs per run, pairs scanned
    bool pick, known;          // pick from the (single) pair; r is known
    int sel;                   // the picked row index, -1: none
};

// Sum over the warp of values below 2^36.
__device__ __forceinline__ unsigned long long warp_total(unsigned long long v) {
    const unsigned lo = __reduce_add_sync(FULL, (unsigned)v & 0xFFFFFFu);
    const unsigned hi = __reduce_add_sync(FULL, (unsigned)(v >> 24));
    return ((unsigned long long)hi << 24) + lo;
}

// Offer one pair (w: bit patterns of uint32 weights, ordered as load_pair
// leaves them: quad k of lane l holds entries 128 k + 4 l + j).
__device__ __forceinline__ void exact_pair(ExactScan& A, const float (&w)[16], int r0, int lane) {
    unsigned long long q[4];
#pragma unroll
    for (int k = 0; k < 4; ++k)
        q[k] = ((unsigned long long)__float_as_uint(w[4 * k]) + __float_as_uint(w[4 * k + 1])) +
               ((unsigned long long)__float_as_uint(w[4 * k + 2]) + __float_as_uint(w[4 * k + 3]));
    const unsigned long long tot = warp_total((q[0] + q[1]) + (q[2] + q[3]));
    A.W += tot;
    if (!A.pick) {
        if (lane == 0) A.sums[A.div == 1 ? A.np : A.np / A.div] += tot;
        ++A.np;
        return;
    }
    if (!A.known) A.r = __umul64hi(A.x, tot);
    if (tot == 0) return;
    // the 128-entry half that holds the crossing, then the lane, then the entry
    unsigned long long r = A.r;
    unsigned long long mine = q[3];
    unsigned e[4] = {__float_as_uint(w[12]), __float_as_uint(w[13]), __float_as_uint(w[14]), __float_as_uint(w[15])};
    int half = 3;
    bool found = false;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const unsigned long long gk = warp_total(q[k]);
        if (!found) {
            if (r < gk) {
                found = true;
                half = k;
                mine = q[k];
#pragma unroll
                for (int j = 0; j < 4; ++j) e[j] = __float_as_uint(w[4 * k + j]);
            } else {
                r -= gk;
            }
        }
    }
    unsigned long long incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long n = __shfl_up_sync(FULL, incl, o);
        if (lane >= o) incl += n;
    }
    const unsigned m = __ballot_sync(FULL, incl > r);
    const int L = m ? __ffs(m) - 1 : 31;  // (always found, as r < tot)
    r -= incl - mine;
    int j = 3;
    if (r < (unsigned long long)e[0]) j = 0;
    else if (r < (unsigned long long)e[0] + e[1]) j = 1;
    else if (r < (unsigned long long)e[0] + e[1] + e[2]) j = 2;
    A.sel = r0 + half * 128 + 4 * L + __shfl_sync(FULL, j, L);
}

// Which of the n sums (in shared memory) holds the crossing of r, r less the
// sums before it; -1 if none.  Warp-collective.
__device__ __noinline__ int find_crossing(const unsigned long long* sums, int n, unsigned long long& r, int lane) {
#pragma unroll 1
    for (int base = 0; base < n; base += 32) {
        const unsigned long long v = base + lane < n ? sums[base + lane] : 0ull;
        unsigned long long incl = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long u = __shfl_up_sync(FULL, incl, o);
            if (lane >= o) incl += u;
        }
        const unsigned m = __ballot_sync(FULL, incl > r);
        if (m) {
            const int L = __ffs(m) - 1;
            r -= __shfl_sync(FULL, incl - v, L);
            return base + L;
        }
        r -= __shfl_sync(FULL, incl, 31);
    }
    return -1;
}

// One lane's quad at row index rel whose last entries lie past the end of the
// arrays (`left` entries of the row's base to their end).  Out of line: it
// runs for the graph's last row only.
__device__ __noinline__ float4 load_quad_tail(const float* wrow, int rel, int left) {
    float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (rel < left) v.x = __ldg(wrow + rel);
    if (rel + 1 < left) v.y = __ldg(wrow + rel + 1);
    if (rel + 2 < left) v.z = __ldg(wrow + rel + 2);
    return v;
}
__device__ __noinline__ int load_labels_tail(const int8_t* lrow, int rel, int left) {
    int l = 0;
    for (int j = 0; j < 4 && rel + j < left; ++j) l |= (int)(uint8_t)__ldg(lrow + rel + j) << (8 * j);
    return l;
}

// This lane's quads of a pair whose first entry is row index r0, weights with
// MetaPath's label rule applied; 0 outside the row indices [0, lim) (only an
// edge pair, the range's first or last, holds such entries).  wrow, lrow: the
// row's first weight and label.
template <bool LAB>
__device__ __forceinline__ void load_pair(const float* __restrict__ wrow, const int8_t* __restrict__ lrow, int want,
                                          int r0, int lim, int left, int lane, float (&w)[16]) {
    const int at = r0 + 4 * lane;
    const float4* q = reinterpret_cast<const float4*>(wrow + at);
    const int* ql = reinterpret_cast<const int*>(lrow + at);
    int l[4] = {0, 0, 0, 0};
    if (r0 >= 0 && r0 + PAIR <= lim) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float4 v = __ldg(q + 32 * k);
            w[4 * k] = v.x; w[4 * k + 1] = v.y; w[4 * k + 2] = v.z; w[4 * k + 3] = v.w;
        }
        if (LAB && lrow) {
#pragma unroll
            for (int k = 0; k < 4; ++k) l[k] = __ldg(ql + 32 * k);
        }
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int rel = at + 128 * k;
            const bool in = rel < lim && rel + 4 <= left;
            const float4 v = ldg_if(q + 32 * k, in);
            if (LAB && lrow) l[k] = ldg_if(ql + 32 * k, in, 0);
            w[4 * k] = v.x; w[4 * k + 1] = v.y; w[4 * k + 2] = v.z; w[4 * k + 3] = v.w;
        }
        if (lim + 3 > left) {
            // a range that ends with the arrays: its last quad may lie across
            // their end
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int rel = at + 128 * k;
                if (rel < lim && rel + 4 > left) {
                    const float4 v = load_quad_tail(wrow, rel, left);
                    w[4 * k] = v.x; w[4 * k + 1] = v.y; w[4 * k + 2] = v.z; w[4 * k + 3] = v.w;
                    if (LAB && lrow) l[k] = load_labels_tail(lrow, rel, left);
                }
            }
            __syncwarp();
        }
#pragma unroll
        for (int j = 0; j < 16; ++j)
            if ((unsigned)(at + 128 * (j >> 2) + (j & 3)) >= (unsigned)lim) w[j] = 0.0f;
    }
    if (LAB && lrow) {
#pragma unroll
        for (int j = 0; j < 16; ++j)
            if ((int)(int8_t)(l[j >> 2] >> (8 * (j & 3))) != want) w[j] = 0.0f;
    }
}

// --------------------------------------------------------------------------
// node2vec membership: which entries of a chunk of N(cur) are also in
// N(prev) = B?  Both rows ascend.  The values of B inside the chunk's range are
// taken 128 at a time, four per lane, and each is located in the staged columns
// by a binary search; a hit sets its entry's byte (the values of B are
// distinct, so no two lanes write one byte).
//
// The four searches of a lane run in lockstep: a step is one shared load, one
// compare and one predicated add each, and the loads of the four overlap.  The
// steps are uneven (489, 251, 131, ...) because even ones put a warp's probes
// on few banks (p + 2^k - 1 with p a multiple of 2^(k+1)); r entries take
// steps s with r -> max(r - s, s - 1), here 1024, 535, 284, 153, 86, 49, 26,
// 13, 6, 3, 1, 0.
// --------------------------------------------------------------------------

template <int OFF>
__device__ __forceinline__ int lds_at(uint32_t a) {
    int v;
    asm volatile("ld.shared.b32 %0, [%1+%2];" : "=r"(v) : "r"(a), "n"(OFF));
    return v;
}

template <int S, int NV>
__device__ __forceinline__ void lb_step(uint32_t (&a)[NV], const int (&x)[NV]) {
#pragma unroll
    for (int i = 0; i < NV; ++i)
        if (lds_at<(S - 1) * 4>(a[i]) < x[i]) a[i] += S * 4;
}

// Move each a[i] from the first staged column to the first that is >= x[i].
// n columns are staged, with values above every x up to staged_cap(n).
template <int NV>
__device__ __forceinline__ void lb_search(uint32_t (&a)[NV], const int (&x)[NV], int n) {
    if (n > 535) lb_step<489>(a, x);
    if (n > 284) lb_step<251>(a, x);
    lb_step<131>(a, x);
    lb_step<67>(a, x);
    lb_step<37>(a, x);
    lb_step<23>(a, x);
    lb_step<13>(a, x);
    lb_step<7>(a, x);
    lb_step<3>(a, x);
    lb_step<2>(a, x);
    lb_step<1>(a, x);
}
__device__ __forceinline__ int staged_cap(int n) { return n > 535 ? CHUNK : (n > 284 ? 536 : 288); }

// Four 32-entry blocks of B from `base` in one round trip (INT_BIG past pd).
__device__ __forceinline__ void load_b128(const int32_t* __restrict__ B, int pd, int base, int lane, int (&v)[4]) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int idx = base + 32 * i + lane;
        v[i] = ldg_if(B + idx, idx < pd, INT_BIG);
    }
}

// Dense windows: B holds more values inside the chunk's range than the chunk
// has entries, so each staged entry x > `above` (entries [ia, n)) searches the
// window B[from, end) instead.  NSPL splitters B[from + (s+1) w - 1] (w =
// ceil((end - from) / NSPL)) are staged; x's lower bound lies in the bracket
// after the splitters below x, and a binary search of that bracket in global
// memory finishes it, four entries per lane in lockstep.  Warp-collective.
__device__ __noinline__ void dense_members(const int32_t* __restrict__ B, int end, int from, int above,
                                           unsigned char* __restrict__ area, int ia, int n, int lane) {
    const int* col = reinterpret_cast<const int*>(area + Area<true>::COL);
    int* spl = reinterpret_cast<int*>(area + Area<true>::SPL);
    const uint32_t sa = smem_u32(spl);
    const int w = (end - from + NSPL - 1) / NSPL;
#pragma unroll 1
    for (int i = lane; i < kSplCap; i += 32)
        spl[i] = i < NSPL ? __ldg(B + min((long long)from + (long long)(i + 1) * w - 1, (long long)end - 1)) : INT_BIG;
    __syncwarp();
#pragma unroll 1
    for (int e0 = lane; e0 < n; e0 += 128) {
        int x[4], a[4], b[4];
        uint32_t s[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int e = e0 + 32 * j;
            x[j] = e >= ia && e < n ? col[e] : -1;
            s[j] = sa;
        }
        // (splitters below x: 153 entries are searched, INT_BIG from NSPL on)
        lb_step<67>(s, x);
        lb_step<37>(s, x);
        lb_step<23>(s, x);
        lb_step<13>(s, x);
        lb_step<7>(s, x);
        lb_step<3>(s, x);
        lb_step<2>(s, x);
        lb_step<1>(s, x);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            a[j] = x[j] > above ? (int)min((long long)from + (long long)((s[j] - sa) >> 2) * w, (long long)end) : end;
            b[j] = (int)min((long long)a[j] + w, (long long)end);
        }
        bool more = true;
#pragma unroll 1
        while (more) {
            more = false;
            int mid[4], v[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                mid[j] = (int)(((unsigned)a[j] + (unsigned)b[j]) >> 1);
                v[j] = ldg_if(B + mid[j], a[j] < b[j], 0);
            }
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (a[j] < b[j]) {
                    more = true;
                    if (v[j] < x[j]) a[j] = mid[j] + 1;
                    else b[j] = mid[j];
                }
        }
        int hit[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) hit[j] = ldg_if(B + a[j], a[j] < end, -1);
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (a[j] < end && hit[j] == x[j]) area[Area<true>::MASK + e0 + 32 * j] = 1;
    }
    __syncwarp();  // the splitters are rewritten by the next dense chunk
}

// Set the membership bytes of a chunk: staged entries [ia, n) of range [amin,
// amax].  pos: cursor into B, every value before it lies below the chunk.
// Returns the smallest value of B above amax (INT_MIN: not known).
// Warp-collective.
__device__ __forceinline__ int chunk_members(const int32_t* __restrict__ B, int pd, int& pos, int amin, int amax, int ia,
                                             int n, unsigned char* __restrict__ area, int lane) {
    const uint32_t col = smem_u32(area + Area<true>::COL), mask = smem_u32(area + Area<true>::MASK);
    uint4* m4 = reinterpret_cast<uint4*>(area + Area<true>::MASK);
    m4[lane] = make_uint4(0u, 0u, 0u, 0u);
    m4[32 + lane] = make_uint4(0u, 0u, 0u, 0u);
    __syncwarp();
    int v[4];
    load_b128(B, pd, pos, lane, v);
    int last = __shfl_sync(FULL, v[3], 31);
    if (last < amin) {
        // the whole block lies below this chunk: jump to the chunk's range
        pos = lower_bound_from(B, pd, pos + 128, amin, lane);
        load_b128(B, pd, pos, lane, v);
        last = __shfl_sync(FULL, v[3], 31);
    }
    bool checked = false;
#pragma unroll 1
    while (pos < pd) {
        int nv[4];
        load_b128(B, pd, pos + 128, lane, nv);  // lands while this block is searched
        uint32_t a[4] = {col, col, col, col};
        lb_search(a, v, n);
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (lds_at<0>(a[i]) == v[i])
                asm volatile("st.shared.u8 [%0], %1;" ::"r"(mask + ((a[i] - col) >> 2)), "r"(1) : "memory");
        if (last > amax) {
            int nb = INT_BIG;
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (v[i] > amax) nb = min(nb, v[i]);
            return __reduce_min_sync(FULL, nb);
        }
        const int first = __shfl_sync(FULL, v[0], 0);
        pos += 128;
        // When, at this block's density, B holds kDenseRatio times as many
        // further values in the chunk's range as the chunk has entries, look
        // where they end and search from the chunk's side.
        const int dense = kDenseRatio * n + kDenseMin;
        if (!checked && (float)(amax - last) * 128.0f > (float)dense * (float)(last - first + 1)) {
            checked = true;
            const int ub = lower_bound_from(B, pd, pos, amax + 1, lane);
            if (ub - pos > dense) {
                dense_members(B, ub, pos, last, area, ia, n, lane);
                pos = ub;
                return INT_MIN;
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = nv[i];
        last = __shfl_sync(FULL, v[3], 31);
    }
    return INT_BIG;
}

// Scan the entries of row indices [r_a, lim) of slot sl's row (r_a a multiple
// of 16 in the CSR arrays, down to -15) as random stream `stream`: weights with
// the rule's factors, offered to the warp's reservoir R (fast mode) or sums X
// (exact mode).  False if a copy never landed.  Warp-collective.
template <bool EXACT, bool N2V, bool LAB>
__device__ __forceinline__ bool scan_range(const GraphDev& g, const Slot& sl, int r_a, int lim, int lane,
                                           unsigned char* area, uint32_t& ph, Res& R, ExactScan& X, int stream) {
    const long long beg = sl.row[0];
    // (exact mode moves the bit patterns of the integer weights about)
    const float* wrow = (EXACT ? reinterpret_cast<const float*>(g.w_u32) : g.w_f32) + beg;
    const int algo = sl.rq.algo;
    const int8_t* lrow = nullptr;
    int want = 0;
    if (LAB && algo == FW_METAPATH) {
        lrow = g.etype + beg;
        want = (int)sl.rq.schema[(uint32_t)sl.t % (uint32_t)sl.rq.schema_len];
    }
    const int left = (int)min(0x7fffff00ll, g.m - beg);  // entries up to the end of the arrays
    const int prev = N2V ? sl.prev : -1;
    const bool n2v = N2V && algo == FW_NODE2VEC && prev >= 0;
    const int32_t* B = N2V ? g.col + sl.pbeg : nullptr;
    int pos = -1, nb = INT_MIN;
    int* col = reinterpret_cast<int*>(area + Area<N2V>::COL);
    unsigned long long* bar = reinterpret_cast<unsigned long long*>(area + Area<N2V>::BAR);
    // whole 16-entry groups inside the arrays, as copies take them
    const int whole = r_a + ((left - r_a) & ~15);
    if (n2v && lane == 0) {
        const int k = min(min(CHUNK, (lim - r_a + 15) & ~15), whole - r_a);
        mbar_arrive_expect_tx(bar, (uint32_t)k * 4u);
        if (k > 0) tma_load_1d(col, g.col + beg + r_a, (uint32_t)k * 4u, bar);
    }
#pragma unroll 1
    for (int r0 = r_a; r0 < lim; r0 += N2V ? CHUNK : PAIR) {
        bool some = false;
        int prevpos = -1;
        if (n2v) {
            if (!mbar_wait_warp(bar, ph)) return false;
            ph ^= 1u;
            // staged entries [ia, n) belong to the row; the others take values
            // that keep the chunk ascending and equal no vertex id
            const int ia = max(0, -r0), n = min(CHUNK, lim - r0);
            bool wrote = false;
            if (whole < r0 + n) {
#pragma unroll 1
                for (int e = max(whole - r0, 0) + lane; e < n; e += 32) col[e] = __ldg(g.col + beg + r0 + e);
                wrote = true;
            }
            const int cap = staged_cap(n);
            if (ia > 0 || n < cap) {
                if (lane < ia) col[lane] = INT_MIN;
                const int n4 = (n + 3) & ~3;
                if (n + lane < n4) col[n + lane] = INT_BIG;
#pragma unroll 1
                for (int e = n4 + 4 * lane; e < cap; e += 128)
                    *reinterpret_cast<int4*>(col + e) = make_int4(INT_BIG, INT_BIG, INT_BIG, INT_BIG);
                wrote = true;
            }
            __syncwarp();
            const int amin = col[ia], amax = col[n - 1];
            if (nb <= amax) {
                if (pos < 0) pos = r_a <= 0 ? 0 : lower_bound_from(B, sl.pdeg, 0, amin, lane);
                nb = chunk_members(B, sl.pdeg, pos, amin, amax, ia, n, area, lane);
                some = true;
            }
            if (prev >= amin && prev <= amax) {
                uint32_t a[1] = {smem_u32(col)};
                const int x[1] = {prev};
                lb_search(a, x, n);
                if (lds_at<0>(a[0]) == prev) prevpos = (int)(a[0] - smem_u32(col)) >> 2;
            }
            if (wrote) fence_proxy_async_cta();  // the columns are overwritten by the next copy
            __syncwarp();
            if (lane == 0 && r0 + CHUNK < lim) {
                const int rn = r0 + CHUNK, k = min(min(CHUNK, (lim - rn + 15) & ~15), whole - rn);
                mbar_arrive_expect_tx(bar, (uint32_t)max(k, 0) * 4u);
                if (k > 0) tma_load_1d(col, g.col + beg + rn, (uint32_t)k * 4u, bar);
                // a long row's weights are asked for a chunk ahead too (R-MAT-25
                // batch: 197.6 -> 190.1 ms)
                if (k == CHUNK) prefetch_l2(wrow + rn, CHUNK * 4);
            }
        }
#pragma unroll 1
        for (int rp = r0; rp < min(lim, r0 + (N2V ? CHUNK : PAIR)); rp += PAIR) {
            float w[16];
            load_pair<LAB>(wrow, lrow, want, rp, lim, left, lane, w);
            if (n2v) {
                const float f1 = sl.rq.fac_f[1], f2 = sl.rq.fac_f[2];
                const unsigned i1 = sl.rq.fac_i[1], i2 = sl.rq.fac_i[2];
                unsigned mk[4] = {0u, 0u, 0u, 0u};
                if (some) {
                    const unsigned* mw = reinterpret_cast<const unsigned*>(area + Area<N2V>::MASK + (rp - r0)) + lane;
#pragma unroll
                    for (int k = 0; k < 4; ++k) mk[k] = mw[32 * k];
                }
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    const bool in = mk[j >> 2] >> (8 * (j & 3)) & 1u;
                    if (EXACT) w[j] = __uint_as_float(__float_as_uint(w[j]) * (in ? i1 : i2));
                    else w[j] = __fmul_rn(w[j], in ? f1 : f2);
                }
                const int pp = prevpos - (rp - r0);
                if (prevpos >= 0 && (unsigned)pp < (unsigned)PAIR) {
                    // the return factor in place of the other two
                    float wp = __ldg(wrow + rp + pp);
                    if (EXACT) wp = __uint_as_float(__float_as_uint(wp) * sl.rq.fac_i[0]);
                    else wp = __fmul_rn(wp, sl.rq.fac_f[0]);
                    const int jp = (pp >> 2 & 31) == lane ? (pp >> 7) * 4 + (pp & 3) : -1;
#pragma unroll
                    for (int j = 0; j < 16; ++j)
                        if (j == jp) w[j] = wp;
                }
            }
            if (EXACT) exact_pair(X, w, rp, lane);
            else offer_pair<N2V>(R, w, rp + STAGE < lim, rp, lane, reinterpret_cast<WarpHead*>(area + Area<N2V>::HEAD)->rec, sl, stream);
        }
        if (N2V) __syncwarp();  // the membership bytes are cleared for the next chunk
    }
    return true;
}

__device__ __forceinline__ int find_req(const ReqDev* __restrict__ reqs, int n_req, long long gq) {
    int lo = 0, hi = n_req - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (reqs[mid].q_begin <= gq) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// Per-warp counts, kept by lane 0 in shared memory; flush_counts turns them
// into the launch's counters.
enum { N_WALKS, N_WARP, N_BLOCK, N_ROWS, N_ROWS_META, N_ROWS_N2V, N_COUNTS };

__device__ __forceinline__ void count_step(unsigned long long* v, int d, int algo, bool hub) {
    v[hub ? N_BLOCK : N_WARP] += 1;
    v[N_ROWS] += (unsigned)d;
    if (algo == FW_METAPATH) v[N_ROWS_META] += (unsigned)d;
    if (algo == FW_NODE2VEC) v[N_ROWS_N2V] += (unsigned)d;
}

__device__ __forceinline__ void flush_counts(const unsigned long long* v, unsigned long long* counters) {
    const unsigned long long steps = v[N_WARP] + v[N_BLOCK];
    if (v[N_WALKS]) atomicAdd(&counters[C_WALKS], v[N_WALKS]);
    if (!steps) return;
    atomicAdd(&counters[C_STEPS], steps);
    atomicAdd(&counters[C_ROWS], v[N_ROWS]);
    atomicAdd(&counters[C_WARP_STEPS], v[N_WARP]);
    atomicAdd(&counters[C_BLOCK_STEPS], v[N_BLOCK]);
    atomicAdd(&counters[C_PROBES], v[N_ROWS_N2V]);
    // columns and weights, MetaPath's labels, row offsets, the path's entry
    atomicAdd(&counters[C_ALGO_BYTES], 8 * v[N_ROWS] + v[N_ROWS_META] + 20 * steps);
}

// Start fetching the offsets of v's row into a slot (waited for by
// cp_async_wait_all of the same thread).
__device__ __forceinline__ void fetch_row(const GraphDev& g, Slot& s, int v) {
    const int64_t* p = g.row_ptr + v;
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(&s.row[0])), "l"(p) : "memory");
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(&s.row[1])), "l"(p + 1) : "memory");
}

__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Commit a move of slot s (one thread): append the entry at row index `sel` to
// the path, advance the walk, apply the PPR stop test and the length limit,
// fetch the next row's offsets, and hand the slot back (READY or FINISH).
// `hub`: the slot may belong to another warp, so the offsets must have landed
// first.
template <bool PPR>
__device__ __forceinline__ void commit(const GraphDev& g, Slot& s, int sel, bool hub) {
    const ReqDev& R = s.rq;
    const long long beg = s.row[0];
    const int d = (int)(s.row[1] - beg);
    const int next = __ldg(g.col + beg + sel);
    fetch_row(g, s, next);
    const int t = s.t;
    bool stop = false;
    if (PPR && R.algo == FW_PPR) stop = step_block(R.seed, (uint64_t)(R.q_id0 + s.q), (uint32_t)t).z < R.t_stop;
    const int k = s.k;
    R.paths[s.q * ((long long)R.max_len + 1) + k] = next;
    s.k = k + 1;
    s.prev = s.cur;
    s.pbeg = beg;
    s.pdeg = d;
    s.cur = next;
    s.t = t + 1;
    stop = stop || t + 1 >= s.lim;
    if (hub) {
        cp_async_wait_all();
        __threadfence_block();
    }
    *(volatile int*)&s.state = stop ? ST_FINISH : ST_READY;
}

// Claim one segment of an open hub task: task << 8 | segment, or -1 if none is
// open.  Warp-collective, uniform result.
__device__ __noinline__ int hub_claim(CtaHead& H0, int lane) {
    int got = -1;
    if (lane == 0) {
#pragma unroll 1
        for (int i = 0; i < NHUB; ++i) {
            HubTask& H = H0.hub[i];
            const unsigned v = *(volatile unsigned*)&H.ctl;
            if ((v & H_STATE) != H_ACTIVE || hub_next(v) >= hub_nseg(v)) continue;
            const unsigned old = atomicAdd(&H.ctl, 1u);
            // a claim counts only if the task was live then; the task cannot
            // be freed before this segment is done, so its fields stay valid
            if ((old & H_STATE) == H_ACTIVE && hub_next(old) < hub_nseg(old)) {
                got = i << 8 | hub_next(old);
                if (hub_next(old) == hub_nseg(old) - 1) atomicSub(&H0.hub_open, 1);
                break;
            }
        }
        __threadfence_block();
    }
    got = __shfl_sync(FULL, got, 0);
    __syncwarp();  // the other lanes read the task behind lane 0's fence (a shuffle orders no memory)
    return got;
}

// The step's 64-bit draw (exact mode).  Unrolled where no membership test
// competes for the instruction cache: the block lies in every step's chain of
// dependent instructions (1,000 exact walks of 80 on a 1,000-vertex graph, as a
// call: 206 us rolled, 198 unrolled; but the R-MAT-20 exact node2vec batch 10.06
// ms rolled, 10.42 unrolled).
template <bool N2V>
__device__ __noinline__ unsigned long long step_draw(const Slot& s) {
    const uint4 o = step_block_by<N2V ? 1 : 10>(s.rq.seed, (uint64_t)(s.rq.q_id0 + s.q), (uint32_t)s.t);
    return (unsigned long long)o.x | (unsigned long long)o.y << 32;
}

// What the engine's out-of-line parts share.
struct Launch {
    const ReqDev* reqs;  // null: the table inside the parameter block
    int n_req;
    long long total;
    unsigned long long* cursor;
    unsigned long long* counters;
    int d_always;   // rows above it are hub tasks whether or not the CTA has a warp without walks
    int claimers;   // warps of a CTA that claim queries (the others only help with hub tasks)
    int seg_q;      // exact mode: quads per hub segment
    unsigned nap;   // sleep of a warp that has no walk left between looks for hub work (ns); 0: it returns
};

// Claim one query for the empty slot sl: the slot's new state, ST_EMPTY if
// nothing is published right now (served form), -1 if no query is left.
// Out of line (once per walk, and it keeps the step loop's code small).
// Warp-collective, uniform result.
template <bool N2V, bool SERVE>
__device__ __noinline__ int claim_query(const GraphDev& g, const ReqDev* __restrict__ reqs, const Launch& L, const ServeDev& sv,
                                        Slot& sl, int lane) {
    // lane 0: r = the query's request, qi = its index inside the request
    long long qi = -1;
    int r = 0;
    if (SERVE) {
        // the oldest published request with queries left hands out its next
        // one; once the host asks the engine to stop, nothing new is claimed
        if (lane == 0 && !*sv.stop) {
#pragma unroll 1
            for (int tries = 0; tries < 64; ++tries) {
                const unsigned long long hd = *(volatile unsigned long long*)sv.head;
                if ((long long)hd >= *sv.pub_r) break;
                const int rs = (int)(hd % (unsigned long long)sv.maxr);
                const unsigned long long old = atomicAdd(&sv.taken[rs], 1ull);
                if (old < kTakenBase) {
                    qi = (long long)(old + (unsigned long long)__ldcg(&sv.ring[rs].n_q) - kTakenBase);
                    r = rs;
                    break;
                }
                atomicCAS(sv.head, hd, hd + 1);  // exhausted: move the head on
            }
        }
        qi = __shfl_sync(FULL, qi, 0);
        if (qi < 0) return ST_EMPTY;
    } else {
        long long gq = 0;
        if (lane == 0) gq = (long long)atomicAdd(L.cursor, 1ull);
        gq = __shfl_sync(FULL, gq, 0);
        if (gq >= L.total) return -1;
        r = find_req(reqs, L.n_req, gq);
        qi = gq - reqs[r].q_begin;
    }
    // the walk's own copy of its request (through L2: a served ring slot is
    // rewritten between requests)
    r = __shfl_sync(FULL, r, 0);
    constexpr int RW = (int)(sizeof(ReqDev) / 8);
    static_assert(sizeof(ReqDev) % 8 == 0 && RW <= 32, "request copy: one word per lane");
    const unsigned long long* src = reinterpret_cast<const unsigned long long*>(&reqs[r]);
    if (lane < RW) reinterpret_cast<unsigned long long*>(&sl.rq)[lane] = SERVE ? __ldcg(src + lane) : src[lane];
    __syncwarp();
    int st = 0;
    if (lane == 0) {
        const ReqDev& Rq = sl.rq;
        const int start = __ldcg(Rq.starts + qi);
        const int pv = Rq.prev ? __ldcg(Rq.prev + qi) : -1;
        const int t0 = Rq.step0 ? __ldcg(Rq.step0 + qi) : 0;
        const int lim = Rq.lengths ? __ldcg(Rq.lengths + qi) : Rq.max_len;
        sl.q = qi;
        sl.req = r;
        sl.k = 0;
        if (start < 0 || start >= g.n || pv < -1 || pv >= g.n || t0 < 0) {
            atomicAdd(&L.counters[C_BAD_INPUT], 1ull);
            st = ST_FINISH;  // written out as an empty path
        } else {
            // the walk that ended in this slot may have left its last row's
            // copies open (commit asks for them before it knows whether the
            // walk goes on); two copies into the same words have no order
            cp_async_wait_all();
            fetch_row(g, sl, start);
            Rq.paths[qi * ((long long)Rq.max_len + 1)] = start;
            sl.k = 1;
            sl.cur = start;
            sl.prev = pv;
            sl.t = t0;
            sl.lim = min(lim, Rq.max_len);
            sl.pbeg = 0;
            sl.pdeg = 0;
            if (N2V && pv >= 0) {
                const long long pb = __ldg(g.row_ptr + pv);
                sl.pbeg = pb;
                sl.pdeg = (int)(__ldg(g.row_ptr + pv + 1) - pb);
            }
            st = t0 >= sl.lim ? ST_FINISH : ST_READY;
        }
        sl.state = st;
    }
    st = __shfl_sync(FULL, st, 0);
    __syncwarp();
    return st;
}

// Retire a finished walk: path_len and -1 padding; the slot is empty then.
// Warp-collective.
template <bool SERVE>
__device__ __noinline__ void retire_walk(const ServeDev& sv, Slot& sl, unsigned long long* cnt, int lane) {
    const ReqDev& Rq = sl.rq;
    const long long width = (long long)Rq.max_len + 1;
    const int k = sl.k;
    int32_t* row = Rq.paths + sl.q * width;
#pragma unroll 1
    for (long long e = k + lane; e < width; e += 32) row[e] = -1;
    if (SERVE) __syncwarp();  // lane 0's fence below is to cover every lane's padding
    if (lane == 0) {
        Rq.path_len[sl.q] = k;
        cnt[N_WALKS] += 1;
        sl.state = ST_EMPTY;
        if (SERVE) {
            // the request's last walk tells the host (all its writes are
            // visible first)
            __threadfence();
            const int rs = sl.req;
            if (atomicAdd(&sv.done[rs], 1ull) + 1 == (unsigned long long)Rq.n_q) {
                __threadfence_system();
                sv.complete[rs] = global_timer_ns() | 1ull;
            }
        }
    }
    __syncwarp();
}

// Publish the step of slot sl as a CTA hub task of nseg segments, if a task
// entry is free; if none is, the walk stays ready and is published on a later
// visit, after this warp has helped the open tasks.  False if the row is not
// worth it: no warp of the CTA is without walks of its own (and `always` does
// not ask for it).  Warp-collective.
__device__ __noinline__ bool hub_publish(CtaHead& head, WarpHead& wh, Slot& sl, int slot, bool always, int nseg,
                                         int lane) {
    if (!always && !__shfl_sync(FULL, *(volatile int*)&head.working < (int)(blockDim.x >> 5), 0)) return false;
    int ok = 0;
    if (lane == 0) {
#pragma unroll 1
        for (int i = 0; i < NHUB; ++i) {
            HubTask& H = head.hub[i];
            const unsigned vv = *(volatile unsigned*)&H.ctl;
            if ((vv & H_STATE) == H_FREE && atomicCAS(&H.ctl, vv, H_SETUP) == vv) {
                H.slot = slot;
                H.done_seg = 0;
                H.best = ~0ull;
                sl.state = ST_HUB;
                __threadfence_block();
                atomicExch(&H.ctl, H_ACTIVE | (unsigned)nseg << 16);
                atomicAdd(&head.hub_open, 1);
                ok = 1;
                break;
            }
        }
    }
    if (!__shfl_sync(FULL, ok, 0)) {
        const unsigned nap = wh.nap;
        __nanosleep(nap);
        __syncwarp();
        if (lane == 0) wh.nap = min(nap * 2u, 1024u);
        __syncwarp();
    }
    return true;
}

// The walk to advance when the next one in turn is not ready: refills empty
// slots, retires finished walks, waits when there is nothing to do.  A slot
// index, PICK_AGAIN (look for hub work first), or PICK_QUIT.  Out of line: a
// call per few steps.  Warp-collective, uniform result.
enum { PICK_QUIT = -1, PICK_AGAIN = -2 };
template <bool N2V, bool SERVE>
__device__ __noinline__ int pick_walk(const GraphDev& g, const ReqDev* __restrict__ reqs, const Launch& L,
                                      const ServeDev& sv, CtaHead& head, WarpHead& wh, Slot* mine, int sw, int rr,
                                      int lane) {
    bool waiting = false;
#pragma unroll 1
    for (int i = 0; i < sw; ++i) {
        int jj = rr + i;
        if (jj >= sw) jj -= sw;
        Slot& sl = mine[jj];
        // another warp may flip a hub-parked slot at any time: let lane 0
        // read it once for the whole warp
        int st = __shfl_sync(FULL, *(volatile int*)&sl.state, 0);
        __syncwarp();
        if (st == ST_EMPTY && !wh.exhausted) {
            st = claim_query<N2V, SERVE>(g, reqs, L, sv, sl, lane);
            if (st < 0) {
                if (lane == 0) wh.exhausted = 1;
                __syncwarp();
            }
        }
        if (st == ST_FINISH) {
            retire_walk<SERVE>(sv, sl, wh.cnt, lane);
            --i;  // revisit this slot: it can be refilled now
            continue;
        }
        if (st == ST_HUB) waiting = true;
        if (st == ST_READY) return jj;
    }
    // Nothing to do now.  Either way a wait lasts 2 s at most.
    if (!SERVE && !waiting) {
        // Batch: no walk is left to claim.  The warp stays to help with hub
        // tasks until no warp of the CTA holds a walk, in a loop of its own
        // that takes few issue slots from the warps that are scanning.
        if (!L.nap) return PICK_QUIT;
        int quit = 0;
        if (lane == 0) {
            if (!wh.done) {
                wh.done = 1;
                atomicSub(&head.working, 1);
            }
            const unsigned long long t0 = global_timer_ns();
#pragma unroll 1
            while (*(volatile int*)&head.hub_open <= 0) {
                quit = *(volatile int*)&head.working <= 0 || *(volatile int*)&head.abort_flag ||
                       global_timer_ns() - t0 > kWaitLimitNs;
                if (quit) break;
                __nanosleep(L.nap);
            }
        }
        return __shfl_sync(FULL, quit, 0) ? PICK_QUIT : PICK_AGAIN;
    }
    // Walks parked at hub tasks: help (the caller looks for hub work first) or
    // wait for them.  Served: poll for new requests; return once the host asks
    // to stop.
    int quit = 0;
    if (lane == 0) {
        const unsigned long long now = global_timer_ns();
        if (wh.idle_since == 0) wh.idle_since = now;
        const bool late = now - wh.idle_since > kWaitLimitNs;
        if (waiting) {
            if (late) {
                atomicAdd(&L.counters[C_TIMEOUT], 1ull);
                head.abort_flag = 1;
            }
            quit = *(volatile int*)&head.abort_flag;
        } else {
            quit = late || *sv.stop;
        }
    }
    if (__shfl_sync(FULL, quit, 0)) return PICK_QUIT;
    // back off: an idle warp's polling takes issue slots from the warps that
    // are scanning
    const unsigned nap = wh.nap;
    __nanosleep(nap);
    __syncwarp();
    if (lane == 0) wh.nap = min(nap * 2u, waiting ? 1024u : 32768u);
    __syncwarp();
    return PICK_AGAIN;
}

// N2V, LAB, PPR: the launch may hold node2vec / MetaPath / PPR requests (a build
// without them is smaller: see the instruction cache above).  Only node2vec
// launches have a build without PPR.  One with PPR and without labels is worth
// its place: the label rule sits in every pair's load, and a small node2vec + PPR
// launch is a chain of those (8 weighted, 32 node2vec and 129 PPR walks on
// R-MAT-20: 611 us on the build with labels, 577 on this one).
// SERVE: the served form's build (queries claimed from the request ring,
// completion stamps, idle polling); the batch build compiles all of that out.
template <bool EXACT, bool N2V, bool LAB, bool PPR, bool SERVE>
// Registers: 64 a thread for first-order launches (32 warps per SM), 80 for
// node2vec (24 warps; 128 registers and 16 warps measured 241 ms against 202
// on the R-MAT-25 batch of 2^18 walks, 64 registers with spills 248).
__global__ void __maxnreg__(N2V ? 80 : 64)
    walk_kernel(const __grid_constant__ GraphDev g, const __grid_constant__ ReqTable tab, const __grid_constant__ Launch L,
                int sw, int d_t, const __grid_constant__ ServeDev sv) {
    const ReqDev* __restrict__ reqs = SERVE ? sv.ring : (L.reqs ? L.reqs : tab.r);
    extern __shared__ __align__(128) unsigned char dyn[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    CtaHead& head = *reinterpret_cast<CtaHead*>(dyn);
    unsigned char* area = dyn + kHeadBytes + warp * Area<N2V>::BYTES;
    Slot* slots = reinterpret_cast<Slot*>(dyn + kHeadBytes + nwarp * Area<N2V>::BYTES);
    unsigned long long* hub_sums = reinterpret_cast<unsigned long long*>(slots + nwarp * sw);
    WarpHead& wh = *reinterpret_cast<WarpHead*>(area + Area<N2V>::HEAD);
    uint32_t ph = 0;  // parity at which the next chunk's columns land
    if (N2V && lane == 0) {
        mbar_init(reinterpret_cast<unsigned long long*>(area + Area<N2V>::BAR), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        reinterpret_cast<int*>(area + Area<N2V>::COL)[CHUNK] = INT_MIN;
    }
    if (lane < N_COUNTS) wh.cnt[lane] = 0;
    if (lane < sw) slots[warp * sw + lane].state = ST_EMPTY;
    if (lane == 0) {
        wh.idle_since = 0;
        wh.nap = 128;
        wh.exhausted = warp >= L.claimers;
        wh.done = warp >= L.claimers;
    }
    if (threadIdx.x < NHUB) head.hub[threadIdx.x].ctl = H_FREE;
    if (threadIdx.x == 0) {
        head.hub_open = 0;
        head.working = min(L.claimers, nwarp);
        head.abort_flag = 0;
    }
    __syncthreads();

    int rr = 0;
#pragma unroll 1
    for (;;) {
        // ------------------------------------------------ choose the work
        // Either one segment of an open hub task (their owners are waiting,
        // so they come first) or one step of one of this warp's own walks.
        int seg = -1, s;
        if (__shfl_sync(FULL, *(volatile int*)&head.hub_open, 0)) seg = hub_claim(head, lane);
        if (seg >= 0) {
            s = head.hub[seg >> 8].slot;
        } else {
            s = rr;
            if (__shfl_sync(FULL, *(volatile int*)&slots[warp * sw + rr].state, 0) != ST_READY) {
                s = pick_walk<N2V, SERVE>(g, reqs, L, sv, head, wh, slots + warp * sw, sw, rr, lane);
                if (s == PICK_QUIT) break;
                if (s < 0) continue;
            }
            rr = s + 1 == sw ? 0 : s + 1;
            s += warp * sw;
            if (lane == 0) cp_async_wait_all();  // the offsets of its row
            __syncwarp();
        }
        Slot& sl = slots[s];
        int lim = (int)(sl.row[1] - sl.row[0]);
        int ra = lim ? -(int)(sl.row[0] & 15) : 0;  // the scan starts on a 16-entry group (a dead end has none)
        int stream = 0;
        const int sq = seg_entries(ra, lim, EXACT ? L.seg_q : kSegQuads);
        if (seg >= 0) {
            stream = seg & 0xFF;
            ra += stream * sq;
            lim = min(lim, ra + sq);
        } else if (lim > d_t && hub_publish(head, wh, sl, s, lim > L.d_always, (lim - ra + sq - 1) / sq, lane)) {
            continue;
        }

        if (lane == 0) {
            wh.idle_since = 0;
            wh.nap = 128;
        }

        // ------------------------------------ stream the row range (one site)
        int sel = -1;        // the picked row index
        bool fin = true;     // the step is done
        bool scanned = true;
        if (!EXACT) {
            // A hub segment is one range.  A row sampled by this warp alone is
            // cut into the hub path's segments, segment j drawing from random
            // stream j, and the step keeps the smallest (race time, index)
            // over them, as a hub task's merge does.
            unsigned long long best = ~0ull;
            ExactScan none;
#pragma unroll 1
            for (; ra < lim; ra += sq) {
                Res R;
                R.init();
                if (!scan_range<EXACT, N2V, LAB>(g, sl, ra, min(lim, ra + sq), lane, area, ph, R, none, stream)) {
                    scanned = false;
                    break;
                }
                if (R.sel >= 0) best = min(best, race_key(R));
                ++stream;
            }
            if (seg >= 0 && lane == 0) {
                // fold the segment into its hub task; the warp that completes
                // the last segment finishes the step
                // (the count is read first: once this segment is added, the
                // task may be finished, freed and another one's)
                HubTask& H = head.hub[seg >> 8];
                const int nseg = hub_nseg(*(volatile unsigned*)&H.ctl);
                if (best != ~0ull) atomicMin(&H.best, best);
                __threadfence_block();
                fin = atomicAdd(&H.done_seg, 1) == nseg - 1;
                __threadfence_block();
                best = *(volatile unsigned long long*)&H.best;
            }
            sel = best == ~0ull ? -1 : (int)(best & 0xFFFFFFFFull);
        } else if (ra < lim) {
            // Sums first, then the run of pairs that r falls into, down to one
            // pair.  A hub segment only adds its total to the task; the warp
            // that completes the last one goes on in the segment of the pick.
            ExactScan X;
            X.sums = hub_sums + NHUB * NSEG_MAX + warp * kSums;
            X.known = false;
            X.sel = -1;
            bool sums_only = seg >= 0;
            if (!sums_only) X.x = step_draw<N2V>(sl);
#pragma unroll 1
            for (;;) {
                const int np = (lim - ra + PAIR - 1) / PAIR;
                X.pick = np == 1 && !sums_only;
                X.div = (np + kSums - 1) / kSums;
                X.np = 0;
                X.W = 0;
                X.sums[lane] = 0;
                X.sums[32 + lane] = 0;
                __syncwarp();
                Res none;
                if (!scan_range<EXACT, N2V, LAB>(g, sl, ra, lim, lane, area, ph, none, X, 0)) {
                    scanned = false;
                    break;
                }
                __syncwarp();
                if (X.pick) break;
                if (sums_only) {
                    sums_only = false;
                    HubTask& H = head.hub[seg >> 8];
                    unsigned long long* hs = hub_sums + (seg >> 8) * NSEG_MAX;
                    const int nseg = hub_nseg(*(volatile unsigned*)&H.ctl);
                    int last = 0;
                    if (lane == 0) {
                        hs[stream] = X.W;
                        __threadfence_block();
                        last = atomicAdd(&H.done_seg, 1) == nseg - 1;
                        __threadfence_block();
                    }
                    last = __shfl_sync(FULL, last, 0);
                    __syncwarp();  // every lane reads the other warps' totals behind lane 0's fence
                    if (!last) {
                        fin = false;
                        break;
                    }
                    unsigned long long W = 0;
                    for (int i = 0; i < nseg; ++i) W += *(volatile unsigned long long*)&hs[i];
                    if (W == 0) break;
                    X.r = __umul64hi(step_draw<N2V>(sl), W);
                    X.known = true;
                    const int i = find_crossing(hs, nseg, X.r, lane);
                    if (i < 0) break;  // never, as r < W
                    ra = -(int)(sl.row[0] & 15) + i * sq;
                    lim = min((int)(sl.row[1] - sl.row[0]), ra + sq);
                    continue;
                }
                if (!X.known) {
                    if (X.W == 0) break;
                    X.r = __umul64hi(X.x, X.W);
                    X.known = true;
                }
                const int i = find_crossing(X.sums, kSums, X.r, lane);
                if (i < 0) break;  // never, as r < W
                ra += i * X.div * PAIR;
                lim = min(lim, ra + X.div * PAIR);
                __syncwarp();
            }
            sel = X.sel;
        }
        if ((EXACT || N2V) && !scanned) {
            if (lane == 0) atomicAdd(&L.counters[C_TIMEOUT], 1ull);
            break;
        }

        // ------------------------------------------------ use the result
        if (lane == 0 && fin) {
            if (sel < 0) {
                __threadfence_block();
                *(volatile int*)&sl.state = ST_FINISH;  // nothing selectable (or a dead end): the walk stops here
            } else {
                count_step(wh.cnt, (int)(sl.row[1] - sl.row[0]), sl.rq.algo, seg >= 0);
                commit<PPR>(g, sl, sel, seg >= 0);
            }
            if (seg >= 0) {
                __threadfence_block();
                atomicExch(&head.hub[seg >> 8].ctl, H_FREE);
            }
        }
        __syncwarp();
    }
    cp_async_wait_all();
    __syncwarp();
    if (lane == 0) flush_counts(wh.cnt, L.counters);
}

}  // namespace
}  // namespace fw
