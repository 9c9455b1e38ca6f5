// The persistent, degree-aware walk engine (FlowWalker Sections 4-5,
// re-designed for sm_103a without block-wide barriers).
//
// Scheduling (Section 5's sampler-centric model and two-level task pools):
//   * Every warp is an independent sampler with a few walk slots of its own
//     in shared memory (its share of the CTA's local task pool P_L).  It
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
// First-order rules (weighted, MetaPath, PPR) need a row's weights (and
// labels) and the one picked column, so only those are read: 4 (5) bytes per
// entry.  A lane takes four 16-byte quads of 512 entries straight into
// registers: with 32 warps per SM (64 registers) the loads in flight cover the
// latency, and the kernel is bound by instruction issue (3.1 of 4 per cycle and
// SM).  Measured on R-MAT-22 (250,007 ragged weighted walks, 5.75e6 steps):
// 37.9 ms with columns and weights through a TMA ring on 16 warps per SM,
// 22.6 ms with the weights alone through the ring on 32, 21.5 ms by direct
// loads (180 -> 75 instructions per 512 entries: no barrier waits, refills and
// shared round trip), 19.5 ms with the per-step code cut down.
#pragma once

#include "fw_device.cuh"

namespace fw {
namespace {

constexpr int SW_MAX = 8;         // walk slots per warp, upper bound
constexpr int NHUB = 4;           // hub tasks open at once per CTA
constexpr int NSEG_MAX = 64;      // segments per hub task
// A row is cut into segments of kSegQuads quads (16384 entries, counted from
// its first aligned 16-entry group), or more for rows past NSEG_MAX such
// segments.  In fast mode segment j draws from random stream j and the step
// takes the smallest race time over the segments, whichever sampler (a warp
// alone, or a CTA hub task) scans the row: the pick depends on the row, not
// on the threshold d_t or the launch shape.
constexpr int kSegQuads = 4096;
constexpr int STAGE = 256;             // entries per reservoir stage: two 128-entry halves, a quad of each per lane
constexpr int PAIR = 2 * STAGE;        // entries of one scan iteration
constexpr int ST_EMPTY = 0, ST_READY = 1, ST_HUB = 2, ST_FINISH = 3;
// hub task control word: state << 24 | segments << 16 | next segment to hand out
constexpr unsigned H_FREE = 0u, H_SETUP = 1u << 24, H_ACTIVE = 2u << 24, H_STATE = 0xFFu << 24;
__device__ __forceinline__ int hub_nseg(unsigned ctl) { return (int)(ctl >> 16 & 0xFFu); }
__device__ __forceinline__ int hub_next(unsigned ctl) { return (int)(ctl & 0xFFFFu); }

// Per-step view of one walk, held in registers by the lanes of its sampler.
struct StepCtx {
    long long beg;
    long long pbeg;
    int d;
    int pdeg;
    int prev;
    int algo;
    int want;   // MetaPath label for this move
    float f0, f1, f2;  // node2vec factors: return, in, out
};

// A CTA hub task: one step of one walk whose row is longer than d_t.
struct HubTask {
    unsigned ctl;     // one atomic claims a segment and tells whether the task
                      // was live and how many segments it has
    int slot;         // owner slot (index into the CTA's slots)
    int seg_e;        // entries per segment
    int done_seg;
    unsigned long long best;  // (race-time bits << 32) | row index
    StepCtx c;
    uint64_t seed;
    uint64_t qid;
    uint32_t t;
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
    int abort_flag;
};

// Per-warp shared memory.
struct WarpHead {
    unsigned long long cnt[C_NUM];
};
constexpr int kHeadBytes = (sizeof(CtaHead) + 127) & ~127;
constexpr int kWarpHeadBytes = (sizeof(WarpHead) + 127) & ~127;

// Offsets inside a warp's area.
template <bool N2V>
struct Area {
    static constexpr int HEAD = 0;
    static constexpr int BYTES = HEAD + kWarpHeadBytes;
};

template <bool N2V>
constexpr size_t cta_smem(int warps, int sw) {
    return (size_t)kHeadBytes + (size_t)warps * ((size_t)sw * sizeof(Slot) + Area<N2V>::BYTES);
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
// starts at row index r_a: kSegQuads quads, or more for rows of more than
// NSEG_MAX such segments; a multiple of 32 quads (one quad per lane).
__device__ __forceinline__ int seg_entries(int r_a, int d) {
    const unsigned nq = ((unsigned)(d - r_a) + 3) >> 2;
    const unsigned sq = max((unsigned)kSegQuads, (nq + NSEG_MAX - 1) / NSEG_MAX);
    return (int)(((sq + 31) & ~31u) << 2);
}

// What the draws of one segment are keyed by.
struct Stream {
    uint64_t seed, qid;
    uint32_t t, id;
};

// Find every record inside a stage, in visiting order (lane by lane, j
// ascending: any fixed order gives the same law), and leave R with the skip
// budget past the stage.  The stage starts at row index e0; w: this lane's
// entries (0: outside the row or excluded), row indices e0 + 4 lane + j
// (j < 4) and e0 + 4 lane + 124 + j (j >= 4); own: their sum.
__device__ __forceinline__ void stage_records(Res& R, const float (&w)[8], float own, int e0, int lane,
                                              const Stream& S) {
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
    unsigned live = 0;  // entries that a record may still fall on
#pragma unroll
    for (int j = 0; j < 8; ++j)
        if (w[j] > 0.0f) live |= 1u << j;
    float target = R.Xh + R.Xl;  // a record falls on the first entry whose cumulative weight reaches target
#pragma unroll 1
    for (;;) {
        // this lane's first entry that reaches target: a binary search of cum
        int j = cum[3] < target ? 4 : 0;
        j += (j ? cum[5] : cum[1]) < target ? 2 : 0;
        j += (j & 4 ? (j & 2 ? cum[6] : cum[4]) : (j & 2 ? cum[2] : cum[0])) < target ? 1 : 0;
        // (j = 7 stands for 7 and for none)
        unsigned hit = live >> j << j;
        if (cum[7] < target) hit = 0u;
        const unsigned m = __ballot_sync(FULL, hit != 0u);
        if (!m) {
            R.Xh = target - tot;
            R.Xl = 0.0f;
            return;
        }
        const int L = __ffs(m) - 1;
        const int jj = __shfl_sync(FULL, __ffs(hit) - 1, L);
        const bool b0 = jj & 1, b1 = jj & 2, b2 = jj & 4;
        const float wj = b2 ? (b1 ? (b0 ? w[7] : w[6]) : (b0 ? w[5] : w[4])) : (b1 ? (b0 ? w[3] : w[2]) : (b0 ? w[1] : w[0]));
        const float cj = b2 ? (b1 ? (b0 ? cum[7] : cum[6]) : (b0 ? cum[5] : cum[4]))
                            : (b1 ? (b0 ? cum[3] : cum[2]) : (b0 ? cum[1] : cum[0]));
        const float wr = __shfl_sync(FULL, wj, L);
        const float cr = __shfl_sync(FULL, cj, L);
        R.sel = e0 + 4 * L + jj + (jj >= 4 ? 124 : 0);
        // later records lie beyond this one
        if (lane < L) live = 0u;
        if (lane == L) live = live >> (jj + 1) << (jj + 1);
        if (R.i == R.have) {
            const uint4 o = lane_block(S.seed, S.qid, S.t, S.id, (uint32_t)(R.i + lane) >> 1);
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
}

// Offer a pair of stages: w[8 h + j] = this lane's entries of stage h, ordered
// as stage_records takes them; two: the second stage has entries of the row.
// A stage's total is the xor butterfly sum of its lanes' sums (the same in
// every lane, as a + b = b + a in IEEE arithmetic); the two butterflies share
// their last four steps, one stage in each half of the warp.
__device__ __forceinline__ void offer_pair(Res& R, const float (&w)[16], bool two, int e0, int lane, const Stream& S) {
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
#pragma unroll 1
    for (int h = 0; h < (two ? 2 : 1); ++h) {
        const float tot = h ? t1 : t0;
        if (R.Xh - tot + R.Xl > 0.0f) {
            const float s = R.Xh - tot;
            R.Xl += (R.Xh - s) - tot;
            R.Xh = s;
            continue;
        }
        float ws[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) ws[j] = h ? w[8 + j] : w[j];
        stage_records(R, ws, h ? own1 : own0, e0 + h * STAGE, lane, S);
    }
}

// This lane's quads of a pair whose first entry is row index r0, weights with
// MetaPath's label rule applied; 0 outside the row indices [0, lim).  Only an
// edge pair (the range's first or last) holds such entries; its quads are
// loaded one by one, so that nothing past the end of the arrays is read.
// wrow, lrow: the row's first weight and label.
__device__ __forceinline__ void load_pair(const float* __restrict__ wrow, const int8_t* __restrict__ lrow, int want,
                                          int r0, int lim, int left, int lane, float (&w)[16]) {
    const int at = r0 + 4 * lane;
    if (r0 >= 0 && r0 + PAIR <= lim) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float4 v = __ldg(reinterpret_cast<const float4*>(wrow + at) + k * 32);
            w[4 * k] = v.x; w[4 * k + 1] = v.y; w[4 * k + 2] = v.z; w[4 * k + 3] = v.w;
        }
        if (lrow) {
            int l[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) l[k] = __ldg(reinterpret_cast<const int*>(lrow + at) + k * 32);
#pragma unroll
            for (int j = 0; j < 16; ++j)
                if ((int)(int8_t)(l[j >> 2] >> (8 * (j & 3))) != want) w[j] = 0.0f;
        }
        return;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
#pragma unroll
        for (int j = 0; j < 4; ++j) w[4 * k + j] = 0.0f;
        if (r0 + 128 * k >= lim) continue;  // the whole warp's quads lie past the range
        const int rel = at + 128 * k;       // row index of the quad's first entry
        float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        int l = 0;
        if (rel + 4 <= left) {
            if (rel < lim) {
                v = __ldg(reinterpret_cast<const float4*>(wrow + rel));
                if (lrow) l = __ldg(reinterpret_cast<const int*>(lrow + rel));
            }
        } else if (rel < lim) {
            // the last quad of arrays whose size is no multiple of 4
            const int some = left - rel;
            v.x = __ldg(wrow + rel);
            if (some > 1) v.y = __ldg(wrow + rel + 1);
            if (some > 2) v.z = __ldg(wrow + rel + 2);
            if (lrow)
                for (int j = 0; j < some; ++j) l |= (int)(uint8_t)__ldg(lrow + rel + j) << (8 * j);
        }
        const float x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if ((unsigned)(rel + j) < (unsigned)lim) w[4 * k + j] = x[j];
        if (lrow) {
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if ((int)(int8_t)(l >> (8 * j)) != want) w[4 * k + j] = 0.0f;
        }
    }
}

// Scan the entries of row indices [r_a, lim) of c's row (r_a a multiple of 16
// in the CSR arrays, down to -15): weights with the rule's factors, offered
// to the warp's reservoir R.  Warp-collective.
template <bool N2V>
__device__ __forceinline__ void scan_range(const GraphDev& g, const StepCtx& c, int r_a, int lim, int lane, Res& R,
                                           const Stream& S) {
    const float* wrow = g.w_f32 + c.beg;
    const int8_t* lrow = c.algo == FW_METAPATH ? g.etype + c.beg : nullptr;
    const int left = (int)min((long long)INT_BIG, g.m - c.beg);  // entries up to the end of the arrays
#pragma unroll 1
    for (int r0 = r_a; r0 < lim; r0 += PAIR) {
        float w[16];
        load_pair(wrow, lrow, c.want, r0, lim, left, lane, w);
        offer_pair(R, w, r0 + STAGE < lim, r0, lane, S);
    }
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

// Commit a move of slot s (one thread): append `next` to the path, advance
// the walk, apply the PPR stop test and the length limit, fetch the next
// row's offsets, and hand the slot back (READY or FINISH).  `hub`: the slot
// may belong to another warp, so the offsets must have landed first.
__device__ __forceinline__ void commit(const GraphDev& g, Slot& s, long long beg, int d, int sel, uint64_t seed,
                                       uint64_t qid, uint32_t t, bool hub) {
    const ReqDev& R = s.rq;
    const int next = __ldg(g.col + beg + sel);
    fetch_row(g, s, next);
    bool stop = false;
    if (R.algo == FW_PPR) stop = step_block(seed, qid, t).z < R.t_stop;
    const int k = s.k;
    R.paths[s.q * ((long long)R.max_len + 1) + k] = next;
    s.k = k + 1;
    s.prev = s.cur;
    s.pbeg = beg;
    s.pdeg = d;
    s.cur = next;
    s.t = (int)t + 1;
    stop = stop || (int)t + 1 >= s.lim;
    if (hub) {
        cp_async_wait_all();
        __threadfence_block();
    }
    *(volatile int*)&s.state = stop ? ST_FINISH : ST_READY;
}

// Claim one segment of an open hub task: (h, j) = task, segment; false if
// none is open.  Warp-collective, uniform result.
__device__ __forceinline__ bool hub_claim(CtaHead& H0, int lane, int& h, int& j) {
    h = -1;
    j = -1;
    if (!__shfl_sync(FULL, *(volatile int*)&H0.hub_open, 0)) return false;
    if (lane == 0) {
        for (int i = 0; i < NHUB; ++i) {
            HubTask& H = H0.hub[i];
            const unsigned v = *(volatile unsigned*)&H.ctl;
            if ((v & H_STATE) != H_ACTIVE || hub_next(v) >= hub_nseg(v)) continue;
            const unsigned old = atomicAdd(&H.ctl, 1u);
            // a claim counts only if the task was live then; the task cannot
            // be freed before this segment is done, so its fields stay valid
            if ((old & H_STATE) == H_ACTIVE && hub_next(old) < hub_nseg(old)) {
                h = i;
                j = hub_next(old);
                if (j == hub_nseg(old) - 1) atomicSub(&H0.hub_open, 1);
                break;
            }
        }
    }
    h = __shfl_sync(FULL, h, 0);
    j = __shfl_sync(FULL, j, 0);
    if (h >= 0) __threadfence_block();
    return h >= 0;
}

// SERVE: the served form's build (queries claimed from the request ring,
// completion stamps, idle polling); the batch build compiles all of that out.
template <bool N2V, bool SERVE>
__global__ void __launch_bounds__(512, N2V ? 1 : 2)
    fast_kernel(GraphDev g, const __grid_constant__ ReqTable tab, int n_req, long long total, unsigned long long* cursor,
                unsigned long long* counters, int sw, int d_t, ServeDev sv) {
    const ReqDev* __restrict__ reqs = SERVE ? sv.ring : (tab.ext ? tab.ext : tab.r);
    extern __shared__ __align__(128) unsigned char dyn[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    CtaHead& head = *reinterpret_cast<CtaHead*>(dyn);
    unsigned char* area = dyn + kHeadBytes + warp * Area<N2V>::BYTES;
    Slot* slots = reinterpret_cast<Slot*>(dyn + kHeadBytes + nwarp * Area<N2V>::BYTES);
    Slot* mine = slots + warp * sw;
    WarpHead& wh = *reinterpret_cast<WarpHead*>(area + Area<N2V>::HEAD);
    unsigned long long* cnt = wh.cnt;
    if (lane < N_COUNTS) cnt[lane] = 0;
    if (lane < sw) mine[lane].state = ST_EMPTY;
    if (threadIdx.x < NHUB) head.hub[threadIdx.x].ctl = H_FREE;
    if (threadIdx.x == 0) {
        head.hub_open = 0;
        head.abort_flag = 0;
    }
    __syncthreads();

    bool exhausted = false;
    int rr = 0;
    unsigned long long idle_since = 0;
    unsigned nap = 128;  // idle back-off (ns)

    for (;;) {
        // ------------------------------------------------ choose the work
        // Either one segment of an open hub task (their owners are waiting,
        // so they come first) or one step of one of this warp's own walks.
        StepCtx c;
        Stream S;
        int ra, lim, sq;  // row indices [ra, lim) to scan, sq at a time
        int h, j, s = -1;
        const bool seg = hub_claim(head, lane, h, j);
        if (seg) {
            const HubTask& H = head.hub[h];
            c = H.c;
            sq = H.seg_e;
            ra = -(int)(c.beg & 15) + j * sq;
            lim = min(c.d, ra + sq);
            S.seed = H.seed;
            S.qid = H.qid;
            S.t = H.t;
            S.id = (uint32_t)j;
        } else {
            // ---- pick a walk: refill empty slots, retire finished ones ----
            bool waiting = false;
            for (int i = 0; i < sw; ++i) {
                int jj = rr + i;
                if (jj >= sw) jj -= sw;
                Slot& sl = mine[jj];
                // another warp may flip a hub-parked slot at any time: let
                // lane 0 read it once for the whole warp
                int st = __shfl_sync(FULL, *(volatile int*)&sl.state, 0);
                if (st == ST_EMPTY && !exhausted) {
                    // claim one query (lane 0): r = its request, qi = its
                    // index inside the request; -1 if none
                    long long qi = -1;
                    int r = 0;
                    if (SERVE) {
                        // the oldest published request with queries left
                        // hands out its next one; once the host asks the
                        // engine to stop, nothing new is claimed
                        if (lane == 0 && !*sv.stop) {
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
                        if (qi < 0) continue;  // nothing published right now: the slot stays empty
                    } else {
                        long long gq = 0;
                        if (lane == 0) gq = (long long)atomicAdd(cursor, 1ull);
                        gq = __shfl_sync(FULL, gq, 0);
                        if (gq >= total) {
                            exhausted = true;
                            continue;
                        }
                        r = find_req(reqs, n_req, gq);
                        qi = gq - reqs[r].q_begin;
                    }
                    // the walk's own copy of its request (through L2: a
                    // served ring slot is rewritten between requests)
                    r = __shfl_sync(FULL, r, 0);
                    constexpr int RW = (int)(sizeof(ReqDev) / 8);
                    static_assert(sizeof(ReqDev) % 8 == 0 && RW <= 32, "request copy: one word per lane");
                    const unsigned long long* src = reinterpret_cast<const unsigned long long*>(&reqs[r]);
                    if (lane < RW)
                        reinterpret_cast<unsigned long long*>(&sl.rq)[lane] = SERVE ? __ldcg(src + lane) : src[lane];
                    __syncwarp();
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
                            atomicAdd(&counters[C_BAD_INPUT], 1ull);
                            st = ST_FINISH;  // written out as an empty path
                        } else {
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
                }
                if (st == ST_FINISH) {
                    // retire: path_len and -1 padding
                    const ReqDev& Rq = sl.rq;
                    const long long width = (long long)Rq.max_len + 1;
                    const int k = sl.k;
                    int32_t* row = Rq.paths + sl.q * width;
                    for (long long e = k + lane; e < width; e += 32) row[e] = -1;
                    if (lane == 0) {
                        Rq.path_len[sl.q] = k;
                        cnt[N_WALKS] += 1;
                        sl.state = ST_EMPTY;
                        if (SERVE) {
                            // the request's last walk tells the host (all its
                            // writes are visible first)
                            __threadfence();
                            const int rs = sl.req;
                            if (atomicAdd(&sv.done[rs], 1ull) + 1 == (unsigned long long)Rq.n_q) {
                                __threadfence_system();
                                sv.complete[rs] = global_timer_ns() | 1ull;
                            }
                        }
                    }
                    __syncwarp();
                    --i;  // revisit this slot: it can be refilled now
                    continue;
                }
                if (st == ST_HUB) waiting = true;
                if (st == ST_READY) {
                    s = jj;
                    rr = jj + 1 == sw ? 0 : jj + 1;
                    break;
                }
            }
            if (s < 0) {
                // nothing to do now.  Batch: done once every slot is empty.
                // Served: poll for new requests; return once the host asks
                // to stop.  Either way a wait lasts 2 s at most.
                if (!waiting && !SERVE) break;
                int quit = 0;
                if (lane == 0) {
                    const unsigned long long now = global_timer_ns();
                    if (idle_since == 0) idle_since = now;
                    const bool late = now - idle_since > kWaitLimitNs;
                    if (!waiting) {
                        quit = late || *sv.stop;
                    } else {
                        if (late) {
                            atomicAdd(&counters[C_TIMEOUT], 1ull);
                            head.abort_flag = 1;
                        }
                        quit = *(volatile int*)&head.abort_flag;
                    }
                }
                if (__shfl_sync(FULL, quit, 0)) break;
                // back off: an idle warp's polling takes issue slots from the
                // warps that are scanning
                __nanosleep(nap);
                nap = min(nap * 2u, waiting ? 1024u : 32768u);
                continue;
            }

            // ---- one step of slot s ----
            Slot& sl = mine[s];
            if (lane == 0) cp_async_wait_all();
            __syncwarp();
            const long long beg = sl.row[0];
            const int d = (int)(sl.row[1] - beg);
            if (d == 0) {  // dead end
                if (lane == 0) sl.state = ST_FINISH;
                __syncwarp();
                continue;
            }
            S.t = (uint32_t)sl.t;
            c.beg = beg;
            c.d = d;
            c.algo = sl.rq.algo;
            c.want = c.algo == FW_METAPATH ? (int)sl.rq.schema[S.t % (uint32_t)sl.rq.schema_len] : -1;
            if (N2V) {
                c.pbeg = sl.pbeg;
                c.pdeg = sl.pdeg;
                c.prev = sl.prev;
                c.f0 = sl.rq.fac_f[0];
                c.f1 = sl.rq.fac_f[1];
                c.f2 = sl.rq.fac_f[2];
            }
            S.qid = (uint64_t)(sl.rq.q_id0 + sl.q);
            S.seed = sl.rq.seed;
            S.id = 0;
            ra = -(int)(beg & 15);  // the scan starts on a 16-entry group
            lim = d;
            sq = seg_entries(ra, d);

            if (d > d_t) {
                // publish as a CTA hub task, if a task entry is free
                int ok = 0;
                if (lane == 0) {
                    for (int i = 0; i < NHUB; ++i) {
                        HubTask& H = head.hub[i];
                        const unsigned vv = *(volatile unsigned*)&H.ctl;
                        if ((vv & H_STATE) == H_FREE && atomicCAS(&H.ctl, vv, H_SETUP) == vv) {
                            H.slot = (int)(&sl - slots);
                            H.seg_e = sq;
                            H.done_seg = 0;
                            H.best = ~0ull;
                            H.c = c;
                            H.seed = S.seed;
                            H.qid = S.qid;
                            H.t = S.t;
                            sl.state = ST_HUB;
                            __threadfence_block();
                            atomicExch(&H.ctl, H_ACTIVE | (unsigned)((d - ra + sq - 1) / sq) << 16);
                            atomicAdd(&head.hub_open, 1);
                            ok = 1;
                            break;
                        }
                    }
                }
                if (!__shfl_sync(FULL, ok, 0)) {
                    // no free task entry: the walk stays ready and is
                    // published on a later visit, after this warp has helped
                    // the open tasks
                    __nanosleep(nap);
                    nap = min(nap * 2u, 1024u);
                }
                continue;
            }
        }
        idle_since = 0;
        nap = 128;

        // ------------------------------------ stream the row range (one site)
        // A hub segment is one range.  A row sampled by this warp alone is
        // cut into the hub path's segments, segment j drawing from random
        // stream j, and the step keeps the smallest (race time, index) over
        // them, as a hub task's merge does.
        unsigned long long best = ~0ull;
        for (; ra < lim; ra += sq) {
            Res R;
            R.init();
            scan_range<N2V>(g, c, ra, min(lim, ra + sq), lane, R, S);
            if (R.sel >= 0) best = min(best, race_key(R));
            ++S.id;
        }

        // ------------------------------------------------ use the result
        if (lane == 0) {
            Slot* sp = &mine[max(s, 0)];
            bool fin = true;
            if (seg) {
                // fold the segment into its hub task; the warp that completes
                // the last segment finishes the step
                HubTask& H = head.hub[h];
                if (best != ~0ull) atomicMin(&H.best, best);
                __threadfence_block();
                fin = atomicAdd(&H.done_seg, 1) == hub_nseg(*(volatile unsigned*)&H.ctl) - 1;
                __threadfence_block();
                sp = &slots[H.slot];
                best = *(volatile unsigned long long*)&H.best;
            }
            if (fin) {
                if (best == ~0ull) {
                    __threadfence_block();
                    *(volatile int*)&sp->state = ST_FINISH;  // nothing selectable: the walk stops here
                } else {
                    count_step(cnt, c.d, c.algo, seg);
                    commit(g, *sp, c.beg, c.d, (int)(best & 0xFFFFFFFFull), S.seed, S.qid, S.t, seg);
                }
                if (seg) {
                    __threadfence_block();
                    atomicExch(&head.hub[h].ctl, H_FREE);
                }
            }
        }
        __syncwarp();
    }
    cp_async_wait_all();
    __syncwarp();
    if (lane == 0) flush_counts(cnt, counters);
}

}  // namespace
}  // namespace fw
