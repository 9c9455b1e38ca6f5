// Parallel weighted samplers side by side (Section 4): the paper's direct
// parallel reservoir sampling (DPRS, Alg. 3) and zig-zag parallel reservoir
// sampling (ZPRS, Alg. 4), and the exponential-jump reservoir the walk engine
// uses (its fast mode), each run by a group of k threads (a warp, k = 32, or a
// CTA, k = 256) drawing one index from one weight array.
//
// Many independent draws run at once (one per sampler group, `reps` in all)
// over the same weights, so the timing measures the samplers' collective and
// random-number costs (Section 4's beta and gamma) rather than DRAM: every
// array here fits in L2.  Each draw r uses random counters of its own, so the
// returned indices are independent draws from w_i / sum(w).
#include <stdarg.h>
#include <stdio.h>

#include "fw_internal.cuh"

using namespace fw;

namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int SAMP_EXPJ = 0, SAMP_DPRS = 1, SAMP_ZPRS = 2;

int fail_s(int status, const char* fmt, ...) {
    char buf[300];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    return set_error(status, buf);
}

// uniform in [0, 1) from 24 random bits
__device__ __forceinline__ float unit24(uint32_t x) { return (float)(x >> 8) * (1.0f / 16777216.0f); }
// uniform in (0, 1): 23 bits centred in their cell
__device__ __forceinline__ float unit_open23(uint32_t x) { return ((float)(x >> 9) + 0.5f) * (1.0f / 8388608.0f); }

// Per-element uniforms for thread j of draw r: one Philox block gives the
// uniforms of the thread's iterations 4c .. 4c + 3.
__device__ __forceinline__ uint4 elem_block(uint64_t seed, uint64_t r, uint32_t j, uint32_t c) {
    return philox4x32_10(make_uint4((uint32_t)r, (uint32_t)(r >> 32), j, c), make_uint2((uint32_t)seed, (uint32_t)(seed >> 32)));
}

// The selection test of Alg. 3 and 4, u < w / S, for four elements: bit q of
// the result.  Rarely by a division: a product u S above w by more than the
// rounding of either side already says no (the summand keeps denormal weights
// on the exact test).
__device__ __forceinline__ unsigned picks(const uint4& x, const float (&w)[4], const float (&S)[4]) {
    const float u[4] = {unit24(x.x), unit24(x.y), unit24(x.z), unit24(x.w)};
    bool maybe[4], any = false;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        maybe[q] = w[q] > 0.0f && !(u[q] * S[q] > __fmaf_rn(w[q], 1.000001f, 1e-30f));
        any = any || maybe[q];
    }
    unsigned m = 0;
    if (any) {
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (maybe[q] && u[q] < w[q] / S[q]) m |= 1u << q;
    }
    return m;
}

__device__ __forceinline__ uint32_t pick_word(const uint4& b, int i) {
    return (i & 3) == 0 ? b.x : (i & 3) == 1 ? b.y : (i & 3) == 2 ? b.z : b.w;
}

// Four weights of thread j: w[b + q K + j], 0 past n.
template <int K>
__device__ __forceinline__ void load4(const float* __restrict__ w, uint32_t n, uint32_t b, uint32_t j, float (&v)[4]) {
    if (b + 4 * K <= n) {
        const float* p = w + b + j;
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] = __ldg(p + q * K);
    } else {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const uint32_t e = b + q * K + j;
            v[q] = 0.0f;
            if (b + q * K < n && e < n) v[q] = __ldg(w + e);
        }
    }
}

__device__ __forceinline__ float warp_incl_scan(float v, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const float n = __shfl_up_sync(FULL, v, o);
        if (lane >= o) v += n;
    }
    return v;
}

// A group of K threads: a warp (K = 32) or a CTA (K = 256, with shared buffers).
template <int K>
struct Group {
    float* fbuf;   // 2 x 4 x 8 floats
    int* ibuf;     // 8 ints
    int tid;

    __device__ __forceinline__ int max_int(int v) {
        v = __reduce_max_sync(FULL, v);
        if (K == 32) return v;
        __syncthreads();
        if ((tid & 31) == 0) ibuf[tid >> 5] = v;
        __syncthreads();
        int m = ibuf[0];
        for (int i = 1; i < K / 32; ++i) m = max(m, ibuf[i]);
        return m;
    }
};

// Inclusive prefix sum of one value per thread over the group.
template <int K>
__device__ __forceinline__ float group_scan(Group<K>& G, float v) {
    const int lane = G.tid & 31, wp = G.tid >> 5;
    v = warp_incl_scan(v, lane);
    if (K == 32) return v;
    __syncthreads();
    if (lane == 31) G.fbuf[wp] = v;
    __syncthreads();
    float before = 0.0f;
    for (int i = 0; i < wp; ++i) before += G.fbuf[i];
    return v + before;
}

// At most one element per thread (n <= K): the selected index is the thread's
// own, so both algorithms end in one maximum; they differ in how they round
// the running total.  (On 2^18 draws of 32 weights at warp width the
// four-element code takes 112 us.)
template <int K, bool ZIG>
__device__ int draw_short(Group<K>& G, const float* __restrict__ w, uint32_t n, uint64_t seed, uint64_t r) {
    const int j = G.tid;
    const float v = j < n ? __ldg(w + j) : 0.0f;
    const float u = unit24(elem_block(seed, r, (uint32_t)j, 0).x);
    const float incl = group_scan<K>(G, v);
    const float S = ZIG ? (incl - v) + v : incl;
    return G.max_int(v > 0.0f && u < v / S ? j : -1);
}

// ZPRS's result: the selection of the highest thread that selected anything.
template <int K>
__device__ __forceinline__ int zprs_winner(Group<K>& G, int C) {
    const int top = G.max_int(C >= 0 ? G.tid : -1);
    // broadcast the winner's C (K <= 256: through the group's int buffer)
    if (K == 32) return top < 0 ? -1 : __shfl_sync(FULL, C, top);
    __syncthreads();
    if (G.tid == top) G.ibuf[0] = C;
    __syncthreads();
    return top < 0 ? -1 : G.ibuf[0];
}

// Few elements per thread: one per iteration (the four-element code below
// pays for its empty places: on 2^18 draws of 33 weights at warp width it takes
// 121 us instead of 89).
template <int K>
__device__ int draw_dprs_few(Group<K>& G, const float* __restrict__ w, uint32_t n, uint64_t seed, uint64_t r) {
    const int j = G.tid, lane = j & 31, wp = j >> 5;
    float wB = 0.0f;
    int C = -1, i = 0;
    uint4 blk = make_uint4(0, 0, 0, 0);
#pragma unroll 1
    for (uint32_t b = 0; b < n; b += K, ++i) {
        const float wl = b + j < n ? __ldg(w + b + j) : 0.0f;
        float S = warp_incl_scan(wl, lane), tot;
        if (K == 32) {
            tot = __shfl_sync(FULL, S, 31);
        } else {
            float* f = G.fbuf + (i & 1) * 32;
            if (lane == 31) f[wp] = S;
            __syncthreads();
            float before = 0.0f;
            tot = 0.0f;
#pragma unroll
            for (int k = 0; k < K / 32; ++k) {
                const float fk = f[k];
                if (k == wp) S += before;
                if (k == K / 32 - 1) tot = fk + before;
                before += fk;
            }
        }
        if ((i & 3) == 0) blk = elem_block(seed, r, (uint32_t)j, (uint32_t)i >> 2);
        if (wl > 0.0f && unit24(pick_word(blk, i)) < wl / (S + wB)) C = (int)(b + j);
        wB += tot;
    }
    return G.max_int(C);
}

template <int K>
__device__ int draw_zprs_few(Group<K>& G, const float* __restrict__ w, uint32_t n, uint64_t seed, uint64_t r) {
    const int j = G.tid;
    float s = 0.0f;
    for (uint32_t e = j; e < n; e += K) s += __ldg(w + e);
    float P = group_scan<K>(G, s) - s;  // exclusive
    int C = -1, i = 0;
    uint4 blk = make_uint4(0, 0, 0, 0);
#pragma unroll 1
    for (uint32_t e = j; e < n; e += K, ++i) {
        const float we = __ldg(w + e);
        P += we;
        if ((i & 3) == 0) blk = elem_block(seed, r, (uint32_t)j, (uint32_t)i >> 2);
        if (we > 0.0f && unit24(pick_word(blk, i)) < we / P) C = (int)e;
    }
    return zprs_winner(G, C);
}

// DPRS (Alg. 3): per iteration, k consecutive weights, their inclusive
// prefix sum plus the weight of the earlier iterations (w_B), one uniform per
// element against w / (W_P + w_B); the largest selected index wins.  Four
// iterations share a Philox block: their scans run side by side (and, at CTA
// width, through one barrier), and the maximum is taken once, at the end (a
// thread's later index is always the larger).
template <int K>
__device__ int draw_dprs(Group<K>& G, const float* __restrict__ w, uint32_t n, uint64_t seed, uint64_t r) {
    const int j = G.tid, lane = j & 31, wp = j >> 5;
    float wB = 0.0f;
    int C = -1;
    int half = 0;
#pragma unroll 1
    for (uint32_t b = 0; b < n; b += 4 * K) {
        const uint4 blk = elem_block(seed, r, (uint32_t)j, b / (4 * K));
        float wl[4], S[4], tot[4];
        load4<K>(w, n, b, (uint32_t)j, wl);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            S[q] = 0.0f;
            tot[q] = 0.0f;
            if (b + q * K < n) S[q] = warp_incl_scan(wl[q], lane);
        }
        if (K == 32) {
#pragma unroll
            for (int q = 0; q < 4; ++q) tot[q] = __shfl_sync(FULL, S[q], 31);
        } else {
            float* f = G.fbuf + half * 32;
            half ^= 1;
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (lane == 31) f[q * 8 + wp] = S[q];
            __syncthreads();
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                if (b + q * K >= n) break;
                float before = 0.0f;
#pragma unroll
                for (int i = 0; i < K / 32; ++i) {
                    const float fi = f[q * 8 + i];
                    if (i == wp) S[q] += before;
                    if (i == K / 32 - 1) tot[q] = fi + before;
                    before += fi;
                }
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            S[q] += wB;
            wB += tot[q];
        }
        const unsigned m = picks(blk, wl, S);
        if (m) C = (int)(b + (31 - __clz((int)m)) * K + j);
    }
    return G.max_int(C);
}

// ZPRS (Alg. 4): thread j sums its strided subsequence S_j, an exclusive
// prefix sum over the threads starts each running total, a second pass tests
// each element against w / (running total), and the selection of the highest
// thread that selected anything wins.  Both passes take four elements at a
// time, whose loads overlap; the second one's share a Philox block.
template <int K>
__device__ int draw_zprs(Group<K>& G, const float* __restrict__ w, uint32_t n, uint64_t seed, uint64_t r) {
    const int j = G.tid;
    float s = 0.0f;
#pragma unroll 4
    for (uint32_t b = 0; b < n; b += 4 * K) {
        float v[4];
        load4<K>(w, n, b, (uint32_t)j, v);
#pragma unroll
        for (int q = 0; q < 4; ++q) s += v[q];
    }
    float P = group_scan<K>(G, s) - s;  // exclusive
    int C = -1;
#pragma unroll 1
    for (uint32_t b = 0; b < n; b += 4 * K) {
        float v[4], S[4];
        load4<K>(w, n, b, (uint32_t)j, v);
        const uint4 blk = elem_block(seed, r, (uint32_t)j, b / (4 * K));
#pragma unroll
        for (int q = 0; q < 4; ++q) S[q] = P += v[q];
        const unsigned m = picks(blk, v, S);
        if (m) C = (int)(b + (31 - __clz((int)m)) * K + j);
    }
    return zprs_winner(G, C);
}

// The engine's sampler: a warp's exponential race with exponential jumps
// over 128-entry chunks (a sum per chunk, a record only when the skip budget
// runs out), X kept as an FP32 two-sum; at CTA width each warp takes a
// contiguous segment with its own random stream and the smallest race time
// wins (ties: smaller index).  Record i uses block i of the stream; lane l
// holds the draws of record have - 32 + l, handed out by shuffles.
struct Race {
    float tau, Xh, Xl;
    int sel;
    uint32_t i, have;
    float u1, nl2;  // this lane's draws: u1 and -log u2
};

// One chunk, at `base`: the skip budget past it, with every record inside it,
// in visiting order; wv: this lane's weights, own: their sum.
__device__ __forceinline__ void race_chunk(Race& R, const float (&wv)[4], float own, int64_t base, int lane,
                                           uint64_t seed, uint64_t r, uint32_t stream) {
    const float incl = warp_incl_scan(own, lane);
    const float tot = __shfl_sync(FULL, incl, 31);
    if (R.Xh - tot + R.Xl > 0.0f) {
        const float sh = R.Xh - tot;
        R.Xl += (R.Xh - sh) - tot;
        R.Xh = sh;
        return;
    }
    float cum[4];
    cum[0] = (incl - own) + wv[0];
#pragma unroll
    for (int q = 1; q < 4; ++q) cum[q] = cum[q - 1] + wv[q];
    float target = R.Xh + R.Xl;
    int last = -1;
#pragma unroll 1
    for (;;) {
        int jj = -1;
#pragma unroll
        for (int q = 3; q >= 0; --q)
            if (lane * 4 + q > last && wv[q] > 0.0f && cum[q] >= target) jj = q;
        const unsigned m = __ballot_sync(FULL, jj >= 0);
        if (!m) {
            R.Xh = target - tot;
            R.Xl = 0.0f;
            return;
        }
        const int L = __ffs(m) - 1;
        const float wj = jj >= 2 ? (jj == 3 ? wv[3] : wv[2]) : (jj == 1 ? wv[1] : wv[0]);
        const float cj = jj >= 2 ? (jj == 3 ? cum[3] : cum[2]) : (jj == 1 ? cum[1] : cum[0]);
        const float wr = __shfl_sync(FULL, wj, L);
        const float cr = __shfl_sync(FULL, cj, L);
        last = L * 4 + __shfl_sync(FULL, jj, L);
        if (R.i == R.have) {
            const uint4 o = philox4x32_10(make_uint4((uint32_t)r, (uint32_t)(r >> 32), 0x80000000u | stream, R.i + lane),
                                          make_uint2((uint32_t)seed, (uint32_t)(seed >> 32)));
            R.u1 = unit_open23(o.x);
            R.nl2 = -logf(unit_open23(o.y));
            R.have += 32;
        }
        const float u1 = __shfl_sync(FULL, R.u1, R.i), nl = __shfl_sync(FULL, R.nl2, R.i);
        ++R.i;
        float e;
        if (isinf(R.tau)) e = -logf(u1);
        else e = -log1pf(u1 * expm1f(-wr * R.tau));
        R.tau = e / wr;
        R.sel = (int)(base + last);
        R.Xh = nl / R.tau;
        target = cr + R.Xh;
    }
}

__device__ __forceinline__ Race race_start() {
    Race R;
    R.tau = __int_as_float(0x7f800000);
    R.Xh = 0.0f;
    R.Xl = 0.0f;
    R.sel = -1;
    R.i = 0;
    R.have = 0;
    return R;
}

// Past the first records, four chunks at a time: a chunk's total is the sum
// that its scan leaves in lane 31, here by an xor butterfly (the same pairs in
// the same order); the four butterflies share all but their first two steps.
// vec: w is 16-byte aligned.
__device__ Race race_segment(const float* __restrict__ w, int64_t a, int64_t b, int lane, uint64_t seed, uint64_t r,
                             uint32_t stream, bool vec) {
    Race R = race_start();
    int64_t base = a;
    while (base < b) {
        if (R.i && base + 512 <= b) {
            float own[4], wv[4][4];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const float* p = w + base + c * 128 + lane * 4;
                if (vec) {
                    const float4 v = __ldg(reinterpret_cast<const float4*>(p));
                    wv[c][0] = v.x; wv[c][1] = v.y; wv[c][2] = v.z; wv[c][3] = v.w;
                } else {
#pragma unroll
                    for (int q = 0; q < 4; ++q) wv[c][q] = __ldg(p + q);
                }
                own[c] = (wv[c][0] + wv[c][1]) + (wv[c][2] + wv[c][3]);
            }
            const bool b0 = lane & 1, b1 = lane & 2;
            float v0 = b0 ? own[1] : own[0], v1 = b0 ? own[3] : own[2];
            v0 += __shfl_xor_sync(FULL, b0 ? own[0] : own[1], 1);
            v1 += __shfl_xor_sync(FULL, b0 ? own[2] : own[3], 1);
            float v = b1 ? v1 : v0;
            v += __shfl_xor_sync(FULL, b1 ? v0 : v1, 2);
#pragma unroll
            for (int o = 4; o < 32; o <<= 1) v += __shfl_xor_sync(FULL, v, o);
            float Xh = R.Xh, Xl = R.Xl;
            bool ok = true;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const float tot = __shfl_sync(FULL, v, c);
                ok = ok && Xh - tot + Xl > 0.0f;
                const float sh = Xh - tot;
                Xl += (Xh - sh) - tot;
                Xh = sh;
            }
            if (ok) {  // no record in any of them (the common case)
                R.Xh = Xh;
                R.Xl = Xl;
                base += 512;
                continue;
            }
        }
        // chunk by chunk: the first ones of a segment, its end, and the four
        // around a record
        const int64_t stop = R.i ? min(b, base + 512) : min(b, base + 128);
#pragma unroll 1
        for (; base < stop; base += 128) {
            float wv[4];
            const int64_t e = base + lane * 4;
#pragma unroll
            for (int q = 0; q < 4; ++q) wv[q] = e + q < b ? __ldg(w + e + q) : 0.0f;
            race_chunk(R, wv, (wv[0] + wv[1]) + (wv[2] + wv[3]), base, lane, seed, r, stream);
        }
    }
    return R;
}

// A segment of at most one chunk: an own kernel, whose fewer registers leave
// room for more warps (2^18 draws at warp width, in us: 4 weights 108 against 134,
// 127 weights 246 against 284; at CTA width 4 weights 290 against 435).
__device__ Race race_short(const float* __restrict__ w, int a, int b, int lane, uint64_t seed, uint64_t r, uint32_t stream) {
    Race R = race_start();
    const int e = a + lane * 4;
    float wv[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) wv[q] = e + q < b ? __ldg(w + e + q) : 0.0f;
    if (a < b) race_chunk(R, wv, (wv[0] + wv[1]) + (wv[2] + wv[3]), a, lane, seed, r, stream);
    return R;
}

template <int K, bool SHORT>
__device__ int draw_expj(Group<K>& G, const float* __restrict__ w, int64_t n, uint64_t seed, uint64_t r) {
    const int lane = G.tid & 31;
    const bool vec = ((uintptr_t)w & 15) == 0;
    if (K == 32) return SHORT ? race_short(w, 0, (int)n, lane, seed, r, 0).sel : race_segment(w, 0, n, lane, seed, r, 0, vec).sel;
    // CTA width: K / 32 contiguous segments (multiples of 128 entries)
    const int wp = G.tid >> 5;
    const int64_t seg = ((n + K / 32 - 1) / (K / 32) + 127) / 128 * 128;
    const int64_t a = min(n, (int64_t)wp * seg), b = min(n, a + seg);
    const Race R = SHORT ? race_short(w, (int)a, (int)b, lane, seed, r, (uint32_t)wp)
                         : race_segment(w, a, b, lane, seed, r, (uint32_t)wp, vec);
    __shared__ unsigned long long best;
    if (G.tid == 0) best = ~0ull;
    __syncthreads();
    if (lane == 0 && R.sel >= 0) atomicMin(&best, ((unsigned long long)__float_as_uint(R.tau) << 32) | (unsigned)R.sel);
    __syncthreads();
    const unsigned long long bv = best;
    __syncthreads();
    return bv == ~0ull ? -1 : (int)(bv & 0xFFFFFFFFull);
}

// Each form of a sampler is a kernel of its own, with the registers it needs (2^18
// draws of 200 weights at warp width by DPRS: 174 us, 195 with all in one kernel):
// one chunk or element per thread (SHORT), few (FEW), any number (LONG).  CTAs
// per SM: the four-chunk race needs 48 registers, a single chunk 40; at CTA
// width 32 with a few spills are better there, as the barriers want more warps
// (2^18 draws of 32 weights: 462 us against 533).  DPRS and ZPRS run on 32
// throughout; their LONG builds at warp width spill a little for it (52 and 16
// bytes) and are faster than on 40 without (2^18 draws of 2,000 weights: DPRS
// 1,051 us against 1,128, ZPRS 727 against 794; only ZPRS at 2^20 weights is
// slower, 6.98 ms against 6.73 for 4,096 draws).
enum Form { SHORT, FEW, LONG };
template <int METHOD, int K, Form FORM>
__global__ void __launch_bounds__(256, METHOD == SAMP_EXPJ && FORM == LONG   ? 5
                                       : K == 32 && METHOD == SAMP_EXPJ ? 6
                                       : 8) sampler_kernel(
    const float* __restrict__ w, int64_t n, int64_t reps, uint64_t seed, int32_t* __restrict__ out) {
    __shared__ float fbuf[64];
    __shared__ int ibuf[8];
    Group<K> G;
    G.fbuf = fbuf;
    G.ibuf = ibuf;
    G.tid = (int)(threadIdx.x % K);
    const int groups = (int)(blockDim.x / K);
    const int gi = (int)(threadIdx.x / K);
    for (int64_t r = (int64_t)blockIdx.x * groups + gi; r < reps; r += (int64_t)gridDim.x * groups) {
        int sel;
        if (METHOD == SAMP_EXPJ) sel = draw_expj<K, FORM == SHORT>(G, w, n, seed, (uint64_t)r);
        else if (FORM == SHORT) sel = draw_short<K, METHOD == SAMP_ZPRS>(G, w, (uint32_t)n, seed, (uint64_t)r);
        else if (METHOD == SAMP_DPRS)
            sel = FORM == FEW ? draw_dprs_few<K>(G, w, (uint32_t)n, seed, (uint64_t)r)
                              : draw_dprs<K>(G, w, (uint32_t)n, seed, (uint64_t)r);
        else
            sel = FORM == FEW ? draw_zprs_few<K>(G, w, (uint32_t)n, seed, (uint64_t)r)
                              : draw_zprs<K>(G, w, (uint32_t)n, seed, (uint64_t)r);
        if (G.tid == 0) out[r] = sel;
    }
}

template <int METHOD, int K, Form FORM>
cudaError_t launch_form(const float* w, int64_t n, int64_t reps, uint64_t seed, int32_t* out, cudaStream_t st) {
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, sampler_kernel<METHOD, K, FORM>, 256, 0);
    if (e != cudaSuccess) return e;
    const int64_t groups = 256 / K;
    int64_t grid = (int64_t)sms * (per_sm > 0 ? per_sm : 1);
    const int64_t need = (reps + groups - 1) / groups;
    if (need < grid) grid = need;
    sampler_kernel<METHOD, K, FORM><<<(unsigned)grid, 256, 0, st>>>(w, n, reps, seed, out);
    return cudaGetLastError();
}

template <int METHOD, int K>
cudaError_t launch_sampler(const float* w, int64_t n, int64_t reps, uint64_t seed, int32_t* out, cudaStream_t st) {
    // (the lines between few and many lie where the two measured equal)
    constexpr int64_t kShort = METHOD != SAMP_EXPJ ? K : K == 32 ? 128 : 1024;  // the race: one chunk per warp
    constexpr int64_t kFew = METHOD == SAMP_EXPJ ? 0 : K == 32 ? 256 : 768;
    if (n <= kShort) return launch_form<METHOD, K, SHORT>(w, n, reps, seed, out, st);
    // (ZPRS at CTA width: five iterations cost less than two groups of four, for
    // 1,025 weights 499 us against 540, up to about here)
    const bool five = METHOD == SAMP_ZPRS && K == 256 && n > 4 * K && n <= 4 * K + K / 2;
    if (METHOD != SAMP_EXPJ && (n <= kFew || five)) return launch_form<METHOD, K, METHOD == SAMP_EXPJ ? LONG : FEW>(w, n, reps, seed, out, st);
    return launch_form<METHOD, K, LONG>(w, n, reps, seed, out, st);
}

}  // namespace

extern "C" int fw_sampler_run(int32_t method, int32_t width, const float* d_w, int64_t n, int64_t reps,
                              uint64_t seed, int32_t* d_out, void* stream, float* ms) {
    if (!d_w || !d_out) return fail_s(FW_EINVAL, "fw_sampler_run: NULL weights or output");
    if (n < 1 || n > 0x7fffffffll || reps < 1) return fail_s(FW_EINVAL, "fw_sampler_run: n must be in [1, 2^31), reps >= 1");
    if (width != 32 && width != 256) return fail_s(FW_EINVAL, "fw_sampler_run: width must be 32 or 256");
    if (method < SAMP_EXPJ || method > SAMP_ZPRS) return fail_s(FW_EINVAL, "fw_sampler_run: unknown method");
    cudaStream_t st = (cudaStream_t)stream;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (ms) {
        cudaEventCreate(&e0);
        cudaEventCreate(&e1);
        cudaEventRecord(e0, st);
    }
    cudaError_t e;
    if (width == 32) {
        e = method == SAMP_DPRS   ? launch_sampler<SAMP_DPRS, 32>(d_w, n, reps, seed, d_out, st)
            : method == SAMP_ZPRS ? launch_sampler<SAMP_ZPRS, 32>(d_w, n, reps, seed, d_out, st)
                                  : launch_sampler<SAMP_EXPJ, 32>(d_w, n, reps, seed, d_out, st);
    } else {
        e = method == SAMP_DPRS   ? launch_sampler<SAMP_DPRS, 256>(d_w, n, reps, seed, d_out, st)
            : method == SAMP_ZPRS ? launch_sampler<SAMP_ZPRS, 256>(d_w, n, reps, seed, d_out, st)
                                  : launch_sampler<SAMP_EXPJ, 256>(d_w, n, reps, seed, d_out, st);
    }
    if (ms) {
        cudaEventRecord(e1, st);
        cudaEventSynchronize(e1);
        float t = 0.0f;
        cudaEventElapsedTime(&t, e0, e1);
        *ms = t;
        cudaEventDestroy(e0);
        cudaEventDestroy(e1);
    }
    if (e != cudaSuccess) return fail_s(FW_ECUDA, "fw_sampler_run: %s", cudaGetErrorString(e));
    return FW_OK;
}
