// Launches of the walk engine, instantiated for fast mode in fw_fast.cu and for
// exact mode in fw_exact.cu (two translation units build in parallel).
#pragma once

#include <string.h>

#include "fw_engine.cuh"

namespace fw {
namespace {

constexpr int kSmemLimit = 227 * 1024;  // dynamic shared memory a CTA may have

// Grid and shared memory of one engine launch: every SM filled as far as the
// kernel's registers and shared memory allow (at most tu.ctas_per_sm CTAs each).
template <typename K>
cudaError_t engine_grid(K kern, int threads, size_t smem, const Tuning& tu, int* sms, int* per_sm) {
    // always the same limit: it belongs to the function, and another thread may be
    // about to launch the same kernel with more than this call needs
    if (smem > (size_t)kSmemLimit) return cudaErrorInvalidConfiguration;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit);
    if (e != cudaSuccess) return e;
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev);
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, kern, threads, smem);
    if (e != cudaSuccess) return e;
    if (*per_sm < 1) return cudaErrorInvalidConfiguration;
    if (tu.ctas_per_sm > 0) *per_sm = min(*per_sm, tu.ctas_per_sm);
    return cudaSuccess;
}

// One walk per warp unless the caller asked for more: a walk that goes on at once
// finds the row it came from (node2vec's N(prev)) still in L2, and its slots'
// shared memory is L1's.  Measured against four walks taken in turn (ms):
// node2vec R-MAT-25 187.1 -> 182.4, R-MAT-20 35.8 -> 33.1, exact 12.9 -> 10.4,
// weighted R-MAT-22 15.8 -> 15.0, MetaPath + PPR 7.9 -> 7.3.
inline int walks_per_warp(const Tuning& tu) {
    return max(1, min(kSlotsPerWarp, tu.slots / (tu.block_threads / 32)));
}

template <bool EXACT, bool N2V, bool LAB, bool PPR>
cudaError_t launch_as(const GraphDev& g, const ReqTable& reqs, int n_req, int64_t total, unsigned long long* cursor,
                      unsigned long long* counters, const Tuning& tu, cudaStream_t stream) {
    auto kern = walk_kernel<EXACT, N2V, LAB, PPR, false>;
    const int sw = walks_per_warp(tu);
    // CTAs of 256 threads unless the caller chose: at 80 registers three of
    // them fill an SM with 24 warps where 512-thread CTAs leave it at 16
    // (R-MAT-25 node2vec: 240 -> 202 ms), and a hub row's last segments hold
    // back 8 warps instead of 16 (PPR from the R-MAT-22 hub: 5.7 -> 4.8 ms).
    int threads = tu.block_threads, use = sw;
    int sms = 0, per_sm = 0;
    cudaError_t e = engine_grid(kern, threads, cta_smem<EXACT, N2V>(threads / 32, sw), tu, &sms, &per_sm);
    if (e != cudaSuccess) return e;
    const int64_t resident = (int64_t)sms * per_sm * (threads / 32);
    int64_t grid = (int64_t)sms * per_sm;
    Launch L = {reqs.ext, n_req, (long long)total, cursor, counters, tu.d_warp, threads / 32, kSegQuads, 4096u};
    int d_t = tu.d_warp;
    if (!tu.own_d()) {
        // Sharing a row costs throughput (hand-offs, fresh N(prev) cursors,
        // waiting owners) and gains latency: unless the caller set d_t, rows
        // from one segment on are shared while the CTA has a warp without walks
        // of its own.  Fast mode does not share otherwise (PPR from the
        // R-MAT-22 hub: 4.7 -> 4.1 ms); exact mode does above the default d_t.
        d_t = 4 * kSegQuads;
        if (!EXACT) L.d_always = 1 << 30;
    }
    if (total < resident) {
        // Fewer walks than resident warps: latency counts.  One walk per warp
        // (a warp advances its walks one after another), spread evenly over
        // the CTAs.  Hub rows begin at one segment (fast mode) or where the
        // pieces are still worth a hand-off (exact mode); where the graph has
        // such rows, one large CTA per SM keeps warps at hand for them, as long
        // as its 24 warps hold all walks: a first-order launch of 25 to 32 walks
        // per SM would run the rest as a second round (4,800 weighted walks of
        // 80 on R-MAT-22, fast 1,416 us with the large CTAs, 1,152 without).
        // Measured (us): 1,000 exact walks of 80 on a 1,000-vertex graph 617
        // (four walks per warp) -> 222 (174 with what came later); 32 node2vec walks of 40 on R-MAT-22,
        // fast 868 -> 777, exact 1,095 -> 712 (helpers); 129 PPR walks on
        // R-MAT-22 222 -> 201.
        use = 1;
        if (!tu.own_d() && EXACT) {
            d_t = 4096;
            L.seg_q = 512;
        }
        if (!tu.own_shape() && g.d_max > d_t) {
            int wide = 0;
            e = engine_grid(kern, 768, cta_smem<EXACT, N2V>(24, use), tu, &sms, &wide);
            if (e != cudaSuccess) return e;
            if (total <= (int64_t)sms * wide * 24) {
                threads = 768;
                per_sm = wide;
            }
        }
        grid = min((int64_t)sms * per_sm, total);
        L.claimers = (int)((total + grid - 1) / grid);
        L.nap = 512u;
    } else {
        use = (int)min((int64_t)sw, total / resident);
    }
    if (g.d_max <= d_t) L.nap = 0u;  // no hub tasks: warps without walks return at once
    const size_t smem = cta_smem<EXACT, N2V>(threads / 32, use);
    ServeDev none;
    memset(&none, 0, sizeof none);
    kern<<<(unsigned)grid, threads, smem, stream>>>(g, reqs, L, use, d_t, none);
    return cudaGetLastError();
}

template <bool EXACT>
cudaError_t launch_mode(const GraphDev& g, const ReqTable& reqs, int n_req, int64_t total, unsigned long long* cursor,
                        unsigned long long* counters, const Tuning& tu, cudaStream_t stream) {
    const bool n2v = reqs.algos >> FW_NODE2VEC & 1u;
    const bool lab = reqs.algos >> FW_METAPATH & 1u, ppr = reqs.algos >> FW_PPR & 1u;
    const auto as = n2v ? (lab ? launch_as<EXACT, true, true, true> : ppr ? launch_as<EXACT, true, false, true> : launch_as<EXACT, true, false, false>)
                        : (lab ? launch_as<EXACT, false, true, true> : launch_as<EXACT, false, false, true>);
    return as(g, reqs, n_req, total, cursor, counters, tu, stream);
}

template <bool EXACT>
cudaError_t serve_mode(const GraphDev& g, const ServeDev& sv, Scratch* scratch, const Tuning& tu, cudaStream_t stream) {
    auto kern = walk_kernel<EXACT, true, true, true, true>;
    // One 768-thread CTA fills an SM (24 warps of 80 registers), so that the
    // eight SMs left out below are wholly free for other streams' kernels.
    // Filling every SM would hold those back for as long as the server runs,
    // and through the hardware queues streams share, the server's own copies
    // queued behind them.
    const int warps = 24, sw = 1;
    const size_t smem = cta_smem<EXACT, true>(warps, sw);
    int sms = 0, per_sm = 0;
    cudaError_t e = engine_grid(kern, warps * 32, smem, tu, &sms, &per_sm);
    if (e != cudaSuccess) return e;
    ReqTable tab;
    memset(&tab, 0, sizeof tab);
    const Launch L = {nullptr, 0, 0ll, &scratch->cursor, scratch->counters, tu.d_warp, warps, kSegQuads, 0u};
    kern<<<(unsigned)(sms - min(8, sms - 1)), warps * 32, smem, stream>>>(g, tab, L, sw, tu.d_warp, sv);
    return cudaGetLastError();
}

}  // namespace
}  // namespace fw
