// Which engine a walk launch goes to, and the engine's tuning.
#include "fw_internal.cuh"

namespace fw {

Tuning default_tuning() { return Tuning{256, 8, 65536, 0}; }

Tuning sanitize_tuning(Tuning t) {
    const Tuning d = default_tuning();
    // (a caller who limits the CTAs per SM gets large ones; slots without a CTA
    // size are counted per 512 threads, whatever size the engine takes)
    if (t.block_threads != 128 && t.block_threads != 256 && t.block_threads != 512) {
        t.block_threads = t.ctas_per_sm > 0 ? 512 : d.block_threads;
        if (t.slots > 0) t.slots = (t.slots > 16 ? t.slots / 16 : 1) * (t.block_threads / 32);
    }
    const int warps = t.block_threads / 32;
    if (t.slots <= 0) t.slots = warps;
    if (t.slots > warps * kSlotsPerWarp) t.slots = warps * kSlotsPerWarp;
    if (t.d_warp <= 0) t.d_warp = d.d_warp;
    if (t.d_warp < 128) t.d_warp = 128;
    if (t.d_warp > (1 << 30)) t.d_warp = 1 << 30;
    if (t.ctas_per_sm < 0) t.ctas_per_sm = 0;
    return t;
}

cudaError_t launch_serve(const GraphDev& g, int mode, const ServeDev& sv, Scratch* scratch, const Tuning& tune,
                         cudaStream_t stream) {
    const Tuning tu = sanitize_tuning(tune);
    return mode == FW_EXACT ? launch_exact_serve(g, sv, scratch, tu, stream) : launch_fast_serve(g, sv, scratch, tu, stream);
}

cudaError_t launch_walk(const GraphDev& g, int mode, const ReqTable& reqs, int n_req, int64_t total,
                        unsigned long long* cursor, unsigned long long* counters, const Tuning& tune,
                        cudaStream_t stream) {
    const Tuning tu = sanitize_tuning(tune);
    if (total <= 0) return cudaSuccess;
    return mode == FW_EXACT ? launch_exact(g, reqs, n_req, total, cursor, counters, tu, stream)
                            : launch_fast(g, reqs, n_req, total, cursor, counters, tu, stream);
}

}  // namespace fw
