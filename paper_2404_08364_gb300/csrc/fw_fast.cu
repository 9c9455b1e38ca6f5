// Launches of the fast-mode walk engine.
#include <string.h>

#include "fw_engine.cuh"

namespace fw {
namespace {

// Grid and shared memory of one engine launch: every SM filled as far as the
// kernel's registers and shared memory allow (at most tu.ctas_per_sm CTAs each).
template <typename K>
cudaError_t engine_grid(K kern, int threads, size_t smem, const Tuning& tu, int* sms, int* per_sm) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
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

}  // namespace

cudaError_t launch_fast(const GraphDev& g, const ReqTable& reqs, int n_req, int64_t total, unsigned long long* cursor,
                        unsigned long long* counters, const Tuning& tu, cudaStream_t stream) {
    auto kern = fast_kernel<false, false>;
    const int warps = tu.block_threads / 32;
    const int sw = max(1, min(SW_MAX, tu.slots / warps));
    const size_t smem = cta_smem<false>(warps, sw);
    int sms = 0, per_sm = 0;
    cudaError_t e = engine_grid(kern, tu.block_threads, smem, tu, &sms, &per_sm);
    if (e != cudaSuccess) return e;
    const int64_t per_cta = (int64_t)sw * warps;
    const int64_t grid = min((int64_t)sms * per_sm, (total + per_cta - 1) / per_cta);
    ServeDev none;
    memset(&none, 0, sizeof none);
    kern<<<(unsigned)grid, tu.block_threads, smem, stream>>>(g, reqs, n_req, (long long)total, cursor, counters, sw,
                                                             tu.d_warp, none);
    return cudaGetLastError();
}

}  // namespace fw
