// The walk engine's exact mode.
#include "fw_launch.cuh"

namespace fw {

cudaError_t launch_exact(const GraphDev& g, const ReqTable& reqs, int n_req, int64_t total, unsigned long long* cursor,
                        unsigned long long* counters, const Tuning& tu, cudaStream_t stream) {
    return launch_mode<true>(g, reqs, n_req, total, cursor, counters, tu, stream);
}

cudaError_t launch_exact_serve(const GraphDev& g, const ServeDev& sv, Scratch* scratch, const Tuning& tu,
                              cudaStream_t stream) {
    return serve_mode<true>(g, sv, scratch, tu, stream);
}

}  // namespace fw
