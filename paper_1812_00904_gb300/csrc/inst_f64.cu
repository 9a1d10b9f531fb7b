// Instantiations of the streaming kernel for double values and double vectors (one translation unit
// per value type, so that the instantiations compile in parallel).
#include "pass_kernel.cuh"
#include "stream_kernel.cuh"

namespace gbk {

cudaError_t launch_stream_f64(int mode, int kb, const LaunchArgs &a) { return launch_mode<double, double>(mode, kb, a); }
cudaError_t launch_pass_f64(bool sc, bool sd, const PassParams &p, int grid, int warps, int smem,
                            cudaStream_t s) {
    return launch_pass<double, double>(sc, sd, p, grid, warps, smem, s);
}
cudaError_t launch_dvalues_f64(const PassParams &p, int grid, int warps, int smem, cudaStream_t s) {
    return launch_dvalues<double, double>(p, grid, warps, smem, s);
}

}  // namespace gbk
