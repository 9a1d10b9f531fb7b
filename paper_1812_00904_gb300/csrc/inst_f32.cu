// Instantiations of the streaming kernel for float values and float vectors (one translation unit
// per value type, so that the instantiations compile in parallel).
#include "pass_kernel.cuh"
#include "stream_kernel.cuh"

namespace gbk {

cudaError_t launch_stream_f32(int mode, int kb, const LaunchArgs &a) { return launch_mode<float, float>(mode, kb, a); }
cudaError_t launch_pass_f32(bool sc, bool sd, const PassParams &p, int grid, int warps, int smem,
                            cudaStream_t s) {
    return launch_pass<float, float>(sc, sd, p, grid, warps, smem, s);
}
cudaError_t launch_mvdot_f32(int kv, bool onchip, const PassParams &p, int grid, int warps, int smem, cudaStream_t s) {
    return launch_mvdot<float>(kv, onchip, p, grid, warps, smem, s);
}
cudaError_t launch_mvscatter_f32(int kv, const PassParams &p, int grid, int warps, int smem, cudaStream_t s) {
    return launch_mvscatter<float>(kv, p, grid, warps, smem, s);
}
cudaError_t launch_dvalues_f32(const PassParams &p, int grid, int warps, int smem, cudaStream_t s) {
    return launch_dvalues<float, float>(p, grid, warps, smem, s);
}

}  // namespace gbk
