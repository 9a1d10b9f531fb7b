// Instantiations of the streaming kernel for __half values and float vectors (one translation unit
// per value type, so that the instantiations compile in parallel).
#include "pass_kernel.cuh"
#include "stream_kernel.cuh"

namespace gbk {

cudaError_t launch_stream_f16(int mode, int kb, const LaunchArgs &a) { return launch_mode<__half, float>(mode, kb, a); }
cudaError_t launch_pass_f16(bool sc, bool sd, const PassParams &p, int grid, int warps, int smem,
                            cudaStream_t s) {
    return launch_pass<__half, float>(sc, sd, p, grid, warps, smem, s);
}
cudaError_t launch_mvdot_f16(int kv, bool onchip, const PassParams &p, int grid, int warps, int smem, cudaStream_t s) {
    return launch_mvdot<__half>(kv, onchip, p, grid, warps, smem, s);
}
cudaError_t launch_mvscatter_f16(int kv, const PassParams &p, int grid, int warps, int smem, cudaStream_t s) {
    return launch_mvscatter<__half>(kv, p, grid, warps, smem, s);
}
cudaError_t launch_dvalues_f16(const PassParams &p, int grid, int warps, int smem, cudaStream_t s) {
    return launch_dvalues<__half, float>(p, grid, warps, smem, s);
}

}  // namespace gbk
