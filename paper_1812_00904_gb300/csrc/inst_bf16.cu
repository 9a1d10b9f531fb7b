// Instantiations of the streaming kernel for __nv_bfloat16 values and float vectors (one translation unit
// per value type, so that the instantiations compile in parallel).
#include "pass_kernel.cuh"
#include "stream_kernel.cuh"

namespace gbk {

cudaError_t launch_stream_bf16(int mode, int kb, const LaunchArgs &a) { return launch_mode<__nv_bfloat16, float>(mode, kb, a); }
cudaError_t launch_pass_bf16(bool sc, bool sd, const PassParams &p, int grid, int warps, int smem,
                            cudaStream_t s) {
    return launch_pass<__nv_bfloat16, float>(sc, sd, p, grid, warps, smem, s);
}
cudaError_t launch_mvdot_bf16(int kv, bool onchip, const PassParams &p, int grid, int warps, int smem, cudaStream_t s) {
    return launch_mvdot<__nv_bfloat16>(kv, onchip, p, grid, warps, smem, s);
}
cudaError_t launch_mvscatter_bf16(int kv, const PassParams &p, int grid, int warps, int smem, cudaStream_t s) {
    return launch_mvscatter<__nv_bfloat16>(kv, p, grid, warps, smem, s);
}
cudaError_t launch_dvalues_bf16(const PassParams &p, int grid, int warps, int smem, cudaStream_t s) {
    return launch_dvalues<__nv_bfloat16, float>(p, grid, warps, smem, s);
}

}  // namespace gbk
