// Cross-chunk combines: the sum of the per-CTA partial short vectors (the
// Allreduce of Sec. III) and the overlap-zone fixup (the per-zone reductions of
// Sec. IV-A).  Both add in FP64 and in a fixed order, so results do not depend
// on which CTA finished first; FP32 partials and (hi, lo) FP32 carry pairs are
// widened to FP64 on read.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>

#include "device_common.cuh"
#include "internal.h"
#include "zones.cuh"

namespace gbk {

struct OutPtrs {
    void *p[VL_MAX];
};
struct InPtrs {
    const void *p[VL_MAX];
};

// The cross-CTA sums after a pass, one launch for both kinds of block:
// - combine: out_b[i] = sum_{q < nparts} part[q * qstride + b * bstride + i].  A block takes 32
//   consecutive elements; its 8 thread rows sum the partials q = row, row + 8, ... in FP64 and the
//   row sums are added in row order: a fixed order, independent of timing.  Partials of any type
//   are widened to FP64 before they are added.  The FP64 additions (2 a cycle per SM) set the
//   floor, 5 us for 152 partials of 20,000 elements; the loads of FIN_CB partials go together.
// - fix-up: the overlap zones' sums (zones.cuh), one thread per zone, into the zones' columns.
// blockIdx.y is the vector.
struct FinishArgs {
    int comb_blocks;  // blocks [0, comb_blocks) combine, the others fix up
    const void *part;
    int nparts, n_minor;
    size_t qstride, bstride;
    const ZoneDev *zones;
    int z, P;
    const void *rec_left, *rec_right;
    OutPtrs short_out, long_out;
};
constexpr int FIN_CB = 10;
template <typename XT, typename PT, typename RT>
__global__ void __launch_bounds__(FIN_X * FIN_ROWS) finish_kernel(const __grid_constant__ FinishArgs p) {
    __shared__ double sh_s[FIN_ROWS][FIN_X];
    const int b = blockIdx.y;
    if ((int)blockIdx.x >= p.comb_blocks) {
        const int k = (blockIdx.x - p.comb_blocks) * (FIN_X * FIN_ROWS) + threadIdx.x;
        const ZoneDev zd = k < p.z ? p.zones[k] : ZoneDev{0, 0, 0, 0};
        grid_wait();  // the records of the pass launched before
        const double t = zone_sum(k < p.z, zd, static_cast<const RT *>(p.rec_left) + (size_t)b * p.P,
                                  static_cast<const RT *>(p.rec_right) + (size_t)b * p.P);
        if (k < p.z) static_cast<XT *>(p.long_out.p[b])[zd.col] = static_cast<XT>(t);
        return;
    }
    const int tx = threadIdx.x & 31, row = threadIdx.x >> 5;
    const int i = blockIdx.x * FIN_X + tx;
    grid_wait();  // the partials
    double s = 0.0;
    if (i < p.n_minor) {
        const PT *src = static_cast<const PT *>(p.part) + (size_t)b * p.bstride + i;
        for (int q = row; q < p.nparts; q += FIN_CB * FIN_ROWS) {
            PT m[FIN_CB];
#pragma unroll
            for (int j = 0; j < FIN_CB; ++j)
                m[j] = q + j * FIN_ROWS < p.nparts ? src[(size_t)(q + j * FIN_ROWS) * p.qstride] : PT(0);
#pragma unroll
            for (int j = 0; j < FIN_CB; ++j)
                if (q + j * FIN_ROWS < p.nparts) s += widen(m[j]);
        }
    }
    sh_s[row][tx] = s;
    __syncthreads();
    if (row == 0 && i < p.n_minor) {
        double t = sh_s[0][tx];
#pragma unroll
        for (int r = 1; r < FIN_ROWS; ++r) t += sh_s[r][tx];
        static_cast<XT *>(p.short_out.p[b])[i] = static_cast<XT>(t);
    }
}

// SMs and most shared memory of a CTA of the current device (asked once per device).
static cudaError_t device_shape(int &sms, int &most) {
    static std::atomic<int> known[MAX_DEVICES][2];
    int device = 0;
    cudaError_t e = cudaGetDevice(&device);
    if (e != cudaSuccess) return e;
    if (device < 0 || device >= MAX_DEVICES) return cudaErrorInvalidDevice;
    sms = known[device][0].load(std::memory_order_relaxed);
    most = known[device][1].load(std::memory_order_relaxed);
    if (sms > 0 && most > 0) return cudaSuccess;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, device);
    if (e != cudaSuccess) return e;
    known[device][0].store(sms, std::memory_order_relaxed);
    known[device][1].store(most, std::memory_order_relaxed);
    return cudaSuccess;
}

// Launched with programmatic serialization: its blocks may become resident while the pass before
// drains (they wait in griddepcontrol.wait), which hides the launch.  They would all settle on
// the SMs that come free first and share those SMs' FP64 pipes (19 us instead of 7 for 20,000
// elements); each asks for so much shared memory that no SM takes more than its share of them.
template <typename XT, typename PT, typename RT>
cudaError_t launch_finish(FinishArgs &p, int kb, cudaStream_t s) {
    p.comb_blocks = (p.n_minor + FIN_X - 1) / FIN_X;
    const int64_t blocks = p.comb_blocks + ((int64_t)p.z + FIN_X * FIN_ROWS - 1) / (FIN_X * FIN_ROWS);
    if (blocks <= 0) return cudaSuccess;
    int sms = 0, most = 0;
    cudaError_t e = device_shape(sms, most);
    if (e != cudaSuccess) return e;
    auto kern = finish_kernel<XT, PT, RT>;
    static SmemLimit lim;
    const int smem = finish_request(blocks * kb, sms, most);
    e = ensure_smem_limit(kern, lim, smem);
    if (e != cudaSuccess) return e;
    return launch_overlapped(kern, dim3((unsigned)blocks, kb), dim3(FIN_X * FIN_ROWS), (size_t)smem, s, p);
}

static void out_ptrs(OutPtrs &o, void *const *out, int kb) {
    for (int b = 0; b < VL_MAX; ++b) o.p[b] = b < kb ? out[b] : nullptr;
}

cudaError_t launch_combine(bool vec_f64, bool part_f64, const void *part, int nparts, int n_minor, int kb,
                           void *const *out, cudaStream_t s, size_t qstride, size_t bstride) {
    if (n_minor <= 0) return cudaSuccess;
    if (kb < 1 || kb > VL_MAX) return cudaErrorInvalidValue;
    FinishArgs p = {};
    out_ptrs(p.short_out, out, kb);
    p.part = part;
    p.nparts = nparts;
    p.n_minor = n_minor;
    p.qstride = qstride ? qstride : (size_t)kb * n_minor;  // (0: [part][vector][element])
    p.bstride = qstride ? bstride : (size_t)n_minor;
    if (vec_f64) return launch_finish<double, double, double2>(p, kb, s);
    if (part_f64) return launch_finish<float, double, float2>(p, kb, s);
    return launch_finish<float, float, float2>(p, kb, s);
}

cudaError_t launch_fixup(bool vec_f64, const ZoneDev *zones, int z, const void *rec_left, const void *rec_right,
                         int P, int kb, void *const *out, cudaStream_t s) {
    if (z <= 0) return cudaSuccess;
    if (kb < 1 || kb > VL_MAX) return cudaErrorInvalidValue;
    FinishArgs p = {};
    out_ptrs(p.long_out, out, kb);
    p.zones = zones;
    p.z = z;
    p.P = P;
    p.rec_left = rec_left;
    p.rec_right = rec_right;
    return vec_f64 ? launch_finish<double, double, double2>(p, kb, s) : launch_finish<float, float, float2>(p, kb, s);
}

cudaError_t launch_combine_fixup(bool f64, const void *part, int nparts, int n_minor, void *short_out, const ZoneDev *zones,
                                 int z, const void *rec_left, const void *rec_right, int P, void *long_out,
                                 cudaStream_t s) {
    FinishArgs p = {};
    p.short_out.p[0] = short_out;
    p.long_out.p[0] = long_out;
    p.part = part;
    p.nparts = nparts;
    p.n_minor = n_minor;
    p.qstride = (size_t)n_minor;
    p.zones = zones;
    p.z = z;
    p.P = P;
    p.rec_left = rec_left;
    p.rec_right = rec_right;
    return f64 ? launch_finish<double, double, double2>(p, 1, s) : launch_finish<float, float, float2>(p, 1, s);
}

// out[i * KB + b] = in_b[i] for b < kb, 0 for kb <= b < KB: k vectors interleaved for the
// multi-vector segmented passes over vectors kept in global memory.  A block moves IT
// consecutive entries of every vector: coalesced reads of each vector into shared memory,
// then coalesced writes of the interleaved rows.
template <typename XT, int KB>
__global__ void __launch_bounds__(256) interleave_kernel(InPtrs in, int kb, int64_t len, XT *out) {
    constexpr int IT = 256;
    constexpr int RS = KB + 1;  // padded row: no bank conflicts in either phase
    __shared__ XT sh[IT * RS];
    grid_release();
    grid_wait();  // (the vectors may come from the kernel before, which may also still read `out`)
    for (int64_t i0 = (int64_t)blockIdx.x * IT; i0 < len; i0 += (int64_t)gridDim.x * IT) {
        const int cnt = (int)(len - i0 < IT ? len - i0 : (int64_t)IT);
#pragma unroll
        for (int b = 0; b < KB; ++b) {
            const XT *src = b < kb ? static_cast<const XT *>(in.p[b]) : nullptr;
            for (int t = threadIdx.x; t < cnt; t += blockDim.x) sh[t * RS + b] = src ? src[i0 + t] : XT(0);
        }
        __syncthreads();
        XT *dst = out + i0 * KB;
        for (int t = threadIdx.x; t < cnt * KB; t += blockDim.x) dst[t] = sh[(t / KB) * RS + t % KB];
        __syncthreads();
    }
}

cudaError_t launch_interleave(bool f64, int kbt, int kb, const void *const *in, int64_t len, void *out,
                              cudaStream_t s) {
    if (len <= 0) return cudaSuccess;
    if (kb < 1 || kb > kbt || kbt > VL_MAX || (f64 && kbt > KB_MAX)) return cudaErrorInvalidValue;
    InPtrs ip;
    for (int b = 0; b < VL_MAX; ++b) ip.p[b] = b < kb ? in[b] : nullptr;
    const int grid = (int)std::min<int64_t>((len + 255) / 256, 152 * 8);
    if (f64) {
        double *o = static_cast<double *>(out);
        if (kbt == 2) return launch_overlapped(interleave_kernel<double, 2>, dim3(grid), dim3(256), 0, s, ip, kb, len, o);
        else if (kbt == 4) return launch_overlapped(interleave_kernel<double, 4>, dim3(grid), dim3(256), 0, s, ip, kb, len, o);
        else return launch_overlapped(interleave_kernel<double, 8>, dim3(grid), dim3(256), 0, s, ip, kb, len, o);
    } else {
        float *o = static_cast<float *>(out);
        if (kbt == 2) return launch_overlapped(interleave_kernel<float, 2>, dim3(grid), dim3(256), 0, s, ip, kb, len, o);
        else if (kbt == 4) return launch_overlapped(interleave_kernel<float, 4>, dim3(grid), dim3(256), 0, s, ip, kb, len, o);
        else return launch_overlapped(interleave_kernel<float, 8>, dim3(grid), dim3(256), 0, s, ip, kb, len, o);
    }
}

}  // namespace gbk
