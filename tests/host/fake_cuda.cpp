// A CUDA runtime for the host-side tests: devices are numbers, device memory is host memory, kernels are
// entries of a log.  Linked with the library's host code (plans, routing, memory, serving) compiled by g++.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>

#include "../../paper_1812_00904_gb300/csrc/plan_impl.h"

namespace {

std::mutex mu;
std::string lines;  // the log: one call or launch a line
thread_local int current = 0;
int sms = 152, optin = 232448;
bool sync_fails = false;
uint64_t room = ~0ull, used = 0, kept = 0;  // device bytes; what plain allocations and pools hold; freed bytes a pool keeps
std::map<void *, size_t> sizes;

void note(const std::string &s) {
    std::lock_guard<std::mutex> lk(mu);
    lines += s + "\n";
}
cudaError_t take(void **p, size_t n, bool pool) {
    std::lock_guard<std::mutex> lk(mu);
    *p = nullptr;
    if (pool && kept >= n)
        kept -= n;
    else if (n > room || used > room - n)
        return cudaErrorMemoryAllocation;
    else
        used += n;
    *p = aligned_alloc(256, (n + 511) / 256 * 256);
    sizes[*p] = n;
    return cudaSuccess;
}
void give(void *p, bool pool) {
    std::lock_guard<std::mutex> lk(mu);
    auto it = sizes.find(p);
    if (it == sizes.end()) return;
    (pool ? kept : used) += pool ? it->second : (uint64_t)0 - it->second;
    sizes.erase(it);
    free(p);
}

}  // namespace

extern "C" {

// ---- what a test sets and reads
void fake_reset(int sm_count, int smem) {
    std::lock_guard<std::mutex> lk(mu);
    lines.clear();
    current = 0;
    sms = sm_count;
    optin = smem;
    sync_fails = false;
    room = ~0ull;
}
void fake_fail_sync(int on) { sync_fails = on != 0; }
// free device bytes from now on (what a pool keeps counts as taken)
void fake_room(uint64_t bytes) { room = used + bytes; }
uint64_t fake_used() { return used; }
const char *fake_log() {
    static std::string out;
    std::lock_guard<std::mutex> lk(mu);
    out.swap(lines);
    lines.clear();
    return out.c_str();
}
void *fake_alloc(size_t n) {
    void *p = nullptr;
    take(&p, n, false);
    return p;
}
// segments seen once and in range: by the blocks that rank them, and by thread `thread` of `threads` in a strided loop
int64_t fake_ranked_segments(int n_major, unsigned block, int64_t *lowest) {
    int64_t n = 0;
    *lowest = INT64_MAX;
    for (unsigned t = 0; t < gbk::SEG_BLOCK / gbk::SEG_IPT; ++t) {
        const int64_t j0 = gbk::seg_rank_first(block, t);
        for (int i = 0; i < gbk::SEG_IPT && j0 + i < n_major; ++i, ++n) *lowest = std::min(*lowest, j0 + i);
    }
    return n;
}
uint64_t fake_plan_bytes_most(int64_t m, int64_t n, int64_t nnz, int val, int vec) {
    return gbk::plan_bytes_most(0, m, n, nnz, SPMV_CSC_WIDE, val, vec);
}
int fake_finish_request(int64_t blocks, int sm_count, int smem_most) { return gbk::finish_request(blocks, sm_count, smem_most); }
int fake_rank_blocks(int n_major) { return gbk::seg_rank_blocks(n_major); }
int64_t fake_strided(int64_t thread, int64_t threads, int64_t n, int64_t *lowest, int64_t *highest) {
    int64_t seen = 0;
    *lowest = INT64_MAX;
    *highest = -1;
    gbk::strided(thread, threads, n, [&](int64_t i) {
        *lowest = std::min(*lowest, i);
        *highest = std::max(*highest, i);
        ++seen;
    });
    return seen;
}

// ---- the runtime
cudaError_t cudaGetDevice(int *d) { return *d = current, cudaSuccess; }
cudaError_t cudaSetDevice(int d) { return current = d, cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? sms : a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? optin : 0;
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() {
    note("sync device " + std::to_string(current));
    return sync_fails ? cudaErrorStreamCaptureUnsupported : cudaSuccess;
}
cudaError_t cudaMalloc(void **p, size_t n) { return take(p, n, false); }
cudaError_t cudaFree(void *p) {
    if (p) note("free");
    return give(p, false), cudaSuccess;
}
cudaError_t cudaMemPoolCreate(cudaMemPool_t *p, const cudaMemPoolProps *) {
    return *p = reinterpret_cast<cudaMemPool_t>(0x100), cudaSuccess;
}
cudaError_t cudaMemPoolDestroy(cudaMemPool_t) { return cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void *) { return cudaSuccess; }
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t, size_t) {
    std::lock_guard<std::mutex> lk(mu);
    lines += "trim\n";
    used -= kept;
    kept = 0;
    return cudaSuccess;
}
cudaError_t cudaMallocFromPoolAsync(void **p, size_t n, cudaMemPool_t, cudaStream_t) { return take(p, n, true); }
cudaError_t cudaFreeAsync(void *p, cudaStream_t) {
    note("pool free");
    return give(p, true), cudaSuccess;
}
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { return memcpy(d, s, n), cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t) {
    return memcpy(d, s, n), cudaSuccess;
}
cudaError_t cudaMemset(void *d, int v, size_t n) { return memset(d, v, n), cudaSuccess; }
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) { return memset(d, v, n), cudaSuccess; }  // (plan memory)
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *) {
    memset(a, 0, sizeof(*a));
    a->type = cudaMemoryTypeDevice;
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { return *s = reinterpret_cast<cudaStream_t>(0x200), cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { return *e = reinterpret_cast<cudaEvent_t>(0x300), cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { return *ms = 0.f, cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return "fake error"; }

}  // extern "C"

// ---- the launches
namespace gbk {

cudaError_t launch_validate(const int32_t *ptr, const int32_t *, int n_major, int, int, int32_t *, int32_t *nempty, cudaStream_t) {
    for (int j = 0; j < n_major; ++j) *nempty += ptr[j + 1] == ptr[j];
    return cudaSuccess;
}
cudaError_t launch_pad_ptr(const int32_t *, int32_t *, int, int, int, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_chunks(const int32_t *, int, int, int, const int32_t *, int, ChunkAux *, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_setup(ChunkAux *, int, ChunkDev *, ZoneDev *, int32_t *, void *, cudaStream_t) { return cudaSuccess; }
size_t setup_scratch_bytes(int) { return 4096; }
cudaError_t launch_tile_bounds(int, int, int, int32_t *, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_masks(const int32_t *, const ChunkAux *, int, int, int, int, uint32_t *, int, uint16_t *, TileMeta *,
                         const int32_t *, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_steps(const TileMeta *, const uint32_t *, int, int, int, const int32_t *, StepRec *, cudaStream_t) {
    return cudaSuccess;
}
cudaError_t launch_seg_ranks(const int32_t *, int, int32_t *, int32_t *, int32_t *, int32_t *, int32_t *, cudaStream_t) {
    return cudaSuccess;
}
int stream_processors(int ntiles, int T, int nnz, int ctas, int C, int32_t *nzb) {
    int np = 0;
    for (int g = 0; g < ctas; ++g) {
        const CtaChunks c = cta_chunks(g, ntiles, ctas, C);
        for (int q = 0; q < c.nq; ++q, ++np) {
            const int64_t t = c.ta + (q < c.nb ? q * C : c.nb * C + q - c.nb);
            if (nzb) nzb[np] = (int)(t * T < nnz ? t * T : nnz);
        }
    }
    if (nzb) nzb[np] = nnz;
    return np;
}

spmv_status build_row_blocks(spmv_plan_s *, int, cudaStream_t) { return SPMV_OK; }
cudaError_t launch_bank_order(const int32_t *, int, int, const int32_t *, const void *, int, int32_t *, void *, int32_t *,
                              int, int, cudaStream_t) { return cudaSuccess; }

// a kernel of the products: "name, warps of a CTA, CTAs"
static cudaError_t kernel(const std::string &name, int warps, int grid) {
    note(name + " " + std::to_string(warps) + " " + std::to_string(grid));
    return cudaSuccess;
}
#define PASSES(T)                                                                                                      \
    cudaError_t launch_stream_##T(int mode, int kb, const LaunchArgs &a) {                                             \
        static const char *const names[] = {"stream scatter", "stream segdot", "stream dvalues", "stream vseg"};       \
        return kernel(names[mode], a.block / 32, a.grid);                                                              \
    }                                                                                                                  \
    cudaError_t launch_dvalues_##T(const PassParams &, int grid, int warps, int, cudaStream_t) {                       \
        return kernel("dvalues", warps, grid);                                                                         \
    }                                                                                                                  \
    cudaError_t launch_pass_##T(bool sc, bool sd, const PassParams &, int grid, int warps, int, cudaStream_t) {        \
        return kernel(sc && sd ? "pass pair" : sc ? "pass scatter" : "pass segdot", warps, grid);                      \
    }
#define BATCH_PASSES(T)                                                                                                \
    cudaError_t launch_mvscatter_##T(int, const PassParams &, int grid, int warps, int, cudaStream_t) {                \
        return kernel("mvscatter", warps, grid);                                                                       \
    }                                                                                                                  \
    cudaError_t launch_mvdot_##T(int, bool, const PassParams &, int grid, int warps, int, cudaStream_t) {              \
        return kernel("mvdot", warps, grid);                                                                           \
    }
PASSES(f64) PASSES(f32) PASSES(bf16) PASSES(f16) BATCH_PASSES(f32) BATCH_PASSES(bf16) BATCH_PASSES(f16)
cudaError_t launch_interleave(bool, int, int, const void *const *, int64_t, void *, cudaStream_t) { return kernel("interleave", 8, 1); }
cudaError_t launch_combine(bool, bool, const void *, int, int, int, void *const *, cudaStream_t, size_t, size_t) {
    return kernel("combine", 8, 1);
}
cudaError_t launch_fixup(bool, const ZoneDev *, int, const void *, const void *, int, int, void *const *, cudaStream_t) {
    return kernel("fixup", 8, 1);
}
cudaError_t launch_combine_fixup(bool, const void *, int, int, void *, const ZoneDev *, int, const void *, const void *, int,
                                 void *, cudaStream_t) { return kernel("combine+fixup", 8, 1); }

}  // namespace gbk
