// Plans from coordinate triples (row, column, value) stored in the matrix's storage
// order -- column-major for a wide CSC matrix, row-major for a tall CSR one -- the
// triple stream the paper's implementation reads (Sec. V).  The compressed
// pointer array is derived on the device (the plan owns it); the minor indices and
// the values are borrowed as they are.  Triples in any order (SPMV_PLAN_COO_UNSORTED)
// are first sorted on the device by (major, minor) index into a plan-owned copy.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <utility>

#include "plan_impl.h"

namespace gbk {
namespace {

// err bit 1: a major index outside [0, n_major); bit 2: major indices decreasing
__global__ void coo_check_kernel(const int32_t *__restrict__ major, int64_t nnz, int n_major, int32_t *err) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < nnz; k += stride) {
        const int32_t j = major[k];
        if (static_cast<uint32_t>(j) >= static_cast<uint32_t>(n_major)) atomicOr(err, 1);
        if (k > 0 && major[k - 1] > j) atomicOr(err, 2);
    }
}

// ptr[j] = number of triples whose major index is below j (binary search of the sorted stream)
__global__ void coo_ptr_kernel(const int32_t *__restrict__ major, int64_t nnz, int n_major, int32_t *__restrict__ ptr) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j <= n_major; j += stride) {
        int64_t lo = 0, hi = nnz;  // first k with major[k] >= j
        while (lo < hi) {
            const int64_t mid = (lo + hi) >> 1;
            if (major[mid] < j)
                lo = mid + 1;
            else
                hi = mid;
        }
        ptr[j] = static_cast<int32_t>(lo);
    }
}

// ---- stable LSD radix sort of 64-bit keys (major * n_minor + minor) with a 32-bit payload (the
// value itself, or the triple's input position for 8-byte values), up to RS_BITS bits per pass.  A
// tile is 4096 keys: warp w of 16 holds tile elements 256 w .. 256 w + 255, lane l of its round j
// element 32 j + l of them, so that every load is coalesced.  Deterministic: every key's
// destination follows from the keys alone.
constexpr int RS_THREADS = 512, RS_WARPS = RS_THREADS / 32, RS_ROUNDS = 8, RS_TILE = RS_THREADS * RS_ROUNDS;
constexpr int RS_BITS = 9, RS_BINS = 1 << RS_BITS;
static_assert(RS_BINS == RS_THREADS, "one thread per digit in the tile's scan");

__device__ __forceinline__ int digit_of(uint64_t key, int shift, int mask) { return (int)(key >> shift) & mask; }

// The lanes of `live` with the same digit, by one vote per bit.  A match instruction takes a round for
// each digit that differs (32 a warp for random keys): 174 us for a pass of 10M keys over the low 9
// bits, 125 with the votes.
__device__ __forceinline__ unsigned same_digit(int d, unsigned live) {
    unsigned m = live;
#pragma unroll
    for (int b = 0; b < RS_BITS; ++b) {
        const bool one = (d >> b) & 1;
        const unsigned v = __ballot_sync(0xffffffffu, one);
        m &= one ? v : ~v;
    }
    return m;
}

// The triples as the caller has them and, after the sort, as the plan takes them.
struct Triples {
    const int32_t *major, *minor;
    const void *vals;
    int vbytes;  // 2, 4 or 8
    int n_major, n_minor;
    uint64_t recip;  // floor((2^64 - 1) / n_minor)
    int32_t *out_major, *out_minor;
    void *out_vals;
};

// The key of triple k; 0 with bit 1 (major index outside [0, n_major)) or bit 4 (minor index
// outside [0, n_minor)) of `bad` set.
__device__ __forceinline__ uint64_t triple_key(const Triples &t, int64_t k, int &bad) {
    const int32_t j = t.major[k], i = t.minor[k];
    const bool okj = static_cast<uint32_t>(j) < static_cast<uint32_t>(t.n_major);
    const bool oki = static_cast<uint32_t>(i) < static_cast<uint32_t>(t.n_minor);
    if (!okj) bad |= 1;
    if (!oki) bad |= 4;
    return okj && oki ? (uint64_t)j * (uint64_t)t.n_minor + (uint64_t)i : 0;
}

// Values of 2 and 4 bytes travel as the payload, those of 8 bytes are gathered by position at the end.
__device__ __forceinline__ uint32_t triple_payload(const Triples &t, int64_t k) {
    return t.vbytes == 4   ? static_cast<const uint32_t *>(t.vals)[k]
           : t.vbytes == 2 ? (uint32_t)static_cast<const uint16_t *>(t.vals)[k]
                           : (uint32_t)k;
}

// Key and payload to their triple's place.  The quotient by the reciprocal is the true one or one
// less: key < 2^62, so that the reciprocal's error takes away less than one.
__device__ __forceinline__ void triple_store(const Triples &t, int64_t pos, int64_t nnz, uint64_t key, uint32_t pay, int32_t *err) {
    uint64_t j = __umul64hi(key, t.recip), i = key - j * (uint64_t)t.n_minor;
    if (i >= (uint64_t)t.n_minor) {
        ++j;
        i -= (uint64_t)t.n_minor;
    }
    t.out_major[pos] = (int32_t)j;
    t.out_minor[pos] = (int32_t)i;
    if (t.vbytes == 4) {
        static_cast<uint32_t *>(t.out_vals)[pos] = pay;
    } else if (t.vbytes == 2) {
        static_cast<uint16_t *>(t.out_vals)[pos] = (uint16_t)pay;
    } else if (pay < nnz) {
        static_cast<uint64_t *>(t.out_vals)[pos] = static_cast<const uint64_t *>(t.vals)[pay];
    } else {
        static_cast<uint64_t *>(t.out_vals)[pos] = 0;
        atomicOr(err, 8);
    }
}

// hist[d * ntiles + tile] = number of keys of the tile whose digit is d.  FIRST: the keys come from
// the triples, whose indices are checked.
template <bool FIRST>
__global__ void __launch_bounds__(RS_THREADS) rs_hist_kernel(const uint64_t *__restrict__ keys,
                                                             const __grid_constant__ Triples tr, int64_t nnz,
                                                             int shift, int mask, int ntiles,
                                                             int32_t *__restrict__ hist, int32_t *err) {
    __shared__ int h[RS_BINS];
    const int t = threadIdx.x;
    h[t] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * RS_TILE;
    uint64_t key[RS_ROUNDS];
    int bad = 0;
#pragma unroll
    for (int j = 0; j < RS_ROUNDS; ++j) {
        const int64_t k = base + (int64_t)j * RS_THREADS + t;
        key[j] = 0;
        if (k < nnz) {
            if constexpr (FIRST)
                key[j] = triple_key(tr, k, bad);
            else
                key[j] = keys[k];
        }
    }
#pragma unroll
    for (int j = 0; j < RS_ROUNDS; ++j)
        if (base + (int64_t)j * RS_THREADS + t < nnz) atomicAdd(&h[digit_of(key[j], shift, mask)], 1);
    if (FIRST && bad) atomicOr(err, bad);
    __syncthreads();
    if (t <= mask) hist[(int64_t)t * ntiles + blockIdx.x] = h[t];
}

// exclusive scan of n int32 values in place: per-block sums, then block scans that each begin by
// adding up the sums before theirs
constexpr int SC_THREADS = 1024, SC_ITEMS = 4, SC_CHUNK = SC_THREADS * SC_ITEMS;

__device__ int block_exclusive_scan(int v, int *warp_tot, int &total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int inc = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int o = __shfl_up_sync(0xffffffffu, inc, d);
        if (lane >= d) inc += o;
    }
    if (lane == 31) warp_tot[w] = inc;
    __syncthreads();
    if (w == 0) {
        int x = lane < nw ? warp_tot[lane] : 0;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int o = __shfl_up_sync(0xffffffffu, x, d);
            if (lane >= d) x += o;
        }
        if (lane < nw) warp_tot[lane] = x;  // inclusive over warps
    }
    __syncthreads();
    total = warp_tot[nw - 1];
    const int before = w > 0 ? warp_tot[w - 1] : 0;
    __syncthreads();  // warp_tot is reused by the next call
    return before + inc - v;
}

__global__ void __launch_bounds__(SC_THREADS) scan_sums_kernel(const int32_t *__restrict__ a, int64_t n,
                                                               int32_t *__restrict__ sums) {
    __shared__ int wt[32];
    const int64_t base = (int64_t)blockIdx.x * SC_CHUNK + (int64_t)threadIdx.x * SC_ITEMS;
    int v = 0;
    for (int e = 0; e < SC_ITEMS; ++e)
        if (base + e < n) v += a[base + e];
    int total;
    block_exclusive_scan(v, wt, total);
    if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

__global__ void __launch_bounds__(SC_THREADS) scan_apply_kernel(int32_t *__restrict__ a, int64_t n,
                                                                const int32_t *__restrict__ sums) {
    __shared__ int wt[32];
    const int64_t base = (int64_t)blockIdx.x * SC_CHUNK + (int64_t)threadIdx.x * SC_ITEMS;
    int v[SC_ITEMS], tot = 0;
    for (int e = 0; e < SC_ITEMS; ++e) {
        v[e] = base + e < n ? a[base + e] : 0;
        tot += v[e];
    }
    int before = 0, total;
    for (int q = threadIdx.x; q < (int)blockIdx.x; q += SC_THREADS) before += sums[q];
    block_exclusive_scan(before, wt, total);
    before = total;
    int run = before + block_exclusive_scan(tot, wt, total);
    for (int e = 0; e < SC_ITEMS; ++e) {
        if (base + e < n) a[base + e] = run;
        run += v[e];
    }
}

// Stable scatter of a tile: every warp ranks its keys among its own of the same digit
// (same_digit, counters per warp), a scan over warps and digits gives their order in the tile, and
// the keys go through shared memory in that order, so that the keys of a digit (8 on average, 64
// bytes) are written side by side to offs[d * ntiles + tile] and on.  The first pass reads the
// triples themselves and the last one writes the sorted triples.  The 24 bytes a key moves set the
// floor, 35 us a pass of 10M keys; the passes take 80 to 125 (104 with match instructions, and
// 140 more for making the keys and taking them apart in kernels of their own; 162 without the
// reordering).
constexpr size_t RS_SMEM = RS_TILE * 12 + RS_WARPS * RS_BINS * 2 + RS_BINS * 8;
template <bool FIRST, bool LAST>
__global__ void __launch_bounds__(RS_THREADS) rs_scatter_kernel(const uint64_t *__restrict__ kin,
                                                                const uint32_t *__restrict__ pin,
                                                                const __grid_constant__ Triples tr, int64_t nnz, int shift,
                                                                int mask, int ntiles, const int32_t *__restrict__ offs,
                                                                uint64_t *__restrict__ kout, uint32_t *__restrict__ pout,
                                                                int32_t *err) {
    extern __shared__ __align__(16) unsigned char sm[];
    uint64_t *skey = reinterpret_cast<uint64_t *>(sm);
    uint32_t *spay = reinterpret_cast<uint32_t *>(sm + RS_TILE * 8);
    uint16_t *wcnt = reinterpret_cast<uint16_t *>(sm + RS_TILE * 12);  // [warp][digit]
    int32_t *lstart = reinterpret_cast<int32_t *>(sm + RS_TILE * 12 + RS_WARPS * RS_BINS * 2);  // in the tile
    int32_t *gdelta = lstart + RS_BINS;  // place in the output less place in the tile
    __shared__ int wt[32];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    for (int q = t; q < RS_WARPS * RS_BINS / 2; q += RS_THREADS) reinterpret_cast<uint32_t *>(wcnt)[q] = 0u;
    const int64_t base = (int64_t)blockIdx.x * RS_TILE;
    const int n = nnz - base < RS_TILE ? (int)(nnz - base) : RS_TILE;
    uint64_t key[RS_ROUNDS];
    uint32_t pl[RS_ROUNDS];
    uint16_t rank[RS_ROUNDS];
#pragma unroll
    for (int j = 0; j < RS_ROUNDS; ++j) {
        const int i = w * (32 * RS_ROUNDS) + 32 * j + lane;
        if constexpr (FIRST) {
            int bad = 0;  // (reported by the histogram)
            key[j] = i < n ? triple_key(tr, base + i, bad) : 0;
            pl[j] = i < n ? triple_payload(tr, base + i) : 0;
        } else {
            key[j] = i < n ? kin[base + i] : 0;
            pl[j] = i < n ? pin[base + i] : 0;
        }
    }
    __syncthreads();
    uint16_t *mine = wcnt + w * RS_BINS;
#pragma unroll
    for (int j = 0; j < RS_ROUNDS; ++j) {
        const bool live = w * (32 * RS_ROUNDS) + 32 * j + lane < n;
        const int d = digit_of(key[j], shift, mask);
        const unsigned peers = same_digit(d, __ballot_sync(0xffffffffu, live));
        const int before = __popc(peers & ((1u << lane) - 1u));
        rank[j] = live ? (uint16_t)(mine[d] + before) : (uint16_t)0;
        __syncwarp();
        if (live && before == 0) mine[d] = (uint16_t)(mine[d] + __popc(peers));
        __syncwarp();
    }
    __syncthreads();
    {  // thread t: digit t
        int c = 0;
#pragma unroll
        for (int q = 0; q < RS_WARPS; ++q) {
            const int v = wcnt[q * RS_BINS + t];
            wcnt[q * RS_BINS + t] = (uint16_t)c;
            c += v;
        }
        int total;
        const int ls = block_exclusive_scan(c, wt, total);
        lstart[t] = ls;
        gdelta[t] = t <= mask ? offs[(int64_t)t * ntiles + blockIdx.x] - ls : 0;
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < RS_ROUNDS; ++j) {
        if (w * (32 * RS_ROUNDS) + 32 * j + lane < n) {
            const int d = digit_of(key[j], shift, mask);
            const int pos = lstart[d] + mine[d] + rank[j];  // (< n: a permutation of the tile)
            skey[pos] = key[j];
            spay[pos] = pl[j];
        }
    }
    __syncthreads();
    for (int i = t; i < n; i += RS_THREADS) {
        const uint64_t k = skey[i];
        const int64_t pos = (int64_t)gdelta[digit_of(k, shift, mask)] + i;
        if (pos >= 0 && pos < nnz) {
            if constexpr (LAST) {
                triple_store(tr, pos, nnz, k, spay[i], err);
            } else {
                kout[pos] = k;
                pout[pos] = spay[i];
            }
        } else {
            atomicOr(err, 8);
        }
    }
}

}  // namespace

CooSort::~CooSort() {
    if (!tmp && !own) return;
    cudaStreamSynchronize(s);
    dev_free(tmp, device);
    dev_free(own, device);
}

cudaError_t launch_coo_ptr(const int32_t *major_sorted, int64_t nnz, int n_major, int32_t *ptr, int grid,
                           cudaStream_t s) {
    coo_ptr_kernel<<<grid, 256, 0, s>>>(major_sorted, nnz, n_major, ptr);
    return cudaGetLastError();
}

// Sorts the triples by (major, minor), stably: the sorted minor indices and values go to the
// plan-owned block, the sorted major indices to the temporary one; all three come back through
// the out-parameters.  Range errors are reported through `err` (read by the caller after a sync).
spmv_status coo_sort(CooSort &cs, const int32_t *major, const int32_t *minor, const void *vals, int sv, int64_t nnz,
                     int n_major, int n_minor, int32_t *err, cudaStream_t s, const int32_t **major_sorted,
                     int32_t **minor_sorted, void **vals_sorted) {
    auto up = [](size_t v) { return (v + 255) / 256 * 256; };
    const int ntiles = (int)((nnz + RS_TILE - 1) / RS_TILE);
    const int64_t nh = (int64_t)RS_BINS * ntiles;
    const int nsc = (int)((nh + SC_CHUNK - 1) / SC_CHUNK);
    const size_t kb = up((size_t)nnz * 8), pb = up((size_t)nnz * 4), hb = up((size_t)nh * 4), sb = up((size_t)nsc * 4);
    cs.s = s;
    if (cudaGetDevice(&cs.device) != cudaSuccess) return set_error(SPMV_ERR_CUDA, "no current device");
    if (dev_alloc(&cs.tmp, 2 * kb + 2 * pb + hb + sb) != cudaSuccess) return set_error(SPMV_ERR_OOM, "sort scratch");
    char *t = static_cast<char *>(cs.tmp);
    uint64_t *ka = reinterpret_cast<uint64_t *>(t), *kb2 = reinterpret_cast<uint64_t *>(t + kb);
    uint32_t *pa = reinterpret_cast<uint32_t *>(t + 2 * kb), *pb2 = reinterpret_cast<uint32_t *>(t + 2 * kb + pb);
    int32_t *hist = reinterpret_cast<int32_t *>(t + 2 * kb + 2 * pb);
    int32_t *sums = reinterpret_cast<int32_t *>(t + 2 * kb + 2 * pb + hb);
    const size_t ib = up((size_t)nnz * 4);
    cs.own_bytes = ib + up((size_t)nnz * sv);
    if (dev_alloc(&cs.own, cs.own_bytes) != cudaSuccess) return set_error(SPMV_ERR_OOM, "sorted triples");

    const uint64_t span = (uint64_t)n_major * (uint64_t)n_minor;
    const int bits = span > 1 ? 64 - __builtin_clzll(span - 1) : 0;
    const int passes = std::max(1, (bits + RS_BITS - 1) / RS_BITS);
    Triples tr = {};
    tr.major = major;
    tr.minor = minor;
    tr.vals = vals;
    tr.vbytes = sv;
    tr.n_major = n_major;
    tr.n_minor = n_minor;
    tr.recip = ~0ull / (uint64_t)n_minor;
    tr.out_minor = static_cast<int32_t *>(cs.own);
    tr.out_vals = static_cast<char *>(cs.own) + ib;
    for (int q = 0, shift = 0; q < passes; ++q) {  // passes of equal width, give or take a bit
        const int width = (bits - shift + passes - q - 1) / (passes - q), mask = (1 << width) - 1;
        const int64_t nhq = (int64_t)(mask + 1) * ntiles;
        const int nscq = (int)((nhq + SC_CHUNK - 1) / SC_CHUNK);
        const bool first = q == 0, last = q == passes - 1;
        auto histogram = first ? rs_hist_kernel<true> : rs_hist_kernel<false>;
        static SmemLimit lim[4];
        auto scatter = first ? (last ? rs_scatter_kernel<true, true> : rs_scatter_kernel<true, false>)
                             : (last ? rs_scatter_kernel<false, true> : rs_scatter_kernel<false, false>);
        if (ensure_smem_limit(scatter, lim[2 * first + last], (int)RS_SMEM) != cudaSuccess)
            return set_error(SPMV_ERR_CUDA, "sort launch failed");
        tr.out_major = reinterpret_cast<int32_t *>(pb2);  // (the last pass writes no payload)
        histogram<<<ntiles, RS_THREADS, 0, s>>>(ka, tr, nnz, shift, mask, ntiles, hist, err);
        scan_sums_kernel<<<nscq, SC_THREADS, 0, s>>>(hist, nhq, sums);
        scan_apply_kernel<<<nscq, SC_THREADS, 0, s>>>(hist, nhq, sums);
        scatter<<<ntiles, RS_THREADS, RS_SMEM, s>>>(ka, pa, tr, nnz, shift, mask, ntiles, hist, kb2, pb2, err);
        std::swap(ka, kb2);
        std::swap(pa, pb2);
        shift += width;
    }
    if (cudaGetLastError() != cudaSuccess) return set_error(SPMV_ERR_CUDA, "sort launch failed");
    *major_sorted = tr.out_major;
    *minor_sorted = tr.out_minor;
    *vals_sorted = tr.out_vals;
    return SPMV_OK;
}

}  // namespace gbk

using namespace gbk;

namespace {

int dsize(int t) { return t == SPMV_F64 ? 8 : t == SPMV_F32 ? 4 : (t == SPMV_BF16 || t == SPMV_F16) ? 2 : 0; }

}  // namespace

extern "C" spmv_status spmv_plan_coo(spmv_plan_t *out, int64_t m, int64_t n, int64_t nnz, int32_t layout,
                                     const int32_t *rows, const int32_t *cols, const void *vals, int32_t val_dtype,
                                     int32_t vec_dtype, void *stream, uint32_t flags, const spmv_plan_opts *opts) {
    if (!out) return set_error(SPMV_ERR_INVALID_ARG, "out is NULL");
    *out = nullptr;
    if (layout != SPMV_CSC_WIDE && layout != SPMV_CSR_TALL) return set_error(SPMV_ERR_INVALID_ARG, "bad layout");
    if (m < 0 || n < 0 || nnz < 0 || m >= (1ll << 31) - 64 || n >= (1ll << 31) - 64 || nnz >= (1ll << 31) - 64)
        return set_error(SPMV_ERR_INVALID_ARG, "m, n and nnz must lie in [0, 2^31 - 64)");
    if (nnz > 0 && (!rows || !cols || !vals)) return set_error(SPMV_ERR_INVALID_ARG, "rows/cols/vals are NULL");
    const bool unsorted = (flags & SPMV_PLAN_COO_UNSORTED) != 0;
    if (unsorted && dsize(val_dtype) == 0) return set_error(SPMV_ERR_INVALID_ARG, "unknown dtype");
    const bool csc = layout == SPMV_CSC_WIDE;
    const int32_t *major = csc ? cols : rows;
    const int32_t *minor = csc ? rows : cols;
    const int n_major = (int)(csc ? n : m);
    const int n_minor = (int)(csc ? m : n);
    if (nnz > 0 && (n_major == 0 || n_minor == 0))
        return set_error(SPMV_ERR_BAD_MATRIX, "nonzeros need a nonempty matrix");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int sms = 0, dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    int32_t *ptr = nullptr, *err = nullptr;
    void *ptr_mem = nullptr;
    if (dev_alloc(&ptr_mem, ((size_t)n_major + 1) * 4 + 16) != cudaSuccess) return set_error(SPMV_ERR_OOM, "pointer array");
    ptr = static_cast<int32_t *>(ptr_mem);
    auto free_ptr = [&] {
        cudaStreamSynchronize(s);
        dev_free(ptr_mem, dev);
    };
    err = reinterpret_cast<int32_t *>(reinterpret_cast<char *>(ptr) + (((size_t)n_major + 1) * 4 + 3) / 4 * 4);
    auto fail = [&](spmv_status st, const char *msg) {
        free_ptr();
        return set_error(st, msg);
    };
    if (cudaMemsetAsync(err, 0, 4, s) != cudaSuccess) return fail(SPMV_ERR_CUDA, "memset");
    const int grid = std::max(1, sms * 8);
    CooSort cs;
    const int32_t *maj_use = major, *min_use = minor;
    const void *vals_use = vals;
    if (unsorted && nnz > 0) {
        int32_t *omin = nullptr;
        void *ovals = nullptr;
        const spmv_status st = coo_sort(cs, major, minor, vals, dsize(val_dtype), nnz, n_major, n_minor, err, s,
                                        &maj_use, &omin, &ovals);
        if (st != SPMV_OK) {
            free_ptr();
            return st;
        }
        min_use = omin;
        vals_use = ovals;
    } else if (nnz > 0) {
        coo_check_kernel<<<grid, 256, 0, s>>>(major, nnz, n_major, err);
    }
    coo_ptr_kernel<<<grid, 256, 0, s>>>(maj_use, nnz, n_major, ptr);
    if (cudaGetLastError() != cudaSuccess) return fail(SPMV_ERR_CUDA, "launch failed");
    int32_t e = 0;
    if (cudaMemcpyAsync(&e, err, 4, cudaMemcpyDeviceToHost, s) != cudaSuccess || cudaStreamSynchronize(s) != cudaSuccess)
        return fail(SPMV_ERR_CUDA, "pointer construction failed");
    if (e & 1) return fail(SPMV_ERR_BAD_MATRIX, "a major index lies outside the matrix");
    if (e & 4) return fail(SPMV_ERR_BAD_MATRIX, "a minor index lies outside the matrix");
    if (e & 2) return fail(SPMV_ERR_BAD_MATRIX, "triples are not in storage order (major index decreases)");
    if (e & 8) return fail(SPMV_ERR_DEVICE, "inconsistent triple sort");
    spmv_status st = spmv_plan_ex(out, m, n, nnz, layout, ptr, min_use, vals_use, val_dtype, vec_dtype, stream,
                                  flags, opts);
    if (st != SPMV_OK) {
        free_ptr();
        return st;
    }
    (*out)->owned_ptr = ptr;  // freed with the plan
    if (cs.own && !(*out)->owned_nz) {
        // the plan multiplies the sorted copy (a bank-ordered plan made its own copy of it instead)
        (*out)->owned_nz = cs.own;
        (*out)->owned_bytes = cs.own_bytes;
        cs.own = nullptr;
    }
    return SPMV_OK;
}
