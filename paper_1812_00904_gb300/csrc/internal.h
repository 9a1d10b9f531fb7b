// Internal declarations shared by the CUDA translation units of libspmv_gb300.
// Not part of the public ABI (include/spmv_gb300.h).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <mutex>

namespace gbk {

// Kernel modes of the streaming kernel (one staged pass over the nonzeros).
enum Mode : int {
    MODE_SCATTER = 0,  // acc[idx[k]] += val[k] * w[major(k)]   (CSC A x, CSR v^T A)
    MODE_SEGDOT = 1,   // out[j] = sum_{k in segment j} val[k] * w[idx[k]]   (CSC v^T A, CSR A x)
    MODE_DVALUES = 2,  // g[k] = minor[idx[k]] * major[seg(k)]
    MODE_VSEG = 3,     // MODE_SEGDOT for several vectors, one per lane of a lane group
};

constexpr int KB_MAX = 8;        // vectors per pass of the multi-vector kernels (but MODE_VSEG)
constexpr int VL_MAX = 8;        // vectors per pass of MODE_VSEG (lane group width)
constexpr int MAX_WARPS = 24;    // warps per CTA of the single-vector passes (80 registers a thread beyond 16)
constexpr int MAX_WARPS_KB = 16; // warps per CTA of the multi-vector passes
constexpr int WARPS_VSEG = 16;   // warps per CTA of MODE_VSEG (up to 128 registers a thread)
constexpr int WARPS_REGS = 16;   // warps per CTA up to which a kernel may use 128 registers a thread
constexpr int MAX_STAGES = 4;    // slots per warp
constexpr int BAR_BYTES = 1024;  // slot barriers at the start of the staging area

// Per-chunk descriptor produced by the set-up (24 bytes).
struct ChunkDev {
    int32_t nz_begin, nz_end;   // nonzeros [nz_begin, nz_end) (Sec. II rule)
    int32_t e_begin, e_end;     // segments whose end event the chunk owns: [e_begin, e_end)
    int32_t jf;                 // first segment j^f (-1 if empty)
    int32_t flags;              // bit0 needLeft, bit1 needRight
};

// Per-chunk quantities of the set-up (Sec. IV-B), device side.
struct ChunkAux {
    int32_t nz_begin, nz_end, jf, jl, e_begin, e_end, ntiles;
    int32_t needLeft, needRight, leftGroupEnd, rightGroup, leftGroup, procsOnLeft, procsOnRight;
};

struct ZoneDev {
    int32_t first, last, col, pad;  // S_k = chunks [first, last], column j_k
};

// What the streaming kernel reads per execution tile (16 bytes).  Tile t covers
// nonzeros [meta[t].nzb, meta[t+1].nzb) and owns the segment end events
// [meta[t].e_begin, meta[t+1].e_begin); meta[ntiles] is the sentinel {nnz, n_major}
// with the number of nonempty segments as its rank.
struct alignas(16) TileMeta {
    int32_t nzb, e_begin;
    int32_t flags;  // bit0 needLeft, bit1 needRight, bit2 an empty segment ends in the tile
    int32_t rank;   // rank among the nonempty segments of the one open before the tile's first head bit
};

// Parameters of the streaming kernel.
struct StreamParams {
    const int32_t *idx;
    const void *vals;
    const int32_t *pptr;     // plan-owned padded copy of the pointer array (general path)
    int32_t nnz, n_major, n_minor;
    const TileMeta *meta;    // ntiles + 1 entries
    const uint32_t *masks;   // per tile: mwp words of segment-start bits
    const uint16_t *pfx;     // per tile: mwq entries, the segment starts before word j (j >= mwp: all of them)
    int32_t ntiles, mwp, mwq;
    int32_t slot_bytes, vec_region_bytes, slots, x_cap;  // per-warp slot bytes, slots per warp, window elements
    int32_t tile_cap, off_val, off_mask, off_x, off_hdr;  // slot layout: indices at 0, values, masks, windows, header
    int32_t off_pfx;         // segmented modes: the tile's head-count prefix table in the slot (at off_x)
    int32_t checked;         // 1: indices not validated by the plan, checked (clamped) on every step
    int32_t kb;              // vectors in this pass (<= KB template)
    const void *vin[KB_MAX]; // SCATTER: major vectors; SEGDOT: minor vectors; DVALUES: vin[0] minor, vin[1] major;
                             // VSEG: vin[0] = the minor vectors interleaved [entry][VL]
    void *vout[VL_MAX];      // SEGDOT, VSEG: major outputs; DVALUES: vout[0] = g
    void *part;              // SCATTER: per-CTA partials [cta][kb][n_minor] (on chip) or FP64 accumulator [kb][n_minor]
    void *rec_left, *rec_right;  // SEGDOT carry records [b * nproc + proc]: (hi, lo) pairs of the accumulation type
    int32_t nproc;           // processors (chunks of tiles) of the plan: the record stride
    int32_t chunk_tiles;     // C, tiles per chunk (before the single-tile tail of every block)
    int32_t blocks_per_cta;  // BPC: the tiles form gridDim.x BPC blocks; a CTA runs BPC of them in turn
    const int2 *win;         // SEGDOT over row-sorted blocks: per CTA (first element, length) of its window of
                             // the input vector; the indices are offsets into the window (NULL: whole vector)
    int32_t *err;
};

// CTA g's chunks (processors) when ntiles tiles are cut over `ctas` CTAs with chunks of C tiles:
// tiles [ta, ta + nct), nb chunks of C tiles, then single-tile ones, nq in all, numbered from proc0.
struct CtaChunks {
    int ta, nct, nb, nq, proc0;
};
__host__ __device__ inline CtaChunks cta_chunks(int g, int ntiles, int ctas, int C) {
    const int tq = ntiles / ctas, tr = ntiles % ctas, tail = MAX_WARPS * C + MAX_WARPS;
    auto big = [&](int n) { return (n - (n < tail ? n : tail)) / C; };
    auto chunks = [&](int n) { return n - (C - 1) * big(n); };
    CtaChunks c;
    c.ta = g * tq + (g < tr ? g : tr);
    c.nct = tq + (g < tr ? 1 : 0);
    c.nb = big(c.nct);
    c.nq = chunks(c.nct);
    c.proc0 = g * chunks(tq) + (g < tr ? g : tr) * (chunks(tq + 1) - chunks(tq));
    return c;
}

// Element-wise loops over segments, of which there may be 2^31 - 65: a thread's elements first,
// first + step, .. below n, counted in 64 bits (a 32-bit counter wraps when its last step crosses 2^31).
template <typename F> __host__ __device__ inline void strided(int64_t first, int64_t step, int64_t n, F f) {
    for (int64_t i = first; i < n; i += step) f(i);
}
// The blocks that rank the nonempty segments take SEG_BLOCK segments each, every thread SEG_IPT in a row.
constexpr int SEG_IPT = 2, SEG_BLOCK = 512;
__host__ __device__ inline int seg_rank_blocks(int n_major) { return (int)(((int64_t)n_major + SEG_BLOCK - 1) / SEG_BLOCK); }
__host__ __device__ inline int64_t seg_rank_first(unsigned block, unsigned thread) {
    return (int64_t)block * SEG_BLOCK + (int64_t)thread * SEG_IPT;
}

// What the one-vector passes (pass_kernel.cuh) read per step of 256 nonzeros beside them.
struct alignas(16) StepRec {
    uint32_t heads[8];  // bit i of word j: a segment starts at position 32 j + i (the tile's masks)
    uint8_t before[8];  // heads of the step before word j
    int32_t first;      // the segment open before the step's first head (-1: none, leading empty ones)
    int32_t flags;      // STEP_* bits; the heads of the step << 16
};
constexpr int STEP_NEED_LEFT = 1;   // the tile's first segment began before it (its first step is asked)
constexpr int STEP_NEED_RIGHT = 2;  // the tile's last segment continues after it (its last step is asked)
constexpr int STEP_ENDS = 4;        // the tile's last step: the open segment ends with the tile
constexpr int STEP_GAPS = 8;        // empty segments lie between the step's segments

// Parameters of the one-vector passes of a validated plan (tiles of T = 256 spt nonzeros).
struct PassParams {
    const int32_t *idx;
    const void *vals;
    const StepRec *steps;
    // the nonempty segments in order and every segment's rank among them (read in steps with gaps)
    const int32_t *seglist, *rank;
    int32_t nnz, n_minor, ntiles, spt, chunk_tiles;
    int32_t slots;           // staging slots per warp
    int32_t lanes;           // SC: 1 = an element of the accumulator for every lane
    int32_t spread;          // pair: a mask of up to 255 below n_minor (places for a last step's empty positions)
    int32_t copies;          // copies of the accumulator (a power of two), shared by the warps in turn
    int32_t acc_bytes, vec_bytes;  // shared memory of one accumulator (0 without SC) and of the input (0 without SD)
    const void *x, *v;       // the long input (SC), the short input (SD)
    void *part;              // SC: per-CTA partials [cta][n_minor]
    void *u;                 // SD: the long output
    void *rec_left, *rec_right;  // SD: carry records [proc], (hi, lo) pairs
    int32_t bpc;             // SD over row-sorted blocks: blocks each CTA runs in turn, and per block its window
    const int2 *win;         // (first element, length) of v (NULL: all of v)
    float *uv[VL_MAX];       // several vectors: their outputs (SD; v then being interleaved [entry][KV]),
    const void *xv[VL_MAX];  // their long inputs (SC)
    int32_t kb, nproc;       // several vectors: how many; records [b * nproc + proc]
    const int32_t *emptylist;  // SD: the empty segments, whose outputs are 0
    int32_t nempty;
    int32_t *err;
};
// Staging of a pass: a slot holds a step's indices, values, record and 16-byte header.
constexpr int PASS_BAR_BYTES = 512;  // slot barriers, PASS_MAX_SLOTS for each of up to 32 warps
constexpr int PASS_MAX_SLOTS = 2;
__host__ __device__ constexpr int pass_slot_bytes(int val_bytes) { return 1024 + 256 * val_bytes + (int)sizeof(StepRec) + 16; }
// Most warps of a pass: 32 of 64 registers a thread; FP64 needs more registers, and its passes gain
// little from more warps (8M nonzeros, n = 4,000, with 16 / 20 / 24: dot products 48 / 48 / 49 us,
// accumulating 42 / 41 / 40, the pair 76 / 77 / 77).
constexpr int pass_warps(int val_bytes) { return val_bytes != 8 ? 32 : 16; }

// Most warps of the dot products of KV vectors (128, 96 and 80 registers a thread).
constexpr int mvdot_warps(int kv) { return kv == 8 ? 16 : kv == 4 ? 20 : 24; }

// Dynamic shared-memory limit of one kernel, raised at most once per device and
// size: the value set so far on each device, read without a lock, raised under it.
constexpr int MAX_DEVICES = 64;
struct SmemLimit {
    std::atomic<int> bytes[MAX_DEVICES];
    std::mutex mu;
    SmemLimit() {
        for (auto &b : bytes) b.store(0, std::memory_order_relaxed);
    }
};
// Make `kern` launchable with `smem` bytes of dynamic shared memory on the current device.
template <typename K>
cudaError_t ensure_smem_limit(K kern, SmemLimit &lim, int smem) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= MAX_DEVICES) return cudaErrorInvalidDevice;
    if (lim.bytes[dev].load(std::memory_order_acquire) >= smem) return cudaSuccess;
    std::lock_guard<std::mutex> lk(lim.mu);
    if (lim.bytes[dev].load(std::memory_order_relaxed) >= smem) return cudaSuccess;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess) lim.bytes[dev].store(smem, std::memory_order_release);
    return e;
}

// Launch with programmatic serialization: the grid may become resident, and run up to its
// griddepcontrol.wait, while the kernel before it in the stream drains.
template <typename... Params, typename... Args>
cudaError_t launch_overlapped(void (*kern)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, Params(args)...);
}

// The combine and fix-up kernel: blocks of FIN_X x FIN_ROWS threads.  The dynamic shared memory that each of
// `blocks` of them asks for so that no SM takes more than its share: with s of them to an SM, 1 / s of what
// an SM has, less 4 KB (a block's static memory, what the system reserves, rounding).
constexpr int FIN_X = 32, FIN_ROWS = 8;
inline int finish_request(int64_t blocks, int sms, int smem_most) {
    const int64_t per_sm = (blocks + sms - 1) / sms;
    if (per_sm < 1 || per_sm >= 2048 / (FIN_X * FIN_ROWS)) return 0;
    const int64_t request = (smem_most - 7 * 1024) / per_sm - 4096;
    return request > 0 ? (int)request : 0;
}

struct LaunchArgs {
    StreamParams sp;
    int grid, block, smem;
    bool smemv;
    cudaStream_t stream;
};

// Dispatchers implemented in the per-value-type translation units.
cudaError_t launch_stream_f64(int mode, int kb, const LaunchArgs &a);
cudaError_t launch_stream_f32(int mode, int kb, const LaunchArgs &a);
cudaError_t launch_stream_bf16(int mode, int kb, const LaunchArgs &a);
cudaError_t launch_stream_f16(int mode, int kb, const LaunchArgs &a);
// One-vector pass: the accumulating product (sc), the dot products (sd) or both; and the values'
// gradient (v the minor, x the major vector, u the gradient).
cudaError_t launch_dvalues_f64(const PassParams &p, int grid, int warps, int smem, cudaStream_t s);
cudaError_t launch_pass_f64(bool sc, bool sd, const PassParams &p, int grid, int warps, int smem, cudaStream_t s);
cudaError_t launch_dvalues_f32(const PassParams &p, int grid, int warps, int smem, cudaStream_t s);
cudaError_t launch_pass_f32(bool sc, bool sd, const PassParams &p, int grid, int warps, int smem, cudaStream_t s);
cudaError_t launch_dvalues_bf16(const PassParams &p, int grid, int warps, int smem, cudaStream_t s);
cudaError_t launch_pass_bf16(bool sc, bool sd, const PassParams &p, int grid, int warps, int smem, cudaStream_t s);
cudaError_t launch_dvalues_f16(const PassParams &p, int grid, int warps, int smem, cudaStream_t s);
cudaError_t launch_pass_f16(bool sc, bool sd, const PassParams &p, int grid, int warps, int smem, cudaStream_t s);

// Accumulating and dot products of up to kv = 2, 4 or 8 vectors (32-bit accumulation).
cudaError_t launch_mvscatter_f32(int kv, const PassParams &p, int grid, int warps, int smem, cudaStream_t s);
cudaError_t launch_mvdot_f32(int kv, bool onchip, const PassParams &p, int grid, int warps, int smem, cudaStream_t s);
cudaError_t launch_mvscatter_bf16(int kv, const PassParams &p, int grid, int warps, int smem, cudaStream_t s);
cudaError_t launch_mvdot_bf16(int kv, bool onchip, const PassParams &p, int grid, int warps, int smem, cudaStream_t s);
cudaError_t launch_mvscatter_f16(int kv, const PassParams &p, int grid, int warps, int smem, cudaStream_t s);
cudaError_t launch_mvdot_f16(int kv, bool onchip, const PassParams &p, int grid, int warps, int smem, cudaStream_t s);
// Small kernels (small_kernels.cu).
// out_b[i] = sum over parts q of part[q * qstride + b * bstride + i], in FP64, in part order
// (qstride = 0: the layout [part][vector][element]).
cudaError_t launch_combine(bool vec_f64, bool part_f64, const void *part, int nparts, int n_minor, int kb,
                           void *const *out, cudaStream_t s, size_t qstride = 0, size_t bstride = 0);
// out[i * kbt + b] = in[b][i] (zeros for kb <= b < kbt), i < len: vectors interleaved for the
// multi-vector segmented passes (kbt = 2, 4 or 8).
cudaError_t launch_interleave(bool f64, int kbt, int kb, const void *const *in, int64_t len, void *out,
                              cudaStream_t s);
cudaError_t launch_fixup(bool vec_f64, const ZoneDev *zones, int z, const void *rec_left, const void *rec_right,
                         int P, int kb, void *const *out, cudaStream_t s);
// Both after a pass over one vector that served both products.
cudaError_t launch_combine_fixup(bool f64, const void *part, int nparts, int n_minor, void *short_out, const ZoneDev *zones,
                                 int z, const void *rec_left, const void *rec_right, int P, void *long_out,
                                 cudaStream_t s);
// Processors of the streaming launches: the chunks of tiles of every CTA's tile range, in
// order (the kernel's numbering, whatever the warp count).  Fills nzb[0..nproc] (if not
// NULL) with their nonzero boundaries; returns nproc.
int stream_processors(int ntiles, int T, int nnz, int ctas, int C, int32_t *nzb);

// Plan kernels (plan.cu).
// Structural checks (bits into *err) and the number of empty segments (into *nempty, zero on entry).
cudaError_t launch_validate(const int32_t *ptr, const int32_t *idx, int n_major, int nnz, int n_minor, int32_t *err,
                            int32_t *nempty, cudaStream_t s);
// rank[j] = nonempty segments before j (j <= n_major); seglist / emptylist: the nonempty and
// the empty segments in order; blk: seg_rank_blocks(n_major) ints of scratch.
cudaError_t launch_seg_ranks(const int32_t *pptr, int n_major, int32_t *rank, int32_t *seglist, int32_t *emptylist,
                             int32_t *blk, int32_t *total, cudaStream_t s);
// The step records of tiles of 256 spt nonzeros, from their masks and descriptors.
cudaError_t launch_steps(const TileMeta *meta, const uint32_t *masks, int mwp, int ntiles, int spt,
                         const int32_t *seglist, StepRec *steps, cudaStream_t s);
cudaError_t launch_pad_ptr(const int32_t *ptr, int32_t *pptr, int n_major, int nnz, int padded, cudaStream_t s);
// Per chunk: bounds by the Sec. II rule over P chunks (nzb == nullptr) or from nzb[0..P], first/last
// segments, owned end events, and the number of execution tiles of at most tmax nonzeros.
cudaError_t launch_chunks(const int32_t *pptr, int n_major, int nnz, int P, const int32_t *nzb, int tmax, ChunkAux *aux,
                          cudaStream_t s);
// The Sec. IV-B set-up over P chunks (multi-block scans): flags, groups, extents, descriptors,
// zones; counts[0] = z, counts[2] = V (must be zero on entry).  scratch: setup_scratch_bytes(P).
cudaError_t launch_setup(ChunkAux *aux, int P, ChunkDev *chunks, ZoneDev *zones, int32_t *counts, void *scratch,
                         cudaStream_t s);
size_t setup_scratch_bytes(int P);
// Execution tile boundaries tile_nzb[t] = min(t * T, nnz), t = 0..ntiles.
cudaError_t launch_tile_bounds(int ntiles, int T, int nnz, int32_t *tile_nzb, cudaStream_t s);
// Per tile: segment-start masks and the kernel's tile descriptors (needLeft / needRight of
// every tile from its neighbours' first and last segments; rank: launch_seg_ranks' array, or
// NULL when no segment is empty).
cudaError_t launch_masks(const int32_t *pptr, const ChunkAux *tiles, int ntiles, int nnz, int n_major, int mwp,
                         uint32_t *masks, int mwq, uint16_t *pfx, TileMeta *meta, const int32_t *rank, cudaStream_t s);

}  // namespace gbk
