// One-vector passes over the nonzeros of a validated plan: the accumulating product (SC: acc[idx[k]] +=
// val[k] * x[seg(k)], A_(i) x_(i) of Sec. III), the dot products (SD: u[j] = sum_k val[k] * v[idx[k]],
// v^T A_(i) of Sec. IV-A), or both from one reading of the matrix; the passes of several vectors and
// the values' gradient over the same steps.
//
// The tiles, chunks (the processors of Sec. II), masks and carry records are those of the
// streaming kernel, and the dot products are formed with its operations in its order (lane
// prefix restarted at every head, butterfly total of a head-free step, segmented Kogge-Stone
// scan, compensated carry), so a vector's dot products are the same bits in either kernel.
#pragma once

#include <algorithm>

#include "device_common.cuh"
#include "internal.h"

namespace gbk {

// What a warp of a pass works off: the steps of its CTA's chunks, staged by bulk copies into slots of
// the warp's own.  The CTA's tiles [ta, ta + nct) (the Sec. II rule over the grid) form nb chunks of
// C tiles, then single-tile ones (the streaming kernel's processors, numbered from proc0).  The
// warps take them in this order from a counter in shared memory: steps with heads cost more than
// head-free ones, and a fixed round-robin left warps waiting at the end (14% of warp time on the
// 50M-nonzero wide matrix).  Whichever warp runs a chunk, its sums are the same.
// A slot receives a step's indices, values and record, one bulk copy each (the nonzeros of a partial
// last step are read from global memory instead), and a header: step, chunk << 2 | first << 1 |
// last; step -1: no more work.
// VALS: the values too.
template <typename VT, bool VALS = true> struct StepFeed {
    static constexpr int SLOT = pass_slot_bytes(sizeof(VT));
    static constexpr int OFF_VAL = 1024, OFF_REC = OFF_VAL + 256 * (int)sizeof(VT), OFF_HDR = OFF_REC + (int)sizeof(StepRec);
    const PassParams &p;
    const int lane;
    uint64_t *bars;
    unsigned char *slots;
    int *next_chunk;
    CtaChunks c;
    bool dead = false;  // a copy did not arrive in time: no more work
    // cursor of the copies: steps [fs, fe) of chunk fq are still to come (lane 0 alone keeps it)
    int fs = 0, fe = 0, fq = -1, ffirst = 0;
    int s = 0;        // slot of the warp's next step
    uint32_t ph = 0;  // phase parity of that slot's barrier

    __device__ __forceinline__ StepFeed(const PassParams &p_, unsigned char *area, int *next_chunk_)
        : p(p_), lane(threadIdx.x & 31), next_chunk(next_chunk_) {
        const int warp = threadIdx.x >> 5;
        bars = reinterpret_cast<uint64_t *>(area) + warp * p.slots;
        slots = area + PASS_BAR_BYTES + warp * p.slots * SLOT;
        if (lane == 0) {
            for (int i = 0; i < p.slots; ++i) mbar_init(&bars[i], 1);
            fence_mbar_init();
        }
    }

    // Begin block gb of `blocks`; again: after another one, whose steps every warp has finished
    // (plans with one slot a warp).  The first copies fly while the vectors are staged.
    __device__ __forceinline__ void start(int gb, int blocks, bool again) {
        c = cta_chunks(gb, p.ntiles, blocks, p.chunk_tiles);
        if (threadIdx.x == 0) *next_chunk = 0;
        __syncthreads();
        if (!again) grid_wait();  // (values and vectors may come from the kernels before)
        if (again) ph ^= 1u;      // the slot's last phase said "no more work"
        if (dead) return;
        for (int i = 0; i < p.slots; ++i) issue(i);
        __syncwarp();
    }

    __device__ __forceinline__ void issue(int i) {
        if (lane != 0) return;
        if (fs == fe) {
            fq = atomicAdd(next_chunk, 1);
            if (fq < c.nq) {
                const int C = p.chunk_tiles;
                const int t0 = fq < c.nb ? c.ta + fq * C : c.ta + c.nb * C + (fq - c.nb);
                fs = t0 * p.spt;
                fe = min((t0 + (fq < c.nb ? C : 1)) * p.spt, p.nnz / 256 + (p.nnz % 256 != 0));
                ffirst = 2;
            }
        }
        unsigned char *slot = slots + i * SLOT;
        int2 hdr = make_int2(-1, 0);
        uint32_t bytes = 0;
        if (fs < fe) {
            hdr = make_int2(fs, (fq << 2) | ffirst | (fs + 1 == fe ? 1 : 0));
            bytes = sizeof(StepRec) + ((p.nnz >> 8) > fs ? 1024u + (VALS ? 256u * (uint32_t)sizeof(VT) : 0u) : 0u);
        }
        *reinterpret_cast<int2 *>(slot + OFF_HDR) = hdr;
        mbar_arrive_expect_tx(&bars[i], bytes);  // releases the header; the bulk bytes complete the phase
        if (fs < fe) {
            bulk_g2s(slot + OFF_REC, p.steps + fs, sizeof(StepRec), &bars[i]);
            if ((p.nnz >> 8) > fs) {
                bulk_g2s(slot, p.idx + (size_t)fs * 256, 1024u, &bars[i]);
                if constexpr (VALS)
                    bulk_g2s(slot + OFF_VAL, static_cast<const VT *>(p.vals) + (size_t)fs * 256,
                             256u * (uint32_t)sizeof(VT), &bars[i]);
            }
            ++fs;
            ffirst = 0;
        }
    }

    // The next step's slot and header, or false: no more work (or a copy did not arrive in time,
    // which is reported; the copies still in flight are let land).
    __device__ __forceinline__ bool next(unsigned char *&slot, int2 &hdr) {
        if (dead) return false;
        slot = slots + s * SLOT;
        bool ok = mbar_wait_bounded(&bars[s], ph, WAIT_LIMIT_NS);
        ok = __all_sync(FULL, ok);
        if (!ok) {
            if (lane == 0) atomicOr(p.err, ERR_WAIT);
            for (int r = 0; r < p.slots; ++r) {
                const int rs = s + r < p.slots ? s + r : s + r - p.slots;
                mbar_wait_bounded(&bars[rs], s + r < p.slots ? ph : ph ^ 1u, WAIT_LIMIT_NS);
            }
            dead = true;
            return false;
        }
        hdr = *reinterpret_cast<const int2 *>(slot + OFF_HDR);
        return hdr.x >= 0;  // (-1: every later slot is empty as well)
    }

    // The slot is read: its next step's copies go into it.  No lane may wait for the slot before
    // lane 0 has armed its barrier.
    __device__ __forceinline__ void release() {
        __syncwarp();
        issue(s);
        __syncwarp();
        if (++s == p.slots) {
            s = 0;
            ph ^= 1u;
        }
    }
};

// 32 warps of 64 registers (FP64: 16 of 128) with one step of 256 nonzeros in flight each: 66 KB, more
// than the latency of memory needs, and warps enough to hide the chains of a step (scan, additions).
// SC and the pair are bound by the shared-memory pipe (76 to 92% of its cycles): an FP32 addition is a
// load and a compare-and-swap that costs two, each with the bank conflicts of 32 rows.  SD alone
// runs near the memory rate, FP64 at the rate of its pipe (2 operations a cycle per SM).  With the
// combine and fix-up, streaming kernel before, this one now (us): 200M FP32 nonzeros, m = 20,000, bank
// order: pair 640 -> 386, SC 362 -> 294, SD 303 -> 261; 150M, n = 2,000: pair 538 -> 372, SC 313 ->
// 262, SD 242 -> 207; 8M FP64, n = 4,000: pair 121 -> 76, SC 62 -> 42, SD 69 -> 48.
// LANES: SC into very short vectors (PASS_LANES_MOST elements): every lane has an element of its own for
// each row, [row][lane], so that the lanes of a warp never add to the same place (one row, 51,000
// nonzeros: 58 us FP64 and 48 FP32 without, the streaming kernel 31 and 26).
template <typename VT, typename XT, bool SC, bool SD, bool LANES, int WB>
__global__ void __launch_bounds__(WB * 32, 1) pass_kernel(const __grid_constant__ PassParams p) {
    using AT = typename Acc<VT>::type;
    using AT2 = typename Pair<AT>::type;
    using Feed = StepFeed<VT>;
    // SC's additions are one attempt each, and what failed (another warp's addition to the same place came
    // between) is tried again after the eight, every lane at its own next one: a loop around each
    // addition repeated nearly all of them for the sake of single lanes (FP64, 8M nonzeros, n = 4,000:
    // 2.3 compare-and-swaps an addition, 16 cycles of the FP64 pipe each; 59 us, now 42; FP32, 10M, m =
    // 15,000: 40 -> 33; 200M, m = 20,000: 305 -> 294).  The FP32 pair has no registers left for it (402
    // against 391), and KV lanes to a nonzero meet too seldom (wide batch of 8: 695 against 670).
    constexpr bool DEFER = sizeof(AT) == 8 || !SD;
    extern __shared__ __align__(128) unsigned char smem[];
    // this warp's copy of the accumulator (warps share p.copies of them)
    AT *acc = reinterpret_cast<AT *>(smem + (threadIdx.x >> 5) % p.copies * p.acc_bytes) + (LANES ? threadIdx.x & 31 : 0);
    auto place = [&](int row) { return acc + (LANES ? 32 * row : row); };
    XT *vs = reinterpret_cast<XT *>(smem + p.copies * p.acc_bytes);
    const int lane = threadIdx.x & 31;
    // the combine and the zone fix-up may be launched: their blocks find room as this grid's CTAs end
    grid_release();
    // ---- the short vectors on chip: the accumulator zeroed (while the kernel before drains), the
    // input staged
    if constexpr (SC) {
        float4 *q = reinterpret_cast<float4 *>(smem);
        const int n16 = p.copies * p.acc_bytes >> 4;
        for (int i = threadIdx.x; i < n16; i += blockDim.x) q[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __shared__ int next_chunk;
    Feed feed(p, smem + p.copies * p.acc_bytes + p.vec_bytes, &next_chunk);
    // (FP64 batches: a grid row for each vector)
    const XT *xg = static_cast<const XT *>(SC && !SD && sizeof(AT) == 8 ? p.xv[blockIdx.y] : p.x);
    const int sh = (lane & 3) << 3;  // the lane's byte of its segment-start word
    const int sw = (lane >> 2) & 1;  // staggered shared-memory loads
    unsigned char *slot;
    int2 hdr;

    // the row-sorted copy's blocks take turns, each with its window of the input; else one block a CTA
    const int bpc = SD && !SC ? p.bpc : 1;
#pragma unroll 1
    for (int turn = 0; turn < bpc; ++turn) {
        const int gb = blockIdx.x * bpc + turn;
        if (turn > 0) __syncthreads();  // every warp is done with the block before
        feed.start(gb, gridDim.x * bpc, turn > 0);
        if constexpr (SD) {
            if (turn == 0)
                strided((int64_t)blockIdx.x * blockDim.x + threadIdx.x, (int64_t)gridDim.x * blockDim.x, p.nempty,
                        [&](int64_t i) { static_cast<XT *>(p.u)[p.emptylist[i]] = XT(0); });
            constexpr int xa = 16 / (int)sizeof(XT);
            const XT *src = static_cast<const XT *>(p.v);
            int len = p.n_minor;
            if (!SC && p.win) {  // (windows begin on 16 bytes)
                const int2 w = p.win[gb];
                src += w.x;
                len = min(w.y, p.n_minor);
            }
            const int n16 = len / xa;
#pragma unroll 4
            for (int i = threadIdx.x; i < n16; i += blockDim.x)
                reinterpret_cast<float4 *>(vs)[i] = call_load(reinterpret_cast<const float4 *>(src) + i);
            for (int i = n16 * xa + threadIdx.x; i < len; i += blockDim.x) vs[i] = call_load(src + i);
        }
        __syncthreads();

        AT chi = AT(0), clo = AT(0);  // open segment's running sum (SD)
        int cfirst = -1;              // the chunk's first segment when its sum goes to the left record
        while (feed.next(slot, hdr)) {
            const int ps = hdr.x << 8;
            const StepRec *rec = reinterpret_cast<const StepRec *>(slot + Feed::OFF_REC);
            const int2 bf = *reinterpret_cast<const int2 *>(&rec->first);  // first, flags
            // the step's segments are columns (rows of a tall matrix) first, first + 1, ..; with empty
            // ones between them they are counted by rank and looked up
            const bool gaps = (bf.y & STEP_GAPS) != 0;
            const int base = gaps && bf.x >= 0 ? plan_load(p.rank + bf.x) : bf.x;
            auto col_of = [&](int c) { return gaps ? plan_load(p.seglist + c) : c; };
            const bool whole = p.nnz - ps >= 256;
            // With SD this lane takes positions 8 lane .. 8 lane + 7, register e holding position
            // e ^ (4 sw) (staggered loads, which touch every bank exactly four times an instruction);
            // SC alone takes positions 32 e + lane (consecutive lanes then hold distinct rows of a
            // segment, and neighbouring entries of the long vector).
            int ix[8];
            AT va[8];
            if (whole && !SD) {
                const int32_t *is = reinterpret_cast<const int32_t *>(slot);
                const VT *vv = reinterpret_cast<const VT *>(slot + Feed::OFF_VAL);
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    ix[e] = is[32 * e + lane];
                    va[e] = to_acc<AT>(vv[32 * e + lane]);
                }
            } else if (whole) {
                stag8_idx(reinterpret_cast<const int32_t *>(slot), 8 * lane, sw, ix);
                Stag8<VT, AT>::run(slot + Feed::OFF_VAL, 8 * lane, sw, va);
            } else {
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const int at = SD ? 8 * lane + (e ^ (4 * sw)) : 32 * e + lane, pos = ps + at;
                    const bool in = pos < p.nnz;
                    // (the pair adds zeros for the positions past the end: to places of their own, for 243
                    // additions to one place took 10 us)
                    ix[e] = in ? call_load(p.idx + pos) : SC && SD ? at & p.spread : 0;
                    va[e] = in ? to_acc<AT>(static_cast<const VT *>(p.vals)[pos]) : AT(0);
                }
            }
            uint32_t hb = 0;
            int L = base;  // segment open before the lane's positions
            uint32_t w[8];
            if constexpr (SD) {
                const uint32_t mw = rec->heads[lane >> 2];
                hb = (mw >> sh) & 0xFFu;
                L += rec->before[lane >> 2] + __popc(mw & ((1u << sh) - 1u));
            } else {
                const uint4 wa = reinterpret_cast<const uint4 *>(rec->heads)[0], wb = reinterpret_cast<const uint4 *>(rec->heads)[1];
                w[0] = wa.x; w[1] = wa.y; w[2] = wa.z; w[3] = wa.w;
                w[4] = wb.x; w[5] = wb.y; w[6] = wb.z; w[7] = wb.w;
            }
            feed.release();
            const unsigned bal = SD ? __ballot_sync(FULL, hb != 0u) : static_cast<unsigned>(bf.y >> 16);  // 0: no head
            AT a[8], c[8];
            if constexpr (SC) {  // the long vector's entries
                if (bal == 0u) {
                    const AT xv = static_cast<AT>(call_load(xg + col_of(L)));
#pragma unroll
                    for (int e = 0; e < 8; ++e) c[e] = xv;
                } else if (!SD) {
                    const uint32_t lane_le = FULL >> (31 - lane);
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        c[e] = static_cast<AT>(call_load(xg + col_of(L + __popc(w[e] & lane_le))));
                        L += __popc(w[e]);
                    }
                } else {
                    const int nlo = __popc(hb & 0xFu);
                    const uint32_t h1 = sw ? hb >> 4 : hb, h2 = sw ? hb : hb >> 4;
                    int cc = sw ? L + nlo : L;
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        if (e == 4) cc = sw ? L : L + nlo;
                        cc += ((e < 4 ? h1 : h2) >> (e & 3)) & 1u;
                        // (-1 in the first step: empty segments before the first nonzero, whose head counts)
                        c[e] = static_cast<AT>(call_load(xg + col_of(cc)));
                    }
                }
            }
            if constexpr (SD) {
                if (hdr.y & 2) cfirst = (bf.y & STEP_NEED_LEFT) ? bf.x : -1;  // (a column)
#pragma unroll
                for (int e = 0; e < 8; ++e) a[e] = static_cast<AT>(vs[ix[e]]);
            }
            if constexpr (sizeof(AT) == 4) {  // (FP64 multiplies in the additions)
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    if constexpr (SC) c[e] *= va[e];
                    if constexpr (SD) a[e] = mul_rn(va[e], a[e]);
                }
            }
            if (!whole) {  // positions past the last nonzero (zero times an infinity is no zero)
                const int nv = p.nnz - ps;
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    if ((SD ? 8 * lane + (e ^ (4 * sw)) : 32 * e + lane) >= nv) {
                        if constexpr (SD) a[e] = AT(0);
                        if constexpr (SC) c[e] = AT(0);
                    }
                }
            }
            if constexpr (SC) {
                [[maybe_unused]] unsigned failed = 0u;
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    if constexpr (!DEFER) {
                        atomicAdd(place(ix[e]), c[e]);
                    } else if (!try_add(place(ix[e]), va[e], c[e])) {
                        failed |= 1u << e;
                    }
                }
                while (failed) {  // each lane its next failed addition
                    const int e = __ffs(failed) - 1;
                    int r = ix[0];
                    AT v = va[0], x = c[0];
#pragma unroll
                    for (int q = 1; q < 8; ++q)
                        if (e == q) {
                            r = ix[q];
                            v = va[q];
                            x = c[q];
                        }
                    if (try_add(place(r), v, x)) failed &= failed - 1u;
                }
            }
            if constexpr (SD) {  // into the order of the positions
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const AT lo = sw ? a[e + 4] : a[e];
                    a[e + 4] = sw ? a[e] : a[e + 4];
                    a[e] = lo;
                    if constexpr (sizeof(AT) == 8) {
                        const AT vl = sw ? va[e + 4] : va[e];
                        va[e + 4] = sw ? va[e] : va[e + 4];
                        va[e] = vl;
                    }
                }
            }
            if constexpr (SD) {
                // position e's term (FP32: its product) added to s, or alone where a segment starts
                auto next_term = [&](int e, AT s, bool restart) -> AT {
                    if constexpr (sizeof(AT) == 8) {
                        return seg_term(va[e], a[e], s, restart);
                    } else {
                        return restart ? a[e] : s + a[e];
                    }
                };
                auto first_term = [&](int e) -> AT { return next_term(e, AT(0), true); };
                if (bal == 0u) {
                    // the open segment runs through the step: butterfly total, compensated carry
                    AT s = first_term(0);
#pragma unroll
                    for (int e = 1; e < 8; ++e) s = next_term(e, s, false);
#pragma unroll
                    for (int d = 16; d >= 1; d >>= 1) s += __shfl_xor_sync(FULL, s, d);
                    carry_in(chi, clo, s);
                } else {
                    // lane prefix restarted at every head; f: what the lane's first head closes
                    const uint32_t h1 = hb & (0u - hb), hr = hb ^ h1;
                    AT s = first_term(0), f = AT(0);
#pragma unroll
                    for (int e = 1; e < 8; ++e) {
                        if ((h1 >> e) & 1u) f = s;
                        s = next_term(e, s, (hb >> e) & 1u);
                    }
                    if (hr) {  // segments inside the lane: closed by its later heads
                        AT q = first_term(0);
                        int cc = L;
#pragma unroll
                        for (int e = 1; e < 8; ++e) {
                            if ((hr >> e) & 1u) {
                                ++cc;
                                static_cast<XT *>(p.u)[col_of(cc)] = static_cast<XT>(q);
                            }
                            q = next_term(e, q, (hb >> e) & 1u);
                        }
                    }
                    // segmented scan of the lanes' open sums
                    const unsigned le = bal & (FULL >> (31 - lane));
                    const int reach = le ? lane - (31 - __clz(le)) : lane;
#pragma unroll
                    for (int d = 1; d < 32; d <<= 1) {
                        // (FP64 additions are worth a vote)
                        if (sizeof(AT) == 8 && !__any_sync(FULL, d <= reach)) break;
                        const AT o = __shfl_up_sync(FULL, s, d);
                        if (d <= reach) s += o;
                    }
                    AT before = __shfl_up_sync(FULL, s, 1);  // open sum at the end of the previous lane
                    if (lane == 0) before = AT(0);
                    if (hb && L >= 0) {  // (-1: empty segments before the first nonzero)
                        const AT lead = before + ((bal & ((1u << lane) - 1u)) ? AT(0) : chi + clo);
                        const AT v = f + lead;
                        const int col = col_of(L);
                        if (col == cfirst)
                            static_cast<AT2 *>(p.rec_left)[feed.c.proc0 + (hdr.y >> 2)] = make_pair2(v, AT(0));
                        else
                            static_cast<XT *>(p.u)[col] = static_cast<XT>(v);
                    }
                    chi = __shfl_sync(FULL, s, 31);
                    clo = AT(0);
                }
            }
            if constexpr (SD) {
                // a segment that ends with the tile is complete; the open one goes on in the chunk's
                // next tile or, at the end of the chunk, to the right record
                const bool ends = (bf.y & STEP_ENDS) != 0, chunk_last = (hdr.y & 1) != 0;
                if (ends || chunk_last) {
                    if (lane == 0) {
                        const int last = col_of(base + (bf.y >> 16));
                        if (ends) {
                            const AT v = chi + clo;
                            if (last == cfirst)
                                static_cast<AT2 *>(p.rec_left)[feed.c.proc0 + (hdr.y >> 2)] = make_pair2(v, AT(0));
                            else
                                static_cast<XT *>(p.u)[last] = static_cast<XT>(v);
                        } else if (bf.y & STEP_NEED_RIGHT) {
                            static_cast<AT2 *>(p.rec_right)[feed.c.proc0 + (hdr.y >> 2)] = make_pair2(chi, clo);
                        }
                    }
                    chi = AT(0);
                    clo = AT(0);
                }
            }
        }
    }

    if constexpr (SC) {
        __syncthreads();
        AT *part = static_cast<AT *>(p.part) + ((size_t)blockIdx.x * gridDim.y + blockIdx.y) * p.n_minor;
        const AT *acc0 = reinterpret_cast<const AT *>(smem);
        if constexpr (LANES) {  // (a warp takes a row: its 32 sums, then a butterfly)
            for (int i = threadIdx.x; i < 32 * p.n_minor; i += blockDim.x) {
                AT t = acc0[i];
                for (int r = 1; r < p.copies; ++r) t += acc0[r * (p.acc_bytes / (int)sizeof(AT)) + i];
#pragma unroll
                for (int d = 16; d >= 1; d >>= 1) t += __shfl_xor_sync(FULL, t, d);
                if (lane == 0) part[i >> 5] = t;
            }
        } else if (p.copies == 1) {
            for (int i = threadIdx.x; i < p.n_minor; i += blockDim.x) part[i] = acc0[i];
        } else {
            for (int i = threadIdx.x; i < p.n_minor; i += blockDim.x) {
                AT t = acc0[i];
                for (int r = 1; r < p.copies; ++r) t += acc0[r * (p.acc_bytes / (int)sizeof(AT)) + i];
                part[i] = t;
            }
        }
    }
}

// KV vectors' entries of index i from the interleaved copy [entry][KV], in shared or global memory.
// On chip the 16-byte halves of an 8-vector entry are swapped in every other group of four
// entries, so that one load instruction's halves fall into all banks (128 lanes' worth of
// conflicts fewer: 48M -> 34M wavefronts on 50M nonzeros).
template <int KV, bool ONCHIP> __device__ __forceinline__ void mv_gather(const float *vt, int i, float (&w)[KV]) {
    const float *q = vt + (size_t)i * KV;
    const int hs = ONCHIP && KV == 8 ? (i >> 2) & 1 : 0;
    if constexpr (!ONCHIP && KV == 8) {
        asm volatile("ld.global.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                     : "=f"(w[0]), "=f"(w[1]), "=f"(w[2]), "=f"(w[3]), "=f"(w[4]), "=f"(w[5]), "=f"(w[6]), "=f"(w[7])
                     : "l"(q));
    } else if constexpr (KV == 2) {
        const float2 t = ONCHIP ? *reinterpret_cast<const float2 *>(q) : call_load(reinterpret_cast<const float2 *>(q));
        w[0] = t.x;
        w[1] = t.y;
    } else {
#pragma unroll
        for (int h = 0; h < KV / 4; ++h) {
            const float4 t = ONCHIP ? reinterpret_cast<const float4 *>(q)[h ^ hs] : call_load(reinterpret_cast<const float4 *>(q) + h);
            w[4 * h] = t.x;
            w[4 * h + 1] = t.y;
            w[4 * h + 2] = t.z;
            w[4 * h + 3] = t.w;
        }
    }
}

// The dot products of up to KV = 2, 4 or 8 vectors in one reading of the matrix (32-bit
// accumulation).  A lane carries all vectors through its 8 positions: one vector load fetches a
// nonzero's KV entries (32 bytes for 8 vectors), GP positions' loads are in flight together, and
// the products, prefixes and scans of a vector are those of pass_kernel, so each vector's result
// equals its single product bit for bit.  Lane b keeps vector b's carry.  With the vectors read
// through L2 (8 of m = 20,000 are 640 KB) the gathers set the pace: one line a cycle and SM from the
// L1 tags.  8 vectors, 50M nonzeros: 261 us (streaming kernel 410); on chip (m = 5,500) 124 for 25M.
// 8 vectors over the row-sorted copy of 200M nonzeros (windows of 38,466 columns): 1,436 us with the
// combine (streaming kernel 2,763); 2 vectors 559 (1,254).
template <typename VT, int KV, bool ONCHIP, int WB>
__global__ void __launch_bounds__(WB * 32, 1) mvdot_kernel(const __grid_constant__ PassParams p) {
    using Feed = StepFeed<VT>;
    constexpr int GP = 4;
    extern __shared__ __align__(128) unsigned char smem[];
    const int lane = threadIdx.x & 31;
    grid_release();
    __shared__ int next_chunk;
    Feed feed(p, smem + p.vec_bytes, &next_chunk);
    const int sh = (lane & 3) << 3;
    const int sw = (lane >> 2) & 1;
    unsigned char *slot;
    int2 hdr;

    // the row-sorted copy's blocks take turns, each with its window of the vectors; else one block a CTA
#pragma unroll 1
    for (int turn = 0; turn < p.bpc; ++turn) {
        const int gb = blockIdx.x * p.bpc + turn;
        if (turn > 0) __syncthreads();  // every warp is done with the block before
        feed.start(gb, gridDim.x * p.bpc, turn > 0);
        if (turn == 0)
            strided((int64_t)blockIdx.x * blockDim.x + threadIdx.x, (int64_t)gridDim.x * blockDim.x, p.nempty, [&](int64_t i) {
                const int col = p.emptylist[i];
                for (int b = 0; b < p.kb; ++b) p.uv[b][col] = 0.f;
            });
        const int2 w = p.win ? p.win[gb] : make_int2(0, p.n_minor);  // (windows begin on four entries)
        const float *vt = static_cast<const float *>(p.v) + (size_t)w.x * KV;
        if constexpr (ONCHIP) {
            const int n8 = min(w.y, p.n_minor) * KV / 2;  // in pairs of values
#pragma unroll 4
            for (int i = threadIdx.x; i < n8; i += blockDim.x)
                reinterpret_cast<float2 *>(smem)[KV == 8 ? i ^ ((i >> 3) & 2) : i] = call_load(reinterpret_cast<const float2 *>(vt) + i);
            vt = reinterpret_cast<const float *>(smem);
            __syncthreads();
        }
        float chi = 0.f, clo = 0.f;  // vector `lane`'s open segment
        int cfirst = -1;
        while (feed.next(slot, hdr)) {
            const int ps = hdr.x << 8;
            const StepRec *rec = reinterpret_cast<const StepRec *>(slot + Feed::OFF_REC);
            const int2 bf = *reinterpret_cast<const int2 *>(&rec->first);
            const bool gaps = (bf.y & STEP_GAPS) != 0;
            const int base = gaps && bf.x >= 0 ? plan_load(p.rank + bf.x) : bf.x;
            auto col_of = [&](int c) { return gaps ? plan_load(p.seglist + c) : c; };
            const bool whole = p.nnz - ps >= 256;
            int ix[8];
            float va[8];
            if (whole) {
                stag8_idx(reinterpret_cast<const int32_t *>(slot), 8 * lane, sw, ix);
                Stag8<VT, float>::run(slot + Feed::OFF_VAL, 8 * lane, sw, va);
#pragma unroll
                for (int e = 0; e < 4; ++e) {  // into the order of the positions
                    const int i0 = sw ? ix[e + 4] : ix[e];
                    const float v0 = sw ? va[e + 4] : va[e];
                    ix[e + 4] = sw ? ix[e] : ix[e + 4];
                    va[e + 4] = sw ? va[e] : va[e + 4];
                    ix[e] = i0;
                    va[e] = v0;
                }
            } else {
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const int pos = ps + 8 * lane + e;
                    const bool in = pos < p.nnz;
                    ix[e] = in ? call_load(p.idx + pos) : 0;
                    va[e] = in ? to_f<VT>(static_cast<const VT *>(p.vals)[pos]) : 0.f;
                }
            }
            const uint32_t mw = rec->heads[lane >> 2];
            const uint32_t hb = (mw >> sh) & 0xFFu;
            const int L = base + rec->before[lane >> 2] + __popc(mw & ((1u << sh) - 1u));
            feed.release();
            const unsigned bal = __ballot_sync(FULL, hb != 0u);
            const int proc = feed.c.proc0 + (hdr.y >> 2);
            if (hdr.y & 2) cfirst = (bf.y & STEP_NEED_LEFT) ? bf.x : -1;

            // the lane's prefix s, restarted at every head; f: what its first head closes; segments
            // inside the lane are closed by its later heads
            const uint32_t h1 = hb & (0u - hb), hr = hb ^ h1;
            float s[KV], f[KV];
            int cc = L;
#pragma unroll
            for (int b = 0; b < KV; ++b) s[b] = f[b] = 0.f;
#pragma unroll
            for (int e0 = 0; e0 < 8; e0 += GP) {
                float w[GP][KV];
#pragma unroll
                for (int g = 0; g < GP; ++g) mv_gather<KV, ONCHIP>(vt, ix[e0 + g], w[g]);
                if (!whole) {  // past the last nonzero (zero times an infinity is no zero)
#pragma unroll
                    for (int g = 0; g < GP; ++g)
                        if (8 * lane + e0 + g >= p.nnz - ps) {
#pragma unroll
                            for (int b = 0; b < KV; ++b) w[g][b] = 0.f;
                        }
                }
#pragma unroll
                for (int g = 0; g < GP; ++g) {
                    const int e = e0 + g;
                    if (e > 0) {
                        if ((hr >> e) & 1u) {
                            const int col = col_of(++cc);
#pragma unroll
                            for (int b = 0; b < KV; ++b)
                                if (b < p.kb) p.uv[b][col] = s[b];
                        }
                        if ((h1 >> e) & 1u) {
#pragma unroll
                            for (int b = 0; b < KV; ++b) f[b] = s[b];
                        }
                    }
                    const bool restart = e == 0 || ((hb >> e) & 1u);
#pragma unroll
                    for (int b = 0; b < KV; ++b) {
                        const float q = mul_rn(va[e], w[g][b]);
                        s[b] = restart ? q : s[b] + q;
                    }
                }
            }
            if (bal == 0u) {
                // butterfly totals, the vectors halved between the lanes as long as there are several
                // (the same pairs are added as by a butterfly of every vector); lane b gets vector b's
                int n = KV, d = 16;
#pragma unroll
                for (; n > 1; n >>= 1, d >>= 1) {
                    const bool up = (lane & d) != 0;
#pragma unroll
                    for (int j = 0; j < KV / 2; ++j)
                        if (j < n / 2) {
                            const float mine = up ? s[j + n / 2] : s[j], other = up ? s[j] : s[j + n / 2];
                            s[j] = mine + __shfl_xor_sync(FULL, other, d);
                        }
                }
#pragma unroll
                for (; d >= 1; d >>= 1) s[0] += __shfl_xor_sync(FULL, s[0], d);
                carry_in(chi, clo, __shfl_sync(FULL, s[0], (lane * (32 / KV)) & 31));
            } else {
                const unsigned le = bal & (FULL >> (31 - lane));
                const int reach = le ? lane - (31 - __clz(le)) : lane;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    if (!__any_sync(FULL, d <= reach)) break;
#pragma unroll
                    for (int b = 0; b < KV; ++b) {
                        const float o = __shfl_up_sync(FULL, s[b], d);
                        if (d <= reach) s[b] += o;
                    }
                }
                const float carry = chi + clo;
                const bool own = hb && L >= 0, inner = (bal & ((1u << lane) - 1u)) != 0u;
                const int col = own ? col_of(L) : 0;
                clo = 0.f;
#pragma unroll
                for (int b = 0; b < KV; ++b) {
                    float before = __shfl_up_sync(FULL, s[b], 1);
                    if (lane == 0) before = 0.f;
                    const float cb = __shfl_sync(FULL, carry, b), end = __shfl_sync(FULL, s[b], 31);
                    if (own && b < p.kb) {
                        const float v = f[b] + (before + (inner ? 0.f : cb));
                        if (col == cfirst)
                            static_cast<float2 *>(p.rec_left)[(size_t)b * p.nproc + proc] = make_float2(v, 0.f);
                        else
                            p.uv[b][col] = v;
                    }
                    if (lane == b) chi = end;
                }
            }
            const bool ends = (bf.y & STEP_ENDS) != 0, chunk_last = (hdr.y & 1) != 0;
            if (ends || chunk_last) {
                if (lane < p.kb) {
                    const int last = col_of(base + (bf.y >> 16));
                    if (ends) {
                        const float v = chi + clo;
                        if (last == cfirst)
                            static_cast<float2 *>(p.rec_left)[(size_t)lane * p.nproc + proc] = make_float2(v, 0.f);
                        else
                            p.uv[lane][last] = v;
                    } else if (bf.y & STEP_NEED_RIGHT) {
                        static_cast<float2 *>(p.rec_right)[(size_t)lane * p.nproc + proc] = make_float2(chi, clo);
                    }
                }
                chi = 0.f;
                clo = 0.f;
            }
        }
    }
}

// The accumulating product of up to KV = 2, 4 or 8 vectors in one reading of the matrix (32-bit
// accumulation), the accumulators interleaved [row][KV] on chip.  KV lanes take one nonzero, a
// vector each, four nonzeros in a row per load; 32 / KV nonzeros per addition then meet fewer
// bank conflicts than 32 rows of one vector do (additions at 980, 1,160, 1,450 G/s for KV = 2, 4, 8
// against 800; a 64- or 128-bit compare-and-swap over 2 or 4 vectors is no faster), and the nonzeros
// are staged once.  8 vectors of 20,000 rows, 50M nonzeros, two a pass: 603 us (866 one by one in the
// streaming kernel).  The partials go out as [cta][vector][row].
template <typename VT, int KV, int WB>
__global__ void __launch_bounds__(WB * 32, 1) mvscatter_kernel(const __grid_constant__ PassParams p) {
    using Feed = StepFeed<VT>;
    constexpr int NG = 32 / KV;  // lane groups
    extern __shared__ __align__(128) unsigned char smem[];
    float *acc = reinterpret_cast<float *>(smem + (threadIdx.x >> 5) % p.copies * p.acc_bytes);
    const int lane = threadIdx.x & 31;
    const int g = lane / KV, b = lane % KV;
    const bool act = b < p.kb;
    grid_release();
    {
        float4 *q = reinterpret_cast<float4 *>(smem);
        const int n16 = p.copies * p.acc_bytes >> 4;
        for (int i = threadIdx.x; i < n16; i += blockDim.x) q[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __shared__ int next_chunk;
    Feed feed(p, smem + p.copies * p.acc_bytes, &next_chunk);
    feed.start(blockIdx.x, gridDim.x, false);
    __syncthreads();
    const float *xb = static_cast<const float *>(p.xv[act ? b : 0]);
    acc += b;
    unsigned char *slot;
    int2 hdr;
    while (feed.next(slot, hdr)) {
        const int ps = hdr.x << 8;
        const StepRec *rec = reinterpret_cast<const StepRec *>(slot + Feed::OFF_REC);
        const int2 bf = *reinterpret_cast<const int2 *>(&rec->first);
        const bool gaps = (bf.y & STEP_GAPS) != 0;
        const int base = gaps && bf.x >= 0 ? plan_load(p.rank + bf.x) : bf.x;
        auto col_of = [&](int c) { return gaps ? plan_load(p.seglist + c) : c; };
        const int left = p.nnz - ps;  // (256 or more but in a partial last step)
        int cprev = -1;
        float x = 0.f;
#pragma unroll 2
        for (int j = 0; j < 64 / NG; ++j) {
            const int pos = 4 * (NG * j + g);
            const uint32_t w = rec->heads[pos >> 5];
            const uint32_t hb = w >> (pos & 31);
            int c = base + rec->before[pos >> 5] + __popc(w & ((1u << (pos & 31)) - 1u));
            int row[4];
            float v[4];
            if (left >= 256) {
                const int4 q = *reinterpret_cast<const int4 *>(slot + 4 * pos);
                row[0] = q.x; row[1] = q.y; row[2] = q.z; row[3] = q.w;
                Load4<VT, float>::run(slot + Feed::OFF_VAL, pos, v);
            } else {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const bool in = pos + i < left;
                    row[i] = in ? call_load(p.idx + ps + pos + i) : -1;
                    v[i] = in ? to_f<VT>(static_cast<const VT *>(p.vals)[ps + pos + i]) : 0.f;
                }
            }
            float xs[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                c += (hb >> i) & 1u;
                if (c != cprev) x = call_load(xb + col_of(c));
                cprev = c;
                xs[i] = x;
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (act && row[i] >= 0) atomicAdd(acc + row[i] * KV, v[i] * xs[i]);
        }
        feed.release();
    }
    __syncthreads();
    float *part = static_cast<float *>(p.part) + (size_t)blockIdx.x * p.kb * p.n_minor;
    const float *acc0 = reinterpret_cast<const float *>(smem);
    for (int i = threadIdx.x; i < p.n_minor * KV; i += blockDim.x) {
        if (i % KV >= p.kb) continue;
        float t = acc0[i];
        for (int r = 1; r < p.copies; ++r) t += acc0[r * (p.acc_bytes / 4) + i];
        part[(size_t)(i % KV) * p.n_minor + i / KV] = t;
    }
}

template <typename VT>
cudaError_t launch_mvscatter(int kv, const PassParams &p, int grid, int warps, int smem, cudaStream_t s) {
    if constexpr (sizeof(VT) == 8) {
        return cudaErrorInvalidValue;
    } else {
        auto go = [&](auto kern, SmemLimit &lim) {
            const cudaError_t e = ensure_smem_limit(kern, lim, smem);
            if (e != cudaSuccess) return e;
            return launch_overlapped(kern, dim3(grid), dim3(warps * 32), smem, s, p);
        };
        static SmemLimit lim[3];
        return kv == 2   ? go(mvscatter_kernel<VT, 2, 32>, lim[0])
               : kv == 4 ? go(mvscatter_kernel<VT, 4, 32>, lim[1])
                         : go(mvscatter_kernel<VT, 8, 32>, lim[2]);
    }
}

template <typename VT, int KV, bool ONCHIP>
cudaError_t launch_mvdot_one(const PassParams &p, int grid, int warps, int smem, cudaStream_t s) {
    auto kern = mvdot_kernel<VT, KV, ONCHIP, mvdot_warps(KV)>;
    static SmemLimit lim;
    const cudaError_t e = ensure_smem_limit(kern, lim, smem);
    if (e != cudaSuccess) return e;
    return launch_overlapped(kern, dim3(grid), dim3(warps * 32), smem, s, p);
}
template <typename VT>
cudaError_t launch_mvdot(int kv, bool onchip, const PassParams &p, int grid, int warps, int smem, cudaStream_t s) {
    if constexpr (sizeof(VT) == 8) {
        return cudaErrorInvalidValue;
    } else {
        if (onchip)
            return kv == 2   ? launch_mvdot_one<VT, 2, true>(p, grid, warps, smem, s)
                   : kv == 4 ? launch_mvdot_one<VT, 4, true>(p, grid, warps, smem, s)
                             : launch_mvdot_one<VT, 8, true>(p, grid, warps, smem, s);
        return kv == 2   ? launch_mvdot_one<VT, 2, false>(p, grid, warps, smem, s)
               : kv == 4 ? launch_mvdot_one<VT, 4, false>(p, grid, warps, smem, s)
                         : launch_mvdot_one<VT, 8, false>(p, grid, warps, smem, s);
    }
}

// Two neighbouring values of the gradient, in the values' type, by one store.
__device__ __forceinline__ void store2(float *g, float a, float b) { *reinterpret_cast<float2 *>(g) = make_float2(a, b); }
__device__ __forceinline__ void store2(double *g, double a, double b) { *reinterpret_cast<double2 *>(g) = make_double2(a, b); }
__device__ __forceinline__ void store2(__nv_bfloat16 *g, float a, float b) {
    *reinterpret_cast<__nv_bfloat162 *>(g) = __halves2bfloat162(__float2bfloat16_rn(a), __float2bfloat16_rn(b));
}
__device__ __forceinline__ void store2(__half *g, float a, float b) {
    *reinterpret_cast<__half2 *>(g) = __halves2half2(__float2half_rn(a), __float2half_rn(b));
}

// The gradient of r^T A x by the stored values, g[k] = minor[idx[k]] * major[seg(k)]: the minor
// vector on chip, a lane taking positions 64 j + 2 lane and the next one (conflict-free index
// loads, whole-line stores).  Reads 4 bytes and writes one value a nonzero; the streaming kernel,
// 128 positions a step, took 108 us for 20M FP16 values (m = 8,003), this one 38.  A minor vector too
// long for the chip is read through L2.
template <typename VT, typename XT, bool ONCHIP, int WB>
__global__ void __launch_bounds__(WB * 32, 1) dvalues_kernel(const __grid_constant__ PassParams p) {
    using AT = typename Acc<VT>::type;
    using Feed = StepFeed<VT, false>;
    extern __shared__ __align__(128) unsigned char smem[];
    XT *vs = reinterpret_cast<XT *>(smem);
    const int lane = threadIdx.x & 31;
    grid_release();
    __shared__ int next_chunk;
    Feed feed(p, smem + p.vec_bytes, &next_chunk);
    feed.start(blockIdx.x, gridDim.x, false);
    const XT *vg = static_cast<const XT *>(p.v);
    auto minor = [&](int i) -> AT {
        if constexpr (ONCHIP)
            return static_cast<AT>(vs[i]);
        else
            return static_cast<AT>(call_load(vg + i));
    };
    if constexpr (ONCHIP) {
        constexpr int xa = 16 / (int)sizeof(XT);
        const XT *src = vg;
        const int n16 = p.n_minor / xa;
#pragma unroll 4
        for (int i = threadIdx.x; i < n16; i += blockDim.x)
            reinterpret_cast<float4 *>(vs)[i] = call_load(reinterpret_cast<const float4 *>(src) + i);
        for (int i = n16 * xa + threadIdx.x; i < p.n_minor; i += blockDim.x) vs[i] = call_load(src + i);
    }
    __syncthreads();
    const XT *xg = static_cast<const XT *>(p.x);
    VT *g = static_cast<VT *>(p.u);
    unsigned char *slot;
    int2 hdr;
    while (feed.next(slot, hdr)) {
        const int ps = hdr.x << 8;
        const StepRec *rec = reinterpret_cast<const StepRec *>(slot + Feed::OFF_REC);
        const int2 bf = *reinterpret_cast<const int2 *>(&rec->first);
        const bool gaps = (bf.y & STEP_GAPS) != 0;
        const int base = gaps && bf.x >= 0 ? plan_load(p.rank + bf.x) : bf.x;
        auto col_of = [&](int c) { return gaps ? plan_load(p.seglist + c) : c; };
        const int left = p.nnz - ps;
        int ix[8];
        AT x[8];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int pos = 64 * j + 2 * lane;
            if (left >= 256) {
                const int2 q = *reinterpret_cast<const int2 *>(slot + 4 * pos);
                ix[2 * j] = q.x;
                ix[2 * j + 1] = q.y;
            } else {
                ix[2 * j] = pos < left ? call_load(p.idx + ps + pos) : 0;
                ix[2 * j + 1] = pos + 1 < left ? call_load(p.idx + ps + pos + 1) : 0;
            }
            const uint32_t w = rec->heads[pos >> 5];
            const int b = pos & 31;  // (even: bit b + 1 exists)
            const int c0 = base + rec->before[pos >> 5] + __popc(w & ((2u << b) - 1u));
            const int c1 = c0 + ((w >> (b + 1)) & 1u);
            x[2 * j] = static_cast<AT>(call_load(xg + col_of(max(c0, 0))));
            x[2 * j + 1] = static_cast<AT>(call_load(xg + col_of(max(c1, 0))));
        }
        feed.release();
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int pos = 64 * j + 2 * lane;
            const AT a = minor(ix[2 * j]) * x[2 * j], c = minor(ix[2 * j + 1]) * x[2 * j + 1];
            if (pos + 1 < left)
                store2(g + ps + pos, a, c);
            else if (pos < left)
                g[ps + pos] = from_d<VT>(static_cast<double>(a));
        }
    }
}

template <typename VT, typename XT, bool ONCHIP>
cudaError_t launch_dvalues_one(const PassParams &p, int grid, int warps, int smem, cudaStream_t s) {
    auto kern = dvalues_kernel<VT, XT, ONCHIP, pass_warps(sizeof(VT))>;
    static SmemLimit lim;
    const cudaError_t e = ensure_smem_limit(kern, lim, smem);
    if (e != cudaSuccess) return e;
    return launch_overlapped(kern, dim3(grid), dim3(warps * 32), smem, s, p);
}

// (p.vec_bytes: 0 for a minor vector in global memory)
template <typename VT, typename XT>
cudaError_t launch_dvalues(const PassParams &p, int grid, int warps, int smem, cudaStream_t s) {
    return p.vec_bytes ? launch_dvalues_one<VT, XT, true>(p, grid, warps, smem, s)
                       : launch_dvalues_one<VT, XT, false>(p, grid, warps, smem, s);
}

template <typename VT, typename XT, bool SC, bool SD, bool LANES>
cudaError_t launch_pass_one(const PassParams &p, int grid, int warps, int smem, cudaStream_t s) {
    constexpr int WB = pass_warps(sizeof(VT));
    auto kern = pass_kernel<VT, XT, SC, SD, LANES, WB>;
    static SmemLimit lim;
    const cudaError_t e = ensure_smem_limit(kern, lim, smem);
    if (e != cudaSuccess) return e;
    const int vectors = SC && !SD && sizeof(VT) == 8 ? std::max(1, p.kb) : 1;
    return launch_overlapped(kern, dim3(grid, vectors), dim3(warps * 32), smem, s, p);
}

template <typename VT, typename XT>
cudaError_t launch_pass(bool sc, bool sd, const PassParams &p, int grid, int warps, int smem, cudaStream_t s) {
    if (sc && sd) {
        if constexpr (sizeof(VT) == 8)
            if (p.lanes) return launch_pass_one<VT, XT, true, true, true>(p, grid, warps, smem, s);
        return launch_pass_one<VT, XT, true, true, false>(p, grid, warps, smem, s);
    }
    if (sc)
        return p.lanes ? launch_pass_one<VT, XT, true, false, true>(p, grid, warps, smem, s)
                       : launch_pass_one<VT, XT, true, false, false>(p, grid, warps, smem, s);
    return launch_pass_one<VT, XT, false, true, false>(p, grid, warps, smem, s);
}

}  // namespace gbk
