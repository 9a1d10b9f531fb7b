// One-vector passes over the nonzeros of a validated plan: the accumulating product (SC: acc[idx[k]] += val[k] * x[seg(k)], A_(i) x_(i) of Sec. III),
// the dot products (SD: u[j] = sum_k val[k] * v[idx[k]], v^T A_(i) of Sec. IV-A), or both from
// one reading of the matrix.
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

template <typename VT, typename XT, bool SC, bool SD, int WB>
__global__ void __launch_bounds__(WB * 32, 1) pass_kernel(const __grid_constant__ PassParams p) {
    using AT = typename Acc<VT>::type;
    using AT2 = typename Pair<AT>::type;
    constexpr int SLOT = pass_slot_bytes(sizeof(VT));
    constexpr int OFF_VAL = 1024, OFF_REC = OFF_VAL + 256 * (int)sizeof(VT), OFF_HDR = OFF_REC + (int)sizeof(StepRec);
    extern __shared__ __align__(128) unsigned char smem[];
    // this warp's copy of the accumulator (warps share p.copies of them)
    AT *acc = reinterpret_cast<AT *>(smem + (threadIdx.x >> 5) % p.copies * p.acc_bytes);
    XT *vs = reinterpret_cast<XT *>(smem + p.copies * p.acc_bytes);
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int W = blockDim.x >> 5;
    const int S = p.slots;
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + p.copies * p.acc_bytes + p.vec_bytes) + warp * S;
    unsigned char *slots = smem + p.copies * p.acc_bytes + p.vec_bytes + PASS_BAR_BYTES + warp * S * SLOT;

    // This CTA's tiles [ta, ta + nct) by the Sec. II rule over the grid: nb chunks of C tiles, then
    // single-tile ones (the streaming kernel's processors, numbered from proc0).  The warps take
    // them in this order from a counter in shared memory: steps with heads cost more than
    // head-free ones, and a fixed round-robin left warps waiting at the end (14% of warp time on
    // the 50M-nonzero wide matrix).  Whichever warp runs a chunk, its sums are the same.
    const int C = p.chunk_tiles;
    const CtaChunks cc_ = cta_chunks(blockIdx.x, p.ntiles, gridDim.x, C);
    const int ta = cc_.ta, nb = cc_.nb, nq = cc_.nq, proc0 = cc_.proc0;
    const int nsteps = p.nnz / 256 + (p.nnz % 256 != 0);  // of the matrix

    // the combine and the zone fix-up may be launched: their blocks find room as this grid's CTAs end
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    __shared__ int next_chunk;
    if (threadIdx.x == 0) next_chunk = 0;
    if (lane == 0) {
        for (int s = 0; s < S; ++s) mbar_init(&bars[s], 1);
        fence_mbar_init();
    }
    __syncthreads();

    // ---- the copies of the next step into slot s: indices, values and the step's record, one bulk
    // copy each (a partial last step's nonzeros are read from global memory instead), and a
    // header: step, chunk << 2 | first << 1 | last; step -1: no more work.  Cursor of the copies:
    // steps [fs, fe) of chunk fq are still to come (lane 0 alone keeps it).
    int fs = 0, fe = 0, fq = -1, ffirst = 0;
    auto issue = [&](int s) {
        if (lane == 0) {
            if (fs == fe) {
                fq = atomicAdd(&next_chunk, 1);
                if (fq < nq) {
                    const int t0 = fq < nb ? ta + fq * C : ta + nb * C + (fq - nb);
                    fs = t0 * p.spt;
                    fe = min((t0 + (fq < nb ? C : 1)) * p.spt, nsteps);
                    ffirst = 2;
                }
            }
            unsigned char *slot = slots + s * SLOT;
            int2 hdr = make_int2(-1, 0);
            uint32_t bytes = 0;
            if (fs < fe) {
                hdr = make_int2(fs, (fq << 2) | ffirst | (fs + 1 == fe ? 1 : 0));
                bytes = sizeof(StepRec) + ((p.nnz >> 8) > fs ? 1024u + 256u * (uint32_t)sizeof(VT) : 0u);
            }
            *reinterpret_cast<int2 *>(slot + OFF_HDR) = hdr;
            mbar_arrive_expect_tx(&bars[s], bytes);  // releases the header; the bulk bytes complete the phase
            if (fs < fe) {
                bulk_g2s(slot + OFF_REC, p.steps + fs, sizeof(StepRec), &bars[s]);
                if ((p.nnz >> 8) > fs) {
                    bulk_g2s(slot, p.idx + (size_t)fs * 256, 1024u, &bars[s]);
                    bulk_g2s(slot + OFF_VAL, static_cast<const VT *>(p.vals) + (size_t)fs * 256,
                             256u * (uint32_t)sizeof(VT), &bars[s]);
                }
                ++fs;
                ffirst = 0;
            }
        }
    };
    for (int s = 0; s < S; ++s) issue(s);  // the first copies fly while the vectors are staged

    // ---- the short vectors on chip: the accumulator zeroed, the input staged
    if constexpr (SC) {
        float4 *q = reinterpret_cast<float4 *>(smem);
        const int n16 = p.copies * p.acc_bytes >> 4;
        for (int i = threadIdx.x; i < n16; i += blockDim.x) q[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    if constexpr (SD) {
        for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < p.nempty; i += gridDim.x * blockDim.x)
            static_cast<XT *>(p.u)[p.emptylist[i]] = XT(0);
        constexpr int xa = 16 / (int)sizeof(XT);
        const XT *src = static_cast<const XT *>(p.v);
        const int n16 = p.n_minor / xa;
#pragma unroll 4
        for (int i = threadIdx.x; i < n16; i += blockDim.x)
            reinterpret_cast<float4 *>(vs)[i] = __ldg(reinterpret_cast<const float4 *>(src) + i);
        for (int i = n16 * xa + threadIdx.x; i < p.n_minor; i += blockDim.x) vs[i] = __ldg(src + i);
    }
    __syncthreads();

    const XT *xg = static_cast<const XT *>(p.x);
    const int sh = (lane & 3) << 3;  // the lane's byte of its segment-start word
    const int sw = (lane >> 2) & 1;  // staggered shared-memory loads

    AT chi = AT(0), clo = AT(0);  // open segment's running sum (SD)
    int cfirst = -1;              // the chunk's first segment when its sum goes to the left record
    int s = 0;
    uint32_t ph = 0;
    while (true) {
        unsigned char *slot = slots + s * SLOT;
        bool okw = mbar_wait_bounded(&bars[s], ph, WAIT_LIMIT_NS);
        okw = __all_sync(FULL, okw);
        if (!okw) {  // report, let the copies in flight land, do no more work
            if (lane == 0) atomicOr(p.err, ERR_WAIT);
            for (int r = 0; r < S; ++r) {
                const int rs = s + r < S ? s + r : s + r - S;
                mbar_wait_bounded(&bars[rs], s + r < S ? ph : ph ^ 1u, WAIT_LIMIT_NS);
            }
            break;
        }
        const int2 hdr = *reinterpret_cast<const int2 *>(slot + OFF_HDR);
        if (hdr.x < 0) break;  // every later slot is empty as well
        const int ps = hdr.x << 8;
        const StepRec *rec = reinterpret_cast<const StepRec *>(slot + OFF_REC);
        const int2 bf = *reinterpret_cast<const int2 *>(&rec->first);  // first, flags
        // the step's segments are columns (rows of a tall matrix) first, first + 1, ..; with empty
        // ones between them they are counted by rank and looked up
        const bool gaps = (bf.y & STEP_GAPS) != 0;
        const int base = gaps && bf.x >= 0 ? __ldg(p.rank + bf.x) : bf.x;
        auto col_of = [&](int c) { return gaps ? __ldg(p.seglist + c) : c; };
        const bool whole = p.nnz - ps >= 256;
        // With SD this lane takes positions 8 lane .. 8 lane + 7, register e holding position
        // e ^ (4 sw) (staggered loads, which touch every bank exactly four times an instruction);
        // SC alone takes positions 32 e + lane (consecutive lanes then hold distinct rows of a
        // segment, and neighbouring entries of the long vector).
        int ix[8];
        AT va[8];
        if (whole && !SD) {
            const int32_t *is = reinterpret_cast<const int32_t *>(slot);
            const VT *vv = reinterpret_cast<const VT *>(slot + OFF_VAL);
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                ix[e] = is[32 * e + lane];
                va[e] = to_acc<AT>(vv[32 * e + lane]);
            }
        } else if (whole) {
            stag8_idx(reinterpret_cast<const int32_t *>(slot), 8 * lane, sw, ix);
            Stag8<VT, AT>::run(slot + OFF_VAL, 8 * lane, sw, va);
        } else {
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int pos = ps + (SD ? 8 * lane + (e ^ (4 * sw)) : 32 * e + lane);
                const bool in = pos < p.nnz;
                ix[e] = in ? __ldg(p.idx + pos) : 0;
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
        __syncwarp();  // the slot is read: its next step's copies go into it
        issue(s);
        __syncwarp();  // no lane may wait for the slot before lane 0 has armed its barrier
        if (++s == S) {
            s = 0;
            ph ^= 1u;
        }
        const unsigned bal = SD ? __ballot_sync(FULL, hb != 0u) : static_cast<unsigned>(bf.y >> 16);  // 0: no head
        AT a[8], c[8];
        if constexpr (SC) {  // the long vector's entries
            if (bal == 0u) {
                const AT xv = static_cast<AT>(__ldg(xg + col_of(L)));
#pragma unroll
                for (int e = 0; e < 8; ++e) c[e] = xv;
            } else if (!SD) {
                const uint32_t lane_le = FULL >> (31 - lane);
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    c[e] = static_cast<AT>(__ldg(xg + col_of(L + __popc(w[e] & lane_le))));
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
                    c[e] = static_cast<AT>(__ldg(xg + col_of(cc)));
                }
            }
        }
        if constexpr (SD) {
            if (hdr.y & 2) cfirst = (bf.y & STEP_NEED_LEFT) ? bf.x : -1;  // (a column)
#pragma unroll
            for (int e = 0; e < 8; ++e) a[e] = static_cast<AT>(vs[ix[e]]);
        }
        if constexpr (SC) {
#pragma unroll
            for (int e = 0; e < 8; ++e) c[e] *= va[e];
        }
        if constexpr (SD && sizeof(AT) == 4) {  // (FP64 multiplies in the prefix)
#pragma unroll
            for (int e = 0; e < 8; ++e) a[e] = mul_rn(va[e], a[e]);
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
#pragma unroll
            for (int e = 0; e < 8; ++e) atomicAdd(acc + ix[e], c[e]);
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
                        static_cast<AT2 *>(p.rec_left)[proc0 + (hdr.y >> 2)] = make_pair2(v, AT(0));
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
                            static_cast<AT2 *>(p.rec_left)[proc0 + (hdr.y >> 2)] = make_pair2(v, AT(0));
                        else
                            static_cast<XT *>(p.u)[last] = static_cast<XT>(v);
                    } else if (bf.y & STEP_NEED_RIGHT) {
                        static_cast<AT2 *>(p.rec_right)[proc0 + (hdr.y >> 2)] = make_pair2(chi, clo);
                    }
                }
                chi = AT(0);
                clo = AT(0);
            }
        }
    }

    if constexpr (SC) {
        __syncthreads();
        AT *part = static_cast<AT *>(p.part) + (size_t)blockIdx.x * p.n_minor;
        const AT *acc0 = reinterpret_cast<const AT *>(smem);
        if (p.copies == 1) {
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

template <typename VT, typename XT, bool SC, bool SD>
cudaError_t launch_pass_one(const PassParams &p, int grid, int warps, int smem, cudaStream_t s) {
    constexpr int WB = pass_warps(sizeof(VT));
    auto kern = pass_kernel<VT, XT, SC, SD, WB>;
    static SmemLimit lim;
    const cudaError_t e = ensure_smem_limit(kern, lim, smem);
    if (e != cudaSuccess) return e;
    kern<<<grid, warps * 32, smem, s>>>(p);
    return cudaGetLastError();
}

template <typename VT, typename XT>
cudaError_t launch_pass(bool sc, bool sd, const PassParams &p, int grid, int warps, int smem, cudaStream_t s) {
    if (sc && sd) return launch_pass_one<VT, XT, true, true>(p, grid, warps, smem, s);
    if (sc) return launch_pass_one<VT, XT, true, false>(p, grid, warps, smem, s);
    return launch_pass_one<VT, XT, false, true>(p, grid, warps, smem, s);
}

}  // namespace gbk
