// The sum of one overlap zone (Sec. IV-A step 2) from the carry records of its chunks.
#pragma once

#include <stdint.h>

#include "internal.h"

namespace gbk {

// An FP32 value widened to FP64 exactly, by integer operations on its bits only: the FP64
// pipe (slow on this part) is left to the additions.  Normal numbers move the sign, the
// exponent (rebiased from 127 to 1023) and the mantissa; a subnormal m 2^-149 is normalised
// at its leading one bit h (exponent h - 149); zeros keep their sign; infinities and NaNs
// take the all-ones exponent with the mantissa bits (a NaN stays a NaN).
__device__ __forceinline__ double widen(float f) {
    const uint32_t u = __float_as_uint(f);
    const uint32_t e = (u >> 23) & 0xFFu;
    const uint32_t mant = u & 0x7FFFFFu;
    const uint64_t sign = static_cast<uint64_t>(u & 0x80000000u) << 32;
    uint64_t d;
    if (e == 0u) {
        const int h = 31 - __clz(mant | 1u);
        d = mant == 0u ? sign
                       : sign | (static_cast<uint64_t>(h + 874) << 52) |
                             (static_cast<uint64_t>(mant ^ (1u << h)) << (52 - h));
    } else {
        const uint64_t ed = e == 0xFFu ? 0x7FFull : static_cast<uint64_t>(e + 896u);
        d = sign | (ed << 52) | (static_cast<uint64_t>(mant) << 29);
    }
    return __longlong_as_double(static_cast<long long>(d));
}
__device__ __forceinline__ double widen(double f) { return f; }

// Zone S_k = [first, last]: u_{j_k} = right record of the first chunk + the records of the middle
// chunks (whole-chunk sums, kept as right records) + left record of the last, in FP64 (the hi and
// the lo parts of the (hi, lo) records in two FP64 sums, added at the end; for FP32 records both
// widen exactly).  Called by whole warps, every lane with a zone of its own (or none: valid
// false); returns the lane's sum.  A lane adds the records of a short zone in order; a zone of
// more than ZONE_LANE records is shared by eight lanes (lane l takes records l, l + 8, .., and the
// lanes' sums are added by a butterfly): the chain of loads and FP64 additions of one lane, 75
// records for the longest columns of a 40M-nonzero matrix, had set the time of the whole fix-up
// (20 us).  Either way the order is fixed by the zone alone.
constexpr int ZONE_LANE = 4;
template <typename RT>
__device__ __forceinline__ double zone_sum(bool valid, const ZoneDev &zd, const RT *rec_left, const RT *rec_right) {
    const int lane = threadIdx.x & 31;
    const int n = valid ? zd.last - zd.first + 1 : 0;
    double sum = 0.0;
    if (n > 0 && n <= ZONE_LANE) {
        RT m[ZONE_LANE];
#pragma unroll
        for (int e = 0; e < ZONE_LANE; ++e)
            if (e < n) m[e] = (e == n - 1 ? rec_left : rec_right)[zd.first + e];
        double sh = widen(m[0].x), sl = widen(m[0].y);
#pragma unroll
        for (int e = 1; e < ZONE_LANE; ++e)
            if (e < n) {
                sh += widen(m[e].x);
                sl += widen(m[e].y);
            }
        sum = sh + sl;
    }
    unsigned todo = __ballot_sync(0xffffffffu, n > ZONE_LANE);
    while (todo) {  // four long zones at a time, eight lanes to each
        unsigned left = todo;
        int src = -1;
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            if (g == lane >> 3 && left) src = __ffs(left) - 1;
            left &= left - 1u;
        }
        todo = left;
        const int first = __shfl_sync(0xffffffffu, zd.first, src & 31), last = __shfl_sync(0xffffffffu, zd.last, src & 31);
        double sh = 0.0, sl = 0.0;
        if (src >= 0) {
            constexpr int ZB = 4;  // loads of 32 records together
            for (int q = first + (lane & 7); q <= last; q += 8 * ZB) {
                RT m[ZB];
#pragma unroll
                for (int j = 0; j < ZB; ++j)
                    if (q + 8 * j <= last) m[j] = (q + 8 * j == last ? rec_left : rec_right)[q + 8 * j];
#pragma unroll
                for (int j = 0; j < ZB; ++j)
                    if (q + 8 * j <= last) {
                        sh += widen(m[j].x);
                        sl += widen(m[j].y);
                    }
            }
        }
#pragma unroll
        for (int d = 4; d >= 1; d >>= 1) {
            sh += __shfl_xor_sync(0xffffffffu, sh, d);
            sl += __shfl_xor_sync(0xffffffffu, sl, d);
        }
        const double t = sh + sl;
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            const int to = __shfl_sync(0xffffffffu, src, 8 * g);
            const double v = __shfl_sync(0xffffffffu, t, 8 * g);
            if (lane == to) sum = v;
        }
    }
    return sum;
}

}  // namespace gbk
