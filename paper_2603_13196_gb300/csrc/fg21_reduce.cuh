// a6: per point, sum the channel-group partials in fixed order and form
// lnL = -1/2 (F T ln(2 pi sigma_n^2) + chi2 / sigma_n^2) (eq. likelihood).  The
// partials (compensated FP32 pairs) are summed in double-float arithmetic
// (Knuth's two-sum on FP32 pairs, about 48 bits) and converted once: FP64 is a
// scarce pipe on this part.
//
// Each request's rows are summed in a form fixed by the row length alone, so a
// request's logL does not depend on what it is batched with:
//  - rows of at most REDUCE_SERIAL_MAX partials (the usual case): one thread per
//    point sums its row in ascending order (double-float);
//  - longer rows (one channel per group at small P): one warp per point, lane l
//    summing partials l, l+32, ... in ascending order, the lanes' sums combined
//    in a fixed butterfly.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "fg21_internal.h"

namespace fg21 {

constexpr int REDUCE_SERIAL_MAX = 32;       // longest partial row summed by one thread

// (sh, sl) += (xh, xl) in double-float arithmetic: Knuth's two-sum of the high
// parts, the low parts added to its error, then renormalised.
__device__ __forceinline__ void df_add(float &sh, float &sl, float xh, float xl) {
    const float s = sh + xh;
    const float bb = s - sh;
    const float err = ((sh - (s - bb)) + (xh - bb)) + (sl + xl);
    sh = s + err;
    sl = err - (sh - s);
}
__device__ __forceinline__ void two_sum_acc(float &s, float &c, float x) {
    const float t = s + x;
    const float z = t - s;
    c += (s - (t - z)) + (x - z);
    s = t;
}

// The logL of point p of request r: by one thread (WARP false, `lane` 0), or by
// a whole warp.  The partials were written by other SMs of the same grid or by
// an earlier kernel: they are read from L2.
template <bool WARP>
__device__ __forceinline__ void reduce_point(const ReqDesc &r, int64_t p, int lane) {
    if (!r.pvalid[p]) {      // prep tested the point (point_valid)
        if (lane == 0) {
            r.logL[p] = -INFINITY;
            atomicAdd(r.invalid, 1ull);
        }
        return;
    }
    float sh = 0.0f, sl = 0.0f;
    const float2 *__restrict__ part = r.partials + (size_t)p * r.n_part;
    if (WARP) {
        for (int g = lane; g < r.n_part; g += 32) {
            const float2 v = __ldcg(part + g);
            two_sum_acc(sh, sl, v.x);
            two_sum_acc(sh, sl, v.y);
        }
        for (int o = 16; o > 0; o >>= 1) {
            const float oh = __shfl_xor_sync(0xffffffffu, sh, o), ol = __shfl_xor_sync(0xffffffffu, sl, o);
            df_add(sh, sl, oh, ol);
        }
        if (lane != 0) return;
    } else {
#pragma unroll 4
        for (int g = 0; g < r.n_part; ++g) {
            const float2 v = __ldcg(part + g);
            two_sum_acc(sh, sl, v.x);
            two_sum_acc(sh, sl, v.y);
        }
    }
    const double chi2 = ((double)sh + (double)sl) * r.chi2_scale;
    if (r.pnorm) {           // sigma_n terms from prep (tensor path)
        const double2 nm = r.pnorm[p];
        r.logL[p] = -0.5 * (nm.x + chi2 * nm.y);
    } else {
        const double sig = r.params[p * (r.NPF + 4) + r.NPF + 3];
        const double n = (double)r.F * (double)r.T;
        r.logL[p] = -0.5 * (n * log(2.0 * 3.141592653589793 * sig * sig) + chi2 / (sig * sig));
    }
}

// Tensor path: the count of a tile's finished work items, in a spare row of its
// point operands (prep zeroes it).
__device__ __forceinline__ int *tile_count(const ReqDesc &r, int tile) {
    return reinterpret_cast<int *>(r.pts32 + ((size_t)tile * r.pts_rows + r.Kp + 1) * TILE_M);
}

}  // namespace fg21
