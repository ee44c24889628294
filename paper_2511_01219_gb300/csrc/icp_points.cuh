// The sensor-frame points of a request's valid beams for the ICP refinement (icp.cu): beam i at range z_i = R_i res / 2^16
// and angle a_i = 2 pi b_i / N_s is (z_i cos a_i, z_i sin a_i), in FP64.  They are the same for every pose, and an FP64
// sine and cosine cost an SM some 150 clocks, so the top-K launch computes them once, 32 beams per CTA, beside the
// ranking.
#pragma once
#include <cuda_runtime.h>
#include <math.h>

#include "relo_internal.h"

namespace relo {

// beams 32 chunk .. 32 chunk + 31, by the first warp of a CTA
__device__ __forceinline__ void icp_points_chunk(const ReqDesc &d, int chunk) {
    const int i = 32 * chunk + (int)threadIdx.x;
    if (threadIdx.x >= 32 || i >= d.scan->n_valid) return;
    const int2 bR = d.vbR[i];
    const double z = __dmul_rn((double)bR.y, d.resd / 65536.0), a = __dmul_rn((double)bR.x, 2.0 * M_PI / (double)d.ns);
    d.icp_pts[2 * i] = __dmul_rn(z, cos(a));
    d.icp_pts[2 * i + 1] = __dmul_rn(z, sin(a));
}

}  // namespace relo
