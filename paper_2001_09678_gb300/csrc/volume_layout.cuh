// volume_layout.cuh -- byte order of the wide volumes (see agg_wide.cu), shared by the cost
// kernel that writes them, winner-take-all and the stage dump.
#pragma once
#include "mpv_internal.cuh"

namespace mpv {

// Byte of label k in a pixel's wide volume: lane k / (4 nq) of the path owns 4 nq consecutive
// labels, packed two per register as (w, w + 2 nq).
__host__ __device__ __forceinline__ int wide_byte(int k, int nq)
{
    const int l = k / (4 * nq), i = k - l * 4 * nq;
    return l * 4 * nq + (i < 2 * nq ? 2 * i : 2 * (i - 2 * nq) + 1);
}

}  // namespace mpv
