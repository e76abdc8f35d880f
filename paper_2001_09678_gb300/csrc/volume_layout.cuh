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

// A step of a warp's scan of wide volumes is 16 nq elements of 8 bytes, lane + 32 k being the
// lane's k-th: whether there is one (with an odd nq the last 16 lanes have one fewer).
__host__ __device__ __forceinline__ bool wide_elem(int nq, int lane, int k)
{
    return lane + 32 * k < 16 * nq;
}

// Byte of label k in a 48-label pixel with byte sums: 4 lanes of 12 labels, the lanes' first 8
// labels, then their last 4.
__host__ __device__ __forceinline__ int bytes48_of(int k)
{
    const int l = k / 12, i = k - l * 12;
    return i < 8 ? l * 8 + i : 32 + l * 4 + (i - 8);
}
__host__ __device__ __forceinline__ int bytes48_label(int b)
{
    return b < 32 ? (b >> 3) * 12 + (b & 7) : ((b - 32) >> 2) * 12 + 8 + (b & 3);
}

}  // namespace mpv
