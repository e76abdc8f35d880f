// cost.cu -- integer SSIM matching-cost volume (Section 3.2, Eq. components, Eq. ssim).
//
// For pixel (x,y) of I0 and disparity u the cost compares the N x N patch of I0
// centred at (x,y) with the patch of I1 centred at (x-u,y), coordinates clamped to the
// image.  With alpha = beta = gamma = 1 and C3 = C2/2, SSIM = A1*A2 / (B1*B2) where, for
// the patch sums Sx, Sy, Sxx, Syy, Sxy and n = N*N,
//     A1 = 2 Sx Sy + c1,              B1 = Sx^2 + Sy^2 + c1,
//     A2 = 2 (n Sxy - Sx Sy) + c2,    B2 = n (Sxx + Syy) - Sx^2 - Sy^2 + c2,
// (c1, c2 = C1, C2 scaled by n^2 and rounded) and the cost is
//     floor(255 (B1 B2 - A1 A2) / (2 B1 B2))  in [0, 255];  255 when x - u < 0.
//
// GPU design ("fast SSIM", Fig. fast_ssim, read as running box sums).  One block per row
// segment and view:
//  * the block stages, in shared memory, every image column its pixels can reach as the
//    N patch-row bytes packed in a 64-bit word, with the patch statistics of the centre whose
//    window that column completes (one 16-byte load per node of I1, 24 broadcast bytes of I0);
//  * each lane owns one label of the window ring and slides along the row: the cross sum Sxy
//    of pixel x follows from pixel x-1 by adding the entering column product (two dp4a) and
//    subtracting the leaving one, kept in a register ring of the last N products;
//  * the quotient is estimated in fp32 from exact float sums and made exact with an int64
//    check only when the estimate lies within 1.2e-4 of an integer (see cost_body.cuh).
// Bound: issue slots (84 % active at full range, 40 warp instructions per 32 nodes; about 65
// with windows, of which staging is a quarter and moved windows another) and shared-memory
// wavefronts (8 per 32 nodes).  Measured on a GB300, both views, per frame: 1280x720, D = 128,
// three scales 233 -> 175 us; 1920x1080, D = 192 860 -> 484 us (48 labels in 1.5 instead of 2
// passes over the pixels); 1280x720, 128 labels at full range 522 -> 291 us.  Segments of 160,
// 320, 480 and 640 pixels took 191, 175, 182 and 178 us; 4, 5 and 6 blocks per SM 180, 175
// and 176 us.
#include "cost_body.cuh"

namespace mpv {

namespace {

constexpr int kCostBlocks = 1216;     // about 8 per SM: two rounds of resident blocks

template <int N, int ST, int ORD>
__global__ void __launch_bounds__(kCostThreads, 5) cost_kernel(LevelArgs a, int uspan_max, int seg)
{
    if (a.gate && *a.gate == 0) return;
    extern __shared__ __align__(16) unsigned char smem[];
    cost_body<N, ST, ORD>(a, uspan_max, seg, blockIdx.x, blockIdx.y, blockIdx.z, threadIdx.x, smem);
}

template <int N, int ST, int ORD = 0>
void launch_cost_n(const LevelArgs &a, cudaStream_t s)
{
    // widest disparity span of a segment: window starts lie in [0, D - Dw]
    const int uspan_max = a.D - 1;
    const CostSmem L = cost_smem_layout(a.N / 2, uspan_max);
    // the widest segments of which the launch still has kCostBlocks blocks: wide ones stage
    // fewer columns per pixel, but a small level needs its blocks spread over the GPU
    const int u = cost_seg_unit(N);
    int seg = cost_seg(a.W, N, cost_seg_max(N));
    while (seg > u && (int64_t)((a.W + seg - 1) / seg) * a.H * a.nviews < kCostBlocks)
        seg = cost_seg(a.W, N, seg - u);
    dim3 grid((a.W + seg - 1) / seg, a.H, a.nviews);
    cudaFuncSetAttribute(cost_kernel<N, ST, ORD>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)L.bytes);
    cost_kernel<N, ST, ORD><<<grid, kCostThreads, L.bytes, s>>>(a, uspan_max, seg);
}

template <int N>
void launch_cost_st(const LevelArgs &a, cudaStream_t s)
{
    if (a.wide_nq) {
        launch_cost_n<N, 0, 1>(a, s);
        return;
    }
    switch (a.Dws) {   // the common strides as constants (store addresses, window wrap)
    case 16: launch_cost_n<N, 16>(a, s); return;
    case 32: launch_cost_n<N, 32>(a, s); return;
    case 48:
        if (a.bytes) launch_cost_n<N, 48, 2>(a, s);
        else launch_cost_n<N, 48>(a, s);
        return;
    default: launch_cost_n<N, 0>(a, s); return;
    }
}

}  // namespace

void launch_cost(const LevelArgs &a, cudaStream_t s)
{
    if (a.N == 5) launch_cost_st<5>(a, s);
    else launch_cost_st<3>(a, s);
}

}  // namespace mpv
