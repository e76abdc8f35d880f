// pyramid.cu -- image pyramid, window seeding, winner-take-all and left-right check.
//
// Section 3.4 of the paper: the pair is down-sampled by 2 per level; only the top
// level searches the full range; each finer level searches a per-pixel window whose
// centre comes from the coarser level's disparities, doubled (the sampling rate), as a
// block mode at intermediate levels and by linear interpolation at the finest level.
#include "pyramid_body.cuh"
#include "volume_layout.cuh"

namespace mpv {

namespace {

__global__ void mirror_kernel(const int *gate, ImageJob j0, ImageJob j1, int W, int H)
{
    if (gate && *gate == 0) return;
    mirror_body(blockIdx.z == 0 ? j0 : j1, W, H, blockIdx.x * blockDim.x + threadIdx.x, blockIdx.y);
}

struct Jobs4 {
    ImageJob j[4];
};

struct PyrJobs4 {
    PyrJob j[4];
};

__global__ void down2_kernel(Jobs4 jobs, int W, int H, const int *gate)
{
    if (gate && *gate == 0) return;
    down2_body(jobs.j[blockIdx.z], W, H, blockIdx.x * blockDim.x + threadIdx.x, blockIdx.y);
}

__global__ void __launch_bounds__(2 * kPyrCols) pyramid2_kernel(PyrJobs4 jobs, int W, int H,
                                                                 const int *gate)
{
    if (gate && *gate == 0) return;
    __shared__ uint8_t t1[2][kPyrCols];
    pyramid2_body(jobs.j[blockIdx.z], W, H, blockIdx.x, blockIdx.y, threadIdx.x, t1);
}

// One block per row (blockIdx.x) and view (blockIdx.y); the threads stride over the row.
__global__ void __launch_bounds__(256) seed_kernel(SeedArgs a)
{
    if (a.gate && *a.gate == 0) return;
#pragma unroll 4
    for (int x = threadIdx.x; x < a.W; x += blockDim.x) seed_body(a, x, blockIdx.x, blockIdx.y);
}

// Four window starts from centres c at p (the row ends after n more); 8 bytes where rows are whole
// groups of four.
__device__ __forceinline__ void seed_store4(const SeedArgs &a, uint16_t *p, int n, const int (&c)[4])
{
    uint32_t lo[4];
#pragma unroll
    for (int x = 0; x < 4; ++x) lo[x] = (uint32_t)min(max(c[x] - (a.Dw >> 1), 0), a.D - a.Dw);
    if ((a.W & 3) == 0) {
        *(uint2 *)p = make_uint2(lo[0] | (lo[1] << 16), lo[2] | (lo[3] << 16));
    } else {
#pragma unroll
        for (int x = 0; x < 4; ++x)
            if (x < n) p[x] = (uint16_t)lo[x];
    }
}

// The two rules of the default pyramid, a thread per 4 window starts of 4 (blocks of 2 x 2 coarse
// pixels) or 2 rows (no blocks), which share its loads and comparisons: both launches of a
// 1280x720 frame 25 -> 14 us against one thread per window start, bound by its
// instructions (now by the launches).
__global__ void __launch_bounds__(128) seed2_kernel(SeedArgs a)
{
    if (a.gate && *a.gate == 0) return;
    const int bx = blockIdx.x * 128 + threadIdx.x, by = blockIdx.y, view = blockIdx.z;
    if (2 * bx >= a.Wp || !MPV_IN(a.err, 2 * by < a.Hp, 11)) return;
    const int best = 2 * seed_mode2(a.dprev[view], a.Wp, a.Hp, 2 * bx, 2 * by);
    const int c[4] = {best, best, best, best};
    uint16_t *p = a.lo[view] + (int64_t)4 * by * a.W + 4 * bx;
#pragma unroll
    for (int r = 0; r < 4; ++r, p += a.W)
        if (4 * by + r < a.H) seed_store4(a, p, a.W - 4 * bx, c);
}

// (seed_body's means of doubled neighbours: of 2, their sum; of 4, half their sum, rounded up)
__global__ void __launch_bounds__(128) seed1_kernel(SeedArgs a)
{
    if (a.gate && *a.gate == 0) return;
    const int bx = blockIdx.x * 128 + threadIdx.x, cy = blockIdx.y, view = blockIdx.z;
    if (2 * bx >= a.Wp || !MPV_IN(a.err, cy < a.Hp, 11)) return;
    const uint16_t *r0 = a.dprev[view] + (int64_t)cy * a.Wp;
    const uint16_t *r1 = a.dprev[view] + (int64_t)min(cy + 1, a.Hp - 1) * a.Wp;
    const int x1 = min(2 * bx + 1, a.Wp - 1), x2 = min(2 * bx + 2, a.Wp - 1);
    const int p0 = r0[2 * bx], p1 = r0[x1], p2 = r0[x2];
    const int q0 = r1[2 * bx], q1 = r1[x1], q2 = r1[x2];
    uint16_t *p = a.lo[view] + (int64_t)2 * cy * a.W + 4 * bx;
    const int even[4] = {2 * p0, p0 + p1, 2 * p1, p1 + p2};
    seed_store4(a, p, a.W - 4 * bx, even);
    if (2 * cy + 1 >= a.H) return;
    const int odd[4] = {p0 + q0, (p0 + p1 + q0 + q1 + 1) >> 1, p1 + q1, (p1 + p2 + q1 + q2 + 1) >> 1};
    seed_store4(a, p + a.W, a.W - 4 * bx, odd);
}

template <int LPP>
__global__ void wta_kernel(LevelArgs a)
{
    if (a.gate && *a.gate == 0) return;
    wta_body<LPP>(a, (int64_t)blockIdx.x * blockDim.x + threadIdx.x, blockIdx.z);
}

// Winner-take-all on wide volumes (agg_wide.cu): S = npaths C + E, ties to the smallest
// disparity.  Four threads per pixel, each with the G NQ consecutive bytes of G / 4 lanes.
// Bound by DRAM (1280x720, 128 labels, both views: 472 MB in 90 us).
template <int G, int NQ>
__global__ void __launch_bounds__(256) wide_wta_kernel(LevelArgs a)
{
    if (a.gate && *a.gate == 0) return;
    constexpr int R = 4 * G * NQ, TPP = 4, NW = G * NQ / 4;   // words per thread
    const ViewLevel &v = a.v[blockIdx.z];
    const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t i = g / TPP;
    const int sub = (int)(g % TPP);
    uint32_t best = 0xFFFFFFFFu;
    const bool in = i < (int64_t)a.W * a.H;
    if (in) {
        const uint8_t *pc = v.C + i * R + sub * (4 * NW), *pe = v.E + i * R + sub * (4 * NW);
        uint32_t qc[NW], qe[NW];
        if (NW % 4 == 0) {
#pragma unroll
            for (int k = 0; k < NW / 4; ++k) {
                const uint4 x = ((const uint4 *)pc)[k], y = ((const uint4 *)pe)[k];
                qc[4 * k] = x.x, qc[(4 * k + 1) % NW] = x.y;
                qc[(4 * k + 2) % NW] = x.z, qc[(4 * k + 3) % NW] = x.w;
                qe[4 * k] = y.x, qe[(4 * k + 1) % NW] = y.y;
                qe[(4 * k + 2) % NW] = y.z, qe[(4 * k + 3) % NW] = y.w;
            }
        } else if (NW % 2 == 0) {
#pragma unroll
            for (int k = 0; k < NW / 2; ++k) {
                const uint2 x = ((const uint2 *)pc)[k], y = ((const uint2 *)pe)[k];
                qc[2 * k] = x.x, qc[(2 * k + 1) % NW] = x.y;
                qe[2 * k] = y.x, qe[(2 * k + 1) % NW] = y.y;
            }
        } else {
#pragma unroll
            for (int k = 0; k < NW; ++k) {
                qc[k] = ((const uint32_t *)pc)[k];
                qe[k] = ((const uint32_t *)pe)[k];
            }
        }
        const uint32_t np = (uint32_t)a.npaths << 16;
#pragma unroll
        for (int k = 0; k < NW; ++k)
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const uint32_t c = (qc[k] >> (8 * b)) & 0xFFu, e = (qe[k] >> (8 * b)) & 0xFFu;
                const int ln = (4 * k + b) / (4 * NQ), j = 4 * k + b - ln * 4 * NQ;
                const int u = sub * (4 * NW) + ln * 4 * NQ + (j >> 1) + (j & 1) * 2 * NQ;
                const uint32_t key = c * np + ((e << 16) | (uint32_t)u);
                if (u < a.Dw) best = min(best, key);
            }
    }
#pragma unroll
    for (int o = 1; o < TPP; o <<= 1) best = min(best, __shfl_xor_sync(0xFFFFFFFFu, best, o));
    if (in && sub == 0) v.d[i] = (uint16_t)(best & 0xFFFFu);
}

template <int NQ>
void launch_wide_wta(const LevelArgs &a, cudaStream_t s)
{
    const int64_t nthreads = 4 * (int64_t)a.W * a.H;
    const dim3 grid((unsigned)((nthreads + 255) / 256), 1, a.nviews);
    if (a.wide_g == 4) wide_wta_kernel<4, NQ><<<grid, 256, 0, s>>>(a);
    else wide_wta_kernel<8, NQ><<<grid, 256, 0, s>>>(a);
}

// Winner-take-all on byte sums: S = npaths C + E, ties to the smallest disparity.  TPP threads
// per pixel, each with the same DWS / TPP bytes of C and of E.  A chunk of 16 labels is compared
// in pairs of 16-bit keys, 16 S + position (S <= 8 * 255 + 255).  Bound by DRAM and L2
// (1280x720, 32 labels, both views, 118 MB: 22 us; with a 32-bit key per label 29 us, 16-bit sums
// 41 us).
template <int DWS, int TPP>
__global__ void __launch_bounds__(256) bytes_wta_kernel(LevelArgs a)
{
    if (a.gate && *a.gate == 0) return;
    constexpr int NV = DWS / TPP / 16;        // 16-byte loads per thread and volume
    const ViewLevel &v = a.v[blockIdx.z];
    const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t i = g / TPP;
    const int sub = (int)(g % TPP);
    uint32_t best = 0xFFFFFFFFu;
    const bool in = i < (int64_t)a.W * a.H;
    int lo = 0;
    if (in) {
        const uint4 *pc = (const uint4 *)(v.C + i * DWS) + sub * NV;
        const uint4 *pe = (const uint4 *)(v.E + i * DWS) + sub * NV;
        uint4 qc[NV], qe[NV];
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            qc[k] = pc[k];
            qe[k] = pe[k];
        }
        lo = v.lo ? (int)v.lo[i] : 0;
        const uint32_t np = 16u * (uint32_t)a.npaths;
        const bool padded = a.Dw < DWS;
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            const uint32_t wc[4] = {qc[k].x, qc[k].y, qc[k].z, qc[k].w};
            const uint32_t we[4] = {qe[k].x, qe[k].y, qe[k].z, qe[k].w};
            // byte b's label, in ascending order of b (TPP = 1 for 48 labels)
            auto label = [&](int b) {
                return DWS == 48 ? bytes48_label(16 * k + b) : (sub * NV + k) * 16 + b;
            };
            uint32_t m = 0xFFFFFFFFu;
#pragma unroll
            for (int b = 0; b < 16; b += 2) {
                const uint32_t sel = (b & 2) ? 0x4342u : 0x4140u;
                const uint32_t c = __byte_perm(wc[b >> 2], 0u, sel);
                const uint32_t e = __byte_perm(we[b >> 2], 0u, sel);
                uint32_t key = c * np + (e * 16u + (uint32_t)(b | ((b + 1) << 16)));
                if (padded)
                    key |= (label(b) < a.Dw ? 0u : 0xFFFFu) | (label(b + 1) < a.Dw ? 0u : 0xFFFF0000u);
                m = __vminu2(m, key);
            }
            const uint32_t one = min(m & 0xFFFFu, m >> 16);
            best = min(best, ((one >> 4) << 16) | (uint32_t)label((int)(one & 15u)));
        }
    }
#pragma unroll
    for (int o = 1; o < TPP; o <<= 1) best = min(best, __shfl_xor_sync(0xFFFFFFFFu, best, o));
    if (in && sub == 0) v.d[i] = (uint16_t)(lo + (best & 0xFFFFu));
}

template <int DWS, int TPP>
void launch_bytes_wta(const LevelArgs &a, cudaStream_t s)
{
    const int64_t nthreads = TPP * (int64_t)a.W * a.H;
    bytes_wta_kernel<DWS, TPP><<<dim3((unsigned)((nthreads + 255) / 256), 1, a.nviews), 256, 0, s>>>(a);
}

// Window-edge hits of the learned proposal: pixels whose minimum sits on an edge of
// their window while the range continues beyond it (k = d - lo is 0 with lo > 0, or
// Dw - 1 with lo + Dw < D).  A fixed grid strides over the pixels and every block adds
// its two counts with one pair of atomics.
constexpr int kEdgeBlocks = 304, kEdgeThreads = 256;

__global__ void __launch_bounds__(kEdgeThreads) edge_kernel(LevelArgs a)
{
    const ViewLevel &v = a.v[blockIdx.z];
    const int64_t npx = (int64_t)a.W * a.H;
    unsigned hits = 0, px = 0;
    for (int64_t i = (int64_t)blockIdx.x * kEdgeThreads + threadIdx.x; i < npx;
         i += (int64_t)kEdgeBlocks * kEdgeThreads) {
        const int lo = v.lo ? (int)v.lo[i] : 0;
        const int k = (int)v.d[i] - lo;
        hits += (k == 0 && lo > 0) || (k == a.Dw - 1 && lo + a.Dw < a.D);
        ++px;
    }
    for (int o = 16; o > 0; o >>= 1) {
        hits += __shfl_xor_sync(0xFFFFFFFFu, hits, o);
        px += __shfl_xor_sync(0xFFFFFFFFu, px, o);
    }
    __shared__ unsigned part[2][kEdgeThreads / 32];
    if ((threadIdx.x & 31) == 0) {
        part[0][threadIdx.x >> 5] = hits;
        part[1][threadIdx.x >> 5] = px;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long h = 0, p = 0;
        for (int w = 0; w < kEdgeThreads / 32; ++w) {
            h += part[0][w];
            p += part[1][w];
        }
        if (p) {
            atomicAdd(a.edge, h);
            atomicAdd(a.edge + 1, p);
        }
    }
}

// Stage dump: C and S in the documented [H][W][Dw] layout (u16 and u32).
__global__ void unpack_kernel(LevelArgs a, int view, uint16_t *cost, uint32_t *sum)
{
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t n = (int64_t)a.W * a.H * a.Dw;
    if (e >= n) return;
    const int64_t pix = e / a.Dw;
    const int k = (int)(e - pix * a.Dw);
    const ViewLevel &v = a.v[view];
    if (a.wide_nq) {
        const int64_t j = pix * (4 * a.wide_g * a.wide_nq) + wide_byte(k, a.wide_nq);
        if (cost) cost[e] = v.C[j];
        if (sum) sum[e] = (uint32_t)a.npaths * v.C[j] + v.E[j];
        return;
    }
    if (a.bytes) {
        const int64_t j = pix * a.Dws + (a.Dws == 48 ? bytes48_of(k) : k);
        if (cost) cost[e] = v.C[j];
        if (sum) sum[e] = (uint32_t)a.npaths * v.C[j] + v.E[j];
        return;
    }
    if (cost) cost[e] = v.C[pix * a.Dws + k];
    if (sum) {
        const int64_t j = pix * a.Dws + k;
        sum[e] = v.S2 ? ((uint32_t)v.S[j] + (uint32_t)v.S2[j]) >> 1 : v.S[j];
    }
}

// Left-right check.  dRm is the right view's map in mirrored coordinates.
__global__ void lr_kernel(const uint16_t *__restrict__ dL, const uint16_t *__restrict__ dRm,
                          int W, int H, int tol, int check, uint16_t *out, int out_pitch,
                          uint16_t *out_right, int right_pitch, const int *gate)
{
    if (gate && *gate == 0) return;
    lr_body(dL, dRm, W, H, tol, check, out, out_pitch, out_right, right_pitch,
            blockIdx.x * blockDim.x + threadIdx.x, blockIdx.y);
}

}  // namespace

void launch_mirror(const ImageJob *jobs, int njobs, int W, int H, cudaStream_t s,
                   const int *gate)
{
    dim3 grid((W + 127) / 128, H, njobs);
    mirror_kernel<<<grid, 128, 0, s>>>(gate, jobs[0], njobs > 1 ? jobs[1] : jobs[0], W, H);
}

void launch_down2(const ImageJob *jobs, int njobs, int W, int H, cudaStream_t s,
                  const int *gate)
{
    Jobs4 j4;
    for (int i = 0; i < 4; ++i) j4.j[i] = jobs[i < njobs ? i : 0];
    const int W2 = (W + 1) / 2, H2 = (H + 1) / 2;
    dim3 grid((W2 + 127) / 128, H2, njobs);
    down2_kernel<<<grid, 128, 0, s>>>(j4, W, H, gate);
}

void launch_pyramid2(const PyrJob *jobs, int njobs, int W, int H, cudaStream_t s,
                     const int *gate)
{
    PyrJobs4 j4;
    for (int i = 0; i < 4; ++i) j4.j[i] = jobs[i < njobs ? i : 0];
    const int W1 = (W + 1) / 2, H1 = (H + 1) / 2;
    dim3 grid((W1 + kPyrCols - 1) / kPyrCols, (H1 + 1) / 2, njobs);
    pyramid2_kernel<<<grid, 2 * kPyrCols, 0, s>>>(j4, W, H, gate);
}

void launch_seed(const SeedArgs &a, cudaStream_t s)
{
    const int bx = ((a.Wp + 1) / 2 + 127) / 128;
    if (a.block == 2) {
        seed2_kernel<<<dim3(bx, (a.Hp + 1) / 2, a.nviews), 128, 0, s>>>(a);
        return;
    }
    if (a.block < 2) {
        seed1_kernel<<<dim3(bx, a.Hp, a.nviews), 128, 0, s>>>(a);
        return;
    }
    seed_kernel<<<dim3(a.H, a.nviews, 1), 256, 0, s>>>(a);
}

void launch_wta(const LevelArgs &a, cudaStream_t s)
{
    switch (a.wide_nq) {
    case 0: break;
    case 3: launch_wide_wta<3>(a, s); return;
    case 4: launch_wide_wta<4>(a, s); return;
    case 5: launch_wide_wta<5>(a, s); return;
    case 6: launch_wide_wta<6>(a, s); return;
    case 7: launch_wide_wta<7>(a, s); return;
    default: launch_wide_wta<8>(a, s); return;
    }
    if (a.bytes) {
        if (a.Dws == 16) launch_bytes_wta<16, 1>(a, s);
        else if (a.Dws == 32) launch_bytes_wta<32, 2>(a, s);
        else if (a.Dws == 48) launch_bytes_wta<48, 1>(a, s);
        else launch_bytes_wta<64, 4>(a, s);
        if (a.edge) edge_kernel<<<dim3(kEdgeBlocks, 1, a.nviews), kEdgeThreads, 0, s>>>(a);
        return;
    }
    const int lpp = a.Dws >= 32 ? 4 : 2;
    const int64_t nthreads = lpp * (int64_t)a.W * a.H;
    dim3 grid((unsigned)((nthreads + 255) / 256), 1, a.nviews);
    if (lpp == 4)
        wta_kernel<4><<<grid, 256, 0, s>>>(a);
    else
        wta_kernel<2><<<grid, 256, 0, s>>>(a);
    if (a.edge) edge_kernel<<<dim3(kEdgeBlocks, 1, a.nviews), kEdgeThreads, 0, s>>>(a);
}

void launch_unpack(const LevelArgs &a, int view, uint16_t *cost, uint32_t *sum, cudaStream_t s)
{
    const int64_t n = (int64_t)a.W * a.H * a.Dw;
    unpack_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(a, view, cost, sum);
}

void launch_lr(const uint16_t *dL, const uint16_t *dRm, int W, int H, int tol, int check,
               uint16_t *out, int out_pitch, uint16_t *out_right, int right_pitch,
               cudaStream_t s, const int *gate)
{
    dim3 grid((W + 127) / 128, H, 1);
    lr_kernel<<<grid, 128, 0, s>>>(dL, dRm, W, H, tol, check, out, out_pitch, out_right,
                                    right_pitch, gate);
}

namespace {

// The fallback decision of a learned-proposal frame: re-match when more than edge_bp of
// every 10000 matched pixels won on a window edge (one thread).
__global__ void fallback_gate_kernel(const unsigned long long *edge, int edge_bp,
                                     FallbackGate *gate, unsigned long long *counters,
                                     cudaGraphConditionalHandle cond, int has_cond)
{
    const unsigned long long hits = edge[0], px = edge[1];
    const int open = hits * 10000ull > (unsigned long long)edge_bp * px ? 1 : 0;
    gate->hits = hits;
    gate->px = px;
    gate->open = open;
    if (counters) {
        atomicAdd(counters, 1ull);
        if (open) atomicAdd(counters + 1, 1ull);
    }
    if (has_cond) cudaGraphSetConditional(cond, (unsigned)open);
}

}  // namespace

void launch_fallback_gate(const unsigned long long *edge, int edge_bp, FallbackGate *gate,
                          unsigned long long *counters, cudaStream_t s,
                          const cudaGraphConditionalHandle *cond)
{
    fallback_gate_kernel<<<1, 1, 0, s>>>(edge, edge_bp, gate, counters,
                                         cond ? *cond : cudaGraphConditionalHandle{}, cond != nullptr);
}

}  // namespace mpv
