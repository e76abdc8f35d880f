// cnn.cu -- the learned disparity-window proposal: a small 3x3 CNN and its training
// kernels (forward, backward, loss, optimizer), plus its input features and its output
// windows.  BF16 activations and weights, FP32 accumulation and FP32 gradients.
//
// Network (trained by paper_2001_09678_gb300/learn.py): six 3x3 convolutions with zero
// padding, 2 + D_top input channels (the top pyramid level's left and right images and
// its full-range cost slice), 32 hidden channels with ReLU, 1 output channel: the
// disparity at full resolution divided by D, at the top level's resolution.
#include <algorithm>
#include <cuda_bf16.h>

#include "mpv_internal.cuh"

namespace mpv {

namespace {

constexpr int kTile = 16;          // output tile side of the convolution kernels

// out[n][co][y][x] = b[co] + sum_{ci,ky,kx} w[co][ci][ky][kx] in[n][ci][y+ky-1][x+kx-1]
// (zero padding), optional ReLU, on the CUDA cores; one thread per output pixel and all output
// channels: one channel (FP32 input, or more BF16 channels than the tensor-core kernel stages), or
// 32 of at most kPixelCin FP32 channels.
__device__ __forceinline__ float ld_act(const __nv_bfloat16 *p, int64_t i) { return __bfloat162float(p[i]); }
__device__ __forceinline__ float ld_act(const float *p, int64_t i) { return p[i]; }

template <int COUT, class TIn>
__global__ void __launch_bounds__(kTile *kTile) conv3x3_pixel_kernel(
    const TIn *__restrict__ in, int Cin, int H, int W,
    const __nv_bfloat16 *__restrict__ w, const float *__restrict__ b, int relu,
    __nv_bfloat16 *__restrict__ out_bf, float *__restrict__ out_f)
{
    extern __shared__ float smem[];
    float *ws = smem;                                   // [Cin*9][COUT]
    float *tile = smem + Cin * 9 * COUT;                // [18][18] of one input channel
    const int n = blockIdx.z;
    const int tx = threadIdx.x % kTile, ty = threadIdx.x / kTile;
    const int x0 = blockIdx.x * kTile, y0 = blockIdx.y * kTile;
    const int x = x0 + tx, y = y0 + ty;
    for (int i = threadIdx.x; i < Cin * 9 * COUT; i += kTile * kTile) {
        const int co = i % COUT, r = i / COUT;         // r = ci*9 + k
        ws[i] = __bfloat162float(w[(int64_t)co * Cin * 9 + r]);
    }
    float acc[COUT];
#pragma unroll
    for (int co = 0; co < COUT; ++co) acc[co] = b ? b[co] : 0.f;
    const int64_t plane = (int64_t)H * W;
    const TIn *src = in + (int64_t)n * Cin * plane;
    for (int ci = 0; ci < Cin; ++ci) {
        __syncthreads();
        for (int i = threadIdx.x; i < 18 * 18; i += kTile * kTile) {
            const int yy = y0 - 1 + i / 18, xx = x0 - 1 + i % 18;
            tile[i] = (yy >= 0 && yy < H && xx >= 0 && xx < W)
                          ? ld_act(src, ci * plane + (int64_t)yy * W + xx)
                          : 0.f;
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            const float v = tile[(ty + k / 3) * 18 + tx + k % 3];
            const float *wr = ws + (ci * 9 + k) * COUT;
#pragma unroll
            for (int co = 0; co < COUT; ++co) acc[co] = fmaf(wr[co], v, acc[co]);
        }
    }
    if (x >= W || y >= H) return;
    const int64_t o = (int64_t)n * COUT * plane + (int64_t)y * W + x;
#pragma unroll
    for (int co = 0; co < COUT; ++co) {
        float v = acc[co];
        if (relu) v = fmaxf(v, 0.f);
        if (out_f) out_f[o + co * plane] = v;
        if (out_bf) out_bf[o + co * plane] = __float2bfloat16(v);
    }
}

// Up to this many FP32 channels conv3x3_pixel_kernel makes 32 channels: the other kernel's chunks
// of 16 staged channels are mostly empty (8 samples of 320 x 180: one channel, the last layer's
// backward pass, 19 us against 27; two 29 against 31; three 38 against 37).
constexpr int kPixelCin = 2;

// Two FP32 multiply-adds in one instruction (each rounded as fmaf), on register pairs.
__device__ __forceinline__ unsigned long long pair(float lo, float hi)
{
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpair(unsigned long long v, float &lo, float &hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ void fma2(unsigned long long &acc, unsigned long long a,
                                     unsigned long long b)
{
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}

// The same for 32 output channels of more FP32 channels (the backward-data pass): 4 pixels of a
// row x 8 channels per thread, a 16 x 16 tile per block, the input tile and the weights of
// kConvChunk channels at a time in shared memory.  A (channel, ky) takes 8 shared loads for 96
// multiply-adds, every operand of a warp in one or two 128-byte rows; the sums run in the same
// order as in conv3x3_pixel_kernel (channel, ky, kx), bit for bit the same.  Bound: the FP32
// pipe (8 samples of 320 x 180, 32 -> 32 channels, 8.5 GFLOP: 295 -> 183 us against one pixel and
// 32 channels per thread and one channel per barrier).
constexpr int kConvChunk = 16, kConvRow = 20;       // channels per chunk; staged row (18 used)
constexpr int kConvW = 36;                          // staged weights of one (channel, tap), 32 used

__global__ void __launch_bounds__(256) conv3x3_f32_kernel(
    const float *__restrict__ in, int Cin, int H, int W, const __nv_bfloat16 *__restrict__ w,
    const float *__restrict__ b, int relu, __nv_bfloat16 *__restrict__ out_bf,
    float *__restrict__ out_f)
{
    __shared__ __align__(16) float tile[kConvChunk * 18 * kConvRow];
    __shared__ __align__(16) float ws[kConvChunk * 9 * kConvW];
    const int n = blockIdx.z;
    // a warp: one group of 8 channels (its weights are one address), 8 rows x 4 groups of pixels
    // (8 lanes' rows, kConvRow floats apart, in different banks)
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int ty = (lane & 7) + 8 * (warp >> 2), tx = 4 * (lane >> 3), co0 = 8 * (warp & 3);
    const int x0 = blockIdx.x * kTile, y0 = blockIdx.y * kTile;
    const int64_t plane = (int64_t)H * W;
    const float *src = in + (int64_t)n * Cin * plane;
    unsigned long long acc[4][4];             // channel pairs x pixels
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int p = 0; p < 4; ++p)
            acc[c][p] = b ? pair(b[co0 + 2 * c], b[co0 + 2 * c + 1]) : pair(0.f, 0.f);
    for (int c0 = 0; c0 < Cin; c0 += kConvChunk) {
        const int nc = min(kConvChunk, Cin - c0);
        __syncthreads();
        // a thread keeps its pixels and walks over the channels
        for (int i = threadIdx.x; i < 18 * 18; i += 256) {
            const int py = i / 18, px = i - py * 18, yy = y0 - 1 + py, xx = x0 - 1 + px;
            const bool in_map = yy >= 0 && yy < H && xx >= 0 && xx < W;
            const float *p = src + (c0 * plane + (int64_t)yy * W + xx);
            float v[kConvChunk];
#pragma unroll
            for (int c = 0; c < kConvChunk; ++c) v[c] = in_map && c < nc ? p[c * plane] : 0.f;
#pragma unroll
            for (int c = 0; c < kConvChunk; ++c) tile[(c * 18 + py) * kConvRow + px] = v[c];
        }
        {
            const int co = threadIdx.x >> 3;
            const __nv_bfloat16 *p = w + (int64_t)co * Cin * 9 + c0 * 9;
#pragma unroll 9
            for (int r = threadIdx.x & 7; r < nc * 9; r += 8)               // r = ci * 9 + k
                ws[r * kConvW + co] = __bfloat162float(p[r]);
        }
        __syncthreads();
        for (int ci = 0; ci < nc; ++ci)
#pragma unroll
            for (int ky = 0; ky < 3; ++ky) {
                const float *t = tile + (ci * 18 + ty + ky) * kConvRow + tx;
                const float4 a = *(const float4 *)t;
                const float2 e = *(const float2 *)(t + 4);
                const unsigned long long v[6] = {pair(a.x, a.x), pair(a.y, a.y), pair(a.z, a.z),
                                                 pair(a.w, a.w), pair(e.x, e.x), pair(e.y, e.y)};
#pragma unroll
                for (int kx = 0; kx < 3; ++kx) {
                    const ulonglong2 *wr =
                        (const ulonglong2 *)(ws + (ci * 9 + ky * 3 + kx) * kConvW + co0);
                    const ulonglong2 w0 = wr[0], w1 = wr[1];
                    const unsigned long long wv[4] = {w0.x, w0.y, w1.x, w1.y};
#pragma unroll
                    for (int c = 0; c < 4; ++c)
#pragma unroll
                        for (int p = 0; p < 4; ++p) fma2(acc[c][p], wv[c], v[p + kx]);
                }
            }
    }
    const int y = y0 + ty;
    if (y >= H) return;
    const bool vec = x0 + tx + 3 < W && W % 4 == 0 && ((uintptr_t)out_f & 15) == 0;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const int64_t o = ((int64_t)n * 32 + co0 + c) * plane + (int64_t)y * W + x0 + tx;
        float v[4];
#pragma unroll
        for (int p = 0; p < 4; ++p) {
            float lo, hi;
            unpair(acc[c >> 1][p], lo, hi);
            v[p] = (c & 1) ? hi : lo;
            if (relu) v[p] = fmaxf(v[p], 0.f);
        }
        if (out_f && vec) *(float4 *)(out_f + o) = make_float4(v[0], v[1], v[2], v[3]);
#pragma unroll
        for (int p = 0; p < 4; ++p) {
            if (x0 + tx + p >= W) break;
            if (out_f && !vec) out_f[o + p] = v[p];
            if (out_bf) out_bf[o + p] = __float2bfloat16(v[p]);
        }
    }
}

// dW[co][ci][k] += sum over a tile of g[n][co][y][x] in[n][ci][y+ky-1][x+kx-1]; db[co] += sum g.
// Any channel counts; one block per (tile, sample), partial sums added atomically.
__global__ void __launch_bounds__(kTile *kTile) conv3x3_wgrad_kernel(
    const __nv_bfloat16 *__restrict__ in, int Cin, const float *__restrict__ g, int Cout,
    int H, int W, float *__restrict__ dw, float *__restrict__ db)
{
    extern __shared__ float smem[];
    float *gt = smem;                         // [Cout][16*16]
    float *it = smem + Cout * kTile * kTile;  // [Cin][18*18]
    const int n = blockIdx.z;
    const int x0 = blockIdx.x * kTile, y0 = blockIdx.y * kTile;
    const int64_t plane = (int64_t)H * W;
    for (int i = threadIdx.x; i < Cout * kTile * kTile; i += kTile * kTile) {
        const int co = i / (kTile * kTile), p = i % (kTile * kTile);
        const int yy = y0 + p / kTile, xx = x0 + p % kTile;
        gt[i] = (yy < H && xx < W) ? g[((int64_t)n * Cout + co) * plane + (int64_t)yy * W + xx]
                                   : 0.f;
    }
    for (int i = threadIdx.x; i < Cin * 18 * 18; i += kTile * kTile) {
        const int ci = i / (18 * 18), p = i % (18 * 18);
        const int yy = y0 - 1 + p / 18, xx = x0 - 1 + p % 18;
        it[i] = (yy >= 0 && yy < H && xx >= 0 && xx < W)
                    ? __bfloat162float(in[((int64_t)n * Cin + ci) * plane + (int64_t)yy * W + xx])
                    : 0.f;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < Cout * Cin * 9; e += kTile * kTile) {
        const int co = e / (Cin * 9), r = e % (Cin * 9), ci = r / 9, k = r % 9;
        const float *gp = gt + co * kTile * kTile;
        const float *ip = it + ci * 18 * 18 + (k / 3) * 18 + (k % 3);
        float s = 0.f;
        for (int py = 0; py < kTile; ++py)
#pragma unroll 4
            for (int px = 0; px < kTile; ++px) s = fmaf(gp[py * kTile + px], ip[py * 18 + px], s);
        atomicAdd(dw + e, s);
    }
    if (db)
        for (int co = threadIdx.x; co < Cout; co += kTile * kTile) {
            float s = 0.f;
            for (int p = 0; p < kTile * kTile; ++p) s += gt[co * kTile * kTile + p];
            atomicAdd(db + co, s);
        }
}

// The same for the network's layers: 32 output channels (CPT 4) or one (CPT 1), Cin <= kWgMaxCin.
// A thread owns CPT output channels x 1 input channel x 9 taps and slides along the tile's rows:
// 4 pixels take CPT + 6 16-byte shared loads for 36 CPT multiply-adds, the loads of a warp (8
// gradient groups, or 8 rows, and 4 input channels) free of bank conflicts.  CPT 1 splits the
// tile's rows among kWgSplit threads per element, added in a fixed order at the end.  Blocks
// stay resident and walk over the tiles, so that their totals meet the shared gradient once per
// block.  Bound: the FP32 pipe and the packing of its operand pairs (8 samples of 320 x 180,
// 32 -> 32 channels, 8.5 GFLOP: 1,070 -> 220 us against two shared loads per multiply-add;
// 32 -> 1: 59 us, its staging).  Staging by an element's index, with its divisions, instead of
// a thread's fixed pixels: 245 us.
constexpr int kWgMaxCin = 40, kWgSplit = 8;
constexpr int kWgGS = 36;                            // floats per staged pixel of 32 gradients
constexpr int kWgIS = 18 * kConvRow;                 // floats per input channel (8 mod 32)

template <int CPT>
__global__ void __launch_bounds__(kWgMaxCin * 8, CPT == 1 ? 3 : 2) wgrad_tile_kernel(
    const __nv_bfloat16 *__restrict__ in, int Cin, const float *__restrict__ g, int H, int W, int tx,
    int ty, int ntiles, float *__restrict__ dw, float *__restrict__ db)
{
    constexpr int Cout = CPT * 8 == 32 ? 32 : 1;
    extern __shared__ __align__(16) float smem[];
    float *gt = smem;                         // CPT 4: [256 pixels][kWgGS], 1: [256]
    float *it = smem + (CPT == 1 ? kTile * kTile : kTile * kTile * kWgGS);   // [Cin][18][kConvRow]
    const int nthr = blockDim.x, t = threadIdx.x;
    // CPT 4: (input channel, channels 4 cg ..); CPT 1: (input channel, rows)
    const int ci = t >> 3, cg = t & 7;
    const bool mine = ci < Cin;
    const int ya = CPT == 1 ? cg : 0, ystep = CPT == 1 ? kWgSplit : 1;
    const int64_t plane = (int64_t)H * W;
    // CPT 4: pairs of channels; CPT 1: (sum over the even pixels, over the odd ones)
    constexpr int NP = CPT == 1 ? 1 : CPT / 2;
    unsigned long long tot[NP][9];
#pragma unroll
    for (int j = 0; j < NP; ++j)
#pragma unroll
        for (int k = 0; k < 9; ++k) tot[j][k] = pair(0.f, 0.f);

    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int n = tile / (tx * ty), r = tile - n * (tx * ty);
        const int y0 = (r / tx) * kTile, x0 = (r % tx) * kTile;
        __syncthreads();
        // a thread keeps its pixels and walks over the channels
        for (int i = t; i < kTile * kTile; i += nthr) {
            const int yy = y0 + i / kTile, xx = x0 + i % kTile;
            const bool in_map = yy < H && xx < W;
            const float *p = g + ((int64_t)n * Cout * plane + (int64_t)yy * W + xx);
            if (CPT == 1) {
                gt[i] = in_map ? *p : 0.f;
            } else {
#pragma unroll
                for (int c = 0; c < Cout; c += 16) {
                    float v[16];
#pragma unroll
                    for (int j = 0; j < 16; ++j) v[j] = in_map ? p[(c + j) * plane] : 0.f;
#pragma unroll
                    for (int j = 0; j < 16; j += 4)
                        *(float4 *)(gt + i * kWgGS + c + j) =
                            make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
                }
            }
        }
        for (int i = t; i < 18 * 18; i += nthr) {
            const int py = i / 18, px = i - py * 18, yy = y0 - 1 + py, xx = x0 - 1 + px;
            const bool in_map = yy >= 0 && yy < H && xx >= 0 && xx < W;
            const __nv_bfloat16 *p = in + ((int64_t)n * Cin * plane + (int64_t)yy * W + xx);
            float *d = it + py * kConvRow + px;
            for (int c = 0; c < Cin; c += 8, p += 8 * plane, d += 8 * kWgIS) {
                float v[8];
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    v[j] = in_map && c + j < Cin ? __bfloat162float(p[j * plane]) : 0.f;
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    if (c + j < Cin) d[j * kWgIS] = v[j];
            }
        }
        __syncthreads();
        // The bias, in conv3x3_wgrad_kernel's partial sums: a tile in row order, every tile
        // added to db by itself.  A loss clipped to +-1/n gives terms of one magnitude, whose
        // partial sums round alike, so that the grouping decides the last bits of the result.
        // One warp, 256 dependent additions: hidden behind the other warps (a training step of
        // 8 x 34 x 180 x 320 2,705 us; with eight sums per channel kept over a block's tiles 2,723).
        if (db && t >= nthr - 32 && t - (nthr - 32) < Cout) {
            const int co = t - (nthr - 32);
            float s = 0.f;
#pragma unroll 16
            for (int p = 0; p < kTile * kTile; ++p) s += gt[CPT == 1 ? p : p * kWgGS + co];
            atomicAdd(db + co, s);
        }
        if (mine) {
            for (int y = ya; y < kTile; y += ystep) {
                const float *ip = it + ci * kWgIS + y * kConvRow;
                const float *gp = gt + y * kTile * (CPT == 1 ? 1 : kWgGS) + (CPT == 1 ? 0 : 4 * cg);
                float4 lo[3];
#pragma unroll
                for (int ky = 0; ky < 3; ++ky) lo[ky] = *(const float4 *)(ip + ky * kConvRow);
#pragma unroll
                for (int x = 0; x < kTile; x += 4) {
                    float v[3][6];
#pragma unroll
                    for (int ky = 0; ky < 3; ++ky) {
                        const float4 hi = *(const float4 *)(ip + ky * kConvRow + x + 4);
                        v[ky][0] = lo[ky].x, v[ky][1] = lo[ky].y, v[ky][2] = lo[ky].z;
                        v[ky][3] = lo[ky].w, v[ky][4] = hi.x, v[ky][5] = hi.y;
                        lo[ky] = hi;
                    }
                    if constexpr (CPT == 1) {
                        const ulonglong2 q = *(const ulonglong2 *)(gp + x);
#pragma unroll
                        for (int k = 0; k < 9; ++k) {
                            const float *vk = v[k / 3] + k % 3;
                            fma2(tot[0][k], q.x, pair(vk[0], vk[1]));
                            fma2(tot[0][k], q.y, pair(vk[2], vk[3]));
                        }
                    } else {
                        unsigned long long vv[3][6];
#pragma unroll
                        for (int k = 0; k < 18; ++k) vv[k / 6][k % 6] = pair(v[k / 6][k % 6], v[k / 6][k % 6]);
#pragma unroll
                        for (int p = 0; p < 4; ++p) {
                            const ulonglong2 q = *(const ulonglong2 *)(gp + (x + p) * kWgGS);
#pragma unroll
                            for (int k = 0; k < 9; ++k) {
                                fma2(tot[0][k], q.x, vv[k / 3][p + k % 3]);
                                fma2(tot[NP - 1][k], q.y, vv[k / 3][p + k % 3]);
                            }
                        }
                    }
                }
            }
        }
    }
    if (CPT == 1) {                           // the split rows' totals in a fixed order
        __syncthreads();
        float *part = smem;                   // [kWgSplit][Cin * 9]
        if (mine)
#pragma unroll
            for (int k = 0; k < 9; ++k) {
                float e, o;
                unpair(tot[0][k], e, o);
                part[(cg * Cin + ci) * 9 + k] = e + o;
            }
        __syncthreads();
        for (int e = t; e < Cin * 9; e += nthr) {
            float s = 0.f;
#pragma unroll
            for (int q = 0; q < kWgSplit; ++q) s += part[q * Cin * 9 + e];
            atomicAdd(dw + e, s);
        }
    } else if (mine) {
#pragma unroll
        for (int j = 0; j < NP; ++j)
#pragma unroll
            for (int k = 0; k < 9; ++k) {
                float lo, hi;
                unpair(tot[j][k], lo, hi);
                float *d = dw + ((int64_t)(4 * cg + 2 * j) * Cin + ci) * 9 + k;
                atomicAdd(d, lo);
                atomicAdd(d + (int64_t)Cin * 9, hi);
            }
    }
}

// g_pre = g * (act > 0) (ReLU backward), bf16 activations; four elements per thread where the
// pointers allow it (bound by DRAM: 14.7 M elements, 147 MB: 57 -> 19 us)
__global__ void relu_mask_kernel(const float *__restrict__ g, const __nv_bfloat16 *__restrict__ act,
                                 float *__restrict__ out, int64_t n)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = __bfloat162float(act[i]) > 0.f ? g[i] : 0.f;
}

__global__ void relu_mask4_kernel(const float4 *__restrict__ g, const uint2 *__restrict__ act,
                                  float4 *__restrict__ out, int64_t n4)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n4) return;
    const float4 v = g[i];
    const uint2 a = act[i];
    // a BF16 value is the upper half of its FP32 bits
    out[i] = make_float4(__uint_as_float(a.x << 16) > 0.f ? v.x : 0.f,
                         __uint_as_float(a.x & 0xFFFF0000u) > 0.f ? v.y : 0.f,
                         __uint_as_float(a.y << 16) > 0.f ? v.z : 0.f,
                         __uint_as_float(a.y & 0xFFFF0000u) > 0.f ? v.w : 0.f);
}

// wt[ci][co][2-ky][2-kx] = w[co][ci][ky][kx]: backward-data weights
__global__ void flip_transpose_kernel(const __nv_bfloat16 *__restrict__ w, int Cout, int Cin,
                                      __nv_bfloat16 *__restrict__ wt)
{
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= Cout * Cin * 9) return;
    const int co = e / (Cin * 9), r = e % (Cin * 9), ci = r / 9, k = r % 9;
    wt[((int64_t)ci * Cout + co) * 9 + (8 - k)] = w[e];
}

// (hi, lo) += (x, y): an FP32 sum with what its additions round off beside it.
__device__ __forceinline__ void pair_add(float &hi, float &lo, float x, float y)
{
    const float u = __fadd_rn(hi, x), z = __fsub_rn(u, hi);
    lo += y + __fadd_rn(__fsub_rn(hi, __fsub_rn(u, z)), __fsub_rn(x, z));
    hi = u;
}

// Huber loss (delta) of prediction p against target t, mean over n; grad = dL/dp.
// The blocks stride over the elements and each adds its losses once: at most kHuberBlocks
// roundings of the loss, and no queue of one addition per warp at its address (460,800 elements
// 23.2 -> 5.5 us, 38,912 3.4 -> 2.5).  A block's sum is a pair of FP32 numbers, as good as a
// 64-bit one, and `per` is 1 / n from the host: FP64 additions and a division, slow on this GPU,
// made calls of 1 to 4,099 elements 2.4 to 3.2 us instead of 1.9 to 2.5 (one addition per warp
// 1.5 to 2.1).
constexpr int kHuberBlocks = 152;

__global__ void __launch_bounds__(256) huber_kernel(const float *__restrict__ p,
                                                    const float *__restrict__ t, float delta,
                                                    int64_t n, double per, float *__restrict__ grad,
                                                    float *__restrict__ loss)
{
    float hi = 0.f, lo = 0.f;
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256) {
        const float r = p[i] - t[i];
        const float a = fabsf(r);
        pair_add(hi, lo, a < delta ? 0.5f * r * r / delta : a - 0.5f * delta, 0.f);
        grad[i] = (a < delta ? r / delta : copysignf(1.f, r)) / (float)n;
    }
    if (!loss) return;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float x = __shfl_down_sync(0xFFFFFFFFu, hi, o), y = __shfl_down_sync(0xFFFFFFFFu, lo, o);
        pair_add(hi, lo, x, y);
    }
    __shared__ float2 part[8];
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = make_float2(hi, lo);
    __syncthreads();
    if (threadIdx.x >= 8) return;
    hi = part[threadIdx.x].x, lo = part[threadIdx.x].y;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
        const float x = __shfl_down_sync(0xFFu, hi, o), y = __shfl_down_sync(0xFFu, lo, o);
        pair_add(hi, lo, x, y);
    }
    if (threadIdx.x == 0) {
        // (an infinite or NaN sum leaves NaN in lo)
        const double sum = isfinite(lo) ? (double)hi + (double)lo : (double)hi;
        atomicAdd(loss, (float)(sum * per));
    }
}

// Adam on fp32 master weights; also refreshes their bf16 copy.
__global__ void adam_kernel(float *__restrict__ w, const float *__restrict__ g,
                            float *__restrict__ m, float *__restrict__ v, int64_t n, float lr,
                            float b1, float b2, float eps, float c1, float c2,
                            __nv_bfloat16 *__restrict__ wbf)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float wi = w[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    w[i] = wi;
    if (wbf) wbf[i] = __float2bfloat16(wi);
}

__global__ void to_bf16_kernel(const float *__restrict__ a, __nv_bfloat16 *__restrict__ b,
                               int64_t n)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) b[i] = __float2bfloat16(a[i]);
}

// Network input at the top level: (I0/255 - 1/2, I1/255 - 1/2, C(k)/255 for k < Dw).
__global__ void features_kernel(const uint8_t *__restrict__ I0, int p0, const uint8_t *__restrict__ I1,
                                int p1, const uint8_t *__restrict__ C, int Dws, int Dw, int W,
                                int H, __nv_bfloat16 *__restrict__ out)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (x >= W) return;
    const int64_t plane = (int64_t)H * W, px = (int64_t)y * W + x;
    out[px] = __float2bfloat16(I0[(int64_t)y * p0 + x] * (1.f / 255.f) - 0.5f);
    out[plane + px] = __float2bfloat16(I1[(int64_t)y * p1 + x] * (1.f / 255.f) - 0.5f);
    const uint8_t *c = C + px * Dws;
    for (int k = 0; k < Dw; ++k) out[(2 + k) * plane + px] = __float2bfloat16(c[k] * (1.f / 255.f));
}

// The same features channels-last, cstr channels per pixel (zero beyond 2 + Dw), written
// in 16-byte pieces: [view][y][x][cstr].
__global__ void features_nhwc_kernel(const uint8_t *__restrict__ I0, int p0,
                                     const uint8_t *__restrict__ I1, int p1,
                                     const uint8_t *__restrict__ C, int Dws, int Dw, int W, int H,
                                     int cstr, __nv_bfloat16 *__restrict__ out)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (x >= W) return;
    const int64_t px = (int64_t)y * W + x;
    const uint8_t *c = C + px * Dws;
    for (int q = 0; q < cstr / 8; ++q) {
        __align__(16) __nv_bfloat16 v[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int ch = 8 * q + e;
            float f = 0.f;
            if (ch == 0) f = I0[(int64_t)y * p0 + x] * (1.f / 255.f) - 0.5f;
            else if (ch == 1) f = I1[(int64_t)y * p1 + x] * (1.f / 255.f) - 0.5f;
            else if (ch - 2 < Dw) f = c[ch - 2] * (1.f / 255.f);
            v[e] = __float2bfloat16(f);
        }
        *(uint4 *)(out + px * cstr + 8 * q) = *(const uint4 *)v;
    }
}

// Training target at the top level's resolution: mean of the f x f block of the
// full-resolution disparity map (blocks clipped at the border), divided by D.
__global__ void target_kernel(const uint16_t *__restrict__ d, int pitch, int W, int H, int f,
                              int Wq, int Hq, float inv_D, float *__restrict__ t)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (x >= Wq) return;
    float s = 0.f;
    int c = 0;
    for (int yy = y * f; yy < min(y * f + f, H); ++yy)
        for (int xx = x * f; xx < min(x * f + f, W); ++xx) {
            s += d[(int64_t)yy * pitch + xx];
            ++c;
        }
    t[(int64_t)y * Wq + x] = c ? s / c * inv_D : 0.f;
}

// Window starts of the finest level from the prediction q (top level, units of D):
// bilinear upsampling by f with pixel centres aligned, c = D q, lo = clamp(rint(c) - Dw/2).
__global__ void proposal_windows_kernel(const float *__restrict__ q, int Wq, int Hq, int f,
                                        int W, int H, int D, int Dw, uint16_t *__restrict__ lo)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (x >= W) return;
    const float u = fminf(fmaxf((x + 0.5f) / f - 0.5f, 0.f), (float)(Wq - 1));
    const float v = fminf(fmaxf((y + 0.5f) / f - 0.5f, 0.f), (float)(Hq - 1));
    const int x0 = (int)u, y0 = (int)v;
    const int x1 = min(x0 + 1, Wq - 1), y1 = min(y0 + 1, Hq - 1);
    const float ax = u - x0, ay = v - y0;
    const float top = q[y0 * Wq + x0] * (1.f - ax) + q[y0 * Wq + x1] * ax;
    const float bot = q[y1 * Wq + x0] * (1.f - ax) + q[y1 * Wq + x1] * ax;
    const float c = (top * (1.f - ay) + bot * ay) * D;
    const int l = (int)rintf(c) - Dw / 2;
    lo[(int64_t)y * W + x] = (uint16_t)min(max(l, 0), D - Dw);
}


// Tensor-core form of the convolution for BF16 input (inference and training forward) on
// the fifth-generation tensor cores: an implicit GEMM
//     D[m][co] = sum_{tap, ci} A[m][(tap, ci)] B[co][(tap, ci)]
// with m one of the 128 pixels of an output tile of 16 rows x 8 columns (M = 128), N = 32
// output channels (16 for the one-channel output layer, its other rows zero weights) and
// K = 9 taps x the input channels rounded up to 16, in k-steps of 16 (kind::f16, BF16
// operands, FP32 accumulation in tensor memory).
//
// Shared memory holds both operands K-major without swizzling, as 8-row x 16-byte core
// matrices.  The input tile with its one-pixel halo (18 x 10 pixels) is stored as planes of
// 8 channels: plane c8 holds channels 8 c8 .. 8 c8 + 7 of every staged pixel, 16 bytes per
// pixel, pixels row-major.  Eight consecutive output pixels of one row then form a core
// matrix for every tap: the A operand of tap (ky, kx) starts at staged pixel ky * 10 + kx,
// its core matrices follow each other along M at one staged row (160 bytes) and along K at
// one plane.  The weights are stored [tap][c8][co][8], so that B's core matrices follow
// each other along N at 8 channels (128 bytes) and along K at one plane of NC x 16 bytes.
// One thread issues the 9 x (K/16) MMAs of a tile and commits them to an mbarrier; the
// four warps read their 32 rows of the accumulator back (tcgen05.ld) for the epilogue.
constexpr int kTcRows = 16, kTcCols = 8;                 // output tile (M = 128 pixels)
constexpr int kTcTR = kTcRows + 2, kTcTC = kTcCols + 2;  // staged input tile, 18 x 10
constexpr int kTcPix = kTcTR * kTcTC;
// bytes of one plane of 8 channels; the extra 16 bytes spread one pixel's planes over banks
constexpr int kTcPlane = kTcPix * 16 + 16;
constexpr int kTcBlocksPerSm = 4;                        // resident blocks the grid aims for
constexpr long long kTcWaitCycles = 2000000000LL;        // about a second

__device__ __forceinline__ uint32_t smem_addr(const void *p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

// Shared-memory matrix descriptor of a K-major operand without swizzling: start address,
// byte distance between core matrices adjacent along K (lbo) and along M or N (sbo), each
// in 16-byte units, and the descriptor version of this architecture (bit 46).
__device__ __forceinline__ uint64_t umma_smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo)
{
    return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}

// Instruction descriptor of kind::f16: FP32 accumulator (bits 4-5), BF16 A and B (bits
// 7-9, 10-12), both K-major (bits 15, 16 clear), N / 8 (bits 17-22), M / 16 (bits 24-28).
template <int M, int N>
__host__ __device__ constexpr uint32_t umma_instr_desc()
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) |
           ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void umma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc,
                                          uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

__device__ __forceinline__ bool mbar_phase_done(uint32_t mbar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(mbar), "r"(parity)
        : "memory");
    return ok != 0;
}

// 32 lanes x X columns of 32 bits from tensor memory: thread t of the warp gets lane
// (warp's first lane + t), columns col .. col + X - 1
template <int X>
struct TmemRow;
template <>
struct TmemRow<32> {
    __device__ __forceinline__ static void ld(uint32_t taddr, uint32_t (&r)[32])
    {
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, "
            "%10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, "
            "%26, %27, %28, %29, %30, %31}, [%32];"
            : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
              "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]),
              "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]),
              "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
              "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]),
              "=r"(r[30]), "=r"(r[31])
            : "r"(taddr));
    }
};
template <>
struct TmemRow<16> {
    __device__ __forceinline__ static void ld(uint32_t taddr, uint32_t (&r)[16])
    {
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, "
            "%10, %11, %12, %13, %14, %15}, [%16];"
            : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
              "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]),
              "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
            : "r"(taddr));
    }
};

size_t tc_smem_bytes(int Cin, int Cout)
{
    const int ncg = tc_planes(Cin), nc = tc_width(Cout);
    return (size_t)ncg * kTcPlane + (size_t)9 * ncg * nc * 16 + 16;
}

// NC: the MMA width N (32, or 16 for the one-channel output layer).
// NHWC: activations [n][y][x][cstr] (cstr a multiple of 8, channels Cin .. cstr - 1 zero)
// and weights pre-arranged [9][tc_planes(Cin)][NC][8] with zero padding (the matcher's own
// buffers); otherwise activations [n][c][y][x] and weights [Cout][Cin][3][3] (the public
// entry points).  err (optional): set to 1 when the wait for the tensor cores ran out; the
// outputs of the block's unfinished tiles are then NaN.
template <int NC, bool NHWC>
__global__ void __launch_bounds__(128) conv3x3_tc_kernel(
    const __nv_bfloat16 *__restrict__ in, int Cin, int cstr, int H, int W, int nimg,
    const __nv_bfloat16 *__restrict__ w, const float *__restrict__ b, int Cout, int relu,
    __nv_bfloat16 *__restrict__ out_bf, float *__restrict__ out_f, int *err)
{
    extern __shared__ __align__(128) unsigned char tsm[];
    const int ncg = tc_planes(Cin), ks = ncg / 2;
    unsigned char *As = tsm;                                   // ncg planes
    unsigned char *Bs = tsm + (size_t)ncg * kTcPlane;          // [9][ncg][NC][8]
    uint64_t *mbar = (uint64_t *)(Bs + (size_t)9 * ncg * NC * 16);
    uint32_t *tslot = (uint32_t *)(mbar + 1);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    // the planes start zero: channels the staging never writes (Cin or cstr up to the
    // k-steps' multiple of 16) stay zero in every tile
    for (int i = tid; i < ncg * kTcPlane / 16; i += 128)
        ((uint4 *)As)[i] = make_uint4(0u, 0u, 0u, 0u);
    if (NHWC) {
        const int nvec = 9 * ncg * NC;
        for (int i = tid; i < nvec; i += 128) ((uint4 *)Bs)[i] = ((const uint4 *)w)[i];
    } else {
        // element (tap, ci, co) at ((tap * ncg + ci / 8) * NC + co) * 8 + ci % 8, zero for
        // absent channels
        __nv_bfloat16 *bw = (__nv_bfloat16 *)Bs;
        const __nv_bfloat16 zero = __float2bfloat16(0.f);
        const int ntot = 9 * ncg * 8 * NC;
        for (int i = tid; i < ntot; i += 128) {
            const int co = i % NC, r = i / NC, ci = r % (ncg * 8), tap = r / (ncg * 8);
            bw[((tap * ncg + ci / 8) * NC + co) * 8 + ci % 8] =
                (co < Cout && ci < Cin) ? w[((int64_t)co * Cin + ci) * 9 + tap] : zero;
        }
    }
    if (warp == 0) {   // 32 columns of tensor memory: the 128 x NC FP32 accumulator
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 32;" ::"r"(
                         smem_addr(tslot))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(mbar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tslot;

    const int tx = (W + kTcCols - 1) / kTcCols, ty = (H + kTcRows - 1) / kTcRows;
    const int ntiles = tx * ty * nimg;
    const int64_t plane = (int64_t)H * W;
    constexpr uint32_t idesc = umma_instr_desc<128, NC>();
    const uint32_t a0 = smem_addr(As), b0 = smem_addr(Bs), mb = smem_addr(mbar);
    uint32_t phase = 0;
    int tile = blockIdx.x;
    bool failed = false;

    for (; tile < ntiles; tile += gridDim.x) {
        const int n = tile / (tx * ty), r = tile - n * (tx * ty);
        const int y0 = (r / tx) * kTcRows, x0 = (r % tx) * kTcCols;
        // the input tile with its one-pixel halo, zero outside the image, in 16-byte pieces
        // (8 channels of one pixel); consecutive threads on consecutive pieces, a batch of
        // loads before the stores
        constexpr int kBatch = 8;
        if (NHWC) {
            const __nv_bfloat16 *src = in + (int64_t)n * cstr * plane;
            // 16-byte pieces per pixel, never more than the planes the operand holds
            // (channels Cin .. cstr - 1 are zero, so those beyond the planes are not needed)
            const int per = min(cstr / 8, ncg), npieces = kTcPix * per;
            for (int i0 = tid; i0 < npieces; i0 += 128 * kBatch) {
                uint4 v[kBatch];
#pragma unroll
                for (int q = 0; q < kBatch; ++q) {
                    const int i = i0 + q * 128;
                    const int pp = i / per, c8 = i - pp * per;
                    const int py = pp / kTcTC, px = pp - py * kTcTC;
                    const int yy = y0 - 1 + py, xx = x0 - 1 + px;
                    v[q] = make_uint4(0u, 0u, 0u, 0u);
                    if (i < npieces && yy >= 0 && yy < H && xx >= 0 && xx < W)
                        v[q] = *(const uint4 *)(src + ((int64_t)yy * W + xx) * cstr + 8 * c8);
                }
#pragma unroll
                for (int q = 0; q < kBatch; ++q) {
                    const int i = i0 + q * 128;
                    if (i >= npieces) break;
                    const int pp = i / per, c8 = i - pp * per;
                    *(uint4 *)(As + c8 * kTcPlane + pp * 16) = v[q];
                }
            }
        } else {
            // piece (plane c8, pixel pp): consecutive threads on consecutive pixels, each
            // gathering its 8 channels from 8 channel planes of the image
            const __nv_bfloat16 *src = in + (int64_t)n * Cin * plane;
            const int cgi = (Cin + 7) / 8, npieces = kTcPix * cgi;
            for (int i = tid; i < npieces; i += 128) {
                const int c8 = i / kTcPix, pp = i - c8 * kTcPix;
                const int py = pp / kTcTC, px = pp - py * kTcTC;
                const int yy = y0 - 1 + py, xx = x0 - 1 + px;
                uint32_t pk[4] = {0u, 0u, 0u, 0u};
                if (yy >= 0 && yy < H && xx >= 0 && xx < W) {
                    const __nv_bfloat16 *s0 = src + (int64_t)(8 * c8) * plane + (int64_t)yy * W + xx;
                    unsigned short h[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e)
                        h[e] = 8 * c8 + e < Cin ? __bfloat16_as_ushort(s0[(int64_t)e * plane]) : 0;
#pragma unroll
                    for (int e = 0; e < 4; ++e) pk[e] = (uint32_t)h[2 * e] | ((uint32_t)h[2 * e + 1] << 16);
                }
                *(uint4 *)(As + c8 * kTcPlane + pp * 16) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
            }
        }
        // the staged tile, written through the generic proxy, before the tensor cores read it
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            for (int tap = 0; tap < 9; ++tap) {
                const uint32_t aoff = (uint32_t)(((tap / 3) * kTcTC + tap % 3) * 16);
                for (int s = 0; s < ks; ++s) {
                    const uint64_t ad =
                        umma_smem_desc(a0 + 2 * s * kTcPlane + aoff, kTcPlane, kTcTC * 16);
                    const uint64_t bd = umma_smem_desc(
                        b0 + (uint32_t)((tap * ncg + 2 * s) * NC * 16), NC * 16, 128);
                    umma_bf16(tmem, ad, bd, idesc, (tap | s) != 0);
                }
            }
            asm volatile(
                "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                    mb)
                : "memory");
        }
        // the products (bounded wait; the block agrees on the outcome)
        bool ok = mbar_phase_done(mb, phase);
        if (!ok) {
            const long long t0 = clock64();
            while (!(ok = mbar_phase_done(mb, phase)) && clock64() - t0 < kTcWaitCycles) {
            }
        }
        phase ^= 1u;
        if (!__syncthreads_and(ok)) {
            failed = true;
            break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        uint32_t acc[NC];
        TmemRow<NC>::ld(tmem + ((uint32_t)(warp * 32) << 16), acc);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        // accumulator row m = 32 warp + lane: output pixel (y0 + m / 8, x0 + m % 8)
        const int m = warp * 32 + lane;
        const int oy = y0 + m / kTcCols, ox = x0 + m % kTcCols;
        if (oy < H && ox < W) {
            const int64_t pix = (int64_t)oy * W + ox;
            bool done = false;
            if constexpr (NC == 32 && NHWC) {
                if (Cout == 32 && out_bf && !out_f) {   // the matcher's hidden layers
                    uint4 *dst = (uint4 *)(out_bf + ((int64_t)n * plane + pix) * 32);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        uint32_t pk[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const int co = 8 * q + 2 * e;
                            float v0 = __uint_as_float(acc[co]) + (b ? b[co] : 0.f);
                            float v1 = __uint_as_float(acc[co + 1]) + (b ? b[co + 1] : 0.f);
                            if (relu) {
                                v0 = fmaxf(v0, 0.f);
                                v1 = fmaxf(v1, 0.f);
                            }
                            const __nv_bfloat162 h2 = __floats2bfloat162_rn(v0, v1);
                            pk[e] = *(const uint32_t *)&h2;
                        }
                        dst[q] = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                    }
                    done = true;
                }
            }
            if (!done) {
#pragma unroll
                for (int co = 0; co < NC; ++co) {
                    if (co >= Cout) break;
                    float v = __uint_as_float(acc[co]) + (b ? b[co] : 0.f);
                    if (relu) v = fmaxf(v, 0.f);
                    const int64_t o = NHWC ? ((int64_t)n * plane + pix) * Cout + co
                                           : ((int64_t)n * Cout + co) * plane + pix;
                    if (out_f) out_f[o] = v;
                    if (out_bf) out_bf[o] = __float2bfloat16(v);
                }
            }
        }
        // every warp's reads of the accumulator and of the staged tile are complete before
        // the next tile overwrites them
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
    }
    if (failed) {
        // the wait ran out: record it, and mark the block's unfinished tiles as NaN
        if (tid == 0 && err) atomicCAS(err, 0, 1);
        for (; tile < ntiles; tile += gridDim.x) {
            const int n = tile / (tx * ty), r = tile - n * (tx * ty);
            const int oy = (r / tx) * kTcRows + tid / kTcCols, ox = (r % tx) * kTcCols + tid % kTcCols;
            if (oy >= H || ox >= W) continue;
            const int64_t pix = (int64_t)oy * W + ox;
            for (int co = 0; co < Cout && co < NC; ++co) {
                const int64_t o = NHWC ? ((int64_t)n * plane + pix) * Cout + co
                                       : ((int64_t)n * Cout + co) * plane + pix;
                if (out_f) out_f[o] = __int_as_float(0x7FC00000);
                if (out_bf) out_bf[o] = __ushort_as_bfloat16((unsigned short)0x7FC0);
            }
        }
    }
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 32;" ::"r"(tmem) : "memory");
}

unsigned blocks(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

size_t conv_smem_bytes(int Cin, int Cout) { return sizeof(float) * ((size_t)Cin * 9 * Cout + 18 * 18); }

template <int COUT, class TIn>
void launch_conv3x3_pixel(const TIn *in, int N, int Cin, int H, int W, const __nv_bfloat16 *w,
                          const float *b, int relu, __nv_bfloat16 *out_bf, float *out_f,
                          cudaStream_t s)
{
    dim3 grid((W + kTile - 1) / kTile, (H + kTile - 1) / kTile, N);
    const size_t smem = conv_smem_bytes(Cin, COUT);
    cudaFuncSetAttribute(conv3x3_pixel_kernel<COUT, TIn>,
                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    conv3x3_pixel_kernel<COUT, TIn><<<grid, kTile * kTile, smem, s>>>(in, Cin, H, W, w, b, relu,
                                                                      out_bf, out_f);
}

void launch_conv3x3_f32(const float *in, int N, int Cin, int H, int W, const __nv_bfloat16 *w,
                        const float *b, int Cout, int relu, __nv_bfloat16 *out_bf, float *out_f,
                        cudaStream_t s)
{
    if (Cout == 1)
        return launch_conv3x3_pixel<1>(in, N, Cin, H, W, w, b, relu, out_bf, out_f, s);
    if (Cin <= kPixelCin)
        return launch_conv3x3_pixel<32>(in, N, Cin, H, W, w, b, relu, out_bf, out_f, s);
    dim3 grid((W + kTile - 1) / kTile, (H + kTile - 1) / kTile, N);
    conv3x3_f32_kernel<<<grid, 256, 0, s>>>(in, Cin, H, W, w, b, relu, out_bf, out_f);
}

int sm_count()
{
    static int n = 0;
    if (!n) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        if (n < 1) n = 1;
    }
    return n;
}

template <bool NHWC>
void launch_tc(const __nv_bfloat16 *in, int N, int Cin, int cstr, int H, int W,
               const __nv_bfloat16 *w, const float *b, int Cout, int relu, __nv_bfloat16 *out_bf,
               float *out_f, int *err, cudaStream_t s)
{
    const int64_t tiles = (int64_t)((W + kTcCols - 1) / kTcCols) * ((H + kTcRows - 1) / kTcRows) * N;
    const int64_t cap = (int64_t)kTcBlocksPerSm * sm_count();
    const unsigned grid = (unsigned)(tiles < cap ? tiles : cap);
    const size_t smem = tc_smem_bytes(Cin, Cout);
    if (Cout == 32) {
        cudaFuncSetAttribute(conv3x3_tc_kernel<32, NHWC>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        conv3x3_tc_kernel<32, NHWC><<<grid, 128, smem, s>>>(in, Cin, cstr, H, W, N, w, b, Cout,
                                                            relu, out_bf, out_f, err);
    } else {
        cudaFuncSetAttribute(conv3x3_tc_kernel<16, NHWC>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        conv3x3_tc_kernel<16, NHWC><<<grid, 128, smem, s>>>(in, Cin, cstr, H, W, N, w, b, Cout,
                                                            relu, out_bf, out_f, err);
    }
}

void launch_conv3x3_nhwc(const __nv_bfloat16 *in, int N, int Cin, int cstr, int H, int W,
                         const __nv_bfloat16 *w, const float *b, int Cout, int relu,
                         __nv_bfloat16 *out_bf, float *out_f, int *err, cudaStream_t s)
{
    launch_tc<true>(in, N, Cin, cstr, H, W, w, b, Cout, relu, out_bf, out_f, err, s);
}

bool conv3x3_tc_ok(int Cin, int Cout)
{
    return (Cout == 32 || Cout == 1) && tc_smem_bytes(Cin, Cout) <= kTcMaxSmem;
}

// Whether some kernel takes a convolution: one channel of any input, 32 of FP32 input, or what the
// tensor-core kernel takes of BF16 input.  (FP32 input is limited as one thread per pixel was.)
bool conv3x3_ok(bool in_f32, int Cin, int Cout)
{
    if (!in_f32 && conv3x3_tc_ok(Cin, Cout)) return true;
    return (Cout == 1 || (Cout == 32 && in_f32)) && conv_smem_bytes(Cin, Cout) <= 200 * 1024;
}

void launch_conv3x3(const __nv_bfloat16 *in, int N, int Cin, int H, int W, const __nv_bfloat16 *w,
                    const float *b, int Cout, int relu, __nv_bfloat16 *out_bf, float *out_f,
                    cudaStream_t s)
{
    // one channel whose operands don't fit in the tensor-core kernel's shared memory on the CUDA
    // cores; 32 have no other kernel (conv3x3_ok)
    if (conv3x3_tc_ok(Cin, Cout))
        launch_tc<false>(in, N, Cin, Cin, H, W, w, b, Cout, relu, out_bf, out_f, nullptr, s);
    else if (Cout == 1)
        launch_conv3x3_pixel<1>(in, N, Cin, H, W, w, b, relu, out_bf, out_f, s);
}

// Whether the tiled kernel takes a weight gradient.  Few input channels leave most of its threads
// idle, and the general kernel is as fast or faster (us, general against tiled): 32 <- 1 channels
// 13.0 / 13.1 with 60 tiles, 13.0 / 18.5 with 120, 64.7 / 69.2 with 1,920; 32 <- 2 channels
// 16.0 / 13.3 with 60 tiles, 16.3 / 18.2 with 120, 28.8 / 33.6 with 320, 53.0 / 41.9 with 784;
// 1 <- 1 channel 5.4 / 4.5 with 320, 11.5 / 12.9 with 1,920.  (Over 65,535 rows of tiles or
// samples the general kernel's launch refuses the call.)
bool wgrad_tiled(int Cin, int Cout, int64_t tiles, int64_t ty, int N)
{
    if ((Cout != 32 && Cout != 1) || Cin > kWgMaxCin || ty > 65535 || N > 65535 ||
        tiles >= 0x7FFFFFFF)
        return false;
    const int64_t sms = sm_count();
    if (Cout == 1) return Cin > 1 || tiles <= 3 * sms;
    if (Cin == 1) return 5 * tiles <= 2 * sms;
    return Cin > 2 || 5 * tiles <= 3 * sms || tiles > 3 * sms;
}

void launch_conv3x3_wgrad(const __nv_bfloat16 *in, int N, int Cin, const float *g, int Cout, int H,
                          int W, float *dw, float *db, cudaStream_t s)
{
    const int64_t tx = (W + kTile - 1) / kTile, ty = (H + kTile - 1) / kTile, tiles = tx * ty * N;
    if (wgrad_tiled(Cin, Cout, tiles, ty, N)) {
        const int64_t resident = (Cout == 1 ? 3 : 2) * (int64_t)sm_count();
        const unsigned blocks = (unsigned)(tiles < resident ? tiles : resident);
        size_t sm = sizeof(float) * ((size_t)kTile * kTile * (Cout == 1 ? 1 : kWgGS) +
                                     (size_t)Cin * kWgIS);
        // 256 threads at least, to stage the tiles (32 <- 3 channels or 1 <- 4 compute with one
        // warp; with 32 threads 1 <- 4 channels took 34 instead of 14 us on 1,920 tiles)
        const int threads = std::max(256, (8 * Cin + 31) / 32 * 32);
        if (Cout == 32) {
            cudaFuncSetAttribute(wgrad_tile_kernel<4>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)sm);
            wgrad_tile_kernel<4><<<blocks, threads, sm, s>>>(in, Cin, g, H, W, (int)tx, (int)ty,
                                                             (int)tiles, dw, db);
        } else {
            const size_t part = sizeof(float) * kWgSplit * 9 * (size_t)Cin;
            if (part > sm) sm = part;
            cudaFuncSetAttribute(wgrad_tile_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)sm);
            wgrad_tile_kernel<1><<<blocks, threads, sm, s>>>(in, Cin, g, H, W, (int)tx, (int)ty,
                                                             (int)tiles, dw, db);
        }
        return;
    }
    dim3 grid((unsigned)tx, (unsigned)ty, N);
    const size_t smem = sizeof(float) * ((size_t)Cout * kTile * kTile + (size_t)Cin * 18 * 18);
    cudaFuncSetAttribute(conv3x3_wgrad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    conv3x3_wgrad_kernel<<<grid, kTile * kTile, smem, s>>>(in, Cin, g, Cout, H, W, dw, db);
}

void launch_features(const uint8_t *I0, int p0, const uint8_t *I1, int p1, const uint8_t *C,
                     int Dws, int Dw, int W, int H, __nv_bfloat16 *out, cudaStream_t s)
{
    features_kernel<<<dim3(blocks(W, 128), H), 128, 0, s>>>(I0, p0, I1, p1, C, Dws, Dw, W, H, out);
}

void launch_features_nhwc(const uint8_t *I0, int p0, const uint8_t *I1, int p1, const uint8_t *C,
                          int Dws, int Dw, int W, int H, int cstr, __nv_bfloat16 *out,
                          cudaStream_t s)
{
    features_nhwc_kernel<<<dim3(blocks(W, 128), H), 128, 0, s>>>(I0, p0, I1, p1, C, Dws, Dw, W,
                                                                 H, cstr, out);
}

void launch_proposal_windows(const float *q, int Wq, int Hq, int f, int W, int H, int D, int Dw,
                             uint16_t *lo, cudaStream_t s)
{
    proposal_windows_kernel<<<dim3(blocks(W, 128), H), 128, 0, s>>>(q, Wq, Hq, f, W, H, D, Dw, lo);
}

}  // namespace mpv

using namespace mpv;

extern "C" {

mpv_status mpv_cnn_conv3x3(const void *in, int32_t in_f32, int32_t n, int32_t cin, int32_t h,
                           int32_t w, const void *weight, const float *bias, int32_t cout,
                           int32_t relu, void *out_bf16, float *out_f32, void *cuda_stream)
{
    if (!in || !weight || n < 1 || cin < 1 || h < 1 || w < 1 || !conv3x3_ok(in_f32 != 0, cin, cout) ||
        (!out_bf16 && !out_f32))
        return MPV_ERR_INVALID_ARG;
    if (in_f32)
        launch_conv3x3_f32((const float *)in, n, cin, h, w, (const __nv_bfloat16 *)weight, bias,
                           cout, relu, (__nv_bfloat16 *)out_bf16, out_f32,
                           (cudaStream_t)cuda_stream);
    else
        launch_conv3x3((const __nv_bfloat16 *)in, n, cin, h, w, (const __nv_bfloat16 *)weight, bias,
                       cout, relu, (__nv_bfloat16 *)out_bf16, out_f32, (cudaStream_t)cuda_stream);
    return cudaGetLastError() == cudaSuccess ? MPV_OK : MPV_ERR_CUDA;
}

mpv_status mpv_cnn_conv3x3_wgrad(const void *in, int32_t n, int32_t cin, const float *grad,
                                 int32_t cout, int32_t h, int32_t w, float *dweight, float *dbias,
                                 void *cuda_stream)
{
    if (!in || !grad || !dweight || n < 1 || cin < 1 || cout < 1 || h < 1 || w < 1 ||
        sizeof(float) * ((size_t)cout * 256 + (size_t)cin * 324) > 200 * 1024)
        return MPV_ERR_INVALID_ARG;
    launch_conv3x3_wgrad((const __nv_bfloat16 *)in, n, cin, grad, cout, h, w, dweight, dbias,
                         (cudaStream_t)cuda_stream);
    return cudaGetLastError() == cudaSuccess ? MPV_OK : MPV_ERR_CUDA;
}

mpv_status mpv_cnn_flip_transpose(const void *weight, int32_t cout, int32_t cin, void *out,
                                  void *cuda_stream)
{
    if (!weight || !out || cout < 1 || cin < 1) return MPV_ERR_INVALID_ARG;
    const int e = cout * cin * 9;
    flip_transpose_kernel<<<blocks(e, 256), 256, 0, (cudaStream_t)cuda_stream>>>(
        (const __nv_bfloat16 *)weight, cout, cin, (__nv_bfloat16 *)out);
    return cudaGetLastError() == cudaSuccess ? MPV_OK : MPV_ERR_CUDA;
}

mpv_status mpv_cnn_relu_backward(const float *grad, const void *act, float *out, int64_t count,
                                 void *cuda_stream)
{
    if (!grad || !act || !out || count < 0) return MPV_ERR_INVALID_ARG;
    if (((uintptr_t)grad | (uintptr_t)out) % 16 == 0 && (uintptr_t)act % 8 == 0 && count % 4 == 0 &&
        count > 0)
        relu_mask4_kernel<<<blocks(count / 4, 256), 256, 0, (cudaStream_t)cuda_stream>>>(
            (const float4 *)grad, (const uint2 *)act, (float4 *)out, count / 4);
    else
        relu_mask_kernel<<<blocks(count, 256), 256, 0, (cudaStream_t)cuda_stream>>>(
            grad, (const __nv_bfloat16 *)act, out, count);
    return cudaGetLastError() == cudaSuccess ? MPV_OK : MPV_ERR_CUDA;
}

mpv_status mpv_cnn_huber(const float *pred, const float *target, float delta, int64_t count,
                         float *grad, float *loss, void *cuda_stream)
{
    if (!pred || !target || !grad || count < 1 || !(delta > 0.f)) return MPV_ERR_INVALID_ARG;
    const unsigned nb = blocks(count, 256);
    huber_kernel<<<nb < kHuberBlocks ? nb : kHuberBlocks, 256, 0, (cudaStream_t)cuda_stream>>>(
        pred, target, delta, count, 1.0 / (double)count, grad, loss);
    return cudaGetLastError() == cudaSuccess ? MPV_OK : MPV_ERR_CUDA;
}

mpv_status mpv_cnn_adam(float *weight, const float *grad, float *m, float *v, int64_t count,
                        float lr, float beta1, float beta2, float eps, int32_t step,
                        void *weight_bf16, void *cuda_stream)
{
    if (!weight || !grad || !m || !v || count < 1 || step < 1) return MPV_ERR_INVALID_ARG;
    const float c1 = 1.f - powf(beta1, (float)step), c2 = 1.f - powf(beta2, (float)step);
    adam_kernel<<<blocks(count, 256), 256, 0, (cudaStream_t)cuda_stream>>>(
        weight, grad, m, v, count, lr, beta1, beta2, eps, c1, c2, (__nv_bfloat16 *)weight_bf16);
    return cudaGetLastError() == cudaSuccess ? MPV_OK : MPV_ERR_CUDA;
}

mpv_status mpv_cnn_to_bf16(const float *in, void *out, int64_t count, void *cuda_stream)
{
    if (!in || !out || count < 0) return MPV_ERR_INVALID_ARG;
    to_bf16_kernel<<<blocks(count, 256), 256, 0, (cudaStream_t)cuda_stream>>>(
        in, (__nv_bfloat16 *)out, count);
    return cudaGetLastError() == cudaSuccess ? MPV_OK : MPV_ERR_CUDA;
}

mpv_status mpv_cnn_target(const uint16_t *disp, int32_t disp_pitch, int32_t width, int32_t height,
                          int32_t factor, int32_t max_disparity, float *target, void *cuda_stream)
{
    if (!disp || !target || factor < 1 || width < 1 || height < 1 || max_disparity < 1)
        return MPV_ERR_INVALID_ARG;
    const int Wq = (width + factor - 1) / factor, Hq = (height + factor - 1) / factor;
    target_kernel<<<dim3(blocks(Wq, 128), Hq), 128, 0, (cudaStream_t)cuda_stream>>>(
        disp, disp_pitch, width, height, factor, Wq, Hq, 1.f / max_disparity, target);
    return cudaGetLastError() == cudaSuccess ? MPV_OK : MPV_ERR_CUDA;
}

}  // extern "C"
