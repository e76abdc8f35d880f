// cost_body.cuh -- the integer SSIM cost volume (see cost.cu), as a device function of
// (block index, thread index) shared by the stand-alone kernel and the batch
// scheduler's persistent kernel.
#pragma once
#include "volume_layout.cuh"

namespace mpv {

namespace {

constexpr int kSegPix = 320;          // pixels per block at most (one row segment)
constexpr int kCostThreads = 256;
constexpr int kCostWarps = kCostThreads / 32;

// The matching cost is evaluated on pixels shifted by -128 (as signed bytes), which leaves
// the covariance and the variances unchanged: with n = N * N, every patch sum is then at
// most 3200 in size, and n Sxy, Sx Sy, n Sxy - Sx Sy and the V = n Sxx - Sx^2 (at most
// n^2 127.5^2 = 10.2 million for N = 5) are integers below 2^24, exact in fp32.
//
// Cost = floor(t), t = 127.5 (1 - num/den), num = A1 A2, den = B1 B2, |num| <= den.  Roundings
// of the fp32 ratio, in units of 2^-24: A1 and A2 one each and their product one; B1 two, B2
// one and their product one; the approximate reciprocal two (rcp.approx.ftz: 2^-23) and the
// last product one.  Ten in all move t by at most 127.5 * 10 * 2^-24 = 7.6e-5, the final
// multiply-add by 2^-17 = 7.7e-6: t is known to 8.4e-5.  t' = t - 1/2 rounded to the nearest
// integer is floor(t) unless t' lies within 8.4e-5 of a half-integer; beyond kQuotientSafe
// from it (a node in 4,000) the integers decide.
constexpr float kQuotientSafe = 0.5f - 1.2e-4f;
constexpr float kRound23 = 12582912.0f;              // 1.5 * 2^23: adding it rounds to an integer
constexpr int kRound23Bits = 0x4B400000;             // its bits: + i is the float kRound23 + i

// The exact floor from the integers (patch sums sx, sy of the unshifted pixels), started
// from an estimate q.
__device__ __forceinline__ int ssim_exact(int q, int A2, int sx, int vx, int sy, int vy, int c1,
                                          int c2)
{
    const long long A1 = 2LL * sx * sy + c1;
    const long long B1 = (long long)sx * sx + (long long)sy * sy + c1;
    const long long B2 = (long long)vx + vy + c2;
    const long long dd = B1 * B2;
    const long long X = 255LL * (dd - A1 * A2);
    const long long Y = 2LL * dd;
    q = min(max(q, 0), 255);
    long long R = X - (long long)q * Y;
    while (R < 0) {
        --q;
        R += Y;
    }
    while (R >= Y) {
        ++q;
        R -= Y;
    }
    return q;
}

// Pixels of a block's row segment: a multiple of 16 N (whole chunks of N pixels for every
// warp and for the two half-warp streams of a 16-label group), at most kSegPix.
__host__ __device__ inline int cost_seg_unit(int N) { return 2 * kCostWarps * N; }
__host__ __device__ inline int cost_seg_max(int N)
{
    return kSegPix / cost_seg_unit(N) * cost_seg_unit(N);
}
// Equal segments of a row of W pixels, each at most seg_max: the widest block sets a
// launch's time.
__host__ __device__ inline int cost_seg(int W, int N, int seg_max)
{
    const int u = cost_seg_unit(N), n = (W + seg_max - 1) / seg_max;
    return ((W + n - 1) / n + u - 1) / u * u;
}

// Shared-memory layout of one block.
struct CostSmem {
    int ncol0, ncol1;     // staged columns of I0 and I1
    size_t off_e1, off_st0, off_col0, bytes;
};

__host__ __device__ inline CostSmem cost_smem_layout(int R, int uspan_max)
{
    CostSmem L;
    L.ncol0 = kSegPix + 2 * R + 2;
    L.ncol1 = kSegPix + 2 * R + 1 + uspan_max;
    size_t o = 0;
    L.off_e1 = o;                          // I1: packed column, statistics (16 bytes)
    o += sizeof(int4) * L.ncol1;
    L.off_st0 = o;                         // I0 statistics of the segment's pixels
    o += sizeof(float4) * kSegPix;
    L.off_col0 = o;                        // I0: packed columns
    o += sizeof(uint2) * L.ncol0;
    L.bytes = o;
    return L;
}

// Product sum of two packed columns (signed bytes; the second word's upper bytes of b are 0).
template <int N>
__device__ __forceinline__ int colprod(int a0, int a1, int b0, int b1)
{
    return N == 5 ? __dp4a(a0, b0, __dp4a(a1, b1, 0)) : __dp4a(a0, b0, 0);
}

// Column xc (clamped) of rows y-R..y+R (clamped), every pixel minus 128 as a signed byte:
// its packed rows, and in `sum` its sums over this column and the N - 1 lanes (columns)
// before it: the sum of squares (below 2^19) plus 2^19 times the sum shifted by 640 per
// column (at most 6375, so that the word holds both exactly).  All lanes of the warp call it.
template <int N>
__device__ __forceinline__ uint2 pack_column(const uint8_t *img, int pitch, int W, int H, int y,
                                             int xc, uint32_t &sum)
{
    constexpr int R = N / 2;
    const int xa = min(max(xc, 0), W - 1);
    uint32_t w0 = 0, w1 = 0;
#pragma unroll
    for (int r = 0; r < N; ++r) {
        const int yy = min(max(y - R + r, 0), H - 1);
        const uint32_t v = img[(int64_t)yy * pitch + xa];
        if (r < 4)
            w0 |= v << (8 * r);
        else
            w1 = v;
    }
    w0 ^= N == 5 ? 0x80808080u : 0x00808080u;
    if (N == 5) w1 ^= 0x80u;
    int s = __dp4a((int)w0, 0x01010101, 640), q = __dp4a((int)w0, (int)w0, 0);
    if (N == 5) {
        const int b = (int)(signed char)w1;
        s += b;
        q += b * b;
    }
    const uint32_t v = (uint32_t)q + ((uint32_t)s << 19);
    uint32_t t = v + __shfl_up_sync(0xFFFFFFFFu, v, 1);
    if (N == 5) {
        t += __shfl_up_sync(0xFFFFFFFFu, t, 2);
        t += __shfl_up_sync(0xFFFFFFFFu, v, 4);
    } else {
        t += __shfl_up_sync(0xFFFFFFFFu, v, 2);
    }
    sum = t;
    return make_uint2(w0, w1);
}

// Patch sum S' (of the shifted pixels) and V = n Sxx - S'^2 from pack_column's word.
template <int N>
__device__ __forceinline__ void patch_stats(uint32_t sum, int &s, int &v)
{
    s = (int)(sum >> 19) - 640 * N;
    v = N * N * (int)(sum & 0x7FFFFu) - s * s;
}

// What the lanes of one label stream share: the block's staging and constants.
struct CostBlock {
    const int4 *e1;       // I1 by staged column: packed column, then S' and V (floats) of the
                          // centre R columns before it
    const float4 *st0;    // I0 by pixel: -S', 2 S, S^2 + c1, V + c2
    const int2 *col0;     // I0 by staged column: packed column; the second word's upper half
                          // holds the window start of the pixel R columns before it and, in
                          // its sign bit, whether that differs from the previous pixel's
    int umax, nb, na;
    int Dw, Dws;
    int stride;           // bytes per pixel of the cost volume
    int nq;               // wide volumes: cost words per lane
    int imin;             // entries before it belong to matches left of the right image
    int c1, c2;
    int *err;
};

// One lane's stream over the pixels xs .. xe - 1 (segment-relative).  The lane owns the
// label u = lo + rel, rel = (slot - lo) mod Dws, of each pixel's window [lo, lo + Dw): its
// disparity stays the same when the window moves, except on the few lanes where the window
// wraps.  The cross sum Sxy follows from pixel to pixel by one entering and one leaving
// column product, kept in a register ring; a lane whose disparity changed sums the previous
// pixel's products anew.  Sxy carries kRound23Bits, so that its bits are a float and no
// conversion is needed.  Nodes whose estimate is too close to an integer are noted and
// decided after each chunk of N pixels.  WIN: the level has windows.  EDGE: some matches fall
// left of the right image or some labels are padding (cost 255).  ST: Dws as a constant, 0:
// B.Dws.  ORD: byte order of a pixel - 0 by label, 1 the wide order and stride (levels without
// windows), 2 the order of 48 labels with byte sums.
template <int N, int ST, int ORD, bool WIN, bool EDGE>
__device__ __forceinline__ void cost_stream(const CostBlock &B, int xs, int xe, int slot,
                                            uint8_t *out)
{
    constexpr int R = N / 2, n = N * N, NR = N;
    const int M = ST ? ST : B.Dws;
    const int MS = ORD == 1 ? B.stride : M;       // bytes per pixel
    const float c1f = (float)B.c1, c2f = (float)B.c2;
    auto window = [&](int x) { return (B.col0[x + 1 + 2 * R].y >> 16) & 0x3FFF; };
    auto label = [&](int lo) {   // rel
        if (ST && (ST & (ST - 1)) == 0) return (slot - lo) & (ST - 1);
        return (int)((unsigned)(slot - lo + (1023 / M + 1) * M) % (unsigned)M);
    };
    // the entry of the column that enters at pixel x: e1 + x + off
    auto entry_off = [&](int lo, int rel) {
        return 1 + 2 * R + B.umax - lo - (EDGE ? min(rel, B.Dw - 1) : rel);
    };
    auto byte_of = [&](int rel) {
        return ORD == 1 ? wide_byte(rel, B.nq) : (ORD == 2 ? bytes48_of(rel) : rel);
    };
    // the integers of one node; exact cost
    auto exact_node = [&](int x) {
        const int lo = window(x), rel = label(lo), off = entry_off(lo, rel);
        int q = 255;
        if (!EDGE || (x + off >= B.imin && rel < B.Dw)) {
            int sxy = 0;
#pragma unroll 1
            for (int d = 0; d < NR; ++d) {
                const int2 a = B.col0[x + 1 + d];
                const int2 b = *(const int2 *)&B.e1[x + off - 2 * R + d];
                sxy += colprod<N>(a.x, a.y, b.x, b.y);
            }
            const float4 s0 = B.st0[x];
            const int4 b = B.e1[x + off];
            const int s1 = (int)__int_as_float(b.z);
            const int A2 = 2 * (n * sxy + (int)s0.x * s1) + B.c2;
            const int sx = (int)(0.5f * s0.y), sy = s1 + 128 * n;
            const int vx = (int)(s0.w - c2f), vy = (int)__int_as_float(b.w);
            const float num = fmaf(s0.y, (float)sy, c1f) * (float)A2;
            const float den = fmaf((float)sy, (float)sy, s0.z) * (s0.w + (float)vy);
            q = ssim_exact((int)(127.5f - 127.5f * (num / den)), A2, sx, vx, sy, vy, B.c1, B.c2);
        }
        out[x * MS + byte_of(rel)] = (uint8_t)q;
    };

    const int xc = xs + (xe - xs) / NR * NR;      // whole chunks end here
    if (xs < xc) {
        int ring[NR], sxy = 0, off = 0, rel = 0;
        // the products of the pixel before x with the label of x; slot (j + d) mod N of the
        // ring holds column d, which the next pixels' entering columns replace in turn
        auto start = [&](int x, int j) {
            sxy = kRound23Bits;
            if (!MPV_IN(B.err, x >= 0 && x + 2 * R < B.na && x - 1 + off - 2 * R >= 0 &&
                                   x - 1 + off < B.nb, 10))
                return;
#pragma unroll
            for (int d = 0; d < NR; ++d) {
                const int2 a = B.col0[x + d];
                const int2 b = *(const int2 *)&B.e1[x - 1 + off - 2 * R + d];
                const int p = colprod<N>(a.x, a.y, b.x, b.y);
                ring[(j + d) % NR] = p;
                sxy += p;
            }
        };
        {
            const int lo = window(xs);
            rel = label(lo);
            off = entry_off(lo, rel);
            start(xs, 0);
        }
        const int2 *c0 = B.col0 + xs + 1 + 2 * R;   // entering I0 column of the chunk's first
        const int4 *e = B.e1 + xs + off;            // pixel, and its I1 entry
        const float4 *st = B.st0 + xs;
        unsigned po = (unsigned)(xs * MS + byte_of(rel));
        int pad = EDGE ? (rel < B.Dw ? B.imin : 0x7FFFFFFF) - off : 0;
        for (int xb = xs; xb < xc; xb += NR) {
            unsigned bad = 0;
#pragma unroll
            for (int j = 0; j < NR; ++j) {
                const int2 a = c0[j];
                if (WIN && a.y < 0) {   // the window moved
                    const int lo = (a.y >> 16) & 0x3FFF;
                    const int r = label(lo), o = entry_off(lo, r);
                    po += (unsigned)(byte_of(r) - byte_of(rel));
                    rel = r;
                    if (o != off) {
                        e += o - off;
                        off = o;
                        start(xb + j, j);
                    }
                    if (EDGE) pad = (rel < B.Dw ? B.imin : 0x7FFFFFFF) - off;
                }
                int4 b = make_int4(0, 0, 0, 0);
                if (MPV_IN(B.err, xb + j + off >= 2 * R && xb + j + off < B.nb &&
                                      xb + j + 1 + 2 * R < B.na, 10))
                    b = e[j];
                const int pr = colprod<N>(a.x, a.y, b.x, b.y);
                sxy += pr - ring[j];
                ring[j] = pr;
                const float4 s0 = st[j];
                const float s1 = __int_as_float(b.z), v1 = __int_as_float(b.w);
                const float nsxy = fmaf((float)n, __int_as_float(sxy), -(float)n * kRound23);
                const float cov = fmaf(s0.x, s1, nsxy);          // n Sxy - Sx Sy, exact
                const float S1 = s1 + 128.0f * n;
                const float num = fmaf(s0.y, S1, c1f) * fmaf(2.0f, cov, c2f);
                const float den = fmaf(S1, S1, s0.z) * (s0.w + v1);
                float r;
                asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(den));
                // (t >= 0 holds exactly: an estimate below 0.0002, the cost of equal patches,
                // is decided already)
                const float t = fmaxf(fmaf(-127.5f, num * r, 127.0f), -0.4998f);
                const float m = t + kRound23;    // its low byte is floor(t + 1/2)
                if (fabsf(t - (m - kRound23)) > kQuotientSafe) bad |= 1u << j;
                int q = __float_as_int(m);
                if (EDGE) q = xb + j < pad ? 255 : q;
                out[po + (unsigned)(j * MS)] = (uint8_t)q;
            }
            c0 += NR;
            e += NR;
            st += NR;
            po += (unsigned)(NR * MS);
            while (bad) {
                exact_node(xb + __ffs(bad) - 1);
                bad &= bad - 1;
            }
        }
    }
    for (int x = max(xs, xc); x < xe; ++x) exact_node(x);   // fewer than N (row ends)
}

// One block of the cost kernel: row segment bx (of seg pixels), row by, view bz; smem: the
// block's dynamic shared memory (cost_smem_layout bytes).
template <int N, int ST, int ORD>
__device__ __forceinline__ void cost_body(const LevelArgs &a, int uspan_max, int seg, int bx,
                                          int by, int bz, int tid, unsigned char *smem)
{
    constexpr int R = N / 2, n = N * N;
    const int view = bz;
    const ViewLevel &V = a.v[view];
    const int W = a.W, H = a.H, Dw = a.Dw, Dws = ST ? ST : a.Dws;
    const int y = by;
    const int x0 = bx * seg;
    const int npx = min(seg, W - x0);
    if (npx <= 0) return;   // (whole block)

    __shared__ int lo_s[kSegPix];
    __shared__ int red[2];
    const CostSmem L = cost_smem_layout(R, uspan_max);
    int4 *e1 = (int4 *)(smem + L.off_e1);
    float4 *st0 = (float4 *)(smem + L.off_st0);
    uint2 *col0 = (uint2 *)(smem + L.off_col0);
    const int lane = tid & 31, warp = tid >> 5;

    const int stride = ORD == 1 ? 4 * a.wide_g * a.wide_nq : Dws;
    if (ORD == 1) {   // this segment's byte sums start at zero, the bytes of no label at cost 255
        const int64_t at = ((int64_t)y * W + x0) * stride;     // a multiple of 16
        const int n16 = npx * (stride / 16);
        uint4 *ez = (uint4 *)(V.E + at), *cz = (uint4 *)(V.C + at);
        const uint32_t f = 0xFFFFFFFFu;
        for (int i = tid; i < n16; i += kCostThreads) {
            ez[i] = make_uint4(0u, 0u, 0u, 0u);
            if (Dws < stride) cz[i] = make_uint4(f, f, f, f);
        }
    } else if (a.bytes) {
        uint4 *ez = (uint4 *)(V.E + ((int64_t)y * W + x0) * Dws);
        const int n16 = npx * Dws / 16;
        for (int i = tid; i < n16; i += kCostThreads) ez[i] = make_uint4(0u, 0u, 0u, 0u);
    } else if (a.zero_s) {   // this segment's summed energies start at zero (16-byte stores)
        uint4 *sz = (uint4 *)(V.S + ((int64_t)y * W + x0) * Dws);
        const int n16 = npx * Dws / 8;     // Dws is a multiple of 16
        for (int i = tid; i < n16; i += kCostThreads) sz[i] = make_uint4(0u, 0u, 0u, 0u);
    }
    int umin = 0, umax = Dw - 1;
    if (V.lo) {   // the segment's window starts and their range
        if (tid == 0) {
            red[0] = 0x7FFFFFFF;
            red[1] = 0;
        }
        __syncthreads();
        int l0 = 0x7FFFFFFF, l1 = 0;
        for (int i = tid; i < npx; i += kCostThreads) {
            const int l = (int)V.lo[(int64_t)y * W + x0 + i];
            lo_s[i] = l;
            l0 = min(l0, l);
            l1 = max(l1, l);
        }
        l0 = __reduce_min_sync(0xFFFFFFFFu, l0);
        l1 = __reduce_max_sync(0xFFFFFFFFu, l1);
        if (lane == 0) {
            atomicMin(&red[0], l0);
            atomicMax(&red[1], l1);
        }
        __syncthreads();
        umin = red[0];
        umax = red[1] + Dw - 1;
    }
    const int uspan = umax - umin;
    const int b0 = x0 - R - 1 - umax;       // first staged I1 column
    const int a0 = x0 - R - 1;              // first staged I0 column
    const int nb = npx + 2 * R + 1 + uspan; // staged I1 columns
    const int na = npx + 2 * R + 2;

    // every warp packs 32 columns at a time, the first 2 R of them for their sums only
    constexpr int kOut = 32 - 2 * R;
    for (int c = warp * kOut; c < na; c += kCostWarps * kOut) {
        const int i = c + lane - 2 * R;
        uint32_t sum;
        uint2 col = pack_column<N>(V.I0, V.pitch0, W, H, y, a0 + i, sum);
        if (lane < 2 * R || i >= na) continue;
        const int x = i - 1 - 2 * R;        // the pixel at which this column enters
        if (x >= 0 && x < npx) {
            int s, v;
            patch_stats<N>(sum, s, v);
            const float S = (float)(s + 128 * n);
            st0[x] = make_float4(-(float)s, 2.0f * S, fmaf(S, S, (float)a.c1), (float)(v + a.c2));
            if (V.lo) {
                const uint32_t l = (uint32_t)lo_s[x];
                col.y |= l << 16;
                if (x > 0 && l != (uint32_t)lo_s[x - 1]) col.y |= 0x80000000u;
            }
        }
        col0[i] = col;
    }
    for (int c = warp * kOut; c < nb; c += kCostWarps * kOut) {
        const int i = c + lane - 2 * R;
        uint32_t sum;
        const uint2 col = pack_column<N>(V.I1, V.pitch1, W, H, y, b0 + i, sum);
        if (lane < 2 * R || i >= nb) continue;
        int s, v;
        patch_stats<N>(sum, s, v);          // (of no centre for the first 2 R columns)
        e1[i] = make_int4((int)col.x, (int)col.y, __float_as_int((float)s), __float_as_int((float)v));
    }
    __syncthreads();

    // (the entry of the centre at the image's first column lies R columns past it)
    const CostBlock B{e1, st0, (const int2 *)col0, umax, nb, na, Dw, Dws, stride, a.wide_nq, R - b0, a.c1, a.c2, a.err};
    // 32 labels of one pixel per warp step; a last group of 16 labels as two streams, half of
    // the warp's pixels each (48 labels in 1.5 passes over the pixels instead of 2)
    const int per_warp = seg / kCostWarps;
    uint8_t *out = V.C + ((int64_t)y * W + x0) * stride;
    const bool edge = x0 - umax < 0 || Dw < Dws;
    for (int k0 = 0; k0 < Dws; k0 += 32) {
        const int half = Dws - k0 < 32;      // a group of 16
        const int len = half ? per_warp / 2 : per_warp;
        const int xs = warp * per_warp + (half && lane >= 16 ? len : 0);
        const int xe = min(xs + len, npx);
        const int slot = k0 + (half ? lane & 15 : lane);
        if (ORD != 1 && V.lo) {
            if (edge) cost_stream<N, ST, ORD, true, true>(B, xs, xe, slot, out);
            else cost_stream<N, ST, ORD, true, false>(B, xs, xe, slot, out);
        } else {
            if (edge) cost_stream<N, ST, ORD, false, true>(B, xs, xe, slot, out);
            else cost_stream<N, ST, ORD, false, false>(B, xs, xe, slot, out);
        }
    }
}

}  // namespace

}  // namespace mpv
