// agg_rows.cuh -- the row directions of levels with byte sums and label strides of 16 or 32.
//
// The row paths are a level's longest chains (W steps): on all but the largest levels their
// time per step is the launch's.  With register prefetch that time was the latency of a load,
// whatever the arithmetic: the loads in flight share a warp's few scoreboards, so a step waited
// for loads issued a step before.  Here a path's costs and window starts come by asynchronous
// copies, kRowChunk pixels at a time (16-byte pieces of 4 rows), one chunk ahead, and a step
// reads shared memory only.
//
// Bound: the chain of one step (77 instructions, 208 cycles with windows when the warp is alone
// on its scheduler; 2.2 of 2.7 cycles per instruction are issue and fixed latencies).
//
// 8 lanes per path, KW words of two labels per lane, 4 paths per warp, as agg_stencil_body
// (same arithmetic, radius at most 2).  With windows the predecessor passes through shared
// memory on every step together with the lanes' minima, behind the same warp barrier, and is
// read back at the step's window shift: no vote, branch, second barrier or halo exchange.
#pragma once
#include "agg_stencil.cuh"

namespace mpv {

namespace {

constexpr int kRowChunk = 8;

template <int KW, bool WIN>
struct RowSmem {                     // one warp's shared memory, in bytes
    static constexpr int DWP = 16 * KW;                       // labels (bytes) per pixel
    static constexpr int ROWB = kRowChunk * DWP + DWP;        // a row's chunk; the pad spreads rows
    static constexpr int PADL = 40;                           // absent labels around a path
    static constexpr int PATHW = (2 * PADL + DWP + 63) / 64 * 32;   // words, a multiple of 32
    static constexpr int off_lo = 2 * 4 * ROWB;               // two chunks of 4 rows
    static constexpr int off_sh = off_lo + (WIN ? 2 * 4 * 32 : 0);   // the chunk's shifts
    static constexpr int off_min = off_sh + (WIN ? 4 * kRowChunk * 8 : 0);
    static constexpr int off_a = off_min + 2 * 32 * 4;
    static constexpr int abuf = (4 * PATHW + 32) * 4;
    static constexpr int bytes = (off_a + (WIN ? 2 * abuf : 0) + 15) / 16 * 16;
    // first word of a path's buffer: lanes KW words apart, paths in different banks
    __device__ static constexpr int path_word(int p)
    {
        return p * PATHW + p % KW + p / KW * (8 * KW) % 32;
    }
};

__device__ __forceinline__ void row_copy(uint32_t dst, const void *src, int bytes, bool on)
{
    if (bytes == 16)
        asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %2, 0;\n"
                     " @p cp.async.cg.shared.global [%0], [%1], 16;\n}" ::"r"(dst),
                     "l"(src), "r"((int)on)
                     : "memory");
    else
        asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %2, 0;\n"
                     " @p cp.async.ca.shared.global [%0], [%1], 4;\n}" ::"r"(dst),
                     "l"(src), "r"((int)on)
                     : "memory");
}

// The rows 4 grp .. 4 grp + 3 in direction (DX, 0); smem: this warp's RowSmem.
template <int KW, bool WIN, int DX>
__device__ __forceinline__ void row_bytes_body(const LevelArgs &a, int grp, int view, int lane,
                                               unsigned char *smem)
{
    using RS = RowSmem<KW, WIN>;
    constexpr int DWP = RS::DWP, K = 2 * KW, NE = KW + 2, CH = kRowChunk;
    const int W = a.W, H = a.H;
    if (4 * grp >= H) return;             // (warp-uniform)
    const int gl = lane & 7, path = lane >> 3;
    const bool valid = 4 * grp + path < H;
    const int y = min(4 * grp + path, H - 1);
    const ViewLevel &V = a.v[view];
    const int nch = (W + CH - 1) / CH;

    // pieces of a chunk: 16 bytes, in the order (row, position); rows past the image repeat the
    // last one
    constexpr int PPR = CH * DWP / 16, NP = 4 * PPR / 32;      // per row, per lane
    const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(smem);
    auto issue = [&](int c) {             // chunk c into stage c & 1
        const int x0 = DX > 0 ? c * CH : W - CH - c * CH;      // (negative at the left edge)
        const uint32_t st = sbase + (c & 1) * (4 * RS::ROWB);
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            const int e = lane + 32 * i, r = e / PPR, q = e % PPR;
            const int yr = min(4 * grp + r, H - 1), x = x0 + q * 16 / DWP;
            const int64_t at = ((int64_t)yr * W + x0) * DWP + q * 16;
            const bool on = x >= 0 && x < W;
            row_copy(st + r * RS::ROWB + q * 16, V.C + at, 16,
                     on && MPV_IN(a.err, at >= 0 && at + 16 <= (int64_t)W * H * DWP, 15));
        }
        if (WIN) {                        // 8 window starts: five aligned words hold them
            const int r = lane / 5, k = lane - 5 * r;
            const int yr = min(4 * grp + r, H - 1);
            const int64_t at = ((((int64_t)yr * W + x0) * 2) & ~(int64_t)3) + 4 * k;
            const bool on = lane < 20 && at >= 0 && at < (int64_t)W * H * 2;
            row_copy(sbase + RS::off_lo + (c & 1) * 128 + r * 32 + 4 * k, (const uint8_t *)V.lo + at,
                     4, on && MPV_IN(a.err, (at & 3) == 0 && r < 4 && 4 * k < 32, 16));
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };

    const uint32_t INF2 = kInf16 * 0x10001u;
    const uint32_t T = (uint32_t)a.trunc;
    const uint32_t Tx2 = T * 0x10001u;
    const uint32_t E1 = min((uint32_t)a.p1, T) * 0x10001u;
    const uint32_t E2 = min(2 * (uint32_t)a.p1, T) * 0x10001u;
    // labels at or beyond Dw are padding: never a predecessor
    uint32_t pad[KW];
#pragma unroll
    for (int i = 0; i < KW; ++i) {
        const int k0 = gl * K + 2 * i;
        pad[i] = INF2 & ((k0 < a.Dw ? 0u : 0x0000FFFFu) | (k0 + 1 < a.Dw ? 0u : 0xFFFF0000u));
    }
    uint32_t *minb = (uint32_t *)(smem + RS::off_min);
    uint32_t *ab = (uint32_t *)(smem + RS::off_a) + RS::path_word(path);
    constexpr int ABW = RS::abuf / 4;     // words from one parity's buffers to the other's
    if (WIN) {
        for (int i = lane; i < 2 * ABW; i += 32) ((uint32_t *)(smem + RS::off_a))[i] = INF2;
        __syncwarp();
    }

    const unsigned char *cs = smem + path * RS::ROWB + gl * K;
    // (the parity of a row's first pixel is the same in every chunk)
    const int x00 = DX > 0 ? 0 : W - CH;
    const unsigned char *ls = smem + RS::off_lo + path * 32 + ((((int64_t)y * W + x00) & 1) ? 2 : 0);
    uint8_t *ep = V.E + ((int64_t)y * W + (DX > 0 ? 0 : W - 1)) * DWP + (KW == 1 ? gl / 2 * 4 : gl * K);
    const bool adds = valid && (KW > 1 || (gl & 1) == 0);

    uint32_t A[KW];
#pragma unroll
    for (int i = 0; i < KW; ++i) A[i] = INF2;     // no predecessor: E = 0 at the first pixel
    int last_lo = 0;                     // window start of lane gl's pixel in the chunk before
    issue(0);
    for (int c = 0; c < nch; ++c) {
        if (c + 1 < nch) issue(c + 1);
        else asm volatile("cp.async.commit_group;" ::: "memory");
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncwarp();                 // chunk c has arrived for every lane
        const unsigned char *cc = cs + (c & 1) * (4 * RS::ROWB);
        const int n = min(CH, W - c * CH);
        if (WIN) {
            // lane gl prepares step gl of its path: the first word and the half-word selection
            // at which the step's labels lie in the predecessor's frame
            const unsigned char *lc = ls + (c & 1) * 128;
            const int lo = *(const uint16_t *)(lc + (DX > 0 ? gl : CH - 1 - gl) * 2);
            int lp = __shfl_up_sync(kFull, lo, 1, 8);
            const int before = __shfl_sync(kFull, last_lo, CH - 1, 8);
            if (gl == 0) lp = c == 0 ? lo : before;
            last_lo = lo;
            const int sc = min(max(lo - lp, -(DWP + 2)), DWP + 2);
            ((uint2 *)(smem + RS::off_sh))[lane] =
                make_uint2((unsigned)((RS::PADL - 2 + sc) >> 1), (sc & 1) ? 0x5432u : 0x3210u);
            __syncwarp();
        }
#pragma unroll
        for (int u = 0; u < CH; ++u) {
            // (the last chunk's steps past the row compute on leftovers and add nothing)
            const int j = DX > 0 ? u : CH - 1 - u;         // position in the chunk
            uint32_t cv[KW];
            if (KW == 1) {
                cv[0] = __byte_perm((uint32_t)*(const uint16_t *)(cc + j * DWP), 0u, 0x4140);
            } else {
#pragma unroll
                for (int i = 0; i < KW / 2; ++i) {
                    const uint32_t w = ((const uint32_t *)(cc + j * DWP))[i];
                    cv[2 * i] = __byte_perm(w, 0u, 0x4140);
                    cv[(2 * i + 1) % KW] = __byte_perm(w, 0u, 0x4342);
                }
            }
            uint2 sh = make_uint2(0u, 0u);
            if (WIN) sh = ((const uint2 *)(smem + RS::off_sh))[path * CH + u];
            // the lanes' minima (and the predecessor), exchanged behind one barrier; buffers
            // alternate by step parity
            uint32_t m2 = A[0];
#pragma unroll
            for (int i = 1; i < KW; ++i) m2 = __vminu2(m2, A[i]);
            m2 = __vminu2(m2, __byte_perm(m2, m2, 0x1032));
            uint32_t *aw = ab + (u & 1) * ABW;
            if (WIN) {
#pragma unroll
                for (int i = 0; i < KW; ++i) aw[RS::PADL / 2 + gl * KW + i] = A[i];
            }
            uint32_t *mw = minb + (u & 1) * 32;
            mw[lane] = m2;
            __syncwarp();
            const uint4 q0 = ((const uint4 *)(mw + path * 8))[0];
            const uint4 q1 = ((const uint4 *)(mw + path * 8))[1];
            uint32_t E[NE];
            if (WIN) {
                // labels -2 .. K + 1 of this step's window in the predecessor's frame
                uint32_t Wd[NE + 1];
                const bool ok = MPV_IN(a.err, (int)sh.x >= 0 && (int)sh.x + gl * KW + NE < RS::PATHW, 3);
                const uint32_t *pw = aw + gl * KW + sh.x;
#pragma unroll
                for (int i = 0; i <= NE; ++i) Wd[i] = ok ? pw[i] : INF2;
#pragma unroll
                for (int i = 0; i < NE; ++i) E[i] = __byte_perm(Wd[i], Wd[i + 1], sh.y);
            } else {
                const uint32_t l = __shfl_up_sync(kFull, A[KW - 1], 1, 8);
                const uint32_t r = __shfl_down_sync(kFull, A[0], 1, 8);
                E[0] = gl == 0 ? INF2 : l;
                E[NE - 1] = gl == 7 ? INF2 : r;
#pragma unroll
                for (int i = 0; i < KW; ++i) E[1 + i] = A[i];
            }
            uint32_t SH[NE - 1];
#pragma unroll
            for (int i = 0; i < NE - 1; ++i) SH[i] = shift1(E[i], E[i + 1]);
            {
                const uint32_t r0 = __vimin3_u16x2(q0.x, q0.y, q0.z);
                const uint32_t r1 = __vimin3_u16x2(q0.w, q1.x, q1.y);
                m2 = __vimin3_u16x2(r0, r1, __vminu2(q1.z, q1.w));
            }
            const uint32_t cap = m2 + Tx2;
            uint32_t inc[KW];
#pragma unroll
            for (int i = 0; i < KW; ++i) {
                uint32_t m = __vimin3_u16x2(E[1 + i], SH[i] + E1, SH[i + 1] + E1);
                m = __vimin3_u16x2(m, E[i] + E2, E[i + 2] + E2);
                inc[i] = __vminu2(m, cap) - m2;            // per half: no borrow, at most T
                A[i] = (cv[i] + inc[i]) | pad[i];
            }
            uint32_t out;
            if (KW == 1) {       // two lanes' labels make a word
                const uint32_t b = __byte_perm(inc[0], 0u, 0x4420);
                out = b | (__shfl_down_sync(kFull, b, 1) << 16);
            } else {
                out = __byte_perm(inc[0], inc[1 % KW], 0x6420);
            }
            uint8_t *dst = ep + u * DX * DWP;
            if (adds && u < n &&
                MPV_IN(a.err, dst >= V.E && dst + 4 <= V.E + (int64_t)W * H * DWP, 17))
                atomicAdd((unsigned int *)dst, out);
        }
        ep += CH * DX * DWP;
        __syncwarp();                 // every lane is done with the stage that is filled next
    }
}

}  // namespace

}  // namespace mpv
