// agg_wide.cu -- the summed directional passes of wide full-range levels (no windows).
//
// Same recursion as aggregate.cu: L = C + E, E(p,u) = M'(u) - min_v L(p-r,v), for label ranges
// beyond the packed stencil's 64.  The directions add E as bytes (byte sums, see
// mpv_internal.cuh).
//
// G lanes own a path, 4 NQ consecutive labels each, packed two per register as (label w, label
// w + 2 NQ): the neighbours of a register's labels are the next registers, only its ends need
// lane exchanges.  The byte order of C and E follows the registers.  The labels past Dw carry
// cost 255, so that their energies are at least 255 and, while the path minimum is at most
// 255 - T, no candidate they offer is below the cap min_v L + T; a path minimum above that
// masks them explicitly (a branch on a warp vote, only where there are such labels).
//
// A warp (one per block, so that positions are warp-uniform registers) owns 32/G paths on
// adjacent pixels: rows for the row directions, columns for the others.  Diagonal paths wrap
// around the image's side and start again there, so every warp of a direction has the same
// length and its pixels stay adjacent (columns beyond the image are idle).  Costs arrive by
// 8-byte asynchronous copies kStages - 1 steps ahead; the packed E of a step is transposed
// through shared memory so that each 64-bit reduction covers 256 contiguous bytes.
//
// Measured on a GB300, 1280x720, 128 labels, 8 paths, both views: 785 us (8 lanes 826 us)
// against 4,600 us for one warp per path on int32 scans with 32-bit reductions into 16-bit
// sums (agg_general, kept for what lies outside the rule in wide_shape).  Bound: HBM (4.1 GB
// of DRAM traffic, 5.2 TB/s; the volumes are four times the L2, and eight directions read C and
// add to E); issue slots 61 %, ALU pipe 45 % active.  4 and 8 cost stages measure the same; the
// step unrolled by 4 lost to instruction fetches.
#include "volume_layout.cuh"

namespace mpv {

namespace {

constexpr unsigned kAll = 0xFFFFFFFFu;
constexpr int kStages = 4;      // cost stages in shared memory; copies run 3 steps ahead

// Warps of one row, column and diagonal direction of one view.
struct WideGrid {
    int nrow, ncol, ndia;
};

__device__ __forceinline__ uint32_t wide_smem(const void *p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

// (predicated instructions: a branch per copy or reduction costs more than they do)
__device__ __forceinline__ void wide_copy8(uint32_t dst, const uint8_t *src, bool on)
{
    asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %2, 0;\n"
                 " @p cp.async.ca.shared.global [%0], [%1], 8;\n}" ::"r"(dst),
                 "l"(src), "r"((int)on)
                 : "memory");
}
__device__ __forceinline__ void wide_add8(uint8_t *dst, unsigned long long v, bool on)
{
    asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %2, 0;\n"
                 " @p red.global.add.u64 [%0], %1;\n}" ::"l"(dst),
                 "l"(v), "r"((int)on)
                 : "memory");
}

// Sets the sentinel bit of every label of the lane whose keep bit is clear; bit i of `keep` is
// label i of the lane.
template <int NQ>
__device__ __forceinline__ void wide_mask(uint32_t (&A)[2 * NQ], uint32_t keep)
{
    const uint32_t inv = ~keep;
#pragma unroll
    for (int w = 0; w < 2 * NQ; ++w) {
        const uint32_t lo = w <= 14 ? inv << (14 - w) : inv >> (w - 14);
        const int hs = 30 - (w + 2 * NQ);
        const uint32_t hi = hs >= 0 ? inv << hs : inv >> -hs;
        A[w] |= (lo & 0x4000u) | (hi & 0x40000000u);
    }
}

// The scan of one warp's paths.  MODE 0: rows (direction (sx, 0)), 1: columns (0, sy), 2:
// diagonals (sx, sy); grp: which paths.  Path i of the warp is active while 0 <= c + i < lim;
// its pixel is i rows or columns past the warp's position.  Rows: c is the first row, fixed.
// Columns: c is the first column, fixed.  Diagonals: c moves by sx and wraps at the ends of wv
// columns.
template <int G, int NQ, int MODE>
__device__ __forceinline__ void wide_scan(const LevelArgs &a, const uint8_t *__restrict__ C,
                                          uint8_t *__restrict__ E, int sx, int sy, int grp, int wv,
                                          unsigned char *cbuf, unsigned char *ebuf)
{
    constexpr int P = 32 / G;             // paths per warp
    constexpr int KW = 2 * NQ;            // packed registers per lane
    constexpr int R = 4 * G * NQ;         // labels (bytes) per pixel
    constexpr int STEP = 128 * NQ;        // bytes of one step of the warp
    constexpr int EPP = R / 8;            // 8-byte elements per pixel
    constexpr int NE = (NQ + 1) / 2;      // elements per lane and step
    constexpr int PF = kStages - 1;
    const int W = a.W, H = a.H;
    const int lane = threadIdx.x, l = lane % G, path = lane / G;
    const int n = MODE == 0 ? W : H;
    const int lim = MODE == 0 ? H : W;
    // pixels from one step to the next, and the position of the first step
    const int dpix = MODE == 0 ? sx : sy * W + (MODE == 2 ? sx : 0);
    const int enter = sx > 0 ? 0 : W - 1;    // column at which a diagonal path starts again
    int c = MODE == 2 ? P * grp - (P - 1) : P * grp;
    int ca = c;                              // the same PF steps ahead
    const int64_t base = MODE == 0 ? (int64_t)c * W + (sx > 0 ? 0 : W - 1)
                                   : (int64_t)(sy > 0 ? 0 : H - 1) * W + c;

    // the lane's elements of a step: lane + 32 k in the order (path, 8-byte element); columns
    // and diagonals have them contiguous in memory
    const bool last = 32 * NE == 16 * NQ || wide_elem(NQ, lane, NE - 1);
    auto elem = [&](int k) { return k + 1 < NE || last; };
    unsigned eo[MODE == 0 ? NE : 1];
    bool eact[MODE == 0 ? NE : 1];
    if (MODE == 0) {
#pragma unroll
        for (int k = 0; k < NE; ++k) {
            const int e = lane + 32 * k, p = e / EPP;
            eo[k % (MODE == 0 ? NE : 1)] = (unsigned)(p * W * R + (e - p * EPP) * 8);
            eact[k % (MODE == 0 ? NE : 1)] = elem(k) && c + p < H;
        }
    }
    const uint8_t *pc = C + base * R + (MODE == 0 ? 0 : lane * 8);
    uint8_t *pe = E + base * R + (MODE == 0 ? 0 : lane * 8);
    const int64_t dstep = (int64_t)dpix * R;
    const int ep0 = lane / EPP, ep1 = (lane + 32) / EPP, ep2 = (lane + 64) / EPP,
              ep3 = (lane + 96) / EPP;
    auto epath = [&](int k) { return k == 0 ? ep0 : k == 1 ? ep1 : k == 2 ? ep2 : ep3; };

    const uint32_t csm = wide_smem(cbuf) + lane * 8;
    // whether element k belongs to a path that is active at first column cc
    auto has = [&](int k, int cc) {
        if (MODE == 0) return eact[k % (MODE == 0 ? NE : 1)];
        return elem(k) && (unsigned)(cc + epath(k)) < (unsigned)lim;
    };
    auto at = [&](int k) -> unsigned {
        return MODE == 0 ? eo[k % (MODE == 0 ? NE : 1)] : (unsigned)(k * 256);
    };
    // costs of the step PF ahead (inside the scan while more)
    auto fetch = [&](bool more, unsigned stage) {
        if (more) {
#pragma unroll
            for (int k = 0; k < NE; ++k) {
                const bool on = has(k, ca);
                const uint8_t *src = pc + at(k);
                wide_copy8(csm + stage * STEP + k * 256, src,
                           on && MPV_IN(a.err, src >= C && src + 8 <= C + (int64_t)W * H * R, 12));
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        pc += dstep;
        if (MODE == 2) {
            ca += sx;
            if (ca > wv - P) {
                ca -= wv;
                pc -= (int64_t)wv * R;
            } else if (ca < -(P - 1)) {
                ca += wv;
                pc += (int64_t)wv * R;
            }
        }
    };

    const uint32_t INF2 = kInf16 * 0x10001u;
    const uint32_t T = (uint32_t)a.trunc;
    const uint32_t Tx2 = T * 0x10001u;
    const uint32_t E1 = min((uint32_t)a.p1, T) * 0x10001u;
    const uint32_t E2 = min(2 * (uint32_t)a.p1, T) * 0x10001u;
    const uint32_t safe_min = 255u - T;
    const bool pads = a.Dw < R;
    const int mine = a.Dw - l * 4 * NQ;         // labels of the lane that exist
    const uint32_t keep = mine >= 32 ? kAll : (mine <= 0 ? 0u : (1u << mine) - 1u);
    const int left = (lane & ~(G - 1)) | ((lane + G - 1) & (G - 1));
    const int right = (lane & ~(G - 1)) | ((lane + 1) & (G - 1));

#pragma unroll 1
    for (int u = 0; u < PF; ++u) fetch(u < n, u);
    uint32_t A[KW];
#pragma unroll
    for (int w = 0; w < KW; ++w) A[w] = INF2;   // no predecessor: E = 0 at the first pixel
    int cp = c;                                 // c of the previous step, at pe

    // the sums of the previous step (stored before the last barrier) into E
    auto flush = [&](unsigned par) {
        const unsigned long long *src = (const unsigned long long *)(ebuf + par * STEP) + lane;
#pragma unroll
        for (int k = 0; k < NE; ++k) {
            // (the element itself, not only its reduction: with an odd NQ the last 16 lanes'
            // would be past the step)
            unsigned long long v = 0;
            if (elem(k) && MPV_IN(a.err, lane + 32 * k < 16 * NQ, 13)) v = src[32 * k];
            const bool on = has(k, cp);
            uint8_t *dst = pe + at(k);
            wide_add8(dst, v, on && MPV_IN(a.err, dst >= E && dst + 8 <= E + (int64_t)W * H * R, 14));
        }
        pe += dstep;
        if (MODE == 2) {
            if (cp + sx > wv - P) pe -= (int64_t)wv * R;
            else if (cp + sx < -(P - 1)) pe += (int64_t)wv * R;
        }
    };
    // the path's minimum, in both halves
    auto minimum = [&]() {
        uint32_t v[KW];
#pragma unroll
        for (int w = 0; w < KW; ++w) v[w] = A[w];
        // three at a time, the partial minima in a tree
#pragma unroll
        for (int s = 1; s < KW; s *= 3)
#pragma unroll
            for (int w = 0; w < KW; w += 3 * s) {
                if (w + 2 * s < KW) v[w] = __vimin3_u16x2(v[w], v[w + s], v[w + 2 * s]);
                else if (w + s < KW) v[w] = __vminu2(v[w], v[w + s]);
            }
        uint32_t m = v[0];
        m = __vminu2(m, __byte_perm(m, m, 0x1032));
#pragma unroll
        for (int o = 1; o < G; o <<= 1) m = __vminu2(m, __shfl_xor_sync(kAll, m, o));
        return m;
    };

    // (one copy of the step: unrolled by 4, the three scans' code no longer fits the
    // instruction caches of an SM whose few warps are all at different places)
#pragma unroll 1
    for (int t = 0; t < n; ++t) {
        const unsigned u = (unsigned)t % kStages;
        asm volatile("cp.async.wait_group %0;" ::"n"(PF - 1) : "memory");
        __syncwarp();    // step t's costs and step t - 1's sums are in shared memory
        if (t > 0) flush((t + 1) & 1);
        fetch(t + PF < n, (u + PF) % kStages);
        uint32_t cw[NQ];
        {
            const uint32_t *cs = (const uint32_t *)(cbuf + u * STEP) + lane * NQ;
            if (NQ % 4 == 0) {
#pragma unroll
                for (int k = 0; k < NQ; k += 4) {
                    const uint4 v = *(const uint4 *)(cs + k);
                    cw[k] = v.x;
                    cw[(k + 1) % NQ] = v.y;
                    cw[(k + 2) % NQ] = v.z;
                    cw[(k + 3) % NQ] = v.w;
                }
            } else if (NQ % 2 == 0) {
#pragma unroll
                for (int k = 0; k < NQ; k += 2) {
                    const uint2 v = *(const uint2 *)(cs + k);
                    cw[k] = v.x;
                    cw[(k + 1) % NQ] = v.y;
                }
            } else {
#pragma unroll
                for (int k = 0; k < NQ; ++k) cw[k] = cs[k];
            }
        }
        if (MODE == 2 && (unsigned)(enter - c) < (unsigned)P) {   // one path starts again
            if (enter - c == path) {
#pragma unroll
                for (int w = 0; w < KW; ++w) A[w] = INF2;
            }
        }
        uint32_t m2 = minimum();
        if (pads) {
            const bool act = (unsigned)(c + path) < (unsigned)lim;
            if (__any_sync(kAll, act && (m2 & 0xFFFFu) > safe_min)) {
                wide_mask<NQ>(A, keep);
                m2 = minimum();
            }
        }
        const uint32_t cap = m2 + Tx2;

        // the registers before the lane's first and after its last
        uint32_t l1 = __shfl_sync(kAll, A[KW - 1], left), l2 = __shfl_sync(kAll, A[KW - 2], left);
        uint32_t r1 = __shfl_sync(kAll, A[0], right), r2 = __shfl_sync(kAll, A[1], right);
        if (l == 0) l1 = l2 = INF2;          // no labels before the first,
        if (l == G - 1) r1 = r2 = INF2;      // after the last
        uint32_t X[KW + 4];
        X[0] = __byte_perm(l2, A[KW - 2], 0x5432);
        X[1] = __byte_perm(l1, A[KW - 1], 0x5432);
#pragma unroll
        for (int w = 0; w < KW; ++w) X[w + 2] = A[w];
        X[KW + 2] = __byte_perm(A[0], r1, 0x5432);
        X[KW + 3] = __byte_perm(A[1], r2, 0x5432);
        uint32_t e[KW];
#pragma unroll
        for (int w = 0; w < KW; ++w) {
            uint32_t m = __vimin3_u16x2(X[w + 2], X[w + 1] + E1, X[w + 3] + E1);
            m = __vimin3_u16x2(m, X[w] + E2, X[w + 4] + E2);
            e[w] = __vminu2(m, cap) - m2;          // per half: no borrow, at most T
        }
        uint32_t *es = (uint32_t *)(ebuf + (t & 1) * STEP) + lane * NQ;
#pragma unroll
        for (int k = 0; k < NQ; ++k) {
            A[2 * k] = __byte_perm(cw[k], 0u, 0x4140) + e[2 * k];
            A[2 * k + 1] = __byte_perm(cw[k], 0u, 0x4342) + e[2 * k + 1];
            es[k] = __byte_perm(e[2 * k], e[2 * k + 1], 0x6420);
        }
        cp = c;
        if (MODE == 2) {
            c += sx;
            if (c > wv - P) c -= wv;
            else if (c < -(P - 1)) c += wv;
        }
    }
    __syncwarp();
    flush((n - 1) & 1);
}

template <int G, int NQ>
__global__ void __launch_bounds__(32) agg_wide(LevelArgs a, WideGrid g)
{
    if (a.gate && *a.gate == 0) return;
    __shared__ __align__(16) unsigned char cbuf[kStages * 128 * NQ];
    __shared__ __align__(16) unsigned char ebuf[2 * 128 * NQ];
    // this warp's direction and paths: rows first (the longest), then columns, diagonals
    const int nv = a.nviews;
    int b = blockIdx.x;
    const int mode = b < 2 * nv * g.nrow ? 0 : (b < 2 * nv * (g.nrow + g.ncol) ? 1 : 2);
    b -= mode == 0 ? 0 : (mode == 1 ? 2 * nv * g.nrow : 2 * nv * (g.nrow + g.ncol));
    const int per = mode == 0 ? g.nrow : (mode == 1 ? g.ncol : g.ndia);
    const int d = b / (nv * per);            // direction of the mode
    b -= d * nv * per;
    const int view = b / per, grp = b - view * per;
    const uint8_t *C = view ? a.v[1].C : a.v[0].C;
    uint8_t *E = view ? a.v[1].E : a.v[0].E;
    const int wv = (32 / G) * g.ndia;
    if (mode == 0)
        wide_scan<G, NQ, 0>(a, C, E, d ? -1 : 1, 0, grp, wv, cbuf, ebuf);
    else if (mode == 1)
        wide_scan<G, NQ, 1>(a, C, E, 0, d ? -1 : 1, grp, wv, cbuf, ebuf);
    else
        wide_scan<G, NQ, 2>(a, C, E, (d & 1) ? -1 : 1, d < 2 ? 1 : -1, grp, wv, cbuf, ebuf);
}

constexpr int64_t kFewLanes = 1824;     // 12 warps per SM

WideGrid wide_grid(const LevelArgs &a, int G)
{
    const int P = 32 / G;
    return {(a.H + P - 1) / P, (a.W + P - 1) / P, (a.W + P - 1 + P - 1) / P};
}

int64_t wide_blocks(const LevelArgs &a, const WideGrid &g)
{
    return a.nviews * (2 * (int64_t)g.nrow + 2 * (int64_t)g.ncol +
                       (a.npaths > 4 ? 4 * (int64_t)g.ndia : 0));
}

template <int G, int NQ>
void launch_wide_k(const LevelArgs &a, cudaStream_t s)
{
    const WideGrid g = wide_grid(a, G);
    agg_wide<G, NQ><<<(unsigned)wide_blocks(a, g), 32, 0, s>>>(a, g);
}

}  // namespace

bool wide_shape(const LevelArgs &a, int &G, int &NQ)
{
    if (a.radius > 2 || a.block_cut > 0 || (int64_t)a.npaths * a.trunc > 255) return false;
    if (a.Dw <= 64 || a.Dw > 256) return false;
    // 4 lanes of up to 32 labels share a step's overhead among more paths, but need enough of
    // them: from kFewLanes warps on (measured: 1280x720 with 96 and 128 labels 674 -> 572 and
    // 826 -> 785 us, 2,288 warps; 640x360 with 72 and 100 labels 211 -> 226 and 223 -> 263 us,
    // 1,148 warps)
    G = 8;
    if (a.Dw <= 128) {
        const WideGrid g = wide_grid(a, 4);
        if (wide_blocks(a, g) >= kFewLanes) G = 4;
    }
    NQ = (a.Dw + 4 * G - 1) / (4 * G);
    // C and E share the region of C and S
    const int R = 4 * G * NQ;
    return 2 * R <= 3 * a.Dws && (int64_t)a.W * a.H * R < (int64_t)1 << 31;
}

void launch_wide(const LevelArgs &a, cudaStream_t s)
{
    if (a.wide_g == 4) {
        switch (a.wide_nq) {
        case 5: launch_wide_k<4, 5>(a, s); return;
        case 6: launch_wide_k<4, 6>(a, s); return;
        case 7: launch_wide_k<4, 7>(a, s); return;
        default: launch_wide_k<4, 8>(a, s); return;
        }
    }
    switch (a.wide_nq) {
    case 3: launch_wide_k<8, 3>(a, s); return;
    case 4: launch_wide_k<8, 4>(a, s); return;
    case 5: launch_wide_k<8, 5>(a, s); return;
    case 6: launch_wide_k<8, 6>(a, s); return;
    case 7: launch_wide_k<8, 7>(a, s); return;
    default: launch_wide_k<8, 8>(a, s); return;
    }
}

}  // namespace mpv
