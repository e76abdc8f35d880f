// agg_layer.cuh -- the layers of the layered merge on levels with label strides of 16 or 32.
//
// A layer is two opposite passes over the data term, which is the cost bytes or the previous
// layer's two volumes, and each layer waits for the one before: few paths are in flight (a
// 1280x720 level has 2,880 row paths, 720 warps), so a layer takes the chain of its longest
// path.  With register prefetch a step of that chain waited for loads issued a step before (the
// loads in flight share a warp's few scoreboards).  Here the data term comes by asynchronous
// copies of 16 bytes, kLayerChunk steps at a time and one chunk ahead, for every direction, and
// a step reads shared memory only.
//
// Bound: the chain of one step; on the largest levels the bytes (a pass reads 128 and writes 64
// per pixel of 32 labels).  Both views, against the packed stencil's layer mode (first layer, second,
// third and fourth): 1280x720, 32 labels, windows 257 -> 172, 122, 137 us; 640x360 108 -> 72, 43,
// 45 us; 320x180 without windows 45 -> 30, 16, 16 us.
//
// 8 lanes per path, KW words of two labels per lane, 4 paths per warp, one warp per block; the
// arithmetic is agg_stencil_body's in its layer mode for radius at most 2 (see there for the
// doubled pass).  With windows the predecessor passes through shared memory on every step
// together with the lanes' minima, behind one warp barrier, and is read back at the step's
// window shift; the doubled pass's suffix minima take a second one.
#pragma once
#include "agg_rows.cuh"

namespace mpv {

namespace {

constexpr int kLayerChunk = 8;

template <int KW, bool WIN, bool PAIR>
struct LayerSmem {                   // one warp's shared memory, in bytes
    static constexpr int DWP = 16 * KW;                       // labels per pixel
    static constexpr int VB = PAIR ? 2 * DWP : DWP;           // bytes of one volume per step
    static constexpr int STEPB = PAIR ? 2 * VB : VB;          // staged bytes per step
    static constexpr int PATHB = kLayerChunk * STEPB + VB;    // a path's chunk; the pad spreads paths
    static constexpr int PADL = 40;                           // absent labels around a path
    static constexpr int PATHW = (2 * PADL + DWP + 63) / 64 * 32;   // words, a multiple of 32
    static constexpr int abuf = (4 * PATHW + 32) * 4;
    static constexpr int off_sh = 2 * 4 * PATHB;              // the chunk's shifts
    static constexpr int off_min = off_sh + (WIN ? 4 * kLayerChunk * 8 : 0);
    static constexpr int off_a = off_min + 2 * 32 * 4;        // predecessors, by step parity
    static constexpr int off_s = off_a + (WIN ? 2 * abuf : 0);   // suffix minima (doubled pass)
    static constexpr int bytes = (off_s + (WIN && !PAIR ? abuf : 0) + 15) / 16 * 16;
    // first word of a path's buffer: lanes KW words apart, paths in different banks
    __device__ static constexpr int path_word(int p)
    {
        return p * PATHW + p % KW + p / KW * (8 * KW) % 32;
    }
};

// Direction dir, paths 4 grp .. 4 grp + 3.  IN: the data term (MergeArgs::in_mode); ASYM: the
// doubled pass.
template <int KW, bool WIN, int IN, bool ASYM>
__device__ __forceinline__ void layer_body(const LevelArgs &a, const MergeArgs &mg, int grp, int dir,
                                           int view, int lane, unsigned char *smem)
{
    constexpr bool PAIR = IN != 0;
    static_assert(!(PAIR && ASYM), "only the first layer has the doubled pass");
    using LS = LayerSmem<KW, WIN, PAIR>;
    constexpr int DWP = LS::DWP, K = 2 * KW, NE = KW + 2, CH = kLayerChunk;
    const int W = a.W, H = a.H;
    const int dx = c_dirs[dir][0], dy = c_dirs[dir][1];
    if (4 * grp >= num_paths_dir(dx, dy, W, H)) return;       // (warp-uniform)
    const int gl = lane & 7, path = lane >> 3;
    const ViewLevel &V = a.v[view];
    const uint16_t *qa = view ? mg.qa[1] : mg.qa[0];
    const uint16_t *qb = view ? mg.qb[1] : mg.qb[0];
    uint16_t *const *outs = view ? mg.out[1] : mg.out[0];
    uint16_t *const outv = (dir & 1) ? outs[1] : outs[0];
    int x0 = 0, y0 = 0, n = 0;
    if (4 * grp + path < num_paths_dir(dx, dy, W, H)) {
        path_start(dx, dy, W, H, 4 * grp + path, x0, y0);
        n = path_length(dx, dy, W, H, x0, y0);
    }
    const int nch = (__reduce_max_sync(kFull, n) + CH - 1) / CH;
    const int64_t pix0 = (int64_t)y0 * W + x0, dpix = (int64_t)dy * W + dx;

    // a chunk's pieces of 16 bytes: lane gl takes piece gl % PPS of every TPI-th step
    constexpr int PPS = LS::VB / 16, TPI = 8 / PPS, NP = CH / TPI;
    const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(smem) + path * LS::PATHB +
                           gl / PPS * LS::STEPB + gl % PPS * 16;
    const int64_t at0 = (pix0 + gl / PPS * dpix) * LS::VB + gl % PPS * 16;
    const uint8_t *pa = (PAIR ? (const uint8_t *)qa : V.C) + at0;
    const uint8_t *pb = PAIR ? (const uint8_t *)qb + at0 : nullptr;
    const int64_t dpiece = TPI * dpix * LS::VB;
    [[maybe_unused]] auto in_volume = [&](const uint8_t *p, const uint8_t *vol) {
        return p >= vol && p + 16 <= vol + (int64_t)W * H * LS::VB;
    };
    auto issue = [&](int c) {             // chunk c into stage c & 1; pa, pb point at it
        const uint32_t st = sbase + (c & 1) * (4 * LS::PATHB);
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            const bool on = c * CH + i * TPI + gl / PPS < n;
            row_copy(st + i * TPI * LS::STEPB, pa, 16,
                     on && MPV_IN(a.err, in_volume(pa, PAIR ? (const uint8_t *)qa : V.C), 18));
            pa += dpiece;
            if (PAIR) {
                row_copy(st + i * TPI * LS::STEPB + LS::VB, pb, 16,
                         on && MPV_IN(a.err, in_volume(pb, (const uint8_t *)qb), 18));
                pb += dpiece;
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    // lane gl holds the window start of step gl of the next chunk
    const uint16_t *lp = WIN ? V.lo + pix0 + gl * dpix : nullptr;
    int lo_next = 0;
    auto issue_lo = [&](int c) {
        if (c * CH + gl < n && MPV_IN(a.err, lp >= V.lo && lp < V.lo + (int64_t)W * H, 19))
            lo_next = (int)ld_pin_u16(lp);
        lp += CH * dpix;
    };

    const uint32_t INF2 = kInf16 * 0x10001u;
    const uint32_t T = (uint32_t)a.trunc;
    const uint32_t Tx2 = T * 0x10001u;
    const uint32_t E1 = min((uint32_t)a.p1, T) * 0x10001u;
    const uint32_t E2 = min(2 * (uint32_t)a.p1, T) * 0x10001u;
    constexpr uint32_t up = ASYM ? 2u : 1u;     // upward jumps and their cap
    const uint32_t U1 = E1 * up, U2 = E2 * up, Tcap = Tx2 * up;
    // labels at or beyond Dw are padding: never a predecessor, stored as 0
    uint32_t pad[KW];
#pragma unroll
    for (int i = 0; i < KW; ++i) {
        const int k0 = gl * K + 2 * i;
        pad[i] = (k0 < a.Dw ? 0u : 0x0000FFFFu) | (k0 + 1 < a.Dw ? 0u : 0xFFFF0000u);
    }
    uint32_t om[7];                       // (doubled pass) all ones at lanes 1 .. 7 not above
#pragma unroll
    for (int l = 0; l < 7; ++l) om[l] = l + 1 > gl ? 0u : 0xFFFFFFFFu;
    uint32_t *minb = (uint32_t *)(smem + LS::off_min);
    uint32_t *ab = (uint32_t *)(smem + LS::off_a) + LS::path_word(path);
    uint32_t *sb = (uint32_t *)(smem + LS::off_s) + LS::path_word(path);
    constexpr int ABW = LS::abuf / 4;     // words from one parity's buffers to the other's
    if (WIN) {
        for (int i = lane; i < (ASYM ? 3 : 2) * ABW; i += 32)
            ((uint32_t *)(smem + LS::off_a))[i] = INF2;
        __syncwarp();
    }

    const unsigned char *cs = smem + path * LS::PATHB + gl * (LS::VB / 8);
    uint16_t *op = outv + (pix0 - dpix) * DWP + gl * K;     // the pixel before step t's
    const int64_t dop = dpix * DWP;

    uint32_t A[KW];
#pragma unroll
    for (int i = 0; i < KW; ++i) A[i] = INF2;     // no predecessor: L = C at the first pixel
    auto store = [&](uint32_t m2) {               // A, normalised by its minimum
        uint32_t v[KW];
#pragma unroll
        for (int i = 0; i < KW; ++i) v[i] = (A[i] - m2) & ~pad[i];   // per half: A >= m2
        if (!MPV_IN(a.err, op >= outv && op + K <= outv + (int64_t)W * H * DWP, 20)) return;
        if (KW == 1) *(uint32_t *)op = v[0];
        else *(uint2 *)op = make_uint2(v[0], v[1 % KW]);
    };
    int last_lo = 0;
    issue(0);
    if (WIN) issue_lo(0);
    for (int c = 0; c < nch; ++c) {
        const int lo = lo_next;
        if (c + 1 < nch) {
            issue(c + 1);
            if (WIN) issue_lo(c + 1);
        } else {
            asm volatile("cp.async.commit_group;" ::: "memory");
        }
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        if (WIN) {
            // lane gl prepares step gl of its path: the first word and the half-word selection
            // at which the step's labels lie in the predecessor's frame
            int before = __shfl_up_sync(kFull, lo, 1, 8);
            const int last = __shfl_sync(kFull, last_lo, CH - 1, 8);
            if (gl == 0) before = c == 0 ? lo : last;
            last_lo = lo;
            const int sc = min(max(lo - before, -(DWP + 2)), DWP + 2);
            ((uint2 *)(smem + LS::off_sh))[lane] =
                make_uint2((unsigned)((LS::PADL - 2 + sc) >> 1), (sc & 1) ? 0x5432u : 0x3210u);
        }
        __syncwarp();                 // chunk c has arrived for every lane, and its shifts
        const unsigned char *cc = cs + (c & 1) * (4 * LS::PATHB);
        // (steps past a path compute on leftovers, and nothing reads or stores them)
#pragma unroll
        for (int u = 0; u < CH; ++u) {
            uint32_t cv[KW];
            if (PAIR) {
                const unsigned char *sa = cc + u * LS::STEPB, *sc = sa + LS::VB;
                uint2 va, vb;
                if (KW == 1) {
                    va.x = va.y = *(const uint32_t *)sa;
                    vb.x = vb.y = *(const uint32_t *)sc;
                } else {
                    va = *(const uint2 *)sa;
                    vb = *(const uint2 *)sc;
                }
                cv[0] = IN == 1 ? __vminu2(va.x, vb.x) : avg_u16x2(va.x, vb.x);
                if (KW == 2) cv[1 % KW] = IN == 1 ? __vminu2(va.y, vb.y) : avg_u16x2(va.y, vb.y);
            } else if (KW == 1) {
                cv[0] = __byte_perm((uint32_t)*(const uint16_t *)(cc + u * LS::STEPB), 0u, 0x4140);
            } else {
                const uint32_t w = *(const uint32_t *)(cc + u * LS::STEPB);
                cv[0] = __byte_perm(w, 0u, 0x4140);
                cv[1 % KW] = __byte_perm(w, 0u, 0x4342);
            }
            uint2 sh = make_uint2(0u, 0u);
            if (WIN) sh = ((const uint2 *)(smem + LS::off_sh))[path * CH + u];
            // the lanes' minima (and the predecessor), exchanged behind one barrier; buffers
            // alternate by step parity
            uint32_t m2 = A[0];
#pragma unroll
            for (int i = 1; i < KW; ++i) m2 = __vminu2(m2, A[i]);
            m2 = __vminu2(m2, __byte_perm(m2, m2, 0x1032));
            uint32_t *aw = ab + (u & 1) * ABW;
            if (WIN) {
#pragma unroll
                for (int i = 0; i < KW; ++i) aw[LS::PADL / 2 + gl * KW + i] = A[i];
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
                const bool ok =
                    MPV_IN(a.err, (int)sh.x >= 0 && (int)sh.x + gl * KW + NE < LS::PATHW, 3);
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
            uint32_t SA[KW];
            if (ASYM) {
                // suffix minima: of the lanes above, then down the lane's own words
                const uint32_t r0 = __vimin3_u16x2(q0.y | om[0], q0.z | om[1], q0.w | om[2]);
                const uint32_t r1 = __vimin3_u16x2(q1.x | om[3], q1.y | om[4], q1.z | om[5]);
                uint32_t ex = __vimin3_u16x2(r0, r1, __vminu2(q1.w | om[6], INF2));
#pragma unroll
                for (int i = KW - 1; i >= 0; --i) {
                    const uint32_t v = __vminu2(A[i], ex);               // (min(lo,r), min(hi,r))
                    SA[i] = __vminu2(v, __byte_perm(v, v, 0x3232));     // low half also <= high
                    ex = __byte_perm(SA[i], SA[i], 0x1010);
                }
                if (WIN) {
                    // label j reads the suffix minimum at j + s: below the predecessor's window
                    // every label is above (the minimum), beyond it none
#pragma unroll
                    for (int i = 0; i < KW; ++i) sb[LS::PADL / 2 + gl * KW + i] = SA[i];
#pragma unroll
                    for (int i = 0; i < 3; ++i)
                        if (i < 2 || gl < LS::PADL / 2 - 16) sb[gl + 8 * i] = m2;
                    __syncwarp();
                    uint32_t Sd[KW + 1];
                    const bool sok =
                        MPV_IN(a.err, (int)sh.x + 1 >= 0 && (int)sh.x + 1 + gl * KW + KW < LS::PATHW, 4);
                    const uint32_t *pw = sb + gl * KW + sh.x + 1;
#pragma unroll
                    for (int i = 0; i <= KW; ++i) Sd[i] = sok ? pw[i] : INF2;
#pragma unroll
                    for (int i = 0; i < KW; ++i) SA[i] = __byte_perm(Sd[i], Sd[i + 1], sh.y);
                }
            }
            if ((unsigned)(c * CH + u - 1) < (unsigned)n) store(m2);   // the pixel before
            op += dop;
            const uint32_t cap = m2 + Tcap;
#pragma unroll
            for (int i = 0; i < KW; ++i) {
                uint32_t m = __vimin3_u16x2(E[1 + i], SH[i] + U1, SH[i + 1] + E1);
                m = __vimin3_u16x2(m, E[i] + U2, E[i + 2] + E2);
                if (ASYM) m = __viaddmin_u16x2(SA[i], Tx2, m);
                m = __vminu2(m, cap);
                A[i] = (cv[i] + m - m2) | (pad[i] & INF2);           // per half: no borrow
            }
        }
        __syncwarp();                 // every lane is done with the stage that is filled next
    }
    // the last pixel of paths that end with their last chunk: nothing followed to store it
    uint32_t m2 = A[0];
#pragma unroll
    for (int i = 1; i < KW; ++i) m2 = __vminu2(m2, A[i]);
    m2 = __vminu2(m2, __byte_perm(m2, m2, 0x1032));
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) m2 = __vminu2(m2, __shfl_xor_sync(kFull, m2, o));
    if (n > 0 && n == nch * CH) store(m2);
}

template <int KW, bool WIN, int IN>
__global__ void __launch_bounds__(32) agg_layer(LevelArgs a, MergeArgs mg)
{
    if (a.gate && *a.gate == 0) return;
    __shared__ __align__(16) unsigned char smem[LayerSmem<KW, WIN, IN != 0>::bytes];
    const int dir = mg.dir0 + blockIdx.y;
    if constexpr (IN == 0)
        if (dir == mg.double_up_dir)
            return layer_body<KW, WIN, 0, true>(a, mg, blockIdx.x, dir, blockIdx.z, threadIdx.x, smem);
    layer_body<KW, WIN, IN, false>(a, mg, blockIdx.x, dir, blockIdx.z, threadIdx.x, smem);
}

template <int KW, bool WIN>
void launch_agg_layer(const LevelArgs &a, const MergeArgs &m, cudaStream_t s)
{
    int paths = 0;
    for (int d = m.dir0; d < m.dir0 + m.ndirs; ++d)
        paths = std::max(paths, d < 2 ? a.H : (d < 4 ? a.W : a.W + a.H - 1));
    const dim3 grid((paths + 3) / 4, m.ndirs, a.nviews);
    if (m.in_mode == 0) agg_layer<KW, WIN, 0><<<grid, 32, 0, s>>>(a, m);
    else if (m.in_mode == 1) agg_layer<KW, WIN, 1><<<grid, 32, 0, s>>>(a, m);
    else agg_layer<KW, WIN, 2><<<grid, 32, 0, s>>>(a, m);
}

}  // namespace

}  // namespace mpv
