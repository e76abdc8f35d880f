// agg_sweep.cuh -- byte sums of the gradient-weighted passes (a slope per step) on levels with
// label strides of 16 or 32.
//
// The envelope of the predecessor A with slope P and cap T is M(u) = min(min_v A(v) + P |u - v|,
// min_v A(v) + T).  4 lanes hold a path, K = 2 KW labels each.  Inside a lane the minimum over
// all its labels takes three rounds (two for K = 4) of 3-input packed minima: over |d| <= 1, then
// the neighbours two and four labels away with 2 P and 4 P, both directions at once.  Across the
// lanes only the values at a lane's two end labels matter: they are exchanged with the lanes'
// minima behind one warp barrier, and what enters a lane from below and from above is a
// minimum over the other three lanes.  Penalties are added on the FMA pipe.  A step whose window
// moved writes the envelope (without its cap) to shared memory, continued at slope P over DWP
// labels past both ends, and reads it back at the shift.  The increments M - min A, at most T, are
// added as bytes.  Costs come by asynchronous copies, 8 steps at a time and one chunk ahead;
// window starts and intensities a chunk ahead in registers, from which each lane prepares the
// slope and shift of two steps.
//
// Bound: issue and L1 on large levels (138 instructions per step of 8 paths; 64 and 73 %), the
// chain of a row step on others.  Both views, 8 paths, against 8 lanes, prefix scans by shuffles
// and 16-bit sums: 1280x720, 32 labels, windows 712 -> 421 us; 640x360 178 -> 130 us; 320x180 without windows
// 83 -> 49 us.  8 lanes for the rows (109 instructions per step of 4 paths) 636 instead of 612 us
// per frame; windows that moved by 2 labels through shuffles 631 us; 12 to 28 resident warps per
// SM within 5 %.
#pragma once
#include "agg_rows.cuh"

namespace mpv {

namespace {

constexpr int kSweepChunk = 8;

template <int KW, bool WIN>
struct SweepSmem {                   // one warp's shared memory, in bytes
    static constexpr int DWP = 8 * KW;                        // labels (bytes) per pixel
    // a path's chunk; the pad spreads the paths over the banks
    static constexpr int PATHB = kSweepChunk * DWP + (KW == 4 ? 32 : 16);
    static constexpr int PAD = DWP + 8;                       // labels past either end of a path
    static constexpr int PATHW = (2 * PAD + DWP) / 2 + 4;     // words (28 or 4 mod 32: paths apart)
    static constexpr int off_step = 2 * 8 * PATHB;            // slopes and shifts of the chunk
    static constexpr int off_x = off_step + 8 * kSweepChunk * 8;   // lanes' minima and end values
    static constexpr int off_lut = off_x + 2 * 32 * 8;        // the table's slopes, at most T
    static constexpr int off_m = off_lut + 256;               // envelopes
    static constexpr int bytes = (off_m + (WIN ? 8 * PATHW * 4 : 0) + 15) / 16 * 16;
};

__device__ __forceinline__ void sweep_store(uint32_t *p, const uint32_t (&v)[4])
{
    *(uint4 *)p = make_uint4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void sweep_store(uint32_t *p, const uint32_t (&v)[2])
{
    *(uint2 *)p = make_uint2(v[0], v[1]);
}

// Paths 8 grp .. 8 grp + 7 of direction dir (at least one).  PD: the level may have padding labels.
template <int KW, bool WIN, bool PD>
__device__ __forceinline__ void sweep_body(const LevelArgs &a, const int *lut, int grp, int dir,
                                           int view, int lane, unsigned char *smem)
{
    static_assert(KW == 2 || KW == 4, "16 or 32 labels");
    using SS = SweepSmem<KW, WIN>;
    constexpr int DWP = SS::DWP, K = 2 * KW, CH = kSweepChunk;
    const int W = a.W, H = a.H;
    const int dx = c_dirs[dir][0], dy = c_dirs[dir][1];
    const int gl = lane & 3, path = lane >> 2;
    const ViewLevel &V = a.v[view];
    const uint32_t T = (uint32_t)a.trunc;
    unsigned char *slut = smem + SS::off_lut;
    for (int i = lane; i < 256; i += 32) slut[i] = (unsigned char)min((uint32_t)lut[i], T);
    __syncwarp();

    int x0 = 0, y0 = 0, n = 0;
    if (8 * grp + path < num_paths_dir(dx, dy, W, H)) {
        path_start(dx, dy, W, H, 8 * grp + path, x0, y0);
        n = path_length(dx, dy, W, H, x0, y0);
    }
    const int nch = (__reduce_max_sync(kFull, n) + CH - 1) / CH;
    const int64_t pix0 = (int64_t)y0 * W + x0, dpix = (int64_t)dy * W + dx;

    // a chunk's pieces of 16 bytes: lane gl takes piece gl % PPS of every TPI-th step
    constexpr int PPS = DWP / 16, TPI = 4 / PPS, NP = CH / TPI;
    const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(smem) + path * SS::PATHB +
                           gl / PPS * DWP + gl % PPS * 16;
    const uint8_t *pc = V.C + (pix0 + gl / PPS * dpix) * DWP + gl % PPS * 16;
    const int64_t dpiece = TPI * dpix * DWP;
    // window starts and intensities of steps 2 gl and 2 gl + 1
    const uint16_t *lp = WIN ? V.lo + pix0 + 2 * gl * dpix : nullptr;
    const int64_t di = (int64_t)dy * V.pitch0 + dx;
    const uint8_t *ip = V.I0 + (int64_t)y0 * V.pitch0 + x0 + 2 * gl * di;
    int lo_n[2] = {0, 0}, in_n[2] = {0, 0};
    auto issue = [&](int c) {             // chunk c into stage c & 1; the pointers point at it
        const uint32_t st = sbase + (c & 1) * (8 * SS::PATHB);
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            const bool on = c * CH + i * TPI + gl / PPS < n;
            row_copy(st + i * TPI * DWP, pc, 16,
                     on && MPV_IN(a.err, pc >= V.C && pc + 16 <= V.C + (int64_t)W * H * DWP, 21));
            pc += dpiece;
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
#pragma unroll
        for (int h = 0; h < 2; ++h)
            if (c * CH + 2 * gl + h < n &&
                MPV_IN(a.err, ip + h * di >= V.I0 && ip + h * di < V.I0 + (int64_t)V.pitch0 * (H - 1) + W &&
                                  (!WIN || (lp + h * dpix >= V.lo && lp + h * dpix < V.lo + (int64_t)W * H)),
                       22)) {
                if (WIN) lo_n[h] = (int)ld_pin_u16(lp + h * dpix);
                in_n[h] = (int)ld_pin_u8(ip + h * di);
            }
        if (WIN) lp += CH * dpix;
        ip += CH * di;
    };

    const uint32_t INF2 = kInf16 * 0x10001u;
    const uint32_t Tx2 = T * 0x10001u;
    uint32_t pad[KW];                     // labels at or beyond Dw: never a predecessor
#pragma unroll
    for (int i = 0; i < KW; ++i) {
        const int k0 = gl * K + 2 * i;
        pad[i] = INF2 & ((k0 < a.Dw ? 0u : 0x0000FFFFu) | (k0 + 1 < a.Dw ? 0u : 0xFFFF0000u));
    }
    // of lane l's end values (top label in the low half, bottom label in the high half): which
    // enters this lane, and the labels between
    uint32_t am[4], dm[4];
#pragma unroll
    for (int l = 0; l < 4; ++l) {
        am[l] = l < gl ? 0x0000FFFFu : (l > gl ? 0xFFFF0000u : 0u);
        dm[l] = l == gl ? 0u : (uint32_t)(K * (abs(gl - l) - 1)) * 0x10001u;
    }
    unsigned char *steps = smem + SS::off_step;
    unsigned char *xch = smem + SS::off_x;
    uint32_t *mb = (uint32_t *)(smem + SS::off_m) + (WIN ? path * SS::PATHW : 0);

    const unsigned char *cs = smem + path * SS::PATHB + gl * K;
    uint8_t *ep = V.E + pix0 * DWP + gl * K;
    const int64_t dep = dpix * DWP;

    uint32_t A[KW];
#pragma unroll
    for (int i = 0; i < KW; ++i) A[i] = INF2;     // no predecessor: E = 0 at the first pixel
    int last_lo = 0, last_in = 0;
    issue(0);
    for (int c = 0; c < nch; ++c) {
        const int lo[2] = {lo_n[0], lo_n[1]}, in[2] = {in_n[0], in_n[1]};
        if (c + 1 < nch) issue(c + 1);
        else asm volatile("cp.async.commit_group;" ::: "memory");
        // slope and window shift of this lane's two steps
        unsigned mv[2] = {0u, 0u};
        {
            int pi = __shfl_up_sync(kFull, in[1], 1, 4);
            const int li = __shfl_sync(kFull, last_in, 3, 4);
            int pl = 0, ll = 0;
            if (WIN) {
                pl = __shfl_up_sync(kFull, lo[1], 1, 4);
                ll = __shfl_sync(kFull, last_lo, 3, 4);
            }
            if (gl == 0) {
                pi = c == 0 ? in[0] : li;
                pl = c == 0 ? lo[0] : ll;
            }
            last_in = in[1];
            last_lo = lo[1];
            int2 st[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const bool on = c * CH + 2 * gl + h < n;
                st[h].x = slut[abs(in[h] - (h ? in[0] : pi)) & 0xFF];
                st[h].y = WIN && on ? lo[h] - (h ? lo[0] : pl) : 0;
                if (WIN) mv[h] = __ballot_sync(kFull, st[h].y != 0);
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) ((int2 *)steps)[(2 * gl + h) * 8 + path] = st[h];
        }
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncwarp();                 // chunk c has arrived for every lane, and its steps
        const unsigned char *cc = cs + (c & 1) * (8 * SS::PATHB);
#pragma unroll
        for (int u = 0; u < CH; ++u) {
            // (steps past a path compute on leftovers and add nothing)
            uint32_t cv[KW];
            if (KW == 4) {
                const uint2 w = *(const uint2 *)(cc + u * DWP);
                cv[0] = __byte_perm(w.x, 0u, 0x4140);
                cv[1] = __byte_perm(w.x, 0u, 0x4342);
                cv[2 % KW] = __byte_perm(w.y, 0u, 0x4140);
                cv[3 % KW] = __byte_perm(w.y, 0u, 0x4342);
            } else {
                const uint32_t w = *(const uint32_t *)(cc + u * DWP);
                cv[0] = __byte_perm(w, 0u, 0x4140);
                cv[1] = __byte_perm(w, 0u, 0x4342);
            }
            const int2 ps = ((const int2 *)steps)[u * 8 + path];
            const uint32_t P = (uint32_t)ps.x;
            const uint32_t C1 = P * 0x10001u, C2 = C1 * 2, C4 = C1 * 4;

            // the envelope over this lane's labels
            uint32_t B[KW];
            {
                uint32_t s[KW + 1];       // (label before, label) pairs, absent at the ends
                s[0] = __byte_perm(A[0], INF2, 0x1054);
                s[KW] = __byte_perm(A[KW - 1], INF2, 0x7632);
#pragma unroll
                for (int w = 1; w < KW; ++w) s[w] = shift1(A[w - 1], A[w]);
#pragma unroll
                for (int w = 0; w <= KW; ++w) s[w] += C1;
#pragma unroll
                for (int w = 0; w < KW; ++w) B[w] = __vimin3_u16x2(A[w], s[w], s[w + 1]);
                uint32_t t[KW];
#pragma unroll
                for (int w = 0; w < KW; ++w) t[w] = B[w] + C2;
#pragma unroll
                for (int w = 0; w < KW; ++w) {
                    if (w == 0) B[w] = __vminu2(B[w], t[1]);
                    else if (w == KW - 1) B[w] = __vminu2(B[w], t[w - 1]);
                    else B[w] = __vimin3_u16x2(B[w], t[w - 1], t[(w + 1) % KW]);
                }
                if (KW == 4) {
#pragma unroll
                    for (int w = 0; w < KW; ++w) t[w] = B[w] + C4;
#pragma unroll
                    for (int w = 0; w < KW; ++w) B[w] = __vminu2(B[w], t[(w + 2) % KW]);
                }
            }
            // the lanes' minima (of A: the envelope's are the same) and end values
            uint32_t lm = B[0];
            if (KW == 4) lm = __vminu2(__vimin3_u16x2(lm, B[1], B[2 % KW]), B[3 % KW]);
            else lm = __vminu2(lm, B[1]);
            unsigned char *xw = xch + (u & 1) * 256;
            // (the paths' lanes 0 and 1, then their lanes 2 and 3: 16 bytes a path)
            *(uint2 *)(xw + gl / 2 * 128 + path * 16 + gl % 2 * 8) =
                make_uint2(lm, shift1(B[KW - 1], B[0]));
            __syncwarp();
            const uint4 q0 = *(const uint4 *)(xw + path * 16);
            const uint4 q1 = *(const uint4 *)(xw + 128 + path * 16);
            const uint32_t fg[4] = {q0.y, q0.w, q1.y, q1.w};
            uint32_t m2 = __vimin3_u16x2(q0.x, q0.z, __vminu2(q1.x, q1.z));
            m2 = __vminu2(m2, __byte_perm(m2, m2, 0x1032));
            uint32_t X;                   // what enters from below and, high half, from above
            {
                uint32_t v[4];
#pragma unroll
                for (int l = 0; l < 4; ++l) v[l] = ((fg[l] & am[l]) | (INF2 & ~am[l])) + P * dm[l];
                X = __vimin3_u16x2(v[0], v[1], __vminu2(v[2], v[3]));
            }
            const uint32_t xf = __byte_perm(X, X, 0x1010), xg = __byte_perm(X, X, 0x3232);
            uint32_t M[KW];
#pragma unroll
            for (int w = 0; w < KW; ++w) {
                // distances from the label below the lane and to the label above it
                const uint32_t du = (uint32_t)(2 * w + 1) | ((uint32_t)(2 * w + 2) << 16);
                const uint32_t dd = (uint32_t)(K - 2 * w) | ((uint32_t)(K - 2 * w - 1) << 16);
                M[w] = __vimin3_u16x2(B[w], P * du + xf, P * dd + xg);
            }
            if (WIN && (mv[u & 1] & (0x11111111u << (u >> 1)))) {
                // a window of the warp moved: re-index.  The path's envelope at its first and
                // last label, and its continuation at slope P over DWP labels to either side
                // (further shifts add theirs: past 255 labels every slope but 0 exceeds T)
                uint32_t v[4];
#pragma unroll
                for (int l = 0; l < 4; ++l)
                    v[l] = fg[l] + P * ((uint32_t)(K * (3 - l)) | ((uint32_t)(K * l) << 16));
                const uint32_t e = __vimin3_u16x2(v[0], v[1], __vminu2(v[2], v[3]));
                const int s = ps.y;
                const uint32_t fu = P * (uint32_t)min(max(s - DWP, 0), 255);
                const uint32_t fd = P * (uint32_t)min(max(-s - DWP, 0), 255);
                const uint32_t up = __byte_perm(e, e, 0x1010) + (fu + P * (uint32_t)(gl * K)) * 0x10001u;
                const uint32_t dn = __byte_perm(e, e, 0x3232) + (fd + P * (uint32_t)(gl * K)) * 0x10001u;
                uint32_t *mw = mb + (SS::PAD + gl * K) / 2;
                uint32_t *lw = mb + (SS::PAD - gl * K) / 2 - KW;
                uint32_t hi[KW], below[KW];
#pragma unroll
                for (int w = 0; w < KW; ++w) {
                    const uint32_t du = (uint32_t)(2 * w + 1) | ((uint32_t)(2 * w + 2) << 16);
                    hi[w] = P * du + up;
                    // labels -(gl K + 2w + 2), -(gl K + 2w + 1)
                    below[KW - 1 - w] = P * __byte_perm(du, du, 0x1032) + dn;
                }
                sweep_store(mw, M);
                sweep_store(mw + DWP / 2, hi);
                sweep_store(lw, below);
                __syncwarp();
                const int j = SS::PAD + gl * K + min(max(s, -DWP), DWP);
                const uint32_t sel = (j & 1) ? 0x5432u : 0x3210u;
                const bool ok = MPV_IN(a.err, j >= 0 && (j >> 1) + KW < SS::PATHW, 5);
                uint32_t Wd[KW + 1];
#pragma unroll
                for (int w = 0; w <= KW; ++w) Wd[w] = ok ? mb[(j >> 1) + w] : INF2;
#pragma unroll
                for (int w = 0; w < KW; ++w) M[w] = __byte_perm(Wd[w], Wd[w + 1], sel);
            }
            const uint32_t cap = m2 + Tx2;
#pragma unroll
            for (int w = 0; w < KW; ++w) {
                M[w] = __vminu2(M[w], cap) - m2;          // per half: no borrow, at most T
                A[w] = cv[w] + M[w];
                if (PD) A[w] |= pad[w];
            }
            if (c * CH + u < n && MPV_IN(a.err, ep >= V.E && ep < V.E + (int64_t)W * H * DWP, 7)) {
                const uint32_t w0 = __byte_perm(M[0], M[1], 0x6420);
                if (KW == 4)
                    atomicAdd((unsigned long long *)ep,
                              ((unsigned long long)__byte_perm(M[2 % KW], M[3 % KW], 0x6420) << 32) | w0);
                else
                    atomicAdd((unsigned int *)ep, w0);
            }
            ep += dep;
        }
        __syncwarp();                 // every lane is done with the stage that is filled next
    }
}

// One warp per block, the row directions first (the longest chains start first).
template <int KW, bool WIN, bool PD>
__global__ void __launch_bounds__(32) agg_sweep(LevelArgs a, const int *lut, int nrow, int ncol)
{
    if (a.gate && *a.gate == 0) return;
    __shared__ __align__(16) unsigned char smem[SweepSmem<KW, WIN>::bytes];
    int b = blockIdx.x;
    const int view = b % a.nviews;
    b /= a.nviews;
    int dir, grp;
    if (b < 2 * nrow) {
        dir = b & 1;
        grp = b >> 1;
    } else if (b < 2 * (nrow + ncol)) {
        b -= 2 * nrow;
        dir = 2 + (b & 1);
        grp = b >> 1;
    } else {
        b -= 2 * (nrow + ncol);
        dir = 4 + (b & 3);
        grp = b >> 2;
    }
    sweep_body<KW, WIN, PD>(a, lut, grp, dir, view, threadIdx.x, smem);
}

template <int KW>
void launch_agg_sweep(const LevelArgs &a, const int *lut, cudaStream_t s)
{
    const int nrow = (a.H + 7) / 8, ncol = (a.W + 7) / 8, ndiag = (a.W + a.H - 1 + 7) / 8;
    const int blocks = a.nviews * (2 * (nrow + ncol) + (a.npaths > 4 ? 4 * ndiag : 0));
    const bool pd = a.Dw < a.Dws;
    if (a.v[0].lo) {
        if (pd) agg_sweep<KW, true, true><<<blocks, 32, 0, s>>>(a, lut, nrow, ncol);
        else agg_sweep<KW, true, false><<<blocks, 32, 0, s>>>(a, lut, nrow, ncol);
    } else {
        if (pd) agg_sweep<KW, false, true><<<blocks, 32, 0, s>>>(a, lut, nrow, ncol);
        else agg_sweep<KW, false, false><<<blocks, 32, 0, s>>>(a, lut, nrow, ncol);
    }
}

}  // namespace

}  // namespace mpv
