// road.cu -- road detection on the disparity map (Section 3.5).
//
// v-disparity Hx[j][i]: the number of pixels of image row j with disparity i (Eq.
// disp_map); u-disparity Hy[j][i]: the same per image column (Eq. hy, read with the
// disparity index); the road profile: the row path j = P(i) over all disparities that
// maximises sum_i Hx[P(i)][i] under 0 < P(i) - P(i-1) < eta (Eqs. e and P_hat), ties to
// the smaller row at the end and at every predecessor.  Pixels whose value is not below
// D (0xFFFF: rejected by the left-right check) are not counted.
#include "mpv_internal.cuh"

namespace mpv {

namespace {

constexpr int kHistThreads = 256;
constexpr int kUCols = 32;               // columns per block of the u-disparity
constexpr int kUThreads = 1024;

// One block per image row: a shared histogram of D bins.
__global__ void __launch_bounds__(kHistThreads) vdisp_kernel(const uint16_t *__restrict__ U,
                                                             int W, int pitch, int D,
                                                             uint32_t *__restrict__ Hx)
{
    extern __shared__ uint32_t hist[];
    const int j = blockIdx.x;
    for (int i = threadIdx.x; i < D; i += kHistThreads) hist[i] = 0;
    __syncthreads();
    const uint16_t *row = U + (int64_t)j * pitch;
    for (int x = threadIdx.x; x < W; x += kHistThreads) {
        const int u = row[x];
        if (u < D) atomicAdd(&hist[u], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < D; i += kHistThreads) Hx[(int64_t)j * D + i] = hist[i];
}

// One block per 32 columns: lane = column, warps stride over the rows.  Few blocks (W / 32), so
// each has 32 warps; a column's bins are D + 1 words apart, so that a row of one disparity (a
// road) meets 32 banks.  (1280x720, D = 128: 15.6 -> 7 us.)
__global__ void __launch_bounds__(kUThreads) udisp_kernel(const uint16_t *__restrict__ U,
                                                          int W, int H, int pitch, int D,
                                                          uint32_t *__restrict__ Hy)
{
    extern __shared__ uint32_t hist[];          // [kUCols][D + 1]
    const int x0 = blockIdx.x * kUCols;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < kUCols * (D + 1); i += kUThreads) hist[i] = 0;
    __syncthreads();
    const int x = x0 + lane;
    constexpr int kRows = kUThreads / 32, kBatch = 8;
    if (x < W)
        for (int y0 = warp; y0 < H; y0 += kRows * kBatch) {
            int u[kBatch];   // the batch's loads are issued before its shared atomics
#pragma unroll
            for (int b = 0; b < kBatch; ++b) {
                const int y = y0 + b * kRows;
                u[b] = y < H ? U[(int64_t)y * pitch + x] : D;
            }
#pragma unroll
            for (int b = 0; b < kBatch; ++b)
                if (u[b] < D) atomicAdd(&hist[lane * (D + 1) + u[b]], 1u);
        }
    __syncthreads();
    const int ncols = min(kUCols, W - x0);
    for (int i = threadIdx.x; i < ncols * D; i += kUThreads) {
        const int c = i / D;
        Hy[(int64_t)x0 * D + i] = hist[i + c];
    }
}

// The road Viterbi in one block: threads own four rows each, the disparities are the
// sequential steps.  A node's key holds its best prefix sum e and its row, ((e + 1) << 12) |
// (4095 - row), 0 when unreachable: the largest key of a window is the predecessor with the
// largest sum, the smaller row on ties.  A thread keeps its own rows' keys in registers and
// reads the rows before them from shared memory, 16 bytes at a time: WM is w & 3 for windows of
// w = eta - 1 >= 4 rows, which says where the four windows begin within the aligned groups, or
// -1 for shorter ones.  Rows of the last thread past H hold garbage that no window of a row
// below H reaches.  The step back from (i, j) is stored as the row difference j - j'
// (1 .. eta-1; nothing for a row that no path reaches), in shared memory when it fits
// (SMEM_BACK) or in the global scratch otherwise.  The histogram comes by asynchronous copies cn
// disparities at a time, transposed, one chunk ahead, issued by kRoadCopy threads of their own
// while the block has room for them, else by every thread; between two chunks only the threads
// with rows meet at a barrier.  Key: 32 bits while the sums stay below 2^20, else 64.
// Bound: the chain of one step (barrier, shared loads, maxima, store) and its instructions'
// issue; 720 rows, D = 128, eta = 8: 112 -> 37 us against one row per
// thread with eta - 1 loads and selects each (64 rows, one warp: 25 us, the chain alone).
constexpr int kRoadChunk = 8;           // at most; fewer when the rows are many
constexpr int kRoadRows = 4;            // rows per thread (kRoadMaxRows / 4 threads at most)
constexpr int kRoadCopy = 256;          // threads that copy the histogram
constexpr int kRoadPad = 256;           // keys before row 0 (all unreachable)

// Rows of the staged arrays: whole threads, 4 mod 32 words so that a disparity's copies of
// neighbouring rows and disparities spread over the banks.
__host__ __device__ inline int road_rows(int H) { return (H + 27) / 32 * 32 + 4; }

// disparities per staged chunk (a power of two; two chunks in at most 96 KB)
__host__ __device__ inline int road_chunk(int H)
{
    int c = kRoadChunk;
    while (c > 1 && (size_t)8 * c * road_rows(H) > 96 * 1024) c >>= 1;
    return c;
}

__device__ __forceinline__ void road_load4(const uint32_t *p, uint32_t (&v)[4])
{
    const uint4 q = *(const uint4 *)p;
    v[0] = q.x, v[1] = q.y, v[2] = q.z, v[3] = q.w;
}
__device__ __forceinline__ void road_load4(const unsigned long long *p, unsigned long long (&v)[4])
{
    const ulonglong2 a = ((const ulonglong2 *)p)[0], b = ((const ulonglong2 *)p)[1];
    v[0] = a.x, v[1] = a.y, v[2] = b.x, v[3] = b.y;
}
__device__ __forceinline__ void road_store4(uint32_t *p, const uint32_t (&v)[4])
{
    *(uint4 *)p = make_uint4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void road_store4(unsigned long long *p, const unsigned long long (&v)[4])
{
    ((ulonglong2 *)p)[0] = make_ulonglong2(v[0], v[1]);
    ((ulonglong2 *)p)[1] = make_ulonglong2(v[2], v[3]);
}

template <class Key>
__device__ __forceinline__ Key road_max(Key a, Key b)
{
    return a > b ? a : b;
}

// The best predecessors of rows j0 .. j0 + 3: pv is row j0 of the step before, k its four keys.
template <int WM, class Key>
__device__ __forceinline__ void road_windows(const Key *pv, int w, const Key (&k)[kRoadRows],
                                             Key (&b)[kRoadRows])
{
    if constexpr (WM < 0) {
        Key v[3 + kRoadRows];            // rows -4 + 1 .. 3
        Key a[4];
        road_load4(pv - 4, a);
#pragma unroll
        for (int x = 0; x < 3; ++x) v[x] = a[x + 1];
#pragma unroll
        for (int x = 0; x < kRoadRows; ++x) v[3 + x] = k[x];
#pragma unroll
        for (int r = 0; r < kRoadRows; ++r) {
            b[r] = v[r + 2];
            if (w >= 2) b[r] = road_max(b[r], v[r + 1]);
            if (w >= 3) b[r] = road_max(b[r], v[r]);
        }
    } else {
        // Row 0's window is rows -w .. -1: n whole groups of four and the last WM rows of the
        // group before.  Its first three rows e leave the windows of rows 1, 2 and 3 in turn;
        // the others lie in all four windows.
        const int n = w >> 2;
        Key q[4], x[4], com = 0;
        road_load4(pv - 4 * n, q);
        if (WM != 0) road_load4(pv - 4 * n - 4, x);
        for (int g = 1; g < n; ++g) {
            Key v[4];
            road_load4(pv - 4 * g, v);
            com = road_max(com, road_max(road_max(v[0], v[1]), road_max(v[2], v[3])));
        }
        Key e[3];
#pragma unroll
        for (int r = 0; r < 3; ++r) e[r] = r < WM ? x[4 - WM + r] : q[r - WM];
#pragma unroll
        for (int r = 3 - WM; r < 4; ++r) com = road_max(com, q[r]);
        const Key e12 = road_max(e[1], e[2]), k01 = road_max(k[0], k[1]);
        b[0] = road_max(com, road_max(e[0], e12));
        b[1] = road_max(com, road_max(e12, k[0]));
        b[2] = road_max(com, road_max(e[2], k01));
        b[3] = road_max(com, road_max(k01, k[2]));
    }
}

template <int WM, bool SMEM_BACK, class Key>
__global__ void __launch_bounds__(1024) road_kernel(const uint32_t *__restrict__ Hx, int H, int D,
                                                    int eta, int cn, int ncopy,
                                                    uint8_t *__restrict__ back_g,
                                                    int32_t *__restrict__ P,
                                                    int64_t *__restrict__ energy)
{
    extern __shared__ __align__(16) unsigned char sm[];
    const int HP = road_rows(H), w = eta - 1;
    const int nt = blockDim.x, t = threadIdx.x, j0 = kRoadRows * t;
    const int ncomp = nt - ncopy;                             // (whole warps)
    const int tc = ncopy ? t - ncomp : t, nc = ncopy ? ncopy : nt;   // copying: thread tc of nc
    const bool own = t < ncomp && j0 < H;
    Key *keys = (Key *)sm;                                    // [2][kRoadPad + HP]
    uint32_t *chunk = (uint32_t *)(keys + 2 * (kRoadPad + HP));   // [2][cn][HP]
    uint8_t *back = (uint8_t *)(chunk + 2 * cn * HP);             // [D][HP]
    const int lc = __ffs(cn) - 1;
    __shared__ Key red[32];
    for (int i = t; i < 2 * (kRoadPad + HP); i += nt) keys[i] = 0;
    const uint32_t csm = (uint32_t)__cvta_generic_to_shared(chunk);
    auto fetch = [&](int i0) {           // disparities i0 .. of every row, transposed
        if (i0 < D) {
            const uint32_t dst = csm + (i0 >> lc & 1) * (cn * HP * 4);
#pragma unroll 4
            for (int e = tc; e < H * cn; e += nc) {
                const int j = e >> lc, c = e & (cn - 1);
                if (i0 + c < D)
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst + (c * HP + j) * 4),
                                 "l"(Hx + (int64_t)j * D + i0 + c)
                                 : "memory");
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    if (tc >= 0) fetch(0);
    Key rk[kRoadRows];                   // the rows' part of the keys
#pragma unroll
    for (int r = 0; r < kRoadRows; ++r) rk[r] = (Key)(4095 - j0 - r);
    Key k[kRoadRows] = {};               // the keys of this thread's rows at the step before
    Key *cur = keys + kRoadPad + j0, *prev = cur + (kRoadPad + HP);
    uint8_t *bk = SMEM_BACK ? back + j0 : back_g + j0;
    for (int i0 = 0; i0 < D; i0 += cn) {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();                 // this chunk is there, the one before is done with
        if (tc >= 0) fetch(i0 + cn);
        if (t < ncomp) {
            const uint32_t *cp = chunk + (i0 >> lc & 1) * (cn * HP) + j0;
            const int steps = min(cn, D - i0);
            for (int c = 0; c < steps; ++c, cp += HP) {
                if (own) {
                    uint32_t cnt[kRoadRows];
                    road_load4(cp, cnt);
                    if (i0 + c == 0) {
#pragma unroll
                        for (int r = 0; r < kRoadRows; ++r) k[r] = (((Key)cnt[r] + 1) << 12) | rk[r];
                    } else {
                        Key b[kRoadRows];
                        road_windows<WM>(prev, w, k, b);
                        uint32_t d[kRoadRows];
#pragma unroll
                        for (int r = 0; r < kRoadRows; ++r) {
                            const Key add = ((Key)cnt[r] << 12) + rk[r];
                            k[r] = b[r] ? (b[r] & ~(Key)4095) + add : 0;
                            d[r] = (uint32_t)(b[r] & 4095) - (uint32_t)rk[r];
                        }
                        if (SMEM_BACK) {
                            *(uint32_t *)bk = __byte_perm(__byte_perm(d[0], d[1], 0x0040),
                                                          __byte_perm(d[2], d[3], 0x0040), 0x5410);
                        } else {
#pragma unroll
                            for (int r = 0; r < kRoadRows; ++r)
                                if (j0 + r < H) bk[r] = (uint8_t)d[r];
                        }
                    }
                    road_store4(cur, k);
                }
                Key *const x = cur;
                cur = prev;
                prev = x;
                bk += SMEM_BACK ? HP : H;
                // the threads with rows only
                asm volatile("barrier.sync 1, %0;" ::"r"(ncomp) : "memory");
            }
        }
    }
    // best final row: the largest key
    Key key = 0;
#pragma unroll
    for (int r = 0; r < kRoadRows; ++r)
        if (own && j0 + r < H) key = road_max(key, k[r]);
    for (int o = 16; o > 0; o >>= 1) key = road_max(key, __shfl_xor_sync(0xFFFFFFFFu, key, o));
    if ((t & 31) == 0) red[t >> 5] = key;
    __syncthreads();
    if (t == 0) {
        Key b = 0;
        for (int x = 0; x < nt / 32; ++x) b = road_max(b, red[x]);
        const int64_t best = (int64_t)(b >> 12) - 1;
        int j = b == 0 ? -1 : 4095 - (int)(b & 4095);
        const uint8_t *row = (SMEM_BACK ? back : back_g) + (int64_t)(D - 1) * (SMEM_BACK ? HP : H);
        for (int i = D - 1; i >= 0; --i) {
            P[i] = j;
            if (j >= 0 && i > 0) j -= row[j];
            row -= SMEM_BACK ? HP : H;
        }
        *energy = best;
    }
}

template <int WM, bool SMEM_BACK, class Key>
void launch_road_w(const uint32_t *Hx, int H, int D, int eta, int32_t *P, int64_t *energy,
                   uint8_t *scratch, cudaStream_t s)
{
    const size_t smem = (sizeof(Key) * 2 * (kRoadPad + (size_t)road_rows(H)) +
                         (size_t)8 * road_chunk(H) * road_rows(H) +
                         (SMEM_BACK ? (size_t)D * road_rows(H) : 0));
    const int rows = ((H + kRoadRows - 1) / kRoadRows + 31) / 32 * 32;   // threads that own rows
    const int ncopy = rows + kRoadCopy <= 1024 ? kRoadCopy : 0;
    cudaFuncSetAttribute(road_kernel<WM, SMEM_BACK, Key>,
                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    road_kernel<WM, SMEM_BACK, Key><<<1, rows + ncopy, smem, s>>>(Hx, H, D, eta, road_chunk(H),
                                                                   ncopy, scratch, P, energy);
}

template <bool SMEM_BACK, class Key>
void launch_road_k(const uint32_t *Hx, int H, int D, int eta, int32_t *P, int64_t *energy,
                   uint8_t *scratch, cudaStream_t s)
{
    const int w = eta - 1;
    if (w < 4) return launch_road_w<-1, SMEM_BACK, Key>(Hx, H, D, eta, P, energy, scratch, s);
    switch (w & 3) {
    case 0: return launch_road_w<0, SMEM_BACK, Key>(Hx, H, D, eta, P, energy, scratch, s);
    case 1: return launch_road_w<1, SMEM_BACK, Key>(Hx, H, D, eta, P, energy, scratch, s);
    case 2: return launch_road_w<2, SMEM_BACK, Key>(Hx, H, D, eta, P, energy, scratch, s);
    default: return launch_road_w<3, SMEM_BACK, Key>(Hx, H, D, eta, P, energy, scratch, s);
    }
}

}  // namespace

size_t road_scratch_bytes(int H, int D) { return (size_t)H * D; }

// (sized for 64-bit keys, whichever run)
bool road_back_in_smem(int H, int D)
{
    const size_t HP = road_rows(H);
    return 16 * (kRoadPad + HP) + (size_t)8 * road_chunk(H) * HP + D * HP <= 200 * 1024;
}

void launch_road(const uint16_t *U, int W, int H, int pitch, int D, int eta, uint32_t *Hx,
                 uint32_t *Hy, int32_t *P, int64_t *energy, uint8_t *scratch, cudaStream_t s)
{
    vdisp_kernel<<<H, kHistThreads, sizeof(uint32_t) * D, s>>>(U, W, pitch, D, Hx);
    if (Hy) {
        const size_t smem = sizeof(uint32_t) * kUCols * (D + 1);
        cudaFuncSetAttribute(udisp_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        udisp_kernel<<<(W + kUCols - 1) / kUCols, kUThreads, smem, s>>>(U, W, H, pitch, D, Hy);
    }
    // a path's sum is at most D rows of W counts
    const bool narrow = (int64_t)W * D < (1 << 20) - 1;
    if (road_back_in_smem(H, D)) {
        if (narrow) launch_road_k<true, uint32_t>(Hx, H, D, eta, P, energy, nullptr, s);
        else launch_road_k<true, unsigned long long>(Hx, H, D, eta, P, energy, nullptr, s);
    } else {
        if (narrow) launch_road_k<false, uint32_t>(Hx, H, D, eta, P, energy, scratch, s);
        else launch_road_k<false, unsigned long long>(Hx, H, D, eta, P, energy, scratch, s);
    }
}

}  // namespace mpv
