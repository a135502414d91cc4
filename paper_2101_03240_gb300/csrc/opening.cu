// opening.cu -- the dilations of morphological-opening drainage (Section
// 2.4.1) on bit planes.
//
// Level i of the opening marks every pore voxel without a level that lies
// within squared distance < Td[i] of the level's trimmed set {W >= T[i]}.
// The sets grow with i.  As long as Td does not, a centre of an earlier
// level marked a larger ball then, so only the centres that are new at
// level i are dilated (a level whose Td is above the one before it takes
// its whole set).
//
//   k_open_planes  one bit per voxel and level: the centres to dilate, 32
//                  voxels along z to a word, for up to 32 levels at once;
//   k_open_dilate  a block holds a tile of 16 x 32 rows of 32 voxels and
//                  walks the levels: the rows of centres within reach go to
//                  shared memory as windows of 64 (or 96) bits around the
//                  tile's 32, and the ball is the union over its disk of
//                  row offsets (dx, dy), each widened along z by
//                  w = isqrt(Td - 1 - dx^2 - dy^2).  With the offsets sorted
//                  by dx^2 + dy^2 the widths fall, so one accumulator per
//                  row, widened by one bit each time w falls by one, does
//                  them all: one shared load and two ORs per offset for 32
//                  voxels.  Where few of the rows hold a centre (the first
//                  levels of an image, most tiles of any level), the rows
//                  with one are stamped instead, a warp each, a lane per
//                  offset, by atomicOr on the tile.
//
// The dilations of 29 levels at 255 x 260 x 277 take 0.85 ms; three EDT passes
// a level took 5.2 ms.
//
// Integer and exact.  The tile is 32 voxels along z because labels and
// planes are read and written in rows; 16 x 32 rows because the halo of a
// radius of 10 then costs 3.7 loads per row, and the windows of a block
// (24 KB at 64 bits) leave six blocks to an SM.  Bound by the shared loads
// of dense tiles (64 bits per offset and lane).
#include <algorithm>

#include "common.cuh"

namespace {

constexpr int kMaxT = 1024;       // largest Td of the tables: w < 32
constexpr int kTX = 16, kTY = 32; // rows of a tile
constexpr int kThreads = 256;
constexpr int kChunk = 32;        // levels per pair of launches
// Rows with a centre that are stamped, at most: 24, 48, 80, 160 and 320 take
// 0.85, 0.89, 1.04, 1.27 and 1.49 ms at 255 x 260 x 277 with radii to 21, and
// 2.82, 2.81, 2.95, 3.91 and 5.37 ms at 260^3 with radii to 26.
constexpr int kSparse = 32;

constexpr int disk_count()
{
    int n = 0;
    for (int x = -31; x <= 31; x++)
        for (int y = -31; y <= 31; y++) n += x * x + y * y < kMaxT;
    return n;
}
constexpr int kDisk = disk_count();

// Window of a row of centres: NW words around the tile's one.
__host__ __device__ constexpr int halo(int nw) { return nw == 2 ? 16 : 32; }
__host__ __device__ constexpr int pitch(int nw) { return kTY + 2 * halo(nw); }
__host__ __device__ constexpr int win_rows(int nw) { return (kTX + 2 * halo(nw)) * pitch(nw); }

// Row offsets with dx^2 + dy^2 < kMaxT by ascending dx^2 + dy^2; cnt[q] of
// them have dx^2 + dy^2 <= q.
struct Disk {
    int8_t dx[kDisk], dy[kDisk];
    uint16_t cnt[kMaxT];
};
struct DiskOffsets {   // the same as index offsets in the window arrays
    int16_t off[2][kDisk];
    uint16_t cnt[kMaxT];
};

constexpr Disk make_disk()
{
    Disk t{};
    int n = 0;
    int start[kMaxT + 1] = {};
    for (int x = -31; x <= 31; x++)
        for (int y = -31; y <= 31; y++)
            if (x * x + y * y < kMaxT) start[x * x + y * y + 1]++;
    for (int q = 0; q < kMaxT; q++) {
        start[q + 1] += start[q];
        t.cnt[q] = (uint16_t)start[q + 1];
    }
    for (int x = -31; x <= 31; x++)
        for (int y = -31; y <= 31; y++)
            if (x * x + y * y < kMaxT) {
                n = start[x * x + y * y]++;
                t.dx[n] = (int8_t)x;
                t.dy[n] = (int8_t)y;
            }
    return t;
}
constexpr DiskOffsets make_offsets()
{
    const Disk d = make_disk();
    DiskOffsets t{};
    for (int i = 0; i < kDisk; i++) {
        t.off[0][i] = (int16_t)(d.dx[i] * pitch(2) + d.dy[i]);
        t.off[1][i] = (int16_t)(d.dx[i] * pitch(3) + d.dy[i]);
    }
    for (int q = 0; q < kMaxT; q++) t.cnt[q] = d.cnt[q];
    return t;
}
__device__ const Disk g_disk = make_disk();              // read by lane
__constant__ const DiskOffsets c_off = make_offsets();   // read by warp

struct Levels {
    int n, first;              // levels of the launch, index of the first
    int prev;                  // radius of the level before the first
    uint32_t whole;            // levels that take their whole set
    int T[kChunk], Td[kChunk];
};

// planes[(l * nzw + zw) * nrows + row]: consecutive rows are consecutive
// words, so that a block of the dilation reads a tile's rows in lines.
// 32 rows of one word each to a block, four to a warp.
__global__ void __launch_bounds__(kThreads) k_open_planes(const int32_t *__restrict__ W, int nrows, int nz, int nzw,
                                                          Levels p, uint32_t *__restrict__ planes)
{
    __shared__ uint32_t s[32][33];
    __shared__ int s_T[kChunk];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int zw = blockIdx.y, z = zw * 32 + lane;
    const int64_t row0 = (int64_t)blockIdx.x * 32;
    int v[4];
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const int64_t row = row0 + warp + 8 * k;
        v[k] = row < nrows && z < nz ? W[row * nz + z] : -1;   // radii are positive: -1 is no centre
    }
    if (threadIdx.x < kChunk) s_T[threadIdx.x] = (int)threadIdx.x < p.n ? p.T[threadIdx.x] : 0;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 4; k++) {
        int l = kChunk;
        if (p.first > 0 && v[k] >= p.prev) {
            l = -1;   // a centre since before this launch
        } else {
            int lo = 0, hi = p.n;   // T is strictly decreasing: first index with T <= v
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (s_T[mid] <= v[k]) hi = mid; else lo = mid + 1;
            }
            if (lo < p.n) l = lo;
        }
        uint32_t mine = 0;
        for (uint32_t rem = __ballot_sync(~0u, l >= 0 && l < kChunk); rem;) {
            const int at = __shfl_sync(~0u, l, __ffs(rem) - 1);
            const uint32_t b = __ballot_sync(~0u, l == at);
            if (lane == at) mine = b;
            rem &= ~b;
        }
        for (uint32_t m = p.whole; m; m &= m - 1) {
            const int at = __ffs(m) - 1;
            const uint32_t b = __ballot_sync(~0u, l <= at);
            if (lane == at) mine = b;
        }
        s[warp + 8 * k][lane] = mine;
    }
    __syncthreads();
    if (row0 + lane < nrows)
        for (int l = warp; l < p.n; l += kThreads / 32)
            planes[((int64_t)l * nzw + zw) * nrows + row0 + lane] = s[lane][l];
}

template <int NW>
struct Window;
template <>
struct Window<2> {
    typedef unsigned long long Bits;
    static __device__ __forceinline__ Bits make(uint32_t a, uint32_t b, uint32_t c)
    {
        return ((Bits)__funnelshift_l(b, c, 16) << 32) | __funnelshift_l(a, b, 16);
    }
    static __device__ __forceinline__ Bits load(const uint32_t *s, int i) { return ((const Bits *)s)[i]; }
    static __device__ __forceinline__ void store(uint32_t *s, int i, Bits v) { ((Bits *)s)[i] = v; }
    static __device__ __forceinline__ uint32_t tile(Bits v) { return (uint32_t)(v >> 16); }
};
template <>
struct Window<3> {
    typedef unsigned __int128 Bits;   // 96 used
    static constexpr int kPlane = win_rows(3);
    static __device__ __forceinline__ Bits make(uint32_t a, uint32_t b, uint32_t c)
    {
        return ((Bits)c << 64) | ((unsigned long long)b << 32) | a;
    }
    static __device__ __forceinline__ Bits load(const uint32_t *s, int i)
    {
        return make(s[i], s[kPlane + i], s[2 * kPlane + i]);
    }
    static __device__ __forceinline__ void store(uint32_t *s, int i, Bits v)
    {
        s[i] = (uint32_t)v;
        s[kPlane + i] = (uint32_t)(v >> 32);
        s[2 * kPlane + i] = (uint32_t)(v >> 64);
    }
    static __device__ __forceinline__ uint32_t tile(Bits v) { return (uint32_t)(v >> 32); }
};

// Every bit with a set bit within w of it (bits near the ends may be missing).
template <class Bits>
__device__ __forceinline__ Bits widened(Bits v, int w)
{
    Bits u = v;   // both ways at once: u to higher bits, v to lower
    for (int have = 0; have < w;) {
        const int step = min(have + 1, w - have);
        u |= u << step;
        v |= v >> step;
        have += step;
    }
    return u | v;
}

template <int NW>
constexpr size_t open_smem()
{
    return (size_t)NW * win_rows(NW) * sizeof(uint32_t);
}

template <int NW>
__global__ void __launch_bounds__(kThreads) k_open_dilate(const uint32_t *__restrict__ planes, int nx, int ny, int nz, int nzw,
                                                          Levels p, int32_t *level)
{
    typedef Window<NW> Win;
    typedef typename Win::Bits Bits;
    constexpr int H = halo(NW), P = pitch(NW);
    extern __shared__ __align__(16) uint32_t s_win[];
    __shared__ uint32_t s_acc[kTX * kTY];
    __shared__ uint16_t s_list[kSparse];
    __shared__ int s_cnt[2];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int zw = blockIdx.x, z = zw * 32 + lane, y0 = blockIdx.y * kTY, x0 = blockIdx.z * kTX;
    const int64_t nrows = (int64_t)nx * ny;
    // this thread's rows: (x0 + warp, y0 + lane) and eight further in x
    uint32_t need[2];
#pragma unroll
    for (int o = 0; o < 2; o++) {
        const int x = x0 + warp + 8 * o;
        uint32_t m = 0;
        if (x < nx)
#pragma unroll 8
            for (int y = 0; y < kTY; y++) {
                const bool b = y0 + y < ny && z < nz && level[((int64_t)x * ny + y0 + y) * nz + z] == -1;
                const uint32_t bits = __ballot_sync(~0u, b);
                if (lane == y) m = bits;
            }
        need[o] = m;
    }
    if (tid < 2) s_cnt[tid] = 0;
    if (!__syncthreads_or(need[0] | need[1])) return;
    for (int l = 0; l < p.n; l++) {
        const int T = p.Td[l];
        int r = 0;
        while ((r + 1) * (r + 1) < T) r++;
        const uint32_t *pl = planes + ((int64_t)l * nzw + zw) * nrows;
        Bits mask = (Bits)0xffffffffu;   // bits of a window within reach of the tile
        mask = ((mask << r | mask) << r | mask) << (H - r);
        for (int xx = warp; xx < kTX + 2 * r; xx += kThreads / 32) {
            const int x = x0 - r + xx;
            for (int yy = lane; yy - lane < kTY + 2 * r; yy += 32) {
                const int y = y0 - r + yy;
                uint32_t a = 0, b = 0, c = 0;
                if (x >= 0 && x < nx && y >= 0 && y < ny && yy < kTY + 2 * r) {
                    const int64_t row = (int64_t)x * ny + y;
                    b = pl[row];
                    if (zw > 0) a = pl[row - nrows];
                    if (zw + 1 < nzw) c = pl[row + nrows];
                }
                const Bits v = Win::make(a, b, c);
                const int at = (xx - r + H) * P + yy - r + H;
                if (yy < kTY + 2 * r) Win::store(s_win, at, v);
                const uint32_t some = __ballot_sync(~0u, (v & mask) != 0);
                if (some) {
                    int base = 0;
                    if (lane == 0) base = atomicAdd(&s_cnt[l & 1], __popc(some));
                    base = __shfl_sync(~0u, base, 0) + __popc(some & ((1u << lane) - 1));
                    if ((some >> lane & 1) && base < kSparse) s_list[base] = (uint16_t)at;
                }
            }
        }
        s_acc[tid] = 0;
        s_acc[tid + kThreads] = 0;
        __syncthreads();
        const int cnt = s_cnt[l & 1];
        if (tid == 0) s_cnt[(l + 1) & 1] = 0;
        uint32_t out[2] = {0, 0};
        if (cnt > kSparse) {
            // what the row's own centres leave
            const int at = (warp + H) * P + lane + H;
            const uint32_t own0 = Win::tile(widened(Win::load(s_win, at), r));
            const uint32_t own1 = Win::tile(widened(Win::load(s_win, at + 8 * P), r));
            out[0] = own0;
            out[1] = own1;
            if (__any_sync(~0u, (need[0] & ~own0) | (need[1] & ~own1))) {
                Bits acc0 = 0, acc1 = 0;
                int k = 0;
                for (int w = r; w >= 0; w--) {
                    acc0 |= acc0 << 1 | acc0 >> 1;
                    acc1 |= acc1 << 1 | acc1 >> 1;
                    const int e = c_off.cnt[T - 1 - w * w];
#pragma unroll 4
                    for (; k < e; k++) {
                        const int i = at + c_off.off[NW - 2][k];
                        acc0 |= Win::load(s_win, i);
                        acc1 |= Win::load(s_win, i + 8 * P);
                    }
                }
                out[0] = Win::tile(acc0);
                out[1] = Win::tile(acc1);
            }
        } else if (cnt > 0) {
            const int nd = c_off.cnt[T - 1];
            for (int j = warp; j < cnt; j += kThreads / 32) {
                const int at = s_list[j];
                const int wx = at / P - H, wy = at % P - H;
                // lane w: the row's centres widened by w, the tile's bits
                const uint32_t wide = Win::tile(widened(Win::load(s_win, at), min(lane, r)));
                int w = r;
                for (int k = lane; k - lane < nd; k += 32) {
                    int x = -1, y = -1;
                    if (k < nd) {
                        const int dx = g_disk.dx[k], dy = g_disk.dy[k];
                        while (w * w + dx * dx + dy * dy >= T) w--;
                        x = wx + dx;
                        y = wy + dy;
                    }
                    const uint32_t bits = __shfl_sync(~0u, wide, w);
                    if (bits && x >= 0 && x < kTX && y >= 0 && y < kTY) atomicOr(&s_acc[x * kTY + y], bits);
                }
            }
            __syncthreads();
            out[0] = s_acc[tid];
            out[1] = s_acc[tid + kThreads];
        }
#pragma unroll
        for (int o = 0; o < 2; o++) {
            const uint32_t got = out[o] & need[o];
            need[o] &= ~got;
            for (uint32_t m = __ballot_sync(~0u, got != 0); m; m &= m - 1) {
                const int y = __ffs(m) - 1;
                const uint32_t bits = __shfl_sync(~0u, got, y);
                if (bits >> lane & 1)
                    level[((int64_t)(x0 + warp + 8 * o) * ny + y0 + y) * nz + z] = p.first + l + 1;
            }
        }
        if (!__syncthreads_or(need[0] | need[1])) return;
    }
}

}  // namespace

// Whether ibip_open_run takes a level.  Up to 16 voxels of reach the windows
// are 64 bits, up to 31 they are 96; the first levels of an image, which have
// the large radii, have few centres.  260^3 with 59 levels to Td = 698 takes
// 2.8 ms against 8.3 ms by EDT passes; the worst found is one level on an open
// image whose centres are the image (250 x 260 x 270, Td = 1024: 0.23 ms
// against 0.16).  Below 16 voxels along z the words are mostly padding.
static bool open_takes(ibip_dims d, int Td) { return d.nz >= 16 && Td <= kMaxT; }

// Levels [i, *next) of the opening on bit planes; *next == i: none of them.
int ibip_open_run(ibip_ctx *ctx, const int32_t *W, ibip_dims d, const int32_t *T, const int32_t *Td, int i, int n,
                  int32_t *level, int *next)
{
    *next = i;
    if (!open_takes(d, Td[i])) return IBIP_OK;
    const int nzw = (d.nz + 31) / 32, nrows = d.nx * d.ny;
    const int64_t words = (int64_t)nzw * nrows;
    const int most = (int)std::min<int64_t>(kChunk, nvox(d) / words);   // the planes take the slot the EDT passes take
    uint32_t *planes = (uint32_t *)ibip_scratch(ctx, SC_G2, nvox(d) * sizeof(int32_t));
    if (!planes) return IBIP_ERR_OOM;
    const bool wide = Td[i] > 289;   // reach above 16 voxels
    Levels p{};
    p.first = i;
    p.prev = i > 0 ? T[i - 1] : 0;
    for (; i < n && p.n < most && open_takes(d, Td[i]) && (Td[i] > 289) == wide; i++) {
        p.T[p.n] = T[i];
        p.Td[p.n] = Td[i];
        if (i > 0 && Td[i] > Td[i - 1]) p.whole |= 1u << p.n;
        p.n++;
    }
    *next = i;
    cudaStream_t s = ctx->stream;
    ibip_prof_begin(ctx, IBIP_K_DILATE);
    k_open_planes<<<dim3((nrows + 31) / 32, nzw), kThreads, 0, s>>>(W, nrows, d.nz, nzw, p, planes);
    IBIP_LAUNCH(ctx);
    const dim3 grid(nzw, (d.ny + kTY - 1) / kTY, (d.nx + kTX - 1) / kTX);
    if (wide) {
        cudaFuncSetAttribute(k_open_dilate<3>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)open_smem<3>());
        k_open_dilate<3><<<grid, kThreads, open_smem<3>(), s>>>(planes, d.nx, d.ny, d.nz, nzw, p, level);
    } else {
        k_open_dilate<2><<<grid, kThreads, open_smem<2>(), s>>>(planes, d.nx, d.ny, d.nz, nzw, p, level);
    }
    IBIP_LAUNCH(ctx);
    ibip_prof_end(ctx, IBIP_K_DILATE);
    return ibip_cuda_status(cudaGetLastError());
}
