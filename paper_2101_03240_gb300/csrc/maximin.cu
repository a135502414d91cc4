// maximin.cu -- widest-path (maximin) values from an image face, used by
// defending-phase trapping (Section 2.2.3) and by the trimming step of
// morphological-opening drainage (Section 2.4.1).
//
// For a value field val (0 = blocked, -1 = +infinity, else the value) and a
// face F, M[v] is the largest, over 6-paths through unblocked voxels from a
// voxel of F to v, of the smallest value on the path (v included); -1 where
// no such path exists.  Trapping thresholds it against seq (a voxel of step
// k is trapped iff M < k); opening keeps {M >= T}.
//
// GPU: M follows from a maximum spanning forest, built by Boruvka rounds on
// basins instead of voxels.
//  * Order voxels by (value, index).  A voxel with a larger neighbour p (the
//    largest one) has M[v] = min(val[v], M[p]): the edge to p is a largest
//    one at v, so some best path starts with it.  Following p leads to a
//    peak, along rising values, so M[v] = min(val[v], M[peak of v]): only
//    the peaks' values are wanted.  Pointers are resolved inside a tile in
//    shared memory first, then from tile to tile.
//  * Basins (the voxels of one peak) are joined through their best edges: of
//    all voxel pairs between a basin and others, and of its face voxels
//    (edges to the outside, of the voxel's own value), the one of largest
//    min(value).  With w its weight and D the basin beyond, M[C] = min(w,
//    M[D]) by the same argument.  Every round hooks each root with an edge
//    to the root beyond it (of two that choose each other the lower stays),
//    and flattens the hooks with the running minimum, until no root has an
//    edge; the outside is a root that never hooks, with M = infinity.
// Ties between edges are broken by the edge's number, so hooks form no cycle.
// After the first round the voxel pairs that still join different roots are
// gathered into a list (or looked at again, if they outnumber it).
//
// The field was propagated before by relaxing 4 x 8 x 32 tiles until nothing
// changed (about 20 activations a tile, 300 bytes a voxel, on a cooperative
// grid or a work queue).  Here each voxel is read in a fixed number of passes
// and everything is ordinary launches, so it runs beside other streams as it
// is.
#include <algorithm>
#include <vector>

#include "common.cuh"

namespace {

typedef unsigned long long u64;

constexpr int TX = 8, TY = 8, TZ = 32;          // tile of the pointer pass
constexpr int kTileVox = TX * TY * TZ;
constexpr int kThreads = 256;
constexpr int kPer = kTileVox / kThreads;       // voxels per thread
constexpr int kRoundsPerSync = 3;               // rounds launched between two looks at the flag
constexpr int kMaxRoundsDev = 64;               // each round at least halves the roots with an edge
constexpr uint32_t kBlocked = 0xffffffffu;
constexpr uint32_t kPeak = 0x80000000u;         // label: kPeak | number of the peak

// One image: its tiles and 32-voxel row segments are numbered globally.
struct MMJob {
    const int32_t *val;
    uint32_t *M;            // pointer (linear index), then label, then the value
    int nx, ny, nz, tx, ty, tz, face, segs;
    int tile0, unit0;       // first tile / segment
    int64_t vox0;           // voxels before this image
};

struct MMWork {
    const MMJob *jobs;
    int njobs, ntiles, nunits;
    u64 *node;              // per basin: parent (low) and the smallest weight on the way there (high); [P] = outside
    u64 *best;              // per root: weight << 33 | edge number of its best edge
    int *ctr;               // [0] peaks, [1] listed edges, [2 + r] roots hooked in round r
    int P;
    int *ea, *eb, *ew;      // list of edges: two roots and the weight
    int *cnt, block;        // entries left in each block of the list, its length
    int cap, listed;        // its length, and the entries in use (-1: not listed)
};

__device__ __forceinline__ int as_val(int v) { return v == -1 ? IBIP_INF32 : v; }

template <class F>
__device__ __forceinline__ int find_mm(int n, F first, int at)
{
    int lo = 0, hi = n;   // largest j with first(j) <= at
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (first(mid) <= at) lo = mid; else hi = mid;
    }
    return lo;
}

__device__ __forceinline__ uint32_t parent_of(const MMWork &w, uint32_t c) { return (uint32_t)__ldcg(w.node + c); }

// Pointers to the largest neighbour, resolved inside the tile: each voxel's
// M gets the label of its peak or the index of the first voxel outside the
// tile on the way there.
__global__ void __launch_bounds__(kThreads) k_mm_tile(MMWork w)
{
    constexpr int HX = TX + 2, HY = TY + 2, HZ = TZ + 2, kHalo = HX * HY * HZ;
    __shared__ int s_val[kHalo];
    __shared__ unsigned short s_ptr[kTileVox];
    __shared__ uint32_t s_tgt[kTileVox];
    const int tid = threadIdx.x, lane = tid & 31;
    const MMJob J = w.jobs[find_mm(w.njobs, [&](int j) { return w.jobs[j].tile0; }, (int)blockIdx.x)];
    const int t = (int)blockIdx.x - J.tile0;
    const int bz = t % J.tz, by = (t / J.tz) % J.ty, bx = t / (J.tz * J.ty);
    const int x0 = bx * TX, y0 = by * TY, z0 = bz * TZ;
    for (int i = tid; i < kHalo; i += kThreads) {
        const int hz = i % HZ, hy = (i / HZ) % HY, hx = i / (HZ * HY);
        const int x = x0 + hx - 1, y = y0 + hy - 1, z = z0 + hz - 1;
        int v = 0;
        if (x >= 0 && y >= 0 && z >= 0 && x < J.nx && y < J.ny && z < J.nz)
            v = as_val(__ldg(J.val + d_lin(x, y, z, J.ny, J.nz)));
        s_val[i] = v;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kPer; k++) {
        const int i = tid + k * kThreads;
        const int lz = i % TZ, ly = (i / TZ) % TY, lx = i / (TZ * TY);
        const int h = ((lx + 1) * HY + ly + 1) * HZ + lz + 1;
        const int v = s_val[h];
        // the largest of the voxel and its neighbours by (value, index): the
        // offsets in order of index are -x -y -z 0 +z +y +x
        const int off[7] = {-HY * HZ, -HZ, -1, 0, 1, HZ, HY * HZ};
        int b = -1, q = 3;
#pragma unroll
        for (int d = 0; d < 7; d++) {
            const int u = s_val[h + off[d]];
            if (u >= b) { b = u; q = d; }
        }
        int to = i;             // itself: a peak, blocked, or the way out of the tile
        uint32_t tgt = kBlocked;
        bool peak = false;
        if (v != 0) {
            if (q == 3) {
                peak = true;
            } else {
                const int dx = q == 0 ? -1 : q == 6 ? 1 : 0, dy = q == 1 ? -1 : q == 5 ? 1 : 0;
                const int dz = q == 2 ? -1 : q == 4 ? 1 : 0;
                const int ux = lx + dx, uy = ly + dy, uz = lz + dz;
                if (ux >= 0 && uy >= 0 && uz >= 0 && ux < TX && uy < TY && uz < TZ) to = (ux * TY + uy) * TZ + uz;
                else tgt = (uint32_t)d_lin(x0 + ux, y0 + uy, z0 + uz, J.ny, J.nz);
            }
        }
        const unsigned m = __ballot_sync(0xffffffffu, peak);
        if (m) {
            int id = 0;
            if (lane == 0) id = atomicAdd(w.ctr, __popc(m));
            id = __shfl_sync(0xffffffffu, id, 0) + __popc(m & ((1u << lane) - 1));
            if (peak) tgt = kPeak | (uint32_t)id;
        }
        s_ptr[i] = (unsigned short)to;
        s_tgt[i] = tgt;
    }
    __syncthreads();
    // follow the pointers to their ends inside the tile (they only rise, so
    // there is no cycle); doubling, at most 11 passes for 2,048 voxels
    for (int pass = 0; pass < 11; pass++) {
        int ch = 0;
#pragma unroll
        for (int k = 0; k < kPer; k++) {
            const int i = tid + k * kThreads;
            const unsigned short p = s_ptr[i], q = s_ptr[p];
            if (q != p) { s_ptr[i] = q; ch = 1; }
        }
        if (!__syncthreads_or(ch)) break;
    }
#pragma unroll
    for (int k = 0; k < kPer; k++) {
        const int i = tid + k * kThreads;
        const int lz = i % TZ, ly = (i / TZ) % TY, lx = i / (TZ * TY);
        const int x = x0 + lx, y = y0 + ly, z = z0 + lz;
        if (x < J.nx && y < J.ny && z < J.nz) J.M[d_lin(x, y, z, J.ny, J.nz)] = s_tgt[s_ptr[i]];
    }
}

// A warp's 32-voxel segment of a row: f(job, row, x, y, z, linear index, inside)
template <class F>
__device__ __forceinline__ void for_segments(const MMWork &w, F f)
{
    const int lane = threadIdx.x & 31, wpb = blockDim.x >> 5;
    for (int u = blockIdx.x * wpb + (threadIdx.x >> 5); u < w.nunits; u += gridDim.x * wpb) {
        const MMJob &J = w.jobs[find_mm(w.njobs, [&](int j) { return w.jobs[j].unit0; }, u)];
        const int i = u - J.unit0, row = i / J.segs, z = (i - row * J.segs) * 32 + lane;
        const int x = row / J.ny, y = row - x * J.ny;
        f(J, x, y, z, (int64_t)row * J.nz + z, z < J.nz);
    }
}

// the rest of the way to the peak, tile by tile
__global__ void __launch_bounds__(kThreads) k_mm_label(MMWork w)
{
    for_segments(w, [&](const MMJob &J, int, int, int, int64_t v, bool in) {
        if (!in) return;
        uint32_t p = __ldcg(J.M + v);
        if (p & kPeak) return;   // a label, or blocked
        while (!(p & kPeak)) p = __ldcg(J.M + p);
        __stcg(J.M + v, p);
    });
}

__global__ void k_mm_nodes(MMWork w)
{
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c <= w.P; c += gridDim.x * blockDim.x) {
        w.node[c] = (u64)IBIP_INF32 << 32 | (uint32_t)c;
        w.best[c] = 0ull;
    }
}

__device__ __forceinline__ void offer(const MMWork &w, uint32_t c, u64 key)
{
    if (key > __ldcg(w.best + c)) atomicMax(w.best + c, key);
}

constexpr int kChunk = 64;   // list entries a warp takes at a time
// List entries that shrink together, at most: fewer where the list does not
// fill the chip with that many to a warp.
constexpr int kBlockEdges = 512;
constexpr int kMaxSms = 256;   // SMs the tables are sized for

// Every voxel pair (the voxel and its +z, +y, +x neighbour) and every face
// voxel as an edge.  LIST: those between different roots are appended to the
// list, of each run of lanes with the same two roots only the largest; else
// they are offered to the two roots (the outside, root P, takes none).
template <bool LIST>
__global__ void __launch_bounds__(kThreads, 8) k_mm_pairs(MMWork w, int round)
{
    if (round > 0 && __ldcg(w.ctr + 2 + round - 1) == 0) return;
    const int lane = threadIdx.x & 31;
    int lbase = 0, lleft = 0;   // list entries of the warp
    bool full = false;          // the list has run out
    const bool first = round == 0;
    for_segments(w, [&](const MMJob &J, int x, int y, int z, int64_t v, bool in) {
        // the loads of all four directions side by side: labels, then values
        // and roots, then the roots' best edges
        const int64_t off[3] = {1, J.nz, (int64_t)J.ny * J.nz};
        const bool ok[3] = {z < J.nz - 1, y < J.ny - 1, x < J.nx - 1};
        const uint32_t lb = in ? __ldcg(J.M + v) : kBlocked;
        uint32_t lu[3];
#pragma unroll
        for (int d = 0; d < 3; d++) lu[d] = in && ok[d] ? __ldcg(J.M + v + off[d]) : kBlocked;
        const int val = lb != kBlocked ? as_val(__ldg(J.val + v)) : 0;
        uint32_t a = lb == kBlocked ? kBlocked : lb & ~kPeak;
        uint32_t bs[4];
        int ws[4];
#pragma unroll
        for (int d = 0; d < 3; d++) {
            bs[d] = kBlocked;
            ws[d] = 0;
            if (lb != kBlocked && lu[d] != kBlocked && lu[d] != lb) {
                bs[d] = lu[d] & ~kPeak;
                ws[d] = as_val(__ldg(J.val + v + off[d]));
                if (!first) bs[d] = parent_of(w, bs[d]);
            }
        }
        if (!first && a != kBlocked) a = parent_of(w, a);
#pragma unroll
        for (int d = 0; d < 3; d++) ws[d] = min(ws[d], val);
        const bool face = a != kBlocked && d_on_face(x, y, z, J.nx, J.ny, J.nz, J.face);
        bs[3] = face ? (uint32_t)w.P : kBlocked;
        ws[3] = val;
        if (!LIST) {
            u64 top = 0, had_b[3], had_a = 0;
            bool any = face && a != (uint32_t)w.P;
#pragma unroll
            for (int d = 0; d < 3; d++) {
                had_b[d] = ~0ull;
                if (bs[d] == kBlocked || bs[d] == a) continue;
                any = true;
                if (bs[d] != (uint32_t)w.P) had_b[d] = __ldcg(w.best + bs[d]);
            }
            if (!any) return;
            if (a != (uint32_t)w.P) had_a = __ldcg(w.best + a);
#pragma unroll
            for (int d = 0; d < 4; d++) {
                if (bs[d] == kBlocked || bs[d] == a) continue;
                const u64 key = (u64)(uint32_t)ws[d] << 33 | (u64)(4 * (J.vox0 + v) + d);
                top = key > top ? key : top;
                if (d < 3 && key > had_b[d]) atomicMax(w.best + bs[d], key);
            }
            if (a != (uint32_t)w.P && top > had_a) atomicMax(w.best + a, top);
            return;
        }
#pragma unroll
        for (int d = 0; d < 4; d++) {
            const uint32_t b = bs[d];
            int wt = ws[d];
            bool edge = b != kBlocked && a != b;
            if (!__any_sync(0xffffffffu, edge)) continue;
            // runs of the same two roots: the largest weight, kept by the
            // last lane of the run
            const uint32_t pa = __shfl_up_sync(0xffffffffu, a, 1), pb = __shfl_up_sync(0xffffffffu, b, 1);
            const bool cont = __shfl_up_sync(0xffffffffu, (int)edge, 1) && lane > 0 && edge && pa == a && pb == b;
            const unsigned heads = __ballot_sync(0xffffffffu, !cont);
            const int start = 31 - __clz(heads & (0xffffffffu >> (31 - lane)));
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(0xffffffffu, wt, o);
                if (lane - o >= start) wt = max(wt, t);
            }
            edge = edge && (lane == 31 || ((heads >> (lane + 1)) & 1u));
            const unsigned m = __ballot_sync(0xffffffffu, edge);
            const int need = __popc(m), k = __popc(m & ((1u << lane) - 1));
            int pos = lbase + k;
            if (lleft < need) {
                int nb = w.cap;
                if (lane == 0 && !full) nb = atomicAdd(w.ctr + 1, kChunk);
                nb = __shfl_sync(0xffffffffu, nb, 0);
                full = nb >= w.cap;   // the counter is left alone then (pairs may number three a voxel)
                nb -= lleft;
                if (k >= lleft) pos = nb + k;
                lbase = nb;
                lleft += kChunk;
            }
            if (edge && pos < w.cap) {
                w.ea[pos] = (int)a;
                w.eb[pos] = (int)b;
                w.ew[pos] = wt;
            }
            lbase += need;
            lleft -= need;
        }
    });
    if (LIST)   // the entries left over are no edges
        for (int i = lane; i < lleft; i += 32)
            if (lbase + i < w.cap) w.ea[lbase + i] = w.eb[lbase + i] = 0;
}

// The listed edges, a block of w.block to a warp: ends moved to their
// roots, then offered.  Edges within one basin leave the list and runs of
// edges between the same two basins (neighbours in the list are neighbours in
// the image) become their largest, so a block shrinks in place from round to
// round (`cnt`: what is left of it).  301 x 323 x 347, 12.6 M edges: the
// rounds' looks at the list took 1,035 us with every entry kept, 490 us so.
__global__ void __launch_bounds__(kThreads) k_mm_edges(MMWork w, int round)
{
    if (__ldcg(w.ctr + 2 + round - 1) == 0) return;
    const int lane = threadIdx.x & 31;
    const int nblk = (w.listed + w.block - 1) / w.block;
    for (int blk = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; blk < nblk; blk += (gridDim.x * blockDim.x) >> 5) {
        const int e0 = blk * w.block;
        const int n = round == 1 ? min(w.listed - e0, w.block) : w.cnt[blk];
        int out = 0;
        for (int i0 = 0; i0 < n; i0 += 32) {
            const int e = e0 + i0 + lane;
            uint32_t a = 0, b = 0;
            int wt = 0;
            if (i0 + lane < n) {
                a = (uint32_t)w.ea[e];
                b = (uint32_t)w.eb[e];
                wt = w.ew[e];
                if (a != b) {
                    a = parent_of(w, a);
                    b = parent_of(w, b);
                    if (a > b) { const uint32_t c = a; a = b; b = c; }
                }
            }
            bool edge = a != b;
            const uint32_t pa = __shfl_up_sync(0xffffffffu, a, 1), pb = __shfl_up_sync(0xffffffffu, b, 1);
            const bool cont = lane > 0 && edge && pa == a && pb == b;
            const unsigned heads = __ballot_sync(0xffffffffu, !cont);
            if (heads != 0xffffffffu) {
                const int start = 31 - __clz(heads & (0xffffffffu >> (31 - lane)));
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int t = __shfl_up_sync(0xffffffffu, wt, o);
                    if (lane - o >= start) wt = max(wt, t);
                }
                edge = edge && (lane == 31 || ((heads >> (lane + 1)) & 1u));
            }
            const unsigned m = __ballot_sync(0xffffffffu, edge);
            if (edge) {
                const int pos = e0 + out + __popc(m & ((1u << lane) - 1));
                w.ea[pos] = (int)a;
                w.eb[pos] = (int)b;
                w.ew[pos] = wt;
                const u64 key = (u64)(uint32_t)wt << 33 | (u64)pos;
                offer(w, a, key);   // (the outside has the largest number)
                if (b != (uint32_t)w.P) offer(w, b, key);
            }
            out += __popc(m);
            __syncwarp();
        }
        if (lane == 0) w.cnt[blk] = out;
    }
}

// each root hooks to the root beyond its best edge
__global__ void __launch_bounds__(kThreads) k_mm_hook(MMWork w, int round)
{
    if (round > 0 && __ldcg(w.ctr + 2 + round - 1) == 0) return;
    const int lane = threadIdx.x & 31;
    for (int c0 = (blockIdx.x * blockDim.x + threadIdx.x) & ~31; c0 < w.P; c0 += gridDim.x * blockDim.x) {
        const int c = c0 + lane;
        bool hook = false;
        if (c < w.P && (uint32_t)w.node[c] == (uint32_t)c) {
            const u64 key = __ldcg(w.best + c);
            if (key) {
                const u64 id = key & ((1ull << 33) - 1);
                uint32_t a, b;
                if (w.listed >= 0) {
                    a = (uint32_t)w.ea[id];
                    b = (uint32_t)w.eb[id];
                } else {
                    const int64_t gv = (int64_t)(id >> 2);
                    const int d = (int)(id & 3);
                    int lo = 0, hi = w.njobs;
                    while (hi - lo > 1) {
                        const int mid = (lo + hi) >> 1;
                        if (w.jobs[mid].vox0 <= gv) lo = mid; else hi = mid;
                    }
                    const MMJob &J = w.jobs[lo];
                    const int64_t v = gv - J.vox0;
                    a = __ldcg(J.M + v) & ~kPeak;
                    b = d == 3 ? (uint32_t)w.P
                               : __ldcg(J.M + v + (d == 0 ? 1 : d == 1 ? (int64_t)J.nz : (int64_t)J.ny * J.nz)) & ~kPeak;
                    if (round > 0) {   // c is one of the two roots: the labels' parents before this round's hooks
                        const uint32_t pa = parent_of(w, a), pb = d == 3 ? b : parent_of(w, b);
                        a = a == (uint32_t)c || pa == (uint32_t)c ? (uint32_t)c : pa;
                        b = b == (uint32_t)c || pb == (uint32_t)c ? (uint32_t)c : pb;
                    }
                }
                const uint32_t o = a == (uint32_t)c ? b : a;
                // (o == c: the other end has hooked to c just now)
                hook = o != (uint32_t)c && !(o != (uint32_t)w.P && __ldcg(w.best + o) == key && (uint32_t)c < o);
                if (hook) __stcg(w.node + c, (key >> 33) << 32 | o);
            }
        }
        const unsigned m = __ballot_sync(0xffffffffu, hook);
        if (m && lane == 0) atomicAdd(w.ctr + 2 + round, __popc(m));
    }
}

// hooks flattened: every basin points at its root, with the smallest weight
// on the way (the pair is one 64-bit word, so a half-done neighbour reads
// consistently)
__global__ void __launch_bounds__(kThreads) k_mm_flatten(MMWork w, int round)
{
    if (__ldcg(w.ctr + 2 + round) == 0) return;
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < w.P; c += gridDim.x * blockDim.x) {
        const u64 x = __ldcg(w.node + c);
        uint32_t p = (uint32_t)x, m = (uint32_t)(x >> 32);
        w.best[c] = 0ull;
        if (p == (uint32_t)c) continue;
        for (;;) {
            const u64 y = __ldcg(w.node + p);
            if ((uint32_t)y == p) break;
            m = min(m, (uint32_t)(y >> 32));
            p = (uint32_t)y;
        }
        __stcg(w.node + c, (u64)m << 32 | p);
    }
}

// M = min(value, the smallest weight to the outside), -1 where it is not reached
__global__ void __launch_bounds__(kThreads) k_mm_value(MMWork w)
{
    for_segments(w, [&](const MMJob &J, int, int, int, int64_t v, bool in) {
        if (!in) return;
        const uint32_t lb = __ldcg(J.M + v);
        const int val = as_val(__ldg(J.val + v));
        int m = -1;
        if (lb != kBlocked) {
            const u64 x = __ldcg(w.node + (lb & ~kPeak));
            if ((uint32_t)x == (uint32_t)w.P) m = min(val, (int)(x >> 32));
        }
        J.M[v] = (uint32_t)m;
    });
}

}  // namespace

// Table bytes for n images of vox voxels: the images, the counters and the
// counts of the list's blocks (at most one per kBlockEdges entries, or two
// per warp of a list that does not fill the chip).
size_t ibip_maximin_table_bytes(int n, int64_t vox)
{
    return (((size_t)n * sizeof(MMJob) + 255) & ~(size_t)255) +
           (2 + kMaxRoundsDev + (size_t)(vox / kBlockEdges) + 1 + 64 * (size_t)kMaxSms) * sizeof(int);
}

// The jobs' voxels together stay below 2^31.
static int mm_group(ibip_ctx *ctx, int n, const IbipMaximinJob *jobs)
{
    std::vector<MMJob> J(n);
    int64_t vox = 0, tiles = 0, units = 0;
    for (int j = 0; j < n; j++) {
        const ibip_dims d = jobs[j].d;
        MMJob &q = J[j];
        q.val = jobs[j].val;
        q.M = (uint32_t *)jobs[j].M;
        q.nx = d.nx; q.ny = d.ny; q.nz = d.nz; q.face = jobs[j].face;
        q.tx = (d.nx + TX - 1) / TX; q.ty = (d.ny + TY - 1) / TY; q.tz = (d.nz + TZ - 1) / TZ;
        q.segs = (d.nz + 31) / 32;
        q.tile0 = (int)tiles; q.unit0 = (int)units; q.vox0 = vox;
        tiles += (int64_t)q.tx * q.ty * q.tz;
        units += (int64_t)d.nx * d.ny * q.segs;
        vox += nvox(d);
    }
    if (tiles >= (1ll << 31) || units >= (1ll << 31)) return IBIP_ERR_ARG;
    cudaStream_t s = ctx->stream;
    const size_t jb = ((size_t)n * sizeof(MMJob) + 255) & ~(size_t)255;
    const size_t cb = (2 + kMaxRoundsDev) * sizeof(int);
    char *t = (char *)ibip_scratch(ctx, SC_TILE, ibip_maximin_table_bytes(n, vox));
    if (!t) return IBIP_ERR_OOM;
    MMWork w = {};
    w.jobs = (const MMJob *)t;
    w.njobs = n;
    w.ntiles = (int)tiles;
    w.nunits = (int)units;
    w.ctr = (int *)(t + jb);
    w.cnt = (int *)(t + jb + cb);
    w.listed = -1;
    ibip_prof_begin(ctx, IBIP_K_MAXIMIN);
    cudaMemcpyAsync(t, J.data(), (size_t)n * sizeof(MMJob), cudaMemcpyHostToDevice, s);
    cudaMemsetAsync(w.ctr, 0, cb, s);
    if (ctx->stream_inv) {
        // server slot: on the high-priority stream, ahead of the wide kernels
        // of the other jobs
        if (cudaEventRecord(ctx->ev_inv, s) != cudaSuccess ||
            cudaStreamWaitEvent(ctx->stream_inv, ctx->ev_inv, 0) != cudaSuccess)
            return ibip_cuda_status(cudaGetLastError());
        s = ctx->stream_inv;
    }
    const int wide = (int)std::min<int64_t>((units + kThreads / 32 - 1) / (kThreads / 32), (int64_t)ctx->sm_count * 32);
    k_mm_tile<<<w.ntiles, kThreads, 0, s>>>(w);
    k_mm_label<<<wide, kThreads, 0, s>>>(w);
    ctx->launches += 2;
    int *h = (int *)ctx->h_pinned;
    cudaMemcpyAsync(h, w.ctr, sizeof(int), cudaMemcpyDeviceToHost, s);
    if (ibip_sync(ctx, s) != cudaSuccess) return ibip_cuda_status(cudaGetLastError());
    w.P = h[0];
    int rounds = 0;
    if (w.P > 0) {
        // The tables share slots with the invasion, the EDT and the curve,
        // none of which runs meanwhile.  No more than half the voxels are
        // peaks; half an edge a voxel is usual.
        int64_t cap = vox;
        if (ctx->arena && ctx->slot[SC_LIST]) cap = std::min<int64_t>(cap, (int64_t)(ctx->slot_bytes[SC_LIST] / 4));
        w.cap = (int)std::min<int64_t>(std::max<int64_t>(cap, 1), 1 << 30);   // places stay below 2^31
        w.node = (u64 *)ibip_scratch(ctx, SC_OKEY, ((size_t)w.P + 1) * sizeof(u64));
        w.best = (u64 *)ibip_scratch(ctx, SC_HIST, ((size_t)w.P + 1) * sizeof(u64));
        w.ea = (int *)ibip_scratch(ctx, SC_RANK, (size_t)w.cap * 4);
        w.eb = (int *)ibip_scratch(ctx, SC_G2, (size_t)w.cap * 4);
        w.ew = (int *)ibip_scratch(ctx, SC_LIST, (size_t)w.cap * 4);
        if (!w.best || !w.node || !w.ea || !w.eb || !w.ew) return IBIP_ERR_OOM;
    }
    const int gp = (int)std::min<int64_t>(((int64_t)w.P + 1 + kThreads - 1) / kThreads, (int64_t)ctx->sm_count * 16);
    if (w.P > 0) {
        k_mm_nodes<<<gp, kThreads, 0, s>>>(w);
        k_mm_pairs<false><<<wide, kThreads, 0, s>>>(w, 0);
        k_mm_hook<<<gp, kThreads, 0, s>>>(w, 0);
        k_mm_flatten<<<gp, kThreads, 0, s>>>(w, 0);
        k_mm_pairs<true><<<std::min(wide, ctx->sm_count * 8), kThreads, 0, s>>>(w, 1);
        ctx->launches += 5;
        cudaMemcpyAsync(h, w.ctr, 3 * sizeof(int), cudaMemcpyDeviceToHost, s);
        if (ibip_sync(ctx, s) != cudaSuccess) return ibip_cuda_status(cudaGetLastError());
        const bool list = h[1] <= w.cap;
        bool more = h[1] > 0 && h[2] > 0;   // the list counts its unused entries too
        if (list) w.listed = h[1];
        const int warps = std::min(ctx->sm_count, kMaxSms) * 32;
        w.block = std::min(std::max((h[1] / warps + 31) & ~31, 32), kBlockEdges);
        const int ge = (int)std::min<int64_t>(((int64_t)h[1] + kThreads - 1) / kThreads + 1, (int64_t)ctx->sm_count * 16);
        rounds = 1;
        while (more) {
            const int r1 = std::min(rounds + kRoundsPerSync, kMaxRoundsDev);
            for (; rounds < r1; rounds++) {
                if (list) k_mm_edges<<<ge, kThreads, 0, s>>>(w, rounds);
                else k_mm_pairs<false><<<wide, kThreads, 0, s>>>(w, rounds);
                k_mm_hook<<<gp, kThreads, 0, s>>>(w, rounds);
                k_mm_flatten<<<gp, kThreads, 0, s>>>(w, rounds);
                ctx->launches += 3;
            }
            cudaMemcpyAsync(h, w.ctr + 2 + rounds - 1, sizeof(int), cudaMemcpyDeviceToHost, s);
            if (ibip_sync(ctx, s) != cudaSuccess) return ibip_cuda_status(cudaGetLastError());
            more = h[0] > 0;
            if (more && rounds == kMaxRoundsDev) {   // cannot happen: 2^63 basins
                ibip_prof_end(ctx, IBIP_K_MAXIMIN);
                return IBIP_ERR_NOT_CONVERGED;
            }
        }
    }
    k_mm_value<<<wide, kThreads, 0, s>>>(w);
    ctx->launches++;
    if (s != ctx->stream) {
        // what follows on the slot's own stream
        if (cudaEventRecord(ctx->ev_inv, s) != cudaSuccess ||
            cudaStreamWaitEvent(ctx->stream, ctx->ev_inv, 0) != cudaSuccess)
            return ibip_cuda_status(cudaGetLastError());
    }
    ibip_prof_end(ctx, IBIP_K_MAXIMIN);
    ctx->inv_stats[30] = rounds;
    ctx->inv_stats[31] = w.P;
    ctx->inv_stats[32] = w.listed;
    return ibip_cuda_status(cudaGetLastError());
}

int ibip_maximin_multi(ibip_ctx *ctx, int n, const IbipMaximinJob *jobs)
{
    for (int j = 0; j < n;) {
        int64_t vox = 0;
        int m = j;
        while (m < n && (m == j || vox + nvox(jobs[m].d) < (1ll << 31))) vox += nvox(jobs[m++].d);
        const int st = mm_group(ctx, m - j, jobs + j);
        if (st) return st;
        j = m;
    }
    return IBIP_OK;
}

int ibip_maximin_launch(ibip_ctx *ctx, const int32_t *val, ibip_dims d, int face, int32_t *M)
{
    IbipMaximinJob j{val, d, face, M};
    return ibip_maximin_multi(ctx, 1, &j);
}
