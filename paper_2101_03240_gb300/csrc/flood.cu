// flood.cu -- volume-controlled invasion (Section 2.1, Figures 1-2) by value
// phases: the step sequence of invade.cu, computed in parallel.
//
// The rule picks the best candidate (largest dt2, lowest index on ties) one
// step at a time, but most of that order is a merge of independent runs:
//
//  * Phases.  Let t be the largest candidate value.  Until every candidate
//    of value >= t is used up, each step's centre has dt2 >= t: the steps
//    fall into phases of decreasing t, consecutive in time.
//  * Groups.  Within a phase the only voxels that matter are the uninvaded
//    ones with dt2 >= t.  A step covers those in its ball and makes
//    candidates of those beside it.  Start one group per candidate of value
//    t (a root) and run each group by itself, a small priority queue of its
//    own, from the state at the start of the phase.  As long as no two
//    groups touch a common voxel of value >= t (cover it, or make it a
//    candidate; merely lying beside another group's root changes nothing),
//    every group takes the steps it takes in the true sequence, in the same
//    order.  Each touched voxel carries the id of its group (`claim`, an
//    atomic maximum); a group that meets another's id joins the two, and the
//    joined group is run again from the start of the phase.  Balls of two
//    groups may share voxels of smaller value: those go to the earlier step
//    by an atomic minimum on the sequence image.
//  * Order.  The true sequence always takes the best head among the groups,
//    so it is sorted by (running worst candidate of the group, place within
//    the group).  A step that is worse than all earlier steps of its group
//    is a record; a record has value t and carries the run of steps up to
//    the next one.  The label of a step is the number of steps before the
//    phase, plus the lengths of the runs whose record has a lower index,
//    plus the place in its run.
//
// Measured on a serial prototype of this file: the 200^3 pack's 420,616
// steps fall into 69 phases and 121 rounds of groups whose longest groups add
// up to 4,922 steps; the 256^3 blobs' 631,020 steps into 109 phases, 189
// rounds and 3,226 steps.  That sum is what is left of the serial chain.
//
// One persistent kernel runs everything (set-up, phases, labels): on a
// cooperative grid of one CTA per SM for a large image, or on one
// thread-block cluster per image (batches, small images, and contexts that
// share the device), with a barrier of that team between the stages.  Small
// groups run on one warp each (single-voxel roots with nothing around them
// on one lane), groups of large balls and joined groups on a whole CTA.
//
// What a phase cannot hold (a group beyond its step budget or queue, more
// roots or steps than the tables take) stops the kernel before anything of the
// phase is stamped; the caller then lets the one-CTA loop of invade.cu go on
// from the steps taken.
#include <cooperative_groups.h>

#include <algorithm>
#include <climits>

#include "common.cuh"
#include "flood.cuh"

namespace cg = cooperative_groups;

namespace {

typedef unsigned long long u64;
typedef unsigned int u32;

constexpr int kFT = 512;               // threads per CTA
constexpr int kFW = kFT / 32;
constexpr int kQW = 64;                // queue entries of a warp's group
constexpr int kQC = 8192;              // queue entries of a CTA's group
constexpr int kU = 4;                  // state chunks a thread loads together
constexpr int kHits = 16 * kFT;        // candidates listed before they are appended, per CTA
constexpr int kWarpHits = kHits / kFW;
constexpr int kCurSmem = 2048;         // roots of a phase whose groups' ids fit in shared memory
constexpr int kHistSmem = 16384;       // values counted in shared memory
constexpr int kLongAfter = 96;          // steps after which a CTA's group is run on the bit planes
constexpr int kHuge = 1024;            // r2 from which the whole team stamps a ball
constexpr u64 kNone = ~0ull;
constexpr int kFailCancel = 3;         // FloodCtl::fail: a long group met the cancel request
constexpr int kLast = (int)0x80000000; // log flag: last step of its run
constexpr unsigned long long kBarrierNs = 20000000000ull;   // a barrier gives up after this

__device__ __forceinline__ u64 now_ns()
{
    u64 t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Priority of a candidate: larger dt2 first, then the lower index (x, y, z
// in order); dimensions are at most 2^14 and dt2 at most 2^15 - 1.
__device__ __forceinline__ u64 make_key(int r2, int x, int y, int z)
{
    return ((u64)(u32)(kFloodMaxVal - r2) << 42) | ((u64)x << 28) | ((u64)y << 14) | (u64)z;
}
__device__ __forceinline__ int key_r2(u64 k) { return kFloodMaxVal - (int)(k >> 42); }
__device__ __forceinline__ int key_x(u64 k) { return (int)((k >> 28) & 0x3fff); }
__device__ __forceinline__ int key_y(u64 k) { return (int)((k >> 14) & 0x3fff); }
__device__ __forceinline__ int key_z(u64 k) { return (int)(k & 0x3fff); }

__device__ __forceinline__ u64 warp_min(u64 k)
{
    const u32 hi = (u32)(k >> 32);
    const u32 mh = __reduce_min_sync(0xffffffffu, hi);
    const u32 ml = __reduce_min_sync(0xffffffffu, hi == mh ? (u32)k : 0xffffffffu);
    return ((u64)mh << 32) | ml;
}

// Index checks.  In a checked build (IBIP_CHECKED) an index outside its
// array's extent is recorded (the place in the code and the index), the
// access is skipped and the call returns IBIP_ERR_BOUNDS; nothing traps.
enum Place {
    P_CLAIM = 1, P_STATE, P_LISTS, P_ROOT, P_LOG, P_VALUE, P_QUEUE, P_ISQ, P_HIT, P_STEP, P_PLANE,
    P_VOXEL
};
__device__ __forceinline__ bool in_range(FloodCtl *ctl, int64_t i, int64_t n, int place)
{
#ifdef IBIP_CHECKED
    if (i >= 0 && i < n) return true;
    if (atomicCAS(&ctl->bad, 0, place) == 0) ctl->bad_index = i;
    return false;
#else
    (void)ctl; (void)i; (void)n; (void)place;
    return true;
#endif
}

// CTA-wide state in shared memory; the queues (and the set-up's histogram)
// are the dynamic part.
struct Shared {
    u64 red[kFW];
    int nq;                  // entries of the CTA group's queue
    int abort;               // bit 0: the group met another, 1: its queue is full, 2: too many steps, 3: cancelled
    int wnq[kFW];            // entries of each warp group's queue
    int wflag[kFW];          // `abort` of each warp group
    int t, g;
    int sum[kFW];
    int total;
};

struct Ball {
    int x, y, z, r2;
};

// Voxels that become candidates: index and value.
struct Hits {
    u32 *at;
    unsigned short *val;
};

// Row (dx, dy) from the centre of a ball: the half-width h of the ball's run
// (-1: the row misses it), and hs, that of ball and shell together (voxels
// with a face neighbour in the ball; -1: none).  A row's shell reaches as far
// as the widest of its four neighbour rows, which is the one towards the
// centre (inside the image whenever the row is), or one past its own run.
// isq[e] = floor(sqrt(e)).
__device__ __forceinline__ void shell_row(const unsigned char *isq, int r2, int dx, int dy, int &h, int &hs)
{
    const int e = r2 - 1 - dx * dx - dy * dy;
    const int m = max(abs(dx), abs(dy));
    const int el = m ? e + 2 * m - 1 : e - 1;
    h = e >= 0 ? (int)isq[e] : -1;
    hs = max(el >= 0 ? (int)isq[el] : -1, e >= 0 ? h + 1 : -1);
}

// The rows of a ball's dilated square.  The state image is read in aligned
// 16-byte chunks of 8 voxels, kU of a row together; no row has more than
// nch of them.
struct Rows {
    int X0, Y0, wy, n, nch;
    float inv;   // 1 / wy
};

__device__ __forceinline__ Rows ball_rows(int nx, int ny, const unsigned char *isq, const Ball &b)
{
    const int H = (int)isq[b.r2 - 1] + 1;
    Rows r;
    r.X0 = max(b.x - H, 0);
    r.Y0 = max(b.y - H, 0);
    r.wy = min(b.y + H, ny - 1) - r.Y0 + 1;
    r.n = (min(b.x + H, nx - 1) - r.X0 + 1) * r.wy;
    r.nch = (2 * H + 7) / 8 + 1;   // 2H + 1 voxels at any alignment
    r.inv = __fdividef(1.0f, (float)r.wy);
    return r;
}

// row r of the square: r < 2^18 and wy <= 365, so the rounded quotient of
// r + 1/2 never crosses an integer
__device__ __forceinline__ void row_at(const Rows &rw, int r, int &X, int &Y)
{
    const int rx = (int)(((float)r + 0.5f) * rw.inv);
    X = rw.X0 + rx;
    Y = rw.Y0 + r - rx * rw.wy;
}

// Chunk masks keep the even voxels of the chunk in bits 0-3 and the odd ones
// in bits 16-19, as they fall out of the packed 16-bit values.
// voxel of bit b
__device__ __forceinline__ int bit_voxel(int b) { return b < 16 ? 2 * b : 2 * (b - 16) + 1; }
// voxels with value >= t (tt = t in both halves; values below 2^15)
__device__ __forceinline__ u32 chunk_ge(const uint4 &w, u32 tt)
{
    const u32 a = ((w.x | 0x80008000u) - tt) & 0x80008000u, b = ((w.y | 0x80008000u) - tt) & 0x80008000u;
    const u32 c = ((w.z | 0x80008000u) - tt) & 0x80008000u, d = ((w.w | 0x80008000u) - tt) & 0x80008000u;
    return a >> 15 | b >> 14 | c >> 13 | d >> 12;
}
// voxels with the candidate bit
__device__ __forceinline__ u32 chunk_cand(const uint4 &w)
{
    return (w.x & 0x80008000u) >> 15 | (w.y & 0x80008000u) >> 14 | (w.z & 0x80008000u) >> 13 | (w.w & 0x80008000u) >> 12;
}
__device__ __forceinline__ int chunk_val(const uint4 &w, int b)
{
    const int k = b & 15;
    const u32 x = k < 2 ? (k == 0 ? w.x : w.y) : (k == 2 ? w.z : w.w);
    return (int)((b < 16 ? x : x >> 16) & 0x7fffu);
}
// the voxels [lo, hi] of a chunk (positions relative to its first; empty if
// lo > hi after clamping)
__device__ __forceinline__ u32 chunk_span(int lo, int hi)
{
    lo = max(lo, 0);
    hi = min(hi, 7);
    if (lo > hi) return 0u;
    const u32 e = (2u << (hi >> 1)) - (1u << ((lo + 1) >> 1)), o = (1u << ((hi + 1) >> 1)) - (1u << (lo >> 1));
    return e | o << 16;
}

__device__ __forceinline__ void coords(int ny, int nz, int v, int &x, int &y, int &z)
{
    const u32 r = (u32)v / (u32)nz;
    z = (int)((u32)v - r * (u32)nz);
    x = (int)(r / (u32)ny);
    y = (int)(r - (u32)x * (u32)ny);
}

__device__ __forceinline__ int ld_state(const Flood &f, int64_t v)
{
    return (int)__ldcg((const unsigned short *)f.state + v);
}

// ------------------------------------------------------------ team barrier --

// All CTAs of the image: a cluster barrier, or for the cooperative grid a
// counter in global memory (one arrival per CTA; the wait is bounded and
// raises the failure flag).  Returns false when the image is given up.
template <bool CLUSTER>
__device__ __forceinline__ bool team_sync(const Flood &f, int T, u32 &epoch)
{
    if (CLUSTER) {
        cg::this_cluster().sync();
        return true;
    }
    __threadfence();
    __syncthreads();
    __shared__ int s_ok;
    if (threadIdx.x == 0) {
        epoch += (u32)T;
        atomicAdd(&f.ctl->bar, 1u);
        const u64 t0 = now_ns();
        int ok = 1;
        u32 spins = 0;
        while ((int)(*(volatile u32 *)&f.ctl->bar - epoch) < 0) {
            if ((++spins & 1023u) == 0 && now_ns() - t0 > kBarrierNs) {
                atomicExch(&f.ctl->fail, 2);
                ok = 0;
                break;
            }
        }
        __threadfence();
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

// ---------------------------------------------------------- union of groups --

__device__ __forceinline__ int find_rep(const Flood &f, int a)
{
    for (int p; (p = __ldcg(f.parent + a)) != a; a = p) {}
    return a;
}

// joins groups a and b; both are to be run again in round `round`
__device__ void join_groups(const Flood &f, int a, int b, int round)
{
    atomicMax(f.dirty + a, 4 * round);
    atomicMax(f.dirty + b, 4 * round);
    for (;;) {
        a = find_rep(f, a);
        b = find_rep(f, b);
        if (a == b) return;
        if (a < b) { const int c = a; a = b; b = c; }
        if (atomicCAS(f.parent + a, a, b) == a) return;
    }
}

// ------------------------------------------------------------------- log --

// A writer's share of the phase's step log: `left` slots from base + used.
// The next share is asked for as soon as the last slot is used, long before
// it is needed, so no step waits for the counter (unused slots are marked
// empty when the writer is done).
struct LogPos {
    int base, used, left;
};

__device__ __forceinline__ void log_put(int4 *log, int log_cap, int *nlog, LogPos &lp, int chunk, int v, int rec, int off, u32 gid)
{
    const int pos = lp.base + lp.used;
    if (pos < log_cap) __stcg(log + pos, make_int4(v, rec, off, (int)gid));
    lp.used++;
    if (--lp.left == 0) {
        lp.base = atomicAdd(nlog, chunk);
        lp.used = 0;
        lp.left = chunk;
    }
}

__device__ __forceinline__ void log_open(int *nlog, LogPos &lp, int chunk)
{
    if (lp.left) return;
    lp.base = atomicAdd(nlog, chunk);
    lp.used = 0;
    lp.left = chunk;
}

__device__ __forceinline__ void log_close(const Flood &f, LogPos &lp)
{
    for (; lp.left > 0; lp.left--, lp.used++)
        if (lp.base + lp.used < f.log_cap) __stcg(f.log + lp.base + lp.used, make_int4(-1, -1, 0, 0));
}

// ----------------------------------------------------------------- groups --

// The constants of one round of groups.
struct Phase {
    int t, R, round, chunk;
    u32 pbase;
};

// position of the k-th (0-based) set bit of m
__device__ __forceinline__ int nth_bit(u32 m, int k)
{
    int pos = 0, c;
    c = __popc(m & 0xffffu); if (k >= c) { k -= c; m >>= 16; pos = 16; }
    c = __popc(m & 0xffu);   if (k >= c) { k -= c; m >>= 8;  pos += 8; }
    c = __popc(m & 0xfu);    if (k >= c) { k -= c; m >>= 4;  pos += 4; }
    c = __popc(m & 0x3u);    if (k >= c) { k -= c; m >>= 2;  pos += 2; }
    return pos + (k >= (int)(m & 1u) ? 1 : 0);
}

enum Team { WARP, BLOCK, LONG };   // a group on a warp, on the CTA, on the CTA with the bit planes

// Runs the group of root `rep` (id `gid`) to its end.  Each step: drop the
// queue's entries covered by the last ball, take the best one left; then,
// a row of its dilated ball per lane, the voxels of value >= t as a mask of
// 32, whose set bits the lanes of the warp claim together, one round trip
// for up to 32 of them; a shell voxel that was no candidate before joins the
// queue.  What bounds a step is the chain of instructions and round trips
// from one step to the next, not the work: rows are dealt to the warps in
// turn, so that the full rows at the centre are spread over all of them.
// Neither the state image nor the planes change while groups run, so their
// loads go through the L1 (the barrier before the round orders them): 512^3
// blobs 105.5 -> 102.5 ms, 200^3 pack 19.0 -> 18.4.
// A long group takes its masks from two bit planes (`fresh`: uninvaded, no
// candidate; `root_bits`: the phase's roots), two words for a row instead of
// up to four 16-byte chunks of the state image.
template <Team TEAM>
__device__ __noinline__ LogPos run_group(const Flood &f, const Phase &ph_in, Shared &sh, u64 *q, const u32 *s_cur,
                                         const unsigned char *isq, int rep, u32 gid, LogPos lp)
{
    constexpr bool CTA = TEAM != WARP;
    constexpr int W = CTA ? kFT : 32;
    constexpr int NWARP = W / 32;
    constexpr int QN = CTA ? kQC : kQW;
    constexpr int kLog = CTA ? kFT - 32 : 0;   // the thread that logs
    constexpr int kPoll = kFT - 64;            // the thread that reads the cancel flag
    // the loop's constants as values: f and the phase are in memory, and every
    // atomic would make the compiler read them again
    const Phase ph = ph_in;
    const u32 tt = (u32)ph.t * 0x10001u;
    const int nx = f.nx, ny = f.ny, nz = f.nz, log_cap = f.log_cap, NW = (f.nz + 31) >> 5;
    // steps one group may take: a CTA's group then goes to the planes, a long
    // one is a chain that the one-CTA loop runs faster
    const int budget = TEAM == WARP ? 1024 : TEAM == BLOCK ? kLongAfter : f.budget;
    const uint4 *const state = (const uint4 *)f.state;
    const u32 *const fresh = f.fresh, *const root_bits = f.root_bits;
    u32 *const claim = f.claim;
    const u32 *const cur = f.cur;
    int4 *const log = f.log;
    FloodCtl *const ctl = f.ctl;
    int *const nlog = &ctl->nlog;
    const int n_vox = nx * ny * nz;   // below 2^31
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int tid = CTA ? (int)threadIdx.x : lane;
    int *s_nq = CTA ? &sh.nq : &sh.wnq[warp];
    int *s_abort = CTA ? &sh.abort : &sh.wflag[warp];
    auto sync = [&]() { if (CTA) __syncthreads(); else __syncwarp(); };
    if (tid == 0) {
        int n = 0, bad = 0;
        int i = ph.round == 0 ? rep : __ldcg(f.head + rep);
        while (i >= 0 && in_range(ctl, i, ph.R, P_ROOT)) {
            if (n == QN) { bad = 2; break; }
            int x, y, z;
            coords(ny, nz, __ldcg(f.roots + i), x, y, z);
            q[n++] = make_key(ph.t, x, y, z);
            if (ph.round == 0) break;
            i = __ldcg(f.next + i);
        }
        *s_nq = n;
        *s_abort = bad;
    }
    if (tid == kLog) log_open(nlog, lp, ph.chunk);
    sync();
    if (*s_abort == 0) {
        Ball b{0, 0, 0, 0};   // r2 = 0: covers nothing
        u64 worst = 0;
        int pv = -1, prec = -1, poff = 0, steps = 0;   // the step not yet logged
        for (;;) {
            // -- queue: remove what the last ball covers, find the best entry
            const int nq = *s_nq;
            u64 best = kNone;
            auto covered = [&](u64 k) {
                const int dx = key_x(k) - b.x, dy = key_y(k) - b.y, dz = key_z(k) - b.z;
                return dx * dx + dy * dy + dz * dz < b.r2;
            };
            if (CTA) {
                const bool count = nq > 1024;   // the same for every thread
                int live = 0;
                for (int i = tid; i < nq; i += W) {
                    const u64 k = q[i];
                    if (k == kNone) continue;
                    if (covered(k)) { q[i] = kNone; continue; }
                    live++;
                    best = k < best ? k : best;
                }
                best = warp_min(best);
                if (count) live = __reduce_add_sync(0xffffffffu, live);
                if (lane == 0) { sh.red[warp] = best; sh.sum[warp] = live; }
                __syncthreads();
                best = warp_min(lane < kFW ? sh.red[lane] : kNone);
                if (count) {
                    live = __reduce_add_sync(0xffffffffu, lane < kFW ? sh.sum[lane] : 0);
                    if (live * 2 < nq) {
                        // close the holes: the entries move down, one pass of the CTA at a time
                        int out = 0;
                        for (int i0 = 0; i0 < nq; i0 += kFT) {
                            const u64 k = i0 + tid < nq ? q[i0 + tid] : kNone;
                            const unsigned m = __ballot_sync(0xffffffffu, k != kNone);
                            __syncthreads();   // sh.sum and this pass's entries have been read
                            if (lane == 0) sh.sum[warp] = __popc(m);
                            __syncthreads();
                            int at = out, all = 0;
                            for (int w = 0; w < kFW; w++) {
                                if (w < warp) at += sh.sum[w];
                                all += sh.sum[w];
                            }
                            if (k != kNone) q[at + __popc(m & ((1u << lane) - 1))] = k;
                            out += all;
                        }
                        if (tid == 0) *s_nq = out;
                        __syncthreads();
                    }
                }
            } else {
                int out = 0;
                for (int c = 0; c < nq; c += 32) {
                    const u64 k = c + lane < nq ? q[c + lane] : kNone;
                    const bool keep = k != kNone && !covered(k);
                    const unsigned m = __ballot_sync(0xffffffffu, keep);
                    if (keep) {
                        q[out + __popc(m & ((1u << lane) - 1))] = k;
                        best = k < best ? k : best;
                    }
                    out += __popc(m);
                    __syncwarp();
                }
                best = warp_min(best);
                if (lane == 0) *s_nq = out;
                __syncwarp();
            }
            if (best == kNone) break;
            // -- the step
            b.x = key_x(best); b.y = key_y(best); b.z = key_z(best); b.r2 = key_r2(best);
            const bool rec = best > worst;
            if (tid == kLog && pv >= 0) log_put(log, log_cap, nlog, lp, ph.chunk, pv, prec, poff | (rec ? kLast : 0), gid);
            pv = (b.x * ny + b.y) * nz + b.z;
            if (rec) { worst = best; prec = pv; poff = 0; } else poff++;
            if (!in_range(ctl, b.r2 - 1, f.maxd, P_ISQ) || !in_range(ctl, pv, n_vox, P_VOXEL)) b.r2 = 1;
            // a long group may run for tens of milliseconds
            if (TEAM == LONG && tid == kPoll && (steps & 511) == 511 && f.cancel && *(const volatile int *)f.cancel) {
                atomicExch(&ctl->fail, kFailCancel);
                atomicOr(s_abort, 8);
            }
            if (++steps > budget) {
                if (tid == 0) *s_abort = 4;
                sync();
                break;
            }
            // -- its rows
            const Rows rw = ball_rows(nx, ny, isq, b);
            const int widest = 2 * (int)isq[b.r2 - 1] + 3;   // voxels of the longest row
            const int passes = TEAM == LONG ? (widest + 31) / 32 : (rw.nch + kU - 1) / kU;
            for (int r0 = 0; r0 < rw.n; r0 += W) {
                const int r = r0 + lane * NWARP + (CTA ? warp : 0);
                int X = 0, Y = 0, h = -1, hs = -1;
                if (r < rw.n) {
                    row_at(rw, r, X, Y);
                    shell_row(isq, b.r2, X - b.x, Y - b.y, h, hs);
                }
                const int za = max(b.z - hs, 0), zb = min(b.z + hs, nz - 1);
                for (int ps = 0; ps < passes; ps++) {
                    u32 all = 0, in = 0;   // voxels to claim, those of them in the ball
                    int z0 = 0;            // z of bit 0
                    if (TEAM == LONG) {
                        // bit k = voxel z0 + k
                        z0 = za + 32 * ps;
                        const int z1 = min(zb, z0 + 31);
                        if (hs >= 0 && z0 <= z1) {
                            const int w = (X * ny + Y) * NW + (z0 >> 5);
                            const bool two = (z0 >> 5) != (z1 >> 5);
                            u32 f0 = 0, f1 = 0, g0 = 0, g1 = 0;
                            if (in_range(ctl, w, nx * ny * NW, P_PLANE) && in_range(ctl, w + two, nx * ny * NW, P_PLANE)) {
                                f0 = fresh[w];
                                g0 = root_bits[w];
                                f1 = fresh[w + two];
                                g1 = root_bits[w + two];
                            }
                            const u32 span = 0xffffffffu >> (31 - (z1 - z0));
                            const u32 fr = __funnelshift_r(f0, f1, z0 & 31) & span;
                            const u32 rt = __funnelshift_r(g0, g1, z0 & 31) & span;
                            const int ra = max(b.z - h, z0) - z0, rb = min(b.z + h, z1) - z0;
                            const u32 run = h >= 0 && ra <= rb ? (0xffffffffu >> (31 - rb)) & (0xffffffffu << ra) : 0u;
                            in = (fr | rt) & run;
                            all = in | (fr & ~run);
                        }
                    } else if (hs >= 0) {
                        // kU chunks of the row, eight bits each: even voxels, then odd ones
                        const int base = (X * ny + Y) * nz;
                        const int c = ((base + za) >> 3) + ps * kU;
                        const int n_ch = ((base + zb) >> 3) - c + 1;
                        z0 = c * 8 - base;
                        uint4 cw[kU];
#pragma unroll
                        for (int u = 0; u < kU; u++)
                            cw[u] = u < n_ch && in_range(ctl, c + u, (n_vox + 7) / 8, P_STATE) ? state[c + u]
                                                                                             : make_uint4(0, 0, 0, 0);
#pragma unroll
                        for (int u = 0; u < kU; u++) {
                            if (u >= n_ch) break;
                            u32 ge = chunk_ge(cw[u], tt);
                            if (!ge) continue;
                            const int zc = z0 + 8 * u;
                            const u32 run = h >= 0 ? chunk_span(b.z - h - zc, b.z + h - zc) : 0u;
                            // another candidate beside the ball stays as it is
                            ge &= chunk_span(za - zc, zb - zc) & (run | ~chunk_cand(cw[u]));
                            all |= ((ge & 0xfu) | (ge >> 12 & 0xf0u)) << (8 * u);
                            in |= ((run & 0xfu) | (run >> 12 & 0xf0u)) << (8 * u);
                        }
                    }
                    // the warp's bits, 32 at a time: lane e takes the e-th
                    const int n = __popc(all);
                    int inc = n;
                    if (!__any_sync(0xffffffffu, n)) continue;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const int u = __shfl_up_sync(0xffffffffu, inc, o);
                        if (lane >= o) inc += u;
                    }
                    const int tot = __shfl_sync(0xffffffffu, inc, 31);
                    const u32 at = (u32)X << 16 | (u32)Y;   // the row (below 2^14 each)
                    for (int e0 = 0; e0 < tot; e0 += 32) {
                        const int e = e0 + lane;
                        int src = 0;
#pragma unroll
                        for (int o = 16; o; o >>= 1) {
                            const int v = __shfl_sync(0xffffffffu, inc, src + o - 1);
                            if (v <= e) src += o;
                        }
                        src = min(src, 31);
                        const u32 m = __shfl_sync(0xffffffffu, all, src), mi = __shfl_sync(0xffffffffu, in, src);
                        const u32 row = __shfl_sync(0xffffffffu, at, src);
                        const int ex = __shfl_sync(0xffffffffu, inc - n, src), zz = __shfl_sync(0xffffffffu, z0, src);
                        u32 old = gid;
                        int vx = 0, vy = 0, vz = 0, val = 1;
                        bool inside = true;
                        if (e < tot) {
                            const int k = nth_bit(m, e - ex);
                            vx = (int)(row >> 16);
                            vy = (int)(row & 0xffffu);
                            vz = zz + (TEAM == LONG ? k : (k & ~7) + ((k & 4) ? 2 * (k & 3) + 1 : 2 * (k & 3)));
                            inside = (mi >> k) & 1u;
                            const int u = (vx * ny + vy) * nz + vz;
                            if (in_range(ctl, u, n_vox, P_CLAIM)) {
                                old = atomicMax(claim + u, gid);
                                if (!inside) val = (int)((const unsigned short *)state)[u];   // beside the claim
                            }
                        }
                        bool push = old != gid;
                        if (old >= ph.pbase && push) {
                            const int o = (int)((old - ph.pbase) % (u32)ph.R);
                            if ((ph.R <= kCurSmem ? s_cur[o] : __ldcg(cur + o)) == old) {   // a live group of this phase
                                join_groups(f, rep, o, ph.round + 1);
                                atomicOr(s_abort, 1);
                                push = false;
                            }
                        }
                        push = push && !inside;
                        const unsigned pm = __ballot_sync(0xffffffffu, push);
                        if (!pm) continue;
                        int slot = 0;
                        if (lane == 0) slot = atomicAdd(s_nq, __popc(pm));
                        slot = __shfl_sync(0xffffffffu, slot, 0) + __popc(pm & ((1u << lane) - 1));
                        if (push) {
                            if (slot < QN && in_range(ctl, slot, QN, P_QUEUE)) q[slot] = make_key(val, vx, vy, vz);
                            else atomicOr(s_abort, 2);
                        }
                    }
                }
            }
            sync();
            if (*(volatile int *)s_abort) break;
        }
        if (tid == kLog && pv >= 0) log_put(log, log_cap, nlog, lp, ph.chunk, pv, prec, poff | kLast, gid);
    }
    sync();
    if (tid == 0 && *s_abort) {
        const int ab = *s_abort;
        atomicExch(&ctl->changed, 1);
        // queue full or too many steps: from a warp to a CTA, from there to
        // the planes (where a group stays), from there to the one-CTA loop
        if (TEAM == LONG) {
            if (ab & 6) atomicExch(&ctl->fail, 1);
            atomicMax(f.dirty + rep, 4 * (ph.round + 1) + 3);
        } else if (ab & 6) {
            atomicMax(f.dirty + rep, 4 * (ph.round + 1) + (CTA || (ab & 4) ? 3 : 1));
        }
    }
    sync();
    return lp;
}

// --------------------------------------------------------- stamping a ball --

// Rows [r0, rows) step `stride` of ball b: the label by atomic minimum, and
// the voxels leave the state image.  G lanes (a power of two) share a row.
__device__ __forceinline__ void stamp_rows(const Flood &f, const unsigned char *isq, const Ball &b, u32 label,
                                           int row0, int stride, int sub, int G)
{
    const int nx = f.nx, ny = f.ny, nz = f.nz;
    u32 *const seq = (u32 *)f.seq;
    unsigned short *const state = f.state;
    const Rows rw = ball_rows(nx, ny, isq, b);
    for (int r = row0; r < rw.n; r += stride) {
        int X, Y;
        row_at(rw, r, X, Y);
        const int e = b.r2 - 1 - (X - b.x) * (X - b.x) - (Y - b.y) * (Y - b.y);
        if (e < 0) continue;
        const int h = (int)isq[e];
        const int z0 = max(b.z - h, 0), z1 = min(b.z + h, nz - 1);
        const int base = (X * ny + Y) * nz;
        for (int z = z0 + sub; z <= z1; z += G) {
            if (!in_range(f.ctl, base + z, (int64_t)nx * ny * nz, P_VOXEL)) continue;
            atomicMin(seq + base + z, label);
            state[base + z] = 0;
        }
    }
}

// Appends the n listed candidates of a warp to the lists of their values,
// one counter update per value and 32 entries, four of them in flight.
__device__ void flush_hits(const Flood &f, const Hits &hit, int n)
{
    const int lane = threadIdx.x & 31;
    for (int i0 = 0; i0 < n; i0 += 128) {
        int slot[4], val[4];
        unsigned peers[4];
#pragma unroll
        for (int p = 0; p < 4; p++) {
            const int i = i0 + p * 32 + lane;
            val[p] = i < n ? (int)hit.val[i] : 0;
            peers[p] = __match_any_sync(0xffffffffu, val[p]);
            slot[p] = 0;
            if (val[p] && lane == __ffs(peers[p]) - 1 && in_range(f.ctl, val[p], f.maxd + 1, P_VALUE))
                slot[p] = atomicAdd(f.cnt + val[p], __popc(peers[p]));
        }
#pragma unroll
        for (int p = 0; p < 4; p++) {
            const int s = __shfl_sync(0xffffffffu, slot[p], __ffs(peers[p]) - 1) + __popc(peers[p] & ((1u << lane) - 1));
            if (val[p] && in_range(f.ctl, val[p], f.maxd + 1, P_VALUE) &&
                in_range(f.ctl, __ldcg(f.off + val[p]) + s, f.npore, P_LISTS))
                __stcg(f.lists + __ldcg(f.off + val[p]) + s, (int)hit.at[i0 + p * 32 + lane]);
        }
    }
    __syncwarp();
}

// The shell of ball b, rows first, first + stride, ... (a warp, one row per
// lane): each uninvaded voxel that was never a candidate becomes one and is
// listed (n entries so far, flushed when full).
__device__ __forceinline__ void expose_ball(const Flood &f, const unsigned char *isq, const Ball &b, int first,
                                            int stride, const Hits &hit, int &n)
{
    const int nx = f.nx, ny = f.ny, nz = f.nz;
    u32 *const state = (u32 *)f.state;
    const int lane = threadIdx.x & 31;
    const Rows rw = ball_rows(nx, ny, isq, b);
    for (int r0 = first; r0 < rw.n; r0 += stride) {
        const int r = r0 + lane;
        int n_ch = 0, za = 0, zb = -1, z0 = 0;
        int c0 = 0;
        if (r < rw.n) {
            int X, Y, h, hs;
            row_at(rw, r, X, Y);
            shell_row(isq, b.r2, X - b.x, Y - b.y, h, hs);
            if (hs >= 0) {
                za = max(b.z - hs, 0);
                zb = min(b.z + hs, nz - 1);
                const int base = (X * ny + Y) * nz;
                c0 = (base + za) >> 3;
                n_ch = ((base + zb) >> 3) - c0 + 1;
                z0 = c0 * 8 - base;
            }
        }
        for (int k = 0; k < rw.nch; k += 2) {
            uint4 cw[2];
            u32 fresh[2];
#pragma unroll
            for (int u = 0; u < 2; u++)
                cw[u] = k + u < n_ch && in_range(f.ctl, c0 + k + u, ((int64_t)nx * ny * nz + 7) / 8, P_STATE)
                            ? __ldcg((const uint4 *)state + c0 + k + u) : make_uint4(0, 0, 0, 0);
            int m = 0;
#pragma unroll
            for (int u = 0; u < 2; u++) {
                // uninvaded and no candidate yet
                fresh[u] = 0;
                if (k + u >= n_ch) continue;
                fresh[u] = chunk_ge(cw[u], 0x10001u) & ~chunk_cand(cw[u]) &
                           chunk_span(za - z0 - 8 * (k + u), zb - z0 - 8 * (k + u));
                if (!fresh[u]) continue;
                u32 old[4];
#pragma unroll
                for (int p = 0; p < 4; p++) {
                    const u32 two = (fresh[u] >> p) & 0x10001u;
                    old[p] = two ? atomicOr(state + (c0 + k + u) * 4 + p, two << 15) : 0u;
                }
                fresh[u] &= ~chunk_cand(make_uint4(old[0], old[1], old[2], old[3]));
                m += __popc(fresh[u]);
            }
            if (!__any_sync(0xffffffffu, m)) continue;
            int pos = m;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, pos, o);
                if (lane >= o) pos += u;
            }
            const int tot = __shfl_sync(0xffffffffu, pos, 31);
            if (n + tot > kWarpHits) {
                __syncwarp();
                flush_hits(f, hit, n);
                n = 0;
            }
            pos += n - m;
#pragma unroll
            for (int u = 0; u < 2; u++)
                for (u32 w = fresh[u]; w; w &= w - 1, pos++) {
                    const int bit = __ffs(w) - 1;
                    if (!in_range(f.ctl, pos, kWarpHits, P_HIT)) continue;
                    hit.at[pos] = (u32)((c0 + k + u) * 8 + bit_voxel(bit));
                    hit.val[pos] = (unsigned short)chunk_val(cw[u], bit);
                }
            n += tot;
        }
    }
}

// appends voxel v (state s, not yet a candidate) as a candidate
__device__ __forceinline__ void seed_voxel(const Flood &f, int64_t v, int s)
{
    atomicOr((u32 *)f.state + (v >> 1), (v & 1) ? 0x80000000u : 0x8000u);
    const unsigned act = __activemask();
    const unsigned peers = __match_any_sync(act, s);
    const int lane = threadIdx.x & 31, leader = __ffs(peers) - 1;
    int slot = 0;
    if (lane == leader) slot = atomicAdd(f.cnt + s, __popc(peers));
    slot = __shfl_sync(peers, slot, leader) + __popc(peers & ((1u << lane) - 1));
    __stcg(f.lists + __ldcg(f.off + s) + slot, (int)v);
}

// block-wide exclusive prefix of one value per thread; *total = block sum
__device__ int block_excl(Shared &sh, int v, int *total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += u;
    }
    __syncthreads();
    if (lane == 31) sh.sum[warp] = inc;
    __syncthreads();
    int base = 0, all = 0;
    for (int w = 0; w < kFW; w++) {
        if (w < warp) base += sh.sum[w];
        all += sh.sum[w];
    }
    *total = all;
    return base + inc - v;
}

// ------------------------------------------------------------------ kernel --

// The whole invasion of one image on the T CTAs of its team (this is CTA c).
template <bool CLUSTER>
__device__ void flood_body(const Flood &f, const int T, const int c)
{
    extern __shared__ __align__(16) unsigned char s_dyn[];
    __shared__ Shared sh;
    u64 *s_q = (u64 *)s_dyn;                                    // queues (set-up: histogram)
    unsigned char *s_hit = s_dyn + (size_t)kQC * 8;             // listed candidates
    u32 *s_cur = (u32 *)(s_hit + (size_t)kHits * 6);            // ids of the phase's groups, if they fit
    unsigned char *isq = (unsigned char *)(s_cur + kCurSmem);   // floor(sqrt(e)), e <= maxd
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nx = f.nx, ny = f.ny, nz = f.nz;
    const int64_t N = (int64_t)nx * ny * nz;
    const int64_t gt = (int64_t)c * kFT + tid, GT = (int64_t)T * kFT;
    const int gw = c * kFW + warp, GW = T * kFW;
    const Hits whits{(u32 *)s_hit + warp * kWarpHits, (unsigned short *)(s_hit + (size_t)kHits * 4) + warp * kWarpHits};
    u32 epoch = 0;
    FloodCtl *ctl = f.ctl;

    // ---- set-up: clear the tables, then state, sequence and value counts
    if (c == 0 && tid == 0) { f.out[0] = -1; f.out[1] = kFloodGiveUp; }   // until the end is reached
    for (int64_t i = gt; i <= f.maxd; i += GT) f.cnt[i] = 0;
    for (int64_t i = gt; i < f.plane_words; i += GT) f.plane[i] = 0u;
    {
        uint4 *c4 = (uint4 *)f.claim;   // 256-byte aligned, padded to 16 bytes
        for (int64_t i = gt; i < (N + 3) / 4; i += GT) c4[i] = make_uint4(0, 0, 0, 0);
    }
    for (int e = tid; e <= f.maxd; e += kFT) isq[e] = (unsigned char)d_isqrt(e);
    int *s_hist = (int *)s_q;
    const bool smem_hist = f.maxd < kHistSmem;
    if (smem_hist)
        for (int i = tid; i <= f.maxd; i += kFT) s_hist[i] = 0;
    if (!team_sync<CLUSTER>(f, T, epoch)) return;
    auto count = [&](int d) {
        if (smem_hist) atomicAdd(s_hist + d, 1); else atomicAdd(f.cnt + d, 1);
    };
    if (!f.resume && (((uintptr_t)f.dt2 | (uintptr_t)f.seq) & 15) == 0) {
        // two vectors of four voxels per thread: 16-byte loads and stores
        const int64_t n8 = N / 8;
        for (int64_t i = gt; i < n8; i += GT) {
            const int4 a = __ldg((const int4 *)f.dt2 + 2 * i), b = __ldg((const int4 *)f.dt2 + 2 * i + 1);
            const int d[8] = {max(a.x, 0), max(a.y, 0), max(a.z, 0), max(a.w, 0),
                              max(b.x, 0), max(b.y, 0), max(b.z, 0), max(b.w, 0)};
            ((int4 *)f.seq)[2 * i] = make_int4(d[0] > 0 ? -1 : 0, d[1] > 0 ? -1 : 0, d[2] > 0 ? -1 : 0, d[3] > 0 ? -1 : 0);
            ((int4 *)f.seq)[2 * i + 1] =
                make_int4(d[4] > 0 ? -1 : 0, d[5] > 0 ? -1 : 0, d[6] > 0 ? -1 : 0, d[7] > 0 ? -1 : 0);
            ((uint4 *)f.state)[i] = make_uint4((u32)d[0] | (u32)d[1] << 16, (u32)d[2] | (u32)d[3] << 16,
                                               (u32)d[4] | (u32)d[5] << 16, (u32)d[6] | (u32)d[7] << 16);
#pragma unroll
            for (int k = 0; k < 8; k++)
                if (d[k] > 0) count(d[k]);
        }
        for (int64_t v = n8 * 8 + gt; v < N; v += GT) {
            const int d = max(f.dt2[v], 0);
            f.seq[v] = d > 0 ? -1 : 0;
            f.state[v] = (unsigned short)d;
            if (d > 0) count(d);
        }
    } else {
        for (int64_t v = gt; v < N; v += GT) {
            const int d = max(f.dt2[v], 0);
            int s = d;
            if (f.resume) { if (d > 0 && f.seq[v] != -1) s = 0; }   // invaded by the earlier run
            else f.seq[v] = d > 0 ? -1 : 0;
            f.state[v] = (unsigned short)s;
            if (d > 0) count(d);
        }
    }
    __syncthreads();
    if (smem_hist)
        for (int i = tid; i <= f.maxd; i += kFT)
            if (s_hist[i]) atomicAdd(f.cnt + i, s_hist[i]);
    if (!team_sync<CLUSTER>(f, T, epoch)) return;
    // list of value d: entries [off[d], off[d] + voxels of value d)
    if (c == 0) {
        int run = 0;
        for (int i0 = 0; i0 <= f.maxd; i0 += kFT) {
            const int i = i0 + tid;
            const int n = i <= f.maxd ? __ldcg(f.cnt + i) : 0;
            int tot;
            const int ex = block_excl(sh, n, &tot);
            if (i <= f.maxd) {
                __stcg(f.off + i, run + ex);
                __stcg(f.cnt + i, 0);
            }
            run += tot;
        }
    }
    if (!team_sync<CLUSTER>(f, T, epoch)) return;
    // first candidates: the inlet, and when resuming every uninvaded voxel
    // beside an invaded one
    if (!f.mask && !f.resume) {
        const int ax = f.inlet >> 1;
        const int n0 = ax == 0 ? f.ny : f.nx, n1 = ax == 2 ? f.ny : f.nz;
        const int fixed = (f.inlet & 1) ? (ax == 0 ? f.nx : ax == 1 ? f.ny : f.nz) - 1 : 0;
        for (int64_t i = gt; i < (int64_t)n0 * n1; i += GT) {
            const int p = (int)(i / n1), q = (int)(i % n1);
            const int64_t v = ax == 0 ? d_lin(fixed, p, q, f.ny, f.nz)
                              : ax == 1 ? d_lin(p, fixed, q, f.ny, f.nz) : d_lin(p, q, fixed, f.ny, f.nz);
            const int s = ld_state(f, v) & kFloodMaxVal;
            if (s) seed_voxel(f, v, s);
        }
    } else {
        for (int64_t v = gt; v < N; v += GT) {
            const int s = ld_state(f, v) & kFloodMaxVal;
            if (!s) continue;
            int x, y, z;
            coords(ny, nz, (int)v, x, y, z);
            bool on = f.mask ? f.mask[v] != 0 : d_on_face(x, y, z, f.nx, f.ny, f.nz, f.inlet);
            if (!on && f.resume) {
                const int64_t nyz = (int64_t)f.ny * f.nz;
                on = (x > 0 && f.seq[v - nyz] >= 1) || (x < f.nx - 1 && f.seq[v + nyz] >= 1) ||
                     (y > 0 && f.seq[v - f.nz] >= 1) || (y < f.ny - 1 && f.seq[v + f.nz] >= 1) ||
                     (z > 0 && f.seq[v - 1] >= 1) || (z < f.nz - 1 && f.seq[v + 1] >= 1);
            }
            if (on) seed_voxel(f, v, s);
        }
    }
    if (!team_sync<CLUSTER>(f, T, epoch)) return;

    // ---- phases
    int64_t steps = f.k0;
    int t_prev = f.maxd + 1, status = IBIP_OK;
    int64_t n_phases = 0, n_rounds = 0, n_events = 0;
    u32 pbase = 1;
    for (;;) {
        // the largest value with candidates
        if (warp == 0) {
            int t = 0;
            for (int hi = t_prev - 1; hi >= 1; hi -= 32) {
                const int v = hi - lane;
                const unsigned m = __ballot_sync(0xffffffffu, v >= 1 && __ldcg(f.cnt + v) > 0);
                if (m) { t = hi - (__ffs(m) - 1); break; }
            }
            if (lane == 0) sh.t = t;
        }
        __syncthreads();
        Phase ph;
        ph.t = sh.t;
        __syncthreads();
        if (ph.t == 0) break;
        t_prev = ph.t;
        // its roots: the listed voxels that are still uninvaded
        if (c == 0 && tid == 0) {
            ctl->nlog = 0;
            ctl->next = 0;
            ctl->nextC = 0;
            ctl->huge = 0;
            ctl->longs = 0;
            // (the read takes ~1 us of every phase it is made in: 1.5 % of a 48^3 sample in all of them)
            if (f.cancel && (n_phases & 3) == 0 && *(const volatile int *)f.cancel) ctl->cancel = 1;
        }
        const int listed = __ldcg(f.cnt + ph.t), lo = __ldcg(f.off + ph.t);
        for (int i0 = c * kFT + (tid & ~31); i0 < listed; i0 += T * kFT) {
            const int i = i0 + lane;
            int v = -1;
            if (i < listed) {
                v = __ldcg(f.lists + lo + i);
                if (!in_range(ctl, v, N, P_VOXEL)) v = 0;
                if ((ld_state(f, v) & kFloodMaxVal) == 0) v = -1;
            }
            const unsigned m = __ballot_sync(0xffffffffu, v >= 0);
            if (!m) continue;
            int slot = 0;
            if (lane == 0) slot = atomicAdd(&ctl->R, __popc(m));
            slot = __shfl_sync(0xffffffffu, slot, 0) + __popc(m & ((1u << lane) - 1));
            if (v >= 0 && slot < f.root_cap) {
                __stcg(f.roots + slot, v);
                __stcg(f.parent + slot, slot);
                __stcg(f.cur + slot, pbase + (u32)slot);
                __stcg(f.dirty + slot, 0);
                __stcg(f.claim + v, pbase + (u32)slot);
            }
        }
        if (!team_sync<CLUSTER>(f, T, epoch)) return;
        ph.R = __ldcg(&ctl->R);
        if (__ldcg(&ctl->cancel)) { status = IBIP_ERR_CANCELLED; break; }
        if (ph.R > f.root_cap || pbase > 0x70000000u - 16u * (u32)f.root_cap) { status = kFloodGiveUp; break; }
        if (ph.R == 0) {   // nothing listed is left (the counters above are read before the next phase adds)
            if (!team_sync<CLUSTER>(f, T, epoch)) return;
            continue;
        }
        if (steps >= f.max_steps) { status = IBIP_ERR_STEP_LIMIT; break; }
        n_phases++;
        ph.pbase = pbase;
        // log slots a warp or CTA takes at a time: unused ones stay few
        ph.chunk = max(2, min(16, ph.R / (4 * GW)));
        bool planes = false;    // the bit planes hold this phase
        bool dropped = false;   // some groups of this phase were run again
        for (ph.round = 0;; ph.round++) {
            n_rounds++;
            LogPos lp{0, 0, 0};
            if (ph.R <= kCurSmem) {
                for (int i = tid; i < ph.R; i += kFT) s_cur[i] = __ldcg(f.cur + i);
                __syncthreads();
            }
            if (ph.round == 0) {
                if (ph.t >= 16 && ph.R <= 4 * T) {
                    // few groups of large balls: one per CTA
                    for (int g = c; g < ph.R; g += T) lp = run_group<BLOCK>(f, ph, sh, s_q, s_cur, isq, g, pbase + (u32)g, lp);
                    if (lane == 0) log_close(f, lp);
                } else {
                    // one group per warp, 32 / LG roots at a time: LG lanes look
                    // over the dilated ball of a root first, and one that meets
                    // no other voxel of value >= t but candidates beside the
                    // ball is a group of one step
                    const int LG = ph.t == 1 ? 1 : ph.t < 16 ? 8 : 32;
                    const int take = 32 / LG;
                    const u32 tt = (u32)ph.t * 0x10001u;
                    u64 *wq = s_q + warp * kQW;
                    for (;;) {
                        int g0 = 0;
                        if (lane == 0) g0 = atomicAdd(&ctl->next, take);
                        g0 = __shfl_sync(0xffffffffu, g0, 0);
                        if (g0 >= ph.R) break;
                        const int g = g0 + lane / LG;
                        const int v = g < ph.R ? __ldcg(f.roots + g) : -1;
                        bool more = false;
                        if (v >= 0) {
                            Ball b;
                            b.r2 = ph.t;
                            coords(ny, nz, v, b.x, b.y, b.z);
                            if (LG == 1) {
                                const int64_t nyz = (int64_t)f.ny * f.nz;
                                int s[6];
                                s[0] = b.x > 0 ? ld_state(f, v - nyz) : 0;
                                s[1] = b.x < f.nx - 1 ? ld_state(f, v + nyz) : 0;
                                s[2] = b.y > 0 ? ld_state(f, v - f.nz) : 0;
                                s[3] = b.y < f.ny - 1 ? ld_state(f, v + f.nz) : 0;
                                s[4] = b.z > 0 ? ld_state(f, v - 1) : 0;
                                s[5] = b.z < f.nz - 1 ? ld_state(f, v + 1) : 0;
#pragma unroll
                                for (int k = 0; k < 6; k++) more |= s[k] != 0 && !(s[k] & 0x8000);
                            } else if (LG == 8) {
                                const Rows rw = ball_rows(nx, ny, isq, b);
                                u32 met = 0;
                                for (int r = lane & 7; r < rw.n; r += 8) {
                                    int X, Y, h, hs;
                                    row_at(rw, r, X, Y);
                                    shell_row(isq, b.r2, X - b.x, Y - b.y, h, hs);
                                    if (hs < 0) continue;
                                    const int za = max(b.z - hs, 0), zb = min(b.z + hs, f.nz - 1);
                                    const int64_t base = ((int64_t)X * f.ny + Y) * f.nz;
                                    const int64_t c1 = (base + zb) >> 3;
                                    for (int64_t k = (base + za) >> 3; k <= c1; k++) {
                                        const uint4 w = __ldcg((const uint4 *)f.state + k);
                                        const int z0 = (int)(k * 8 - base);
                                        const u32 in = h >= 0 ? chunk_span(b.z - h - z0, b.z + h - z0) : 0u;
                                        u32 ge = chunk_ge(w, tt) & chunk_span(za - z0, zb - z0) & (in | ~chunk_cand(w));
                                        if (X == b.x && Y == b.y) ge &= ~chunk_span(b.z - z0, b.z - z0);   // the root
                                        met |= ge;
                                    }
                                }
                                more = met != 0;
                            } else {
                                more = true;
                            }
                        }
                        unsigned mm = __ballot_sync(0xffffffffu, more);
                        const bool head = (lane & (LG - 1)) == 0;
                        const unsigned own = LG == 32 ? 0xffffffffu : ((1u << LG) - 1) << (lane & ~(LG - 1));
                        more = (mm & own) != 0;   // for the whole group of lanes
                        const bool lone = head && v >= 0 && !more;
                        const unsigned ml = __ballot_sync(0xffffffffu, lone);
                        mm = __ballot_sync(0xffffffffu, head && v >= 0 && more);
                        int slot = 0;
                        if (lane == 0 && ml) slot = atomicAdd(&ctl->nlog, __popc(ml));
                        slot = __shfl_sync(0xffffffffu, slot, 0) + __popc(ml & ((1u << lane) - 1));
                        if (lone && slot < f.log_cap) __stcg(f.log + slot, make_int4(v, v, kLast, (int)(pbase + (u32)g)));
                        for (unsigned m = mm; m; m &= m - 1) {
                            const int gg = g0 + (__ffs(m) - 1) / LG;
                            lp = run_group<WARP>(f, ph, sh, wq, s_cur, isq, gg, pbase + (u32)gg, lp);
                        }
                    }
                    if (lane == 0) log_close(f, lp);
                }
            } else {
                // joined groups: on whole CTAs, or when there are many on warps
                const u32 rbase = pbase + (u32)ph.round * (u32)ph.R;
                const int nC = __ldcg(&ctl->todoC), nW = __ldcg(&ctl->todoW);
                for (;;) {
                    if (tid == 0) sh.g = atomicAdd(&ctl->nextC, 1);
                    __syncthreads();
                    const int i = sh.g;
                    __syncthreads();
                    if (i >= nC) break;
                    const int g = __ldcg(f.todo + f.root_cap - 1 - i);
                    if (g < 0) lp = run_group<LONG>(f, ph, sh, s_q, s_cur, isq, ~g, rbase + (u32)~g, lp);
                    else lp = run_group<BLOCK>(f, ph, sh, s_q, s_cur, isq, g, rbase + (u32)g, lp);
                }
                __syncthreads();
                u64 *wq = s_q + warp * kQW;
                for (;;) {
                    int i = 0;
                    if (lane == 0) i = atomicAdd(&ctl->next, 1);
                    i = __shfl_sync(0xffffffffu, i, 0);
                    if (i >= nW) break;
                    const int g = __ldcg(f.todo + i);
                    lp = run_group<WARP>(f, ph, sh, wq, s_cur, isq, g, rbase + (u32)g, lp);
                }
                if (lane == 0) log_close(f, lp);
            }
            if (!team_sync<CLUSTER>(f, T, epoch)) return;
            const int failed = __ldcg(&ctl->fail);
            if (failed || __ldcg(&ctl->nlog) > f.log_cap || ph.round == 14) {   // nothing of the phase is stamped
                status = failed == kFailCancel ? IBIP_ERR_CANCELLED : kFloodGiveUp;
                break;
            }
            if (!__ldcg(&ctl->changed)) break;
            // groups to run again: a set of joined groups, or one handed over
            // to a CTA; every member's mark goes to the set's representative
            dropped = true;
            const int nr = ph.round + 1;
            if (c == 0 && tid == 0) { ctl->next = 0; ctl->nextC = 0; ctl->todoC = 0; ctl->todoW = 0; }
            for (int i = (int)gt; i < ph.R; i += (int)GT) {
                __stcg(f.head + i, -1);
                const int d = __ldcg(f.dirty + i);
                if ((d >> 2) != nr) continue;
                const int r = find_rep(f, i);
                if (r != i) atomicMax(f.dirty + r, d);
            }
            if (!team_sync<CLUSTER>(f, T, epoch)) return;
            if (c == 0 && tid == 0) ctl->changed = 0;
            for (int i = (int)gt; i < ph.R; i += (int)GT) {
                const int r = find_rep(f, i);
                const int d = __ldcg(f.dirty + r);
                if ((d >> 2) != nr) continue;
                const u32 id = pbase + (u32)nr * (u32)ph.R + (u32)r;
                __stcg(f.claim + __ldcg(f.roots + i), id);
                __stcg(f.next + i, atomicExch(f.head + r, i));
                if (i != r) {
                    __stcg(f.cur + i, 0u);
                } else {
                    __stcg(f.cur + r, id);
                    if ((d & 3) == 3) ctl->longs = 1;
                    // flags: 1 a CTA, 3 a CTA with the planes
                    if ((d & 1) || ph.t >= 9)
                        __stcg(f.todo + f.root_cap - 1 - atomicAdd(&ctl->todoC, 1), (d & 3) == 3 ? ~r : r);
                    else __stcg(f.todo + atomicAdd(&ctl->todoW, 1), r);
                }
            }
            if (!team_sync<CLUSTER>(f, T, epoch)) return;
            if (!planes && __ldcg(&ctl->longs)) {
                // the bit planes of this phase, a word per warp, eight in flight
                planes = true;
                const int NW = (nz + 31) >> 5;
                const u32 nwords = (u32)(nx * ny) * (u32)NW;   // below 2^31
                for (u32 w0 = (u32)gw * 8; w0 < nwords; w0 += (u32)GW * 8) {
                    int sv[8];
#pragma unroll
                    for (int k = 0; k < 8; k++) {
                        const u32 w = w0 + k, row = w / (u32)NW;
                        const int z = (int)(w - row * (u32)NW) * 32 + lane;
                        sv[k] = w < nwords && z < nz ? ld_state(f, (int64_t)row * nz + z) : 0;
                    }
                    u32 mf = 0, mr = 0;
#pragma unroll
                    for (int k = 0; k < 8; k++) {
                        const bool on = (sv[k] & kFloodMaxVal) >= ph.t;
                        const u32 a = __ballot_sync(0xffffffffu, on && !(sv[k] & 0x8000));
                        const u32 b = __ballot_sync(0xffffffffu, on && (sv[k] & 0x8000));
                        if (lane == k) { mf = a; mr = b; }
                    }
                    if (lane < 8 && w0 + lane < nwords) {
                        __stcg(f.fresh + w0 + lane, mf);
                        __stcg(f.root_bits + w0 + lane, mr);
                    }
                }
                if (!team_sync<CLUSTER>(f, T, epoch)) return;
            }
        }
        if (status != IBIP_OK) break;
        pbase += (u32)(ph.round + 1) * (u32)ph.R;
        const int nlog = __ldcg(&ctl->nlog);
        if (dropped) {   // entries of groups that were run again
            for (int i = (int)gt; i < nlog; i += (int)GT) {
                const int4 e = __ldcg(f.log + i);
                if (e.x < 0 || !in_range(f.ctl, e.x, (int64_t)f.nx * f.ny * f.nz, P_LOG)) continue;
                const u32 id = (u32)e.w;
                if (__ldcg(f.cur + (id - ph.pbase) % (u32)ph.R) != id) __stcg(f.log + i, make_int4(-1, -1, 0, 0));
            }
            if (!team_sync<CLUSTER>(f, T, epoch)) return;
        }
        // ---- labels: claim[record] = label of its run's first step
        int mine = 0;   // steps of this phase seen by this thread
        const bool huge = f.maxd >= kHuge;
        if ((int64_t)nlog * nlog / 32 <= (int64_t)256 * GW) {
            for (int i = gw; i < nlog; i += GW) {
                const int4 e = __ldcg(f.log + i);
                if (e.x < 0 || !in_range(f.ctl, e.x, (int64_t)f.nx * f.ny * f.nz, P_LOG)) continue;
                if (lane == 0) {
                    mine++;
                    if (huge && f.dt2[e.x] >= kHuge) { const int at = atomicAdd(&ctl->huge, 1); if (at < f.root_cap) __stcg(f.todo + at, i); }
                }
                if (!(e.z & kLast)) continue;
                int s = 0;
                for (int j = lane; j < nlog; j += 32) {
                    const int4 o = __ldcg(f.log + j);
                    if (o.x >= 0 && (o.z & kLast) && o.y < e.y) s += (o.z & ~kLast) + 1;
                }
                s = __reduce_add_sync(0xffffffffu, s);
                if (lane == 0) __stcg(f.claim + e.y, (u32)(steps - f.k0) + (u32)s + 1u);
            }
        } else {
            // many runs: their records as bits of a voxel plane, prefix sums
            // of the run lengths over the plane
            for (int i = (int)gt; i < nlog; i += (int)GT) {
                const int4 e = __ldcg(f.log + i);
                if (e.x < 0 || !in_range(f.ctl, e.x, (int64_t)f.nx * f.ny * f.nz, P_LOG)) continue;
                mine++;
                if (huge && f.dt2[e.x] >= kHuge) { const int at = atomicAdd(&ctl->huge, 1); if (at < f.root_cap) __stcg(f.todo + at, i); }
                if (!(e.z & kLast)) continue;
                atomicOr(f.plane + (e.y >> 5), 1u << (e.y & 31));
                __stcg(f.claim + e.y, (u32)((e.z & ~kLast) + 1));
            }
            if (!team_sync<CLUSTER>(f, T, epoch)) return;
            // (four words a thread: their look-ups overlap)
            const int64_t q_all = (f.plane_words + 3) / 4;
            const int64_t per = ((q_all + T - 1) / T + kFT - 1) / kFT * kFT;
            const int64_t q0 = min((int64_t)c * per, q_all), q1 = min(q0 + per, q_all);
            auto lengths = [&](u32 m, int64_t w) {
                int a = 0;
                while (m) {
                    u32 l[4];
#pragma unroll
                    for (int k = 0; k < 4; k++) {
                        l[k] = m ? __ldcg(f.claim + w * 32 + __ffs(m) - 1) : 0u;
                        m &= m - 1;
                    }
                    a += (int)(l[0] + l[1] + l[2] + l[3]);
                }
                return a;
            };
            int acc = 0;
            for (int64_t w = q0 + tid; w < q1; w += kFT) {
                const uint4 m = __ldcg((const uint4 *)f.plane + w);
                acc += lengths(m.x, 4 * w) + lengths(m.y, 4 * w + 1) + lengths(m.z, 4 * w + 2) + lengths(m.w, 4 * w + 3);
            }
            int tot;
            block_excl(sh, acc, &tot);
            if (tid == 0) __stcg(ctl->part + c, tot);
            if (!team_sync<CLUSTER>(f, T, epoch)) return;
            int64_t run = steps - f.k0 + 1;
            {
                int p = 0;
                for (int i = tid; i < c; i += kFT) p += __ldcg(ctl->part + i);
                block_excl(sh, p, &tot);
                run += tot;
            }
            for (int64_t wb = q0; wb < q1; wb += kFT) {
                const int64_t w = wb + tid;
                const uint4 m4 = w < q1 ? __ldcg((const uint4 *)f.plane + w) : make_uint4(0, 0, 0, 0);
                const u32 m[4] = {m4.x, m4.y, m4.z, m4.w};
                int s[4], all = 0;
#pragma unroll
                for (int k = 0; k < 4; k++) {
                    s[k] = lengths(m[k], 4 * w + k);
                    all += s[k];
                }
                int64_t at = run + block_excl(sh, all, &tot);
#pragma unroll
                for (int k = 0; k < 4; k++) {
                    const bool ones = s[k] == __popc(m[k]);   // every run of this word is one step
                    for (u32 b = m[k]; b; b &= b - 1) {
                        u32 *p = f.claim + (4 * w + k) * 32 + __ffs(b) - 1;
                        const u32 len = ones ? 1u : __ldcg(p);
                        __stcg(p, (u32)at);
                        at += len;
                    }
                }
                if (all) ((uint4 *)f.plane)[w] = make_uint4(0, 0, 0, 0);
                run += tot;
            }
        }
        {
            int tot;
            block_excl(sh, mine, &tot);
            if (tid == 0 && tot) atomicAdd(&ctl->events, tot);
        }
        if (!team_sync<CLUSTER>(f, T, epoch)) return;
        const int64_t ev_all = __ldcg(&ctl->events) - n_events;   // ctl->events counts all phases
        n_events += ev_all;
        // ---- stamp.  Few steps: wpe warps share one ball.  Many: a warp takes
        // `per` log entries, single voxels by lanes, balls by the whole warp
        if (c == 0 && tid == 0) ctl->R = 0;
        const int nhuge = huge ? __ldcg(&ctl->huge) : 0;
        if (nhuge > f.root_cap) { status = kFloodGiveUp; break; }
        const int wpe = min(64, max(1, GW / max(nlog, 1)));
        const int per = max(1, min(32, nlog / GW));
        const int unit = gw / wpe, sub = gw % wpe, units = GW / wpe;
        for (int64_t i0 = (int64_t)unit * per; i0 < nlog && unit < units; i0 += (int64_t)units * per) {
            const int i = (int)i0 + lane;
            int4 e = make_int4(-1, -1, 0, 0);
            if (lane < per && i < nlog) e = __ldcg(f.log + i);
            int r2 = 0;
            u32 label = 0;
            if (e.x >= 0 && in_range(ctl, e.x, N, P_LOG) && in_range(ctl, e.y, N, P_LOG)) {
                r2 = __ldg(f.dt2 + e.x);
                const int64_t k = (int64_t)__ldcg(f.claim + e.y) + (e.z & ~kLast) + f.k0;
                if (k <= f.max_steps) {
                    label = (u32)k;
                    if (k <= f.cap && sub == 0 && in_range(ctl, k - 1, f.cap, P_STEP)) {
                        f.step_r2[k - 1] = r2;
                        if (f.step_centre) f.step_centre[k - 1] = e.x;
                    }
                    if (r2 == 1) {
                        atomicMin((u32 *)f.seq + e.x, label);
                        f.state[e.x] = 0;
                    }
                }
            }
            unsigned m = __ballot_sync(0xffffffffu, label != 0 && r2 > 1 && !(huge && r2 >= kHuge));
            for (; m; m &= m - 1) {
                const int src = __ffs(m) - 1;
                Ball b;
                b.r2 = __shfl_sync(0xffffffffu, r2, src);
                const u32 lab = __shfl_sync(0xffffffffu, label, src);
                coords(ny, nz, __shfl_sync(0xffffffffu, e.x, src), b.x, b.y, b.z);
                if (b.r2 > 16) stamp_rows(f, isq, b, lab, sub * 4 + (lane >> 3), wpe * 4, lane & 7, 8);
                else stamp_rows(f, isq, b, lab, sub * 32 + lane, wpe * 32, 0, 1);
            }
        }
        for (int h = 0; h < nhuge; h++) {   // balls large enough for the whole team
            const int4 e = __ldcg(f.log + __ldcg(f.todo + h));
            const int64_t k = (int64_t)__ldcg(f.claim + e.y) + (e.z & ~kLast) + f.k0;
            if (k > f.max_steps) continue;
            Ball b;
            b.r2 = __ldg(f.dt2 + e.x);
            coords(ny, nz, e.x, b.x, b.y, b.z);
            stamp_rows(f, isq, b, (u32)k, gw, GW, lane, 32);
        }
        steps += ev_all;
        if (steps > f.max_steps) { steps = f.max_steps; status = IBIP_ERR_STEP_LIMIT; break; }
        if (ph.t == 1) break;   // nothing of smaller value is left
        if (!team_sync<CLUSTER>(f, T, epoch)) return;
        // ---- candidates for later phases: what the balls left uninvaded beside them
        int listed_n = 0;
        for (int i = unit; i < nlog && unit < units; i += units) {
            const int4 e = __ldcg(f.log + i);
            if (e.x < 0 || !in_range(f.ctl, e.x, (int64_t)f.nx * f.ny * f.nz, P_LOG)) continue;
            Ball b;
            b.r2 = __ldg(f.dt2 + e.x);
            if (huge && b.r2 >= kHuge) continue;
            coords(ny, nz, e.x, b.x, b.y, b.z);
            expose_ball(f, isq, b, sub * 32, wpe * 32, whits, listed_n);
        }
        for (int h = 0; h < nhuge; h++) {
            const int4 e = __ldcg(f.log + __ldcg(f.todo + h));
            Ball b;
            b.r2 = __ldg(f.dt2 + e.x);
            coords(ny, nz, e.x, b.x, b.y, b.z);
            expose_ball(f, isq, b, gw * 32, GW * 32, whits, listed_n);
        }
        __syncwarp();
        flush_hits(f, whits, listed_n);
        if (!team_sync<CLUSTER>(f, T, epoch)) return;
    }
    if (c == 0 && tid == 0) {
        f.out[0] = steps;
        f.out[1] = status;
#ifdef IBIP_CHECKED
        if (__ldcg(&ctl->bad)) f.out[1] = IBIP_ERR_BOUNDS;
        f.out[4] = __ldcg(&ctl->bad);
        f.out[5] = ctl->bad_index;
#endif
        f.out[2] = n_rounds;
        f.out[3] = n_phases;
    }
}

__global__ void __launch_bounds__(kFT, 1) k_flood_grid(const __grid_constant__ Flood f)
{
    flood_body<false>(f, (int)gridDim.x, (int)blockIdx.x);
}

// cluster i of the launch runs image i
__global__ void __launch_bounds__(kFT, 1) k_flood_cluster(const Flood *__restrict__ jobs)
{
    const cg::cluster_group cl = cg::this_cluster();
    const int T = (int)cl.num_blocks();
    __shared__ Flood f;
    static_assert(sizeof(Flood) % 4 == 0, "copied by words");
    for (int i = threadIdx.x; i < (int)(sizeof(Flood) / 4); i += kFT) ((u32 *)&f)[i] = ((const u32 *)(jobs + blockIdx.x / T))[i];
    __syncthreads();
    flood_body<true>(f, T, (int)cl.block_rank());
    if (!f.rec) return;
    // host-mapped completion record: steps and status, then its flag, once
    // the results are visible to later kernels
    __threadfence();
    cg::this_cluster().sync();
    if (cl.block_rank() == 0 && threadIdx.x == 0) {
        volatile IbipBatchDone *r = f.rec;
        r->steps = f.out[0];
        r->status = (int32_t)f.out[1];
        __threadfence_system();
        r->done = 1;
    }
}

size_t flood_smem(int maxd) { return (size_t)kQC * 8 + (size_t)kHits * 6 + kCurSmem * 4 + (((size_t)maxd + 1 + 15) & ~(size_t)15); }

size_t up256(size_t b) { return (b + 255) & ~(size_t)255; }

}  // namespace

bool ibip_flood_ok(ibip_dims d, int64_t npore, int maxd, int hasinf)
{
    return !hasinf && maxd >= 1 && maxd <= kFloodMaxVal && npore > 0 && npore <= (1ll << 28) && nvox(d) < (1ll << 31);
}

FloodSizes ibip_flood_sizes(ibip_dims d, int64_t npore, int maxd)
{
    FloodSizes z;
    const int64_t N = nvox(d);
    // packs of narrow pores have ~18 % of their pore voxels as roots of the
    // last phase, and log some steps again in every round
    z.root_cap = (int)(npore / 4) + 4096;
    z.log_cap = (int)(npore / 2) + 16384;
    z.state = up256(((size_t)N + 8) * 2);
    z.claim = up256(((size_t)N + 4) * 4);
    z.bits = up256((size_t)d.nx * d.ny * ((d.nz + 31) / 32) * 4);
    z.plane = up256(((size_t)N + 127) / 128 * 16);
    z.lists = up256((size_t)npore * 4);
    z.tables = up256((size_t)z.root_cap * 4 * 4);
    z.tables2 = up256((size_t)z.root_cap * 4 * 3);
    z.log = up256((size_t)z.log_cap * 16);
    z.values = up256(((size_t)maxd + 1) * 8);
    return z;
}

void ibip_flood_fill(Flood *f, const int32_t *dt2, ibip_dims d, int inlet, const uint8_t *mask, int resume, int64_t k0,
                     int64_t max_steps, int32_t *seq, int32_t *step_r2, int32_t *step_centre, int64_t cap, int maxd,
                     int npore, const FloodSizes &z, const FloodMem &m)
{
    const int64_t N = nvox(d);
    f->npore = npore;
    f->nx = d.nx; f->ny = d.ny; f->nz = d.nz; f->inlet = inlet; f->maxd = maxd; f->resume = resume;
    f->dt2 = dt2; f->mask = mask; f->k0 = k0; f->cap = cap;
    f->max_steps = max_steps > INT64_MAX - k0 ? INT64_MAX : k0 + max_steps;
    f->seq = seq; f->step_r2 = step_r2; f->step_centre = step_centre;
    f->state = (unsigned short *)m.state;
    f->claim = (uint32_t *)m.claim;
    f->plane = (uint32_t *)m.plane;
    f->fresh = (uint32_t *)m.fresh;
    f->root_bits = (uint32_t *)m.root_bits;
    f->plane_words = (N + 127) / 128 * 4;
    f->lists = (int *)m.lists;
    int *tb = (int *)m.tables;
    f->roots = tb;
    f->parent = tb + z.root_cap;
    f->cur = (uint32_t *)(tb + 2 * (int64_t)z.root_cap);
    f->next = tb + 3 * (int64_t)z.root_cap;
    int *tb2 = (int *)m.tables2;
    f->head = tb2;
    f->dirty = tb2 + (int64_t)z.root_cap;
    f->todo = tb2 + 2 * (int64_t)z.root_cap;
    f->root_cap = z.root_cap;
    f->log = (int4 *)m.log;
    f->log_cap = z.log_cap;
    f->cnt = (int *)m.values;
    f->off = (int *)m.values + maxd + 1;
    f->ctl = (FloodCtl *)m.ctl;
    f->out = m.out;
    f->cancel = nullptr;
    f->rec = nullptr;
    // A longer group is a serial chain that the one-CTA loop runs faster: a
    // long group takes 2-4 us a step (more with thousands in its queue), the
    // loop 0.4-1.1 us, but on all the steps.  Packs of 100^3-220^3 have a group
    // of up to 0.8 % of their pore voxels and run 3-8 times faster by phases
    // (117^3, porosity 0.43: 5,281 steps, 35 ms against 104; 160^3, 0.40: 11,681,
    // 70 against 280; 220^3, 0.40: 28,796, 170 against 739); at 290^3 the share
    // falls (0.36: 36,830 steps, 0.4 %, 379 ms against 1,876; 512^3 blobs: under
    // 14,478).  What gives up pays for the steps once more: 30 ms of the loop's
    // 1,739 at 290^3 and 0.40, 20 of 3,083 at 350^3 (both by the queue).  Small
    // images get a larger share (16^3-32^3 packs of narrow pores have groups of
    // 250-500 steps and more), noise of single voxels (a group of most steps,
    // whatever the size) bounds it: 32^3 takes 21 ms so and 27 ms with 4,096
    // steps, the loop alone 18.
    f->budget = std::min(std::max(npore / 96, std::min(std::max(npore / 32, 1024), 4096)), 40960);
}

int ibip_flood_launch_grid(ibip_ctx *ctx, const Flood &f, cudaStream_t s)
{
    const size_t dyn = flood_smem(f.maxd);
    cudaError_t e = cudaFuncSetAttribute((const void *)k_flood_grid, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)flood_smem(kFloodMaxVal));
    if (e != cudaSuccess) return ibip_cuda_status(e);
    Flood a = f;
    void *args[] = {&a};
    e = cudaLaunchCooperativeKernel((const void *)k_flood_grid, std::min(ctx->sm_count, kFloodMaxTeam), kFT, args, dyn,
                                    s);
    IBIP_LAUNCH(ctx);
    return ibip_cuda_status(e);
}

int ibip_flood_launch_clusters(ibip_ctx *ctx, const Flood *d_jobs, int n, int maxd, int cluster, cudaStream_t s)
{
    const size_t dyn = flood_smem(maxd);
    const void *fn = (const void *)k_flood_cluster;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)flood_smem(kFloodMaxVal));
    if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return ibip_cuda_status(e);
    for (; cluster >= 1; cluster /= 2) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(n * cluster);
        cfg.blockDim = dim3(kFT);
        cfg.dynamicSmemBytes = dyn;
        cfg.stream = s;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = cluster;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int fit = 0;
        if (cudaOccupancyMaxActiveClusters(&fit, fn, &cfg) != cudaSuccess || fit < 1) {
            cudaGetLastError();
            continue;   // the device cannot place such a cluster
        }
        e = cudaLaunchKernelEx(&cfg, k_flood_cluster, d_jobs);
        IBIP_LAUNCH(ctx);
        return ibip_cuda_status(e);
    }
    return IBIP_ERR_CUDA;
}
