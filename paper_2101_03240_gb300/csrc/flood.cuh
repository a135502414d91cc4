// flood.cuh -- the invasion by value phases (flood.cu) as invade.cu uses it.
#pragma once

#include "common.cuh"

constexpr int kFloodMaxVal = 32767;    // largest dt2 the 15-bit state holds
constexpr int kFloodMaxTeam = 256;     // CTAs of one image at most
constexpr int kFloodGiveUp = -100;     // status of a run that outgrew its tables

// Counters of one image, zero before the launch.
struct FloodCtl {
    unsigned int bar;   // arrivals at the grid barrier
    int fail;           // a group (1) or a barrier (2) gave up, or a group was cancelled (3)
    int R;              // roots of the phase
    int nlog;           // log slots taken
    int next, nextC;    // work counters of the round (warps, CTAs)
    int todoW, todoC;   // groups to run again on warps / on CTAs
    int changed;        // some group has to be run again
    int cancel;
    int events;         // steps so far
    int longs;          // some group is to be run on the bit planes
    int huge;           // balls of this phase the whole team stamps
    int part[kFloodMaxTeam];
    int bad;             // checked build: place of the first index outside its array
    long long bad_index;
};

// One image of the kernel.
struct Flood {
    int nx, ny, nz, inlet, maxd, npore, resume, pad;
    const int32_t *dt2;
    const uint8_t *mask;        // inlet voxels, or null: the inlet face
    int64_t k0, max_steps;      // steps taken before (resume), limit on the total
    int64_t cap;                // length of the step arrays
    int32_t *seq, *step_r2, *step_centre;
    unsigned short *state;      // dt2 while uninvaded, else 0; bit 15: candidate
    uint32_t *claim;            // per voxel: last group that touched it; of a record, its run's label
    uint32_t *fresh, *root_bits;   // bit planes (rows padded to words) of a phase with a long group
    uint32_t *plane;            // per voxel one bit: records of a large phase (zero between phases)
    int64_t plane_words;
    int *lists;                 // candidates by value: entries off[d] .. off[d] + cnt[d]
    int *cnt, *off;
    int *roots, *parent, *next, *head, *dirty, *todo;   // per root of the phase
    uint32_t *cur;                                      // per root: the live id of its group
    int root_cap;
    int4 *log;                  // steps of the phase: voxel, record, place | last, group id
    int log_cap;
    int budget;                 // steps one group may take
    FloodCtl *ctl;
    int64_t *out;               // [0] steps, [1] status, [2] rounds, [3] phases
    const int *cancel;          // host-mapped cancel flag, or null
    IbipBatchDone *rec;         // completion record (host-mapped), or null
};

// Device bytes of one image's tables.
struct FloodSizes {
    int root_cap, log_cap;
    size_t state, claim, plane, bits, lists, tables, tables2, log, values;
    size_t total() const { return state + claim + plane + 2 * bits + lists + tables + tables2 + log + values; }
};

struct FloodMem {
    void *state, *claim, *plane, *fresh, *root_bits, *lists, *tables, *tables2, *log, *values, *ctl;
    int64_t *out;
};

// Whether the kernel takes an image with these statistics: values that fit
// the state image, and some solid (an image without solid is one step).
bool ibip_flood_ok(ibip_dims d, int64_t npore, int maxd, int hasinf);
FloodSizes ibip_flood_sizes(ibip_dims d, int64_t npore, int maxd);
void ibip_flood_fill(Flood *f, const int32_t *dt2, ibip_dims d, int inlet, const uint8_t *mask, int resume, int64_t k0,
                     int64_t max_steps, int32_t *seq, int32_t *step_r2, int32_t *step_centre, int64_t cap, int maxd,
                     int npore, const FloodSizes &z, const FloodMem &m);
// One image on a cooperative grid of one CTA per SM.
int ibip_flood_launch_grid(ibip_ctx *ctx, const Flood &f, cudaStream_t s);
// n images (device table), one cluster of up to `cluster` CTAs each.
int ibip_flood_launch_clusters(ibip_ctx *ctx, const Flood *d_jobs, int n, int maxd, int cluster, cudaStream_t s);
