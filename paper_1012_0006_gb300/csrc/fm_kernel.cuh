// Two-way FM (TopGain) before the flows of a round's pairs: device state and launch.
#pragma once

#include <cuda_runtime.h>

#include "fm_limits.h"
#include "fr_internal.cuh"

namespace fr {

constexpr int kFmMaxBuckets = 2048;   // gain buckets per block: gains in [-1023, 1023]
constexpr int kFmSortSmem = 4096;     // boundary entries a pair sorts in shared memory

// Result of one pair's FM search (what fr_pair_result reports).
struct FmRes {
    long long cut0, wA0, wB0;   // pair cut and block weights before
    long long cut1, wA1, wB1;   // after the rollback to the best prefix
    int kept, tried;            // moves kept / made
};

// Device state of the FM searches of one round (pairs of one graph).
struct FmDev {
    // [n] vertex records, written by every round's gather: {weight to the own block | weight
    // to the pair's other block << 10 | degree << 20, latest stack entry + 1 (0: not queued),
    // block (-1: not in a pair of the round, or moved), row begin}
    int4 *rec;
    int *vlist;                 // [n] per pair region: boundary vertices
    int *mlog;                  // [n] per pair region: vertices moved, in order
    int *blockn, *blockarcs;    // [k] vertex and arc counts of the blocks (zeroed by fm_offsets)
    long long *voff, *eoff;     // [P], [P + 1] region offsets: vertices (vlist, mlog), stack entries
    int *np, *bcnt;             // [P] pair vertex counts, boundary vertices gathered
    int2 *ent;                  // [ecap] bucket stack entries: {vertex, or -1 once dead; entry below}
    unsigned long long *skey;   // [scap] sort scratch for boundaries beyond shared memory
    int *sbkt, *sv;             // [scap]
    FmRes *res;                 // [P]
    const int *maxwdeg;         // max weighted degree of the graph (from prep): bounds |gain|
    long long ecap, scap;
    int permille;
};

__host__ __device__ constexpr int fm_in(int x) { return x & kFmMaxDeg; }
__host__ __device__ constexpr int fm_ext(int x) { return (x >> 10) & kFmMaxDeg; }
__host__ __device__ constexpr int fm_deg(int x) { return (x >> 20) & kFmMaxDeg; }

// Enqueues the FM searches of the round described by w (one graph with k blocks,
// w.npairs pairs): block counts, pair regions, boundary gather, one CTA per pair.
// *nl += kernels launched.
cudaError_t launch_fm(const Work &w, const FmDev &f, int k, int sms, cudaStream_t st, int *nl);
size_t fm_pair_smem();

}  // namespace fr
