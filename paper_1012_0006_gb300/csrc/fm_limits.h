// Limits of the two-way FM search, as plain C++ (checked without a device).
#pragma once

#include <climits>

#ifdef __CUDACC__
#define FR_HD __host__ __device__
#else
#define FR_HD
#endif

namespace fr {

// Ten bits hold a connection weight or a degree in a vertex record: |gain| <= weighted
// degree, and arc weights are at least 1.
constexpr int kFmMaxDeg = 1023;

// End of the row [j0, j1) as a warp that reads ahead of the moves walks it.  It takes both ends
// from a queue entry that the moving warp may be writing again at that moment, so they may
// belong to two rows: never more arcs than a row has, none past the adjacency.
FR_HD constexpr int fm_row_end(int j0, int j1, int nnz) {
    const int end = j1 < nnz ? j1 : nnz;
    return end - j0 > kFmMaxDeg ? j0 + kFmMaxDeg : end;
}

// Stack entries are counted in 32 bits: at most one per vertex and arc of the graph, and a
// move looks up to 32 entries past the last one.
FR_HD constexpr bool fm_entries_fit(long long n, long long nnz) { return n + nnz <= INT_MAX - 64; }

}  // namespace fr
