// Limits of the two-way FM search, as plain C++ (checked without a device).
#pragma once

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

}  // namespace fr
