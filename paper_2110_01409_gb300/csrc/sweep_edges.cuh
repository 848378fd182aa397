// Which parts of the edge array a warp tile's copy of its edge sources reads (sweep_warp.cuh). Plain arithmetic, also
// compiled for the host by a test.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define DAG_HD __host__ __device__ __forceinline__
#else
#define DAG_HD inline
#endif

namespace dag {

// The tile's edges [b0, b1) are copied in 16-byte granules of memory, from the one that holds b0 to the one that holds
// b1 - 1. lead: the place of element b0, at address `at`, in its granule.
DAG_HD int edge_lead(uintptr_t at) { return (int)(at >> 2) & 3; }
DAG_HD int edge_granules(int lead, int edges) { return (lead + edges + 3) >> 2; }

// Whole granules, with the neighbouring tiles' elements they may hold, lie inside the array of m elements. At its ends they
// may reach over it (a caller's array may be a part of a larger one), and the tile is copied element by element. (Tested
// for the last granule itself instead of the three elements it may reach past b1, the copies took 3% of a small banded
// graph's sweeps.)
DAG_HD bool edge_granules_inside(int lead, int b0, int b1, int m) { return lead <= b0 && b1 <= m - 3; }

}  // namespace dag
