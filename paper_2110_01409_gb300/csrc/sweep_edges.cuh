// Which parts of the edge array a warp tile's copy of its edge sources reads (sweep_warp.cuh). Plain arithmetic, also
// compiled for the host by a test.
#pragma once

#ifdef __CUDACC__
#define DAG_HD __host__ __device__ __forceinline__
#else
#define DAG_HD inline
#endif

namespace dag {

// The tile's edges [b0, b1) are copied in 16-byte granules of memory, from the one that holds b0 to the one that holds
// b1 - 1. mis: the elements by which colidx lies past a 16-byte boundary, so element b0 lies (b0 + mis) mod 4 into its
// granule.
DAG_HD int edge_lead(int mis, int b0) { return (b0 + mis) & 3; }
DAG_HD int edge_granules(int mis, int b0, int b1) { return (edge_lead(mis, b0) + (b1 - b0) + 3) >> 2; }

// Whole granules, with the neighbouring tiles' elements they may hold, lie inside the array of m elements; at its ends
// they may reach over it (a caller's array may be a part of a larger one), and the tile is copied element by element.
DAG_HD bool edge_granules_inside(int mis, int b0, int b1, int m)
{
    return edge_lead(mis, b0) <= b0 && 4 * edge_granules(mis, b0, b1) - edge_lead(mis, b0) <= m - b0;
}

}  // namespace dag
