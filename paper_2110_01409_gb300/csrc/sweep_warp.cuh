// Warp tiles shared by the warp-worker sweeps (sweep_warp.cu) and the
// warp-tile frontier Bellman-Ford (sweep_warp_frontier.cu): per-warp shared
// buffers, the staged inputs of a warp tile, its fetch (edge stream two tiles
// ahead by cp.async, gathers one tile ahead), the row sums with a shuffle
// segmented scan, and the bounded wait on a partial another warp publishes.
#pragma once

#include <climits>
#include <cstdint>

#include "sweep_common.cuh"
#include "sweep_edges.cuh"

namespace dag {

// Warp tile shapes: items per lane (odd: fewer bank conflicts in the walk);
// the plan picks one (dag_plan_set_warp_tile), WIPT_DEFAULT unless told.
constexpr int WIPT_DEFAULT = 7;
constexpr int WWARPS = NWARP;        // warps per CTA (block reductions and the grid barrier are per CTA)
constexpr int WMINBLOCKS = 4;        // CTAs per SM the register budget is sized for
constexpr int LIVE_EVERY = 8;        // async / delayed PageRank: a warp reads and adds to the live sum every 8
                                     // tiles (1,792 items, the CTA-tile kernels' tile), not every tile

// A tile's merge-path coordinates: rows [a0, a1) end in it, edges [b0, b1).
struct WCoord {
    int a0, b0, a1, b1;
};

template <int MODE, int WIPT>
struct WarpShared {
    static constexpr int WTILE = 32 * WIPT;
    alignas(16) int col[WWARPS][WTILE + 8];                              // edge sources of the next tile
    uint32_t val[WWARPS][WTILE];                                         // edge terms, then row sums (wwalk)
    uint16_t end[WWARPS][WTILE];                                         // tile-relative row ends
    uint32_t mark[WWARPS][WTILE / 4 + 4];                                // byte j: edge j is the last of its row
    double red0[NWARP];
    double red1[NWARP];
    double res, gprev, T;
    // a warp's own val, which it is done with at the end of its tiles
    __device__ __forceinline__ float& part(int k, int w, int l) { return ((float*)val[w])[32 * k + l]; }
};

__device__ __forceinline__ WCoord wcoord(const SweepParams& p, int t)
{
    return {p.tile_row[t], p.tile_nz[t], p.tile_row[t + 1], p.tile_nz[t + 1]};
}

// Inputs of the next warp tile, loaded while the current one is walked.
template <int MODE, int WIPT>
struct WStage {
    int a0, b0, NA, NB;
    int rp0;              // rowptr[a0]: the tile starts inside row a0 when b0 > rp0
    int re0;              // rowptr[a0 + lane + 1]: the end of the tile's row `lane` (lane < NA)
    uint32_t xv[WIPT];    // terms of edges lane + 32 q: gathered value, with the edge's weight / value
    uint32_t xo;          // old value of row a0 + lane
    float dg;             // its out-degree (PageRank)
    float bv;             // its base term (PageRank, adjoint)
    long long gs;         // one stripe of the live global sum (async / delayed PageRank)
};

__device__ __forceinline__ void wcp16(void* dst, uintptr_t src, uint64_t pol)
{
    asm volatile("cp.async.cg.shared.global.L2::cache_hint [%0], [%1], 16, %2;"
                 ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "l"(pol) : "memory");
}

__device__ __forceinline__ void wcp4(void* dst, const int* src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;"
                 ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}

// Starts the copies of tile c's edge sources into the warp's buffer: whole 16-byte granules around the wanted
// elements, whatever the array's alignment, or at the array's ends the wanted elements (sweep_edges.cuh).
template <int MODE, int WIPT>
__device__ __forceinline__ void wissue_col(WarpShared<MODE, WIPT>& sh, const SweepParams& p, const WCoord& c, int wl, int lane,
                                           uint64_t pol_edge)
{
    if (c.b1 <= c.b0) return;
    const uintptr_t at = (uintptr_t)(p.colidx + c.b0);
    const int lead = edge_lead(at), n = edge_granules(lead, c.b1 - c.b0);
    if (edge_granules_inside(lead, c.b0, c.b1, p.m)) {
        for (int k = lane; k < n; k += 32) wcp16((char*)sh.col[wl] + 16 * k, (at & ~(uintptr_t)15) + 16 * k, pol_edge);
    } else {
#pragma unroll 1
        for (int j = lane; j < c.b1 - c.b0; j += 32) wcp4(sh.col[wl] + lead + j, p.colidx + c.b0 + j);
    }
}
__device__ __forceinline__ void wcommit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// The warp's copies have landed, and every lane is done with what it read before.
__device__ __forceinline__ void wlanded()
{
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncwarp();
}

// Old value, out-degree and base term of row v (only this warp writes it, so a value loaded ahead is still the
// current one).
template <int MODE>
__device__ __forceinline__ void wrow_inputs(const SweepParams& p, const uint32_t* xin, int v, uint64_t pol_vertex,
                                            uint32_t& xo, float& dg, float& bv)
{
    constexpr bool BF = MODE == MODE_BF || MODE == MODE_BF8;
    xo = ld_weak_keep_b32(xin + v, pol_vertex);
    if constexpr (!BF) {
        dg = __uint_as_float(ld_vertex_b32(p.degf + v, pol_vertex));
        bv = row_base<MODE>(p, v);
    }
}

// Issues the gathers, weights / edge values and row inputs of tile c, whose edge sources have landed (wlanded). Every lane has read the
// warp's col buffer when this returns.
template <int MODE, int WIPT>
__device__ __forceinline__ void wgather(WStage<MODE, WIPT>& st, WarpShared<MODE, WIPT>& sh, const SweepParams& p,
                                        const uint32_t* xin, const WCoord& c, int wl, int lane, int rmode, bool live,
                                        uint64_t pol_edge, uint64_t pol_vertex)
{
    st.a0 = c.a0;
    st.b0 = c.b0;
    st.NA = c.a1 - c.a0;
    st.NB = c.b1 - c.b0;
    st.rp0 = (int)ld_vertex_b32(p.rowptr + st.a0, pol_vertex);
    st.re0 = lane < st.NA ? (int)ld_vertex_b32(p.rowptr + st.a0 + lane + 1, pol_vertex) : 0;
    const int* col = sh.col[wl] + edge_lead((uintptr_t)(p.colidx + c.b0));
    uint32_t aux[MODE == MODE_PR ? 1 : WIPT];
#pragma unroll
    for (int q = 0; q < WIPT; ++q) {
        const int j = lane + 32 * q;
        st.xv[q] = Op<MODE>::identity();
        if (j < st.NB) {
            const uint32_t* x = xin + col[j];
            st.xv[q] = rmode == READ_COHERENT ? ld_relaxed_keep_b32(x, pol_vertex) : ld_weak_keep_b32(x, pol_vertex);
        }
    }
    if constexpr (MODE != MODE_PR) {
#pragma unroll
        for (int q = 0; q < WIPT; ++q) {
            const int j = lane + 32 * q;
            aux[q] = 0u;
            if (j < st.NB) {
                if constexpr (MODE == MODE_BF8) aux[q] = ld_edge_u8(p.w8 + st.b0 + j, pol_edge);
                else if constexpr (MODE == MODE_BF) aux[q] = ld_edge_b32(p.w + st.b0 + j, pol_edge);
                else aux[q] = ld_edge_b32(p.val + st.b0 + j, pol_edge);
            }
        }
    }
    if constexpr (MODE != MODE_PR) {
#pragma unroll
        for (int q = 0; q < WIPT; ++q) {
            if constexpr (MODE == MODE_BF || MODE == MODE_BF8) st.xv[q] = relax(st.xv[q], aux[q]);
            else st.xv[q] = __float_as_uint(__uint_as_float(aux[q]) * __uint_as_float(st.xv[q]));
        }
    }
    st.xo = 0u;
    st.dg = 0.0f;
    st.bv = 0.0f;
    if (lane < st.NA) wrow_inputs<MODE>(p, xin, st.a0 + lane, pol_vertex, st.xo, st.dg, st.bv);
    if (live) st.gs = ld_relaxed_i64(&p.sync->stripe[lane * GSTRIDE]);
    __syncwarp();
}

// A gathered tile into the warp's buffers: edge terms (identity past the last), row ends (the first 32 came with the
// gathers, the rest, a tile of mostly empty rows, are loaded here), no marks.
template <int MODE, int WIPT>
__device__ __forceinline__ void wstage(WarpShared<MODE, WIPT>& sh, const WStage<MODE, WIPT>& st, const SweepParams& p, int wl,
                                       int lane, uint64_t pol_vertex)
{
    uint32_t* val = sh.val[wl];
#pragma unroll
    for (int q = 0; q < WIPT; ++q) {
        val[lane + 32 * q] = st.xv[q];
    }
    if (lane < st.NA) sh.end[wl][lane] = (uint16_t)(st.re0 - st.b0);
    for (int i = lane + 32; i < st.NA; i += 32)
        sh.end[wl][i] = (uint16_t)((int)ld_vertex_b32(p.rowptr + st.a0 + i + 1, pol_vertex) - st.b0);
    for (int i = lane; i < 8 * WIPT + 4; i += 32) sh.mark[wl][i] = 0u;
}

// The sum of tile row r after wwalk: the walk leaves it at the row's last edge; a row without edges in the tile has
// the tile's carry (its first row) or nothing.
template <int MODE>
__device__ __forceinline__ uint32_t wrow_sum(const uint32_t* val, const uint16_t* end, int r, uint32_t carry)
{
    const int e = end[r], b = r > 0 ? end[r - 1] : 0;
    return e > b ? val[e - 1] : r == 0 ? carry : Op<MODE>::identity();
}

// Row sums of one warp tile, left in val at each row's last edge (wrow_sum). Lane l adds edges l WIPT .. + WIPT - 1
// and closes a row where its mark is set; a shuffle segmented scan over the lanes joins the rows that span lanes.
// carry: the partial of the row continuing from the previous tile; returns the partial of the row left unfinished.
// The edges are split over the lanes and the row ends found as marks, instead of walking rows and edges together
// (a merge-path walk, whose two kinds of steps diverge): a 224-item tile took about 590 warp instructions that way
// and takes about 400. Marks are bytes, stored without conflict; as bits set by shared-memory atomics, one lane at a
// time, the tiles of many short rows took twice as long as the rest and held up the sweep.
template <int MODE, int WIPT>
__device__ __forceinline__ uint32_t wwalk(const uint16_t* end, uint32_t* val, uint32_t* mark, int NA, uint32_t carry,
                                          int lane)
{
    using O = Op<MODE>;
    constexpr int NW = (WIPT + 3) / 4;  // words of a lane's marks
    for (int r = lane; r < NA; r += 32) {
        const int e = end[r], b = r > 0 ? end[r - 1] : 0;
        if (e > b) ((uint8_t*)mark)[e - 1] = 1;
    }
    const bool first_done = NA > 0 && end[0] == 0;  // the continuing row ends before the tile's first edge
    __syncwarp();
    const int j0 = lane * WIPT;
    uint32_t m[NW];
    {
        uint32_t w = mark[j0 >> 2];
#pragma unroll
        for (int k = 0; k < NW; ++k) {
            const uint32_t w1 = mark[(j0 >> 2) + k + 1];
            m[k] = __funnelshift_r(w, w1, 8 * (j0 & 3));
            w = w1;
        }
        if (WIPT & 3) m[NW - 1] &= (1u << (8 * (WIPT & 3))) - 1u;
    }
    int first = -1;  // the first row end among the lane's edges
    uint32_t acc = (lane == 0 && !first_done) ? carry : O::identity();
#pragma unroll
    for (int q = 0; q < WIPT; ++q) {
        acc = O::combine(acc, val[j0 + q]);
        if ((m[q >> 2] >> (8 * (q & 3))) & 1u) {
            val[j0 + q] = acc;
            acc = O::identity();
            if (first < 0) first = q;
        }
    }
    // inclusive scan of the lanes' open partials, restarting at each lane that closed a row
    const unsigned closed = __ballot_sync(0xffffffffu, first >= 0) & (0xffffffffu >> (31 - lane));
    const int from = closed ? 31 - __clz(closed) : 0;
    uint32_t sv = acc;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t ov = __shfl_up_sync(0xffffffffu, sv, o);
        if (lane - o >= from) sv = O::combine(sv, ov);
    }
    const uint32_t cin = __shfl_up_sync(0xffffffffu, sv, 1);
    if (lane > 0 && first >= 0) {
        uint32_t* f = val + j0 + first;
        *f = O::combine(*f, cin);
    }
    return __shfl_sync(0xffffffffu, sv, 31);
}

__device__ __forceinline__ void st_relaxed_u64(unsigned long long* p, unsigned long long v)
{
    asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// The partial that warp k published for sweep `stamp` (waits, bounded); false
// when the wait ran out or another CTA recorded an error.
__device__ __forceinline__ bool wait_published(const unsigned long long* pub, int k, unsigned stamp, SyncBlock* sb,
                                               long long timeout_ns, uint32_t* out)
{
    const unsigned long long t0 = globaltimer_ns();
    unsigned spins = 0;
    for (;;) {
        const unsigned long long v = ld_relaxed_u64(pub + k);
        if ((unsigned)(v >> 32) == stamp) {
            *out = (uint32_t)v;
            return true;
        }
        if (ld_relaxed_i32(&sb->err) != 0) return false;
        if ((++spins & 15u) == 0 && (long long)(globaltimer_ns() - t0) > timeout_ns) {
            atomicCAS(&sb->err, 0, DAG_ERR_BARRIER_TIMEOUT);
            return false;
        }
        __nanosleep(64);
    }
}

}  // namespace dag
