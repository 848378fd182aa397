// Warp-worker pull sweep: PageRank (plain and weighted), its adjoint and
// Bellman-Ford in the synchronous, asynchronous and delayed-asynchronous
// forms, with one warp per worker and no CTA-wide barrier inside a sweep.
//
// Paper mapping (Blanco, McMillan, Low, HPEC 2021):
//  * worker = one warp. The merge path of the whole graph (rows and in-edges
//    in vertex order, Merrill & Garland) is cut into warp tiles of WTILE items
//    and every worker takes a run of consecutive tiles of equal weight
//    (in-degree + 2 or 3 per row, Sec. III-A's balance with a row's
//    cost on this machine) and owns the rows whose end item lies in its run (contiguous in vertex order). A row whose
//    in-edges span two runs (a hub, or a cut inside a row) is owned by the run
//    that ends it; the earlier runs' partial sums reach it at the end of the
//    sweep through a bounded look-back (below);
//  * pull update of each owned vertex from its in-neighbours (Sec. III-A);
//  * sync: values go to the second array (Sec. I); async: values are written
//    in place as soon as a warp tile completes them (Sec. I); delayed: values
//    go to the warp's buffer in shared memory and reach the global array when
//    it holds >= delta values or the run is done (Sec. III, III-B); reads come
//    from the global array (the "global read" form, Sec. III-C);
//  * one grid barrier per iteration (Sec. I) and the stopping rules of Sec. IV.
//
// Why warps: the CTA-tile kernels (sweep.cu, sweep_tma.cu) stop all eight
// warps at two barriers per 1,792-item tile, so each tile waits for its
// slowest gather; here each warp sums its own 224-item tiles with a
// shuffle-only segmented scan, copies edge sources two tiles ahead (cp.async)
// and issues the next tile's gathers before the current one's sums or after
// them, so the SM's 32 warps keep their gathers in flight independently.
//
// What bounds it: one gather per clock through an SM's L1 (65 M edges: 0.19 to
// 0.21 ms a sweep for 4 M RMAT vertices), then instructions and the slowest
// run. Against a merge-path walk of each tile with the edge stream loaded one
// tile ahead and runs of equal item counts, ms per solve: ordered PageRank (4 M
// vertices) 3.76 -> 3.35 (466 -> 372 us per sweep, one sweep more), uniform
// graph (2 M) 1.55 -> 1.38, synchronous (2 M) 1.77 -> 1.55, banded (4 M) 4.22 ->
// 3.58, weighted PageRank (2 M, RMAT) 2.75 -> 1.95, its adjoint 2.3 -> 1.79.
//
// Row straddling two runs. At the end of its run a warp publishes the partial
// of the row it leaves unfinished (one 64-bit word: sweep stamp and value).
// A warp whose run starts inside a row holds back that row's value and, after
// its own run, adds the partials published by the preceding warps back to the
// one where the row starts (several when a hub spans whole runs); each wait is
// bounded by the launch's timeout. The row then gets its new value like any
// other, so every row is computed once per sweep; only its write comes at the
// end of the sweep.
#include <algorithm>
#include <climits>
#include <cstdint>

#include "sweep_warp.cuh"

namespace dag {

template <int MODE, int VAR, int WIPT>
__global__ void __launch_bounds__(NT, WMINBLOCKS) sweep_warp_kernel(const SweepParams p)
{
    constexpr int WTILE = 32 * WIPT;
    using O = Op<MODE>;
    constexpr bool BF = MODE == MODE_BF || MODE == MODE_BF8;
    constexpr bool SYNC = VAR == DAG_SYNC;
    constexpr bool ASYNC = VAR == DAG_ASYNC;
    constexpr bool DELAYED = VAR == DAG_DELAYED;
    constexpr bool LIVE_G = !SYNC && !BF;  // async/delayed PageRank-type: live global sum
    constexpr unsigned FULL = 0xffffffffu;

    __shared__ WarpShared<MODE, WIPT> sh;
    extern __shared__ __align__(16) uint32_t w_buf[];  // delayed: p.buf_cap values per warp

    const int c = blockIdx.x, tid = threadIdx.x, lane = tid & 31, wl = tid >> 5;
    const int w = c * WWARPS + wl;  // this worker
    SyncBlock* sb = p.sync;
    unsigned long long bar_target = 0;
    uint32_t* X0 = (uint32_t*)p.x0;
    uint32_t* X1 = (uint32_t*)p.x1;
    const int row_lo = p.cta_row[w], row_hi = p.cta_row[w + 1];  // rows whose end item lies in the run
    const int t_lo = p.cta_tile[w], t_hi = p.cta_tile[w + 1];
    uint16_t* end = sh.end[wl];
    uint32_t* val = sh.val[wl];
    uint32_t* buf = w_buf + (size_t)wl * (DELAYED ? p.buf_cap : 0);
    // the run starts inside a row: its first row waits for the earlier runs' partials
    const bool mid0 = t_lo < t_hi && p.tile_nz[t_lo] > p.rowptr[p.tile_row[t_lo]];
    const bool head = mid0 && row_hi > row_lo;

    // ---------------- initial values, a grid-stride pass (a row-range sweep is given them) ----------------
    if (!p.shard) {
        double gpart = 0.0, tpart = 0.0;
        init_values<MODE>(p, X0, gpart, tpart);
        if constexpr (!BF) {
            block_sum2(sh, gpart, tpart);
            if (tid == 0) {
                atomicAdd(&sb->acc_g[2], gpart);
                atomicAdd(&sb->T, tpart);
            }
        }
    }
    if (p.skip_barrier_cta0 && c == 0) return;  // test hook: the others' waits must run out
    if (!p.shard && !grid_barrier(sb, p.nblocks, bar_target, p.timeout_ns, p.cluster)) return;

    double T = 1.0;
    if (tid == 0 && !BF) {
        sh.T = p.shard ? p.shard_T : ld_relaxed_f64(&sb->T);
        sh.gprev = p.shard ? p.shard_N : ld_relaxed_f64(&sb->acc_g[2]);
    }
    __syncthreads();
    if constexpr (!BF) T = (MODE == MODE_ADJ || p.base || p.shard) ? sh.T : 1.0;  // a uniform teleport sums to 1
    double gprev = BF ? 0.0 : sh.gprev;
    AdjOffset A{gprev, 0.0, 0.0f, 0.0, 0.0, 0};  // adjoint: sum lambda, deflation offset
    LiveSum L{};
    if constexpr (LIVE_G) L = live_sum_setup<MODE>(p, T, gprev);
    const double tol = (MODE == MODE_ADJ) ? p.tol * T : p.tol;
    // gathers: sync reads the previous iterate with ordinary loads; async reads the live array
    // in L2 (DAG_READ_CACHED: ordinary loads, refreshed by the grid barrier); delayed per p.read_mode
    const int rmode = SYNC ? READ_CACHED : ASYNC ? (p.read_mode == READ_CACHED ? READ_CACHED : READ_COHERENT)
                                                  : p.read_mode;
    const uint64_t pol_edge = policy_evict_first();
    const uint64_t pol_vertex = policy_evict_last();
    long long flushes = 0;
    int it = 0;
    bool converged = false;
    double last_res = 0.0;

    for (; it < p.max_iters; ++it) {
        const int slot = it % 3;
        const unsigned stamp = (unsigned)it + 1u;
        const uint32_t* xin = SYNC ? ((it & 1) ? X1 : X0) : X0;
        uint32_t* xout = SYNC ? ((it & 1) ? X0 : X1) : X0;
        // per-lane partial sums in FP32 (few rows each); FP64 from the block reduction on
        float res_part = 0.0f, g_part = 0.0f, dg_part = 0.0f;
        uint32_t carry = O::identity();
        bool head_pending = head;
        uint32_t head_part = O::identity();
        int buf_first = row_lo + (head ? 1 : 0), buf_cnt = 0;
        float gt = 0.0f;
        if constexpr (SYNC && !BF)
            gt = (MODE == MODE_ADJ) ? (float)((double)p.g_coef * gprev) : (float)((double)p.g_coef * (T - gprev));

        // pipeline: tile t + 2's edge sources are copied and tile t + 1's gathers are in flight while tile t is summed
        // and its rows finished. (Gathers after this tile's stores, as in the ordered sweep, read newer values, but
        // cost 4% per sweep on a banded graph and 3% with a product per edge, for one sweep less on the former.)
        WStage<MODE, WIPT> nx;
        WCoord c1;  // of tile t + 1
        if (t_lo < t_hi) {
            const WCoord c0 = wcoord(p, t_lo);
            c1 = wcoord(p, min(t_lo + 1, t_hi - 1));
            wissue_col(sh, p, c0, wl, lane, pol_edge);
            wcommit();
            wlanded();
            wgather(nx, sh, p, xin, c0, wl, lane, rmode, LIVE_G, pol_edge, pol_vertex);
            if (t_lo + 1 < t_hi) wissue_col(sh, p, c1, wl, lane, pol_edge);
            wcommit();
        }
        for (int t = t_lo; t < t_hi; ++t) {
            const int a0 = nx.a0, NA = nx.NA;
            const uint32_t pf_xo = nx.xo;
            const float pf_dg = nx.dg, pf_bv = nx.bv;
            if constexpr (LIVE_G) {  // the global term, from the live sum read with every LIVE_EVERY-th tile
                if (((t - t_lo) & (LIVE_EVERY - 1)) == 0) gt = live_term<MODE>(L, warp_sum(nx.gs));
            }
            __syncwarp();  // the previous tile's epilogue is done with end / val
            wstage(sh, nx, p, wl, lane, pol_vertex);
            const WCoord c2 = wcoord(p, min(t + 2, t_hi - 1));
            if (t + 1 < t_hi) {
                wlanded();
                wgather(nx, sh, p, xin, c1, wl, lane, rmode, LIVE_G && ((t + 1 - t_lo) & (LIVE_EVERY - 1)) == 0, pol_edge,
                        pol_vertex);
                if (t + 2 < t_hi) wissue_col(sh, p, c2, wl, lane, pol_edge);
                wcommit();
                c1 = c2;
            }
            __syncwarp();
            const uint32_t carry_in = carry;
            carry = wwalk<MODE, WIPT>(end, val, sh.mark[wl], NA, carry, lane);
            __syncwarp();

            // -------- new values of the rows this tile completed --------
            const int skip = (head_pending && NA > 0) ? 1 : 0;  // the run's first row waits for the look-back
            if (skip && lane == 0) head_part = wrow_sum<MODE>(val, end, 0, carry_in);
            head_pending = head_pending && NA == 0;
            auto finish = [&](int r, uint32_t xo, float dg, float bv) {
                const int v = a0 + r;
                const uint32_t xnew = row_update_b<MODE>(p, v, wrow_sum<MODE>(val, end, r, carry_in), xo, dg, gt, bv, A.off_f,
                                                         res_part, g_part, dg_part);
                if constexpr (SYNC) st_weak_b32(xout + v, xnew);
                else if constexpr (ASYNC) st_relaxed_b32(X0 + v, xnew);
                else buf[v - buf_first] = xnew;
            };
            if (lane < NA && !(lane == 0 && skip)) finish(lane, pf_xo, pf_dg, pf_bv);
            constexpr int WROWS = 4;  // rows per lane whose inputs are in flight together (a tile of mostly empty rows)
            for (int r = lane + 32; r < NA; r += 32 * WROWS) {
                uint32_t xo[WROWS];
                float dg[WROWS], bv[WROWS];
#pragma unroll
                for (int u = 0; u < WROWS; ++u) {
                    xo[u] = 0u;
                    dg[u] = bv[u] = 0.0f;
                    if (r + 32 * u < NA) wrow_inputs<MODE>(p, xin, a0 + r + 32 * u, pol_vertex, xo[u], dg[u], bv[u]);
                }
#pragma unroll
                for (int u = 0; u < WROWS; ++u)
                    if (r + 32 * u < NA) finish(r + 32 * u, xo[u], dg[u], bv[u]);
            }
            if constexpr (ASYNC && LIVE_G) {
                if (((t - t_lo) & (LIVE_EVERY - 1)) == LIVE_EVERY - 1) {  // this warp's change of N
                    const float s = warp_sum(dg_part);
                    dg_part = 0.0f;
                    if (lane == 0 && s != 0.0f) live_add(sb, w % GSTRIPES, s, L.S);
                }
            }
            if constexpr (DELAYED) {
                buf_cnt += NA - skip;
                if (buf_cnt >= p.delta || t == t_hi - 1 || (p.buf_clamped && buf_cnt > p.buf_cap - WTILE)) {
                    __syncwarp();  // the buffer's values are written
                    for (int k = lane; k < buf_cnt; k += 32) st_relaxed_b32(X0 + buf_first + k, buf[k]);
                    if constexpr (LIVE_G) {
                        const float s = warp_sum(dg_part);
                        dg_part = 0.0f;
                        __syncwarp();
                        if (lane == 0 && s != 0.0f) {
                            __threadfence();  // this warp's flushed values before its share of N
                            live_add(sb, w % GSTRIPES, s, L.S);
                        }
                    }
                    if (lane == 0) {
                        // refresh this SM's view: later ordinary loads see what other workers published
                        if (rmode == READ_CACHED_REFRESH) asm volatile("fence.acq_rel.gpu;" ::: "memory");
                        ++flushes;
                    }
                    buf_first += buf_cnt;
                    buf_cnt = 0;
                    __syncwarp();  // the buffer is free again
                }
            }
        }  // tiles

        // -------- the row this run leaves unfinished, and the one it started inside --------
        if (lane == 0) st_relaxed_u64(p.wpub + w, ((unsigned long long)stamp << 32) | carry);
        if (head) {
            uint32_t s = __shfl_sync(FULL, head_part, 0);
            bool ok = true;
            for (int k = w - 1; k >= 0; --k) {
                uint32_t pk = 0u;
                if (lane == 0) ok = wait_published(p.wpub, k, stamp, sb, p.timeout_ns, &pk);
                ok = __shfl_sync(FULL, ok, 0);
                pk = __shfl_sync(FULL, pk, 0);
                if (!ok) break;
                s = O::combine(s, pk);
                // the row starts in run k unless run k ends no row and itself starts inside the row
                const int tk0 = p.cta_tile[k], tk1 = p.cta_tile[k + 1];
                const bool k_emits = p.cta_row[k + 1] > p.cta_row[k];
                const bool k_mid = tk0 >= tk1 || p.tile_nz[tk0] > p.rowptr[p.tile_row[tk0]];
                if (k_emits || !k_mid) break;
            }
            if (ok && lane == 0) {
                const int v = row_lo;
                const uint32_t xo = ld_weak_b32(xin + v);
                const float dg = BF ? 0.0f : p.degf[v];
                if constexpr (LIVE_G) gt = live_term<MODE>(L, stripes_total(sb));  // the live term as the row is computed
                const uint32_t xnew = row_update<MODE>(p, v, s, xo, dg, gt, A.off_f, res_part, g_part, dg_part);
                if constexpr (SYNC) st_weak_b32(xout + v, xnew);
                else st_relaxed_b32(X0 + v, xnew);
            }
        }
        if constexpr (LIVE_G) {  // the rest of this warp's change of N
            const float s = warp_sum(dg_part);
            dg_part = 0.0f;
            if (lane == 0 && s != 0.0f) live_add(sb, w % GSTRIPES, s, L.S);
        }

        // -------- end of sweep: residual, barrier, stopping rule --------
        __syncwarp();  // (block_add uses the warp's val)
        block_add(sh, res_part, &sb->acc_res[slot], g_part, ((SYNC || MODE == MODE_ADJ) && !BF) ? &sb->acc_g[slot] : nullptr);
        if (!grid_barrier(sb, p.nblocks, bar_target, p.timeout_ns, p.cluster)) return;
        if (tid == 0) {
            sh.res = sweep_residual(sb, slot);
            sh.gprev = ld_relaxed_f64(&sb->acc_g[slot]);
            if (c == 0) {
                const int dead = (it + 2) % 3;  // read by everyone before this barrier
                sb->acc_res[dead] = 0.0;
                sb->acc_g[dead] = 0.0;
            }
        }
        __syncthreads();
        if (sweep_failed(sh.res)) return;  // an error was recorded
        last_res = sh.res;
        gprev = sh.gprev;
        if (last_res <= tol) {
            converged = true;
            ++it;
            break;
        }
        if constexpr (MODE == MODE_ADJ) adjoint_deflate(p, A, gprev, SYNC);  // the slow mode along 1, as an offset
    }

    // ---------------- output, a grid-stride pass (a row-range sweep leaves them in x1) ----------------
    if (!p.shard) {
        const uint32_t* xf = SYNC ? ((it & 1) ? X1 : X0) : X0;
        write_output<MODE>(p, xf, A.off_f);
    }
    if (lane == 0 && flushes) atomicAdd((unsigned long long*)&sb->flushes, (unsigned long long)flushes);
    if (tid == 0 && c == 0) {
        sb->iters = it;
        sb->residual = last_res;
        sb->converged = converged ? 1 : 0;
    }
}

// ---------------------------------------------------------------------------
// Ordered warp sweep (asynchronous form, DAG_WARP_ORDERED): the warps take the
// tiles of the whole merge path in turn instead of each walking a run of its
// own, tile t to warp t mod W, so at any moment the GPU works on one window of
// W consecutive tiles and a sweep visits the vertices in order across the GPU:
// one in-order stream, as a single thread's asynchronous sweep (Sec. I) with
// every warp on it. A row whose in-edges
// span tiles is finished with a decoupled look-back over per-tile published
// partials (Merrill & Garland's single-pass scan): every tile publishes the
// partial of the row it leaves unfinished at once (inclusive when that row
// starts inside the tile, else an aggregate, upgraded to inclusive later), and
// the tile that ends a row begun earlier adds the published partials back to
// the first inclusive one, 32 tiles per step (one per lane). A warp resolves
// its tile's look-back after walking its next tile, by when the tiles before
// it have published (a tile publishes before its warp resolves anything
// older, so the lowest pending tile can always finish); each wait is bounded
// by the launch's timeout.
// ---------------------------------------------------------------------------
constexpr unsigned TPUB_INCL = 0x80000000u;  // the published value is the row's partial from its start

// The word tile j published in sweep `stamp` (waits, bounded); false when the wait ran out or another CTA
// recorded an error.
__device__ __forceinline__ bool wait_tile(const unsigned long long* pub, int j, unsigned stamp, SyncBlock* sb,
                                          long long timeout_ns, unsigned long long* out)
{
    const unsigned long long t0 = globaltimer_ns();
    unsigned spins = 0;
    for (;;) {
        const unsigned long long v = ld_relaxed_u64(pub + j);
        if (((unsigned)(v >> 32) & ~TPUB_INCL) == stamp) {
            *out = v;
            return true;
        }
        if (ld_relaxed_i32(&sb->err) != 0) return false;
        if ((++spins & 15u) == 0 && (long long)(globaltimer_ns() - t0) > timeout_ns) {
            atomicCAS(&sb->err, 0, DAG_ERR_BARRIER_TIMEOUT);
            return false;
        }
        __nanosleep(32);
    }
}

template <int MODE, int WIPT>
__global__ void __launch_bounds__(NT, WMINBLOCKS) sweep_ordered_kernel(const SweepParams p)
{
    using O = Op<MODE>;
    constexpr int WTILE = 32 * WIPT;
    constexpr bool BF = MODE == MODE_BF || MODE == MODE_BF8;
    constexpr bool LIVE_G = !BF;
    constexpr unsigned FULL = 0xffffffffu;
    (void)WTILE;

    __shared__ WarpShared<MODE, WIPT> sh;
    const int c = blockIdx.x, tid = threadIdx.x, lane = tid & 31, wl = tid >> 5;
    const int w = c * WWARPS + wl;
    const int W = p.nblocks * WWARPS, T = p.ntiles;  // warp w takes tiles w, w + W, w + 2W, ...
    SyncBlock* sb = p.sync;
    unsigned long long bar_target = 0;
    uint32_t* X = (uint32_t*)p.x0;
    unsigned long long* pub = p.wpub;  // [T]
    uint16_t* end = sh.end[wl];
    uint32_t* val = sh.val[wl];

    // ---------------- initial values (any thread any row: nothing reads them before the barrier) ----------------
    {
        double gpart = 0.0, tpart = 0.0;
        init_values<MODE>(p, X, gpart, tpart);
        if constexpr (!BF) {
            block_sum2(sh, gpart, tpart);
            if (tid == 0) {
                atomicAdd(&sb->acc_g[2], gpart);
                atomicAdd(&sb->T, tpart);
            }
        }
    }
    if (p.skip_barrier_cta0 && c == 0) return;  // test hook: the others' waits must run out
    if (!grid_barrier_call(sb, p.nblocks, bar_target, p.timeout_ns, p.cluster)) return;

    double T_tot = 1.0;
    if (tid == 0 && !BF) {
        sh.T = ld_relaxed_f64(&sb->T);
        sh.gprev = ld_relaxed_f64(&sb->acc_g[2]);
    }
    __syncthreads();
    if constexpr (!BF) T_tot = (MODE == MODE_ADJ || p.base) ? sh.T : 1.0;
    LiveSum L{};
    if constexpr (LIVE_G) L = live_sum_setup<MODE>(p, T_tot, sh.gprev);
    AdjOffset A{BF ? 0.0 : sh.gprev, 0.0, 0.0f, 0.0, 0.0, 0};  // adjoint: sum lambda, deflation offset
    const double tol = (MODE == MODE_ADJ) ? p.tol * T_tot : p.tol;
    const int rmode = p.read_mode == READ_CACHED ? READ_CACHED : READ_COHERENT;
    const uint64_t pol_edge = policy_evict_first();
    const uint64_t pol_vertex = policy_evict_last();
    int it = 0;
    bool converged = false;
    double last_res = 0.0;

    for (; it < p.max_iters; ++it) {
        const int slot = it % 3;
        const unsigned stamp = (unsigned)it + 1u;
        float res_part = 0.0f, g_part = 0.0f, dg_part = 0.0f;
        float gt = 0.0f;
        // the look-back this warp still owes (warp-uniform): tile, its first row, the tile's partial of it,
        // whether the row ends in the tile (else the tile's published aggregate is upgraded), its inputs
        int pend_t = -1, pend_row = 0, pend_fin = 0;
        uint32_t pend_val = 0u, pend_xo = 0u;
        float pend_dg = 0.0f;
        bool ok = true;

        // Adds the partials published by the tiles before pend_t back to the first inclusive one, then
        // finishes the pending row or publishes the tile's inclusive partial. The warp looks back 32
        // tiles at a time, one per lane (lane i reads tile hi - i), as in a single-pass scan's look-back:
        // the nearest inclusive entry ends the walk, the partials after it are reduced over the lanes.
        auto resolve = [&]() {
            if (pend_t < 0) return;
            uint32_t C = O::identity();
            for (int hi = pend_t - 1; ok;) {
                const int j = hi - lane;
                unsigned long long v = 0ull;
                bool got = true;
                if (j >= 0) got = wait_tile(pub, j, stamp, sb, p.timeout_ns, &v);
                ok = __all_sync(FULL, got) != 0;
                if (!ok) break;
                const unsigned incl = __ballot_sync(FULL, j >= 0 && (((unsigned)(v >> 32)) & TPUB_INCL) != 0);
                const int stop = incl ? __ffs(incl) - 1 : 31;  // the nearest inclusive entry, else the whole window
                uint32_t mine = (j >= 0 && lane <= stop) ? (uint32_t)v : O::identity();
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) mine = O::combine(mine, __shfl_xor_sync(FULL, mine, o));
                C = O::combine(C, mine);
                if (incl || hi < 32) break;  // tile 0 is always inclusive, so the walk ends by then
                hi -= 32;
            }
            if (ok && lane == 0) {
                const uint32_t total = O::combine(C, pend_val);
                if (pend_fin) {
                    const uint32_t xnew =
                        row_update<MODE>(p, pend_row, total, pend_xo, pend_dg, gt, A.off_f, res_part, g_part, dg_part);
                    st_relaxed_b32(X + pend_row, xnew);
                } else {
                    st_relaxed_u64(pub + pend_t, ((unsigned long long)(stamp | TPUB_INCL) << 32) | total);
                }
            }
            pend_t = -1;
        };

        WStage<MODE, WIPT> nx;
        WCoord c1;  // of this warp's next tile
        int k = 0;  // its tiles so far in the sweep
        if (w < T) {
            const WCoord c0 = wcoord(p, w);
            c1 = wcoord(p, min(w + W, T - 1));
            wissue_col(sh, p, c0, wl, lane, pol_edge);
            wcommit();
            wlanded();
            wgather(nx, sh, p, X, c0, wl, lane, rmode, LIVE_G, pol_edge, pol_vertex);
            if (w + W < T) wissue_col(sh, p, c1, wl, lane, pol_edge);
            wcommit();
        }
        for (int t = w; t < T && ok; t += W, ++k) {
            const int a0 = nx.a0, b0 = nx.b0, NA = nx.NA;
            const bool cont = b0 > nx.rp0;  // the tile starts inside row a0
            const uint32_t pf_xo = nx.xo;
            const float pf_dg = nx.dg, pf_bv = nx.bv;
            if constexpr (LIVE_G) {
                if ((k & (LIVE_EVERY - 1)) == 0) gt = live_term<MODE>(L, warp_sum(nx.gs));
            }
            __syncwarp();
            wstage(sh, nx, p, wl, lane, pol_vertex);
            const bool more2 = T - t > 2LL * W;
            const WCoord c2 = wcoord(p, more2 ? t + 2 * W : T - 1);
            __syncwarp();
            const uint32_t trail = wwalk<MODE, WIPT>(end, val, sh.mark[wl], NA, O::identity(), lane);
            __syncwarp();
            // the partial of the row left unfinished: inclusive unless the tile lies inside a row begun before
            const bool incl = NA > 0 || !cont;
            if (lane == 0)
                st_relaxed_u64(pub + t, ((unsigned long long)(stamp | (incl ? TPUB_INCL : 0u)) << 32) | trail);

            // -------- rows this tile completed (its first one, begun before, waits for the look-back) --------
            const int skip = (cont && NA > 0) ? 1 : 0;
            const uint32_t first_sum = NA > 0 ? wrow_sum<MODE>(val, end, 0, O::identity()) : 0u;
            auto finish = [&](int r, uint32_t xo, float dg, float bv) {
                const int v = a0 + r;
                const uint32_t xnew = row_update_b<MODE>(p, v, wrow_sum<MODE>(val, end, r, O::identity()), xo, dg, gt, bv,
                                                         A.off_f, res_part, g_part, dg_part);
                st_relaxed_b32(X + v, xnew);
            };
            if (lane < NA && !(lane == 0 && skip)) finish(lane, pf_xo, pf_dg, pf_bv);
            constexpr int WROWS = 2;  // rows per lane whose inputs are in flight together (a tile of mostly empty rows)
            for (int r = lane + 32; r < NA; r += 32 * WROWS) {
                uint32_t xo[WROWS];
                float dg[WROWS], bv[WROWS];
#pragma unroll
                for (int u = 0; u < WROWS; ++u) {
                    xo[u] = 0u;
                    dg[u] = bv[u] = 0.0f;
                    if (r + 32 * u < NA) wrow_inputs<MODE>(p, X, a0 + r + 32 * u, pol_vertex, xo[u], dg[u], bv[u]);
                }
#pragma unroll
                for (int u = 0; u < WROWS; ++u)
                    if (r + 32 * u < NA) finish(r + 32 * u, xo[u], dg[u], bv[u]);
            }
            // -------- the next tile's gathers (after this tile's stores: in flight earlier, they read older values and
            // a sweep took 397 instead of 372 us at 4 M vertices, RMAT) --------
            if (t + W < T) {
                wlanded();
                wgather(nx, sh, p, X, c1, wl, lane, rmode, LIVE_G && ((k + 1) & (LIVE_EVERY - 1)) == 0, pol_edge, pol_vertex);
                if (more2) wissue_col(sh, p, c2, wl, lane, pol_edge);
                wcommit();
                c1 = c2;
            }
            // -------- the previous tile's look-back, then this tile's becomes pending --------
            resolve();
            if (cont) {
                pend_t = t;
                pend_row = a0;
                pend_fin = NA > 0 ? 1 : 0;
                pend_val = NA > 0 ? first_sum : trail;
                pend_xo = __shfl_sync(FULL, pf_xo, 0);
                pend_dg = __shfl_sync(FULL, pf_dg, 0);
            }
            if constexpr (LIVE_G) {
                if ((k & (LIVE_EVERY - 1)) == LIVE_EVERY - 1) {  // this warp's change of N
                    const float s = warp_sum(dg_part);
                    dg_part = 0.0f;
                    if (lane == 0 && s != 0.0f) live_add(sb, w % GSTRIPES, s, L.S);
                }
            }
        }  // tiles
        wlanded();  // (a look-back that gave up leaves copies in flight)
        resolve();
        if constexpr (LIVE_G) {
            const float s = warp_sum(dg_part);
            dg_part = 0.0f;
            if (lane == 0 && s != 0.0f) live_add(sb, w % GSTRIPES, s, L.S);
        }

        // -------- end of sweep: residual, barrier, stopping rule --------
        __syncwarp();  // (block_add uses the warp's val)
        block_add(sh, res_part, &sb->acc_res[slot], g_part, MODE == MODE_ADJ ? &sb->acc_g[slot] : nullptr);
        if (!grid_barrier_call(sb, p.nblocks, bar_target, p.timeout_ns, p.cluster)) return;
        if (tid == 0) {
            sh.res = sweep_residual(sb, slot);
            if (MODE == MODE_ADJ) sh.gprev = ld_relaxed_f64(&sb->acc_g[slot]);
            if (c == 0) {
                const int dead = (it + 2) % 3;  // read by everyone before this barrier
                sb->acc_res[dead] = 0.0;
                sb->acc_g[dead] = 0.0;
            }
        }
        __syncthreads();
        if (sweep_failed(sh.res)) return;  // an error was recorded
        last_res = sh.res;
        if (last_res <= tol) {
            converged = true;
            ++it;
            break;
        }
        if constexpr (MODE == MODE_ADJ) adjoint_deflate(p, A, sh.gprev, false);  // the slow mode along 1, as an offset
    }

    // ---------------- output ----------------
    write_output<MODE>(p, X, A.off_f);
    if (tid == 0 && c == 0) {
        sb->iters = it;
        sb->residual = last_res;
        sb->converged = converged ? 1 : 0;
    }
}

const void* sweep_ordered_kernel_ptr(int mode, int ipt)
{
#define DAG_ORD_ROW(I)                                                                                        \
    {(const void*)sweep_ordered_kernel<MODE_PR, I>, (const void*)sweep_ordered_kernel<MODE_PRW, I>,         \
     (const void*)sweep_ordered_kernel<MODE_ADJ, I>, (const void*)sweep_ordered_kernel<MODE_BF, I>,         \
     (const void*)sweep_ordered_kernel<MODE_BF8, I>}
    static const void* const table[3][5] = {DAG_ORD_ROW(5), DAG_ORD_ROW(7), DAG_ORD_ROW(11)};
#undef DAG_ORD_ROW
    const int k = ipt == 5 ? 0 : ipt == 7 ? 1 : ipt == 11 ? 2 : -1;
    return k < 0 ? nullptr : table[k][mode];
}

// Kernel of (mode, variant, items per lane); nullptr for a shape not built.
const void* sweep_warp_kernel_ptr(int mode, int variant, int ipt)
{
#define DAG_WARP_ROW(M, I)                                                                                    \
    {(const void*)sweep_warp_kernel<M, DAG_SYNC, I>, (const void*)sweep_warp_kernel<M, DAG_ASYNC, I>,       \
     (const void*)sweep_warp_kernel<M, DAG_DELAYED, I>}
#define DAG_WARP_SHAPE(I) \
    {DAG_WARP_ROW(MODE_PR, I), DAG_WARP_ROW(MODE_PRW, I), DAG_WARP_ROW(MODE_ADJ, I), DAG_WARP_ROW(MODE_BF, I), \
     DAG_WARP_ROW(MODE_BF8, I)}
    static const void* const table[3][5][3] = {DAG_WARP_SHAPE(5), DAG_WARP_SHAPE(7), DAG_WARP_SHAPE(11)};
#undef DAG_WARP_SHAPE
#undef DAG_WARP_ROW
    const int k = ipt == 5 ? 0 : ipt == 7 ? 1 : ipt == 11 ? 2 : -1;
    return k < 0 ? nullptr : table[k][mode][variant];
}

// Launch shape of a warp-worker sweep: CTAs resident at once (cooperative
// launch), warps = CTAs * WWARPS workers, and the delayed form's buffer of
// min(delta - 1 + WTILE, rows of the longest run) values per warp, clamped to
// what fits in shared memory (flushed when the next tile might not fit).
enum WarpKind { WARP_RUNS = 0, WARP_ORDERED = 1, WARP_FRONTIER = 2 };

static const void* warp_kernel(int kind, int mode, int variant, int ipt, bool ordered = false)
{
    if (kind == WARP_ORDERED) return sweep_ordered_kernel_ptr(mode, ipt);
    if (kind == WARP_FRONTIER) return sweep_warp_frontier_kernel_ptr(mode, ipt, ordered);
    return sweep_warp_kernel_ptr(mode, variant, ipt);
}

// A row's weight in the warps' runs beside its in-edges (Sec. III-A weighs in-degree + 1, for a CPU thread's work):
// a row's update costs a warp about twice an in-edge more than the row's item did in the tiles' cut. Where a graph's
// rows without in-edges lie together (RMAT: half the rows), runs of equal item counts held up to 6,600 rows against a
// mean of 430 and the sweep waited for them. Weights 1, 2, 3, 4, RMAT, ms: CTA-ordered frontier Bellman-Ford (4 M
// vertices) 2.99, 2.19-2.5, 2.05-2.35, 2.3-2.55; weighted PageRank and its adjoint (2 M) 2.78 + 2.4, 2.05 + 1.9,
// 1.95 + 1.79, 1.99 + 1.98. Bellman-Ford on warp runs, whose edges cost more (a weight each) and rows less (no degree),
// RMAT, 4 M vertices, four-byte weights, 224-item tiles, weights 1, 2, 3: sync 4.34, 3.91, 3.97, delta 16 4.03, 3.83, 3.60,
// delta 256 with cached reads 4.41, 3.95, 4.36, async 3.88, 3.45, 3.48; one-byte weights the same order, 2 to 5% less. Graphs
// without skew do not move. (Each figure is of one plan: where a plan's arrays land in memory moves RMAT's solves by up to
// 9%. Over ten placements, 4 M vertices, four-byte weights, us a sweep, against the tiles' merge-path walk over runs of
// equal item counts: sync 265.5 and 265.3, delta 16 284 and 293, delta 256 cached 300 and 293, async 282 and 291; 1 M 5 to
// 8% less but delta 256 1% more, uniform and banded graphs 4 to 26% less.)
static int warp_row_weight(int kind, int mode)
{
    return kind == WARP_RUNS && (mode == MODE_BF || mode == MODE_BF8) ? 2 : 3;
}

static int warp_shape(dag_plan* plan, int mode, int variant, int delta, int* nb_out, int* cap_out, int* clamped_out,
                      Partition** part_out, cudaStream_t s, int kind, bool ordered = false)
{
    const int WTILE = 32 * plan->warp_ipt;
    const void* k = warp_kernel(kind, mode, variant, plan->warp_ipt, ordered);
    if (!k) return set_error(DAG_ERR_INVALID, "no warp tile of that shape");
    const auto key = std::make_tuple(1 + kind + (ordered ? 8 : 0), mode, variant, variant == DAG_DELAYED ? delta : 0,
                                     plan->worker_cap, plan->warp_ipt);
    const auto hit = plan->shapes.find(key);
    if (hit != plan->shapes.end()) {
        const Shape& sh = hit->second;
        *nb_out = sh.nb;
        *cap_out = sh.cap;
        *clamped_out = sh.clamped;
        *part_out = sh.part;
        return apply_shape(sh);
    }
    Shape sh;
    cudaFuncAttributes fa{};
    DAG_CUDA(cudaFuncGetAttributes(&fa, k));
    int max_dyn = 0;
    DAG_CUDA(cudaDeviceGetAttribute(&max_dyn, cudaDevAttrMaxSharedMemoryPerBlockOptin, plan->device));
    const long long max_cap = ((long long)max_dyn - (long long)fa.sharedSizeBytes) / (4LL * WWARPS);
    int cap = 0, clamped = 0, nb = 0;
    Partition* part = nullptr;
    auto resident = [&](int cap_elems, int* out) -> int {
        const size_t dyn = (size_t)WWARPS * (size_t)cap_elems * 4;
        DAG_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn));
        DAG_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, 100));
        int per_sm = 0;
        DAG_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, NT, dyn));
        if (per_sm < 1) return set_error(DAG_ERR_INVALID, "warp sweep cannot be resident with this delta");
        const int rc = set_l1_carveout(k, plan->device, NT, fa.sharedSizeBytes, dyn, per_sm, &sh.carveout);
        if (rc) return rc;
        sh.dyn = (int)dyn;
        int n_cta = per_sm * plan->num_sms;
        // a small graph's sweep is its grid barrier: one tile per warp (two CTAs at least), as settle_shape; 5,000
        // vertices in 608 CTAs took 545 us, the runs' look-back waiting along runs without a tile, in 34 112
        const long long tiles = ((long long)plan->n + plan->m + WTILE - 1) / WTILE;
        n_cta = (int)std::min((long long)n_cta, std::max(2LL, (tiles + WWARPS - 1) / WWARPS));
        if (plan->worker_cap > 0) n_cta = std::min(n_cta, plan->worker_cap);  // the cap counts CTAs
        *out = n_cta;
        return DAG_OK;
    };
    int rc = resident(0, &nb);
    if (rc) return rc;
    bool settled = false;  // CTAs per SM only fall, so a few passes settle the shape
    for (int iter = 0; iter < 6 && !settled; ++iter) {
        rc = get_warp_partition(plan, nb * WWARPS, WTILE, warp_row_weight(kind, mode), &part, s);
        if (rc) return rc;
        settled = true;
        if (variant != DAG_DELAYED) break;
        const long long want = std::min((long long)delta - 1 + WTILE, (long long)std::max(part->max_rows, 1));
        const long long need = std::min(want, max_cap);
        clamped = need < want ? 1 : 0;
        if (clamped && need < WTILE + 1) return set_error(DAG_ERR_INVALID, "delay buffer does not fit in shared memory");
        cap = (int)std::max(need, 1LL);
        int nb2 = 0;
        rc = resident(cap, &nb2);
        if (rc) return rc;
        if (nb2 < nb) {
            nb = nb2;
            settled = false;
        }
    }
    if (!settled) return set_error(DAG_ERR_INVALID, "warp sweep launch shape did not settle");
    *nb_out = nb;
    *cap_out = cap;
    *clamped_out = clamped;
    *part_out = part;
    sh.nb = nb;
    sh.cap = cap;
    sh.clamped = clamped;
    sh.part = part;
    sh.kernels[0] = k;
    plan->shapes.emplace(key, sh);
    return DAG_OK;
}

// The frontier maps of the warp partition a frontier solve of this plan would use (built once, outside the
// timed solve, as the CTA-tile frontier's are).
int warp_frontier_maps(dag_plan* plan, int mode, cudaStream_t s)
{
    int nb = 0, cap = 0, clamped = 0;
    Partition* part = nullptr;
    int rc = warp_shape(plan, mode, DAG_ASYNC, 0, &nb, &cap, &clamped, &part, s, WARP_FRONTIER);
    if (rc) return rc;
    return frontier_maps(plan, part, s, false);
}

int launch_warp_sweep(dag_plan* plan, int mode, int variant, int delta, SweepParams& p, cudaStream_t s,
                      int* out_nblocks)
{
    if (p.local_read || p.own_l1) return set_error(DAG_ERR_INVALID, "local and own-block reads run the CTA-tile sweeps");
    const bool ordered = p.ordered != 0;
    if (ordered && variant != DAG_ASYNC)
        return set_error(DAG_ERR_INVALID, "ordered warp sweeps run the asynchronous form (delta 0)");
    if (p.frontier && (variant != DAG_ASYNC || (mode != MODE_BF && mode != MODE_BF8)))
        return set_error(DAG_ERR_INVALID, "the warp-tile frontier runs the asynchronous Bellman-Ford form");
    const int kind = p.frontier ? WARP_FRONTIER : ordered ? WARP_ORDERED : WARP_RUNS;
    int nb = 0, cap = 0, clamped = 0;
    Partition* part = nullptr;
    int rc = warp_shape(plan, mode, variant, delta, &nb, &cap, &clamped, &part, s, kind, ordered);
    if (rc) return rc;
    if (kind == WARP_ORDERED && !part->tpub)
        DAG_CUDA(cudaMalloc(&part->tpub, (size_t)part->tiles * sizeof(unsigned long long)));
    if (p.frontier) {
        rc = frontier_maps(plan, part, s, false);
        if (rc) return rc;
        p.fr_orow = plan->fr_orow;
        p.fr_otile = part->fr_otile;
        p.fr_oend = part->fr_oend;
        p.fr_act = part->fr_act;
        p.fr_alist = part->fr_alist;
        p.fr_chg = part->fr_chg;
        p.fr_glist = part->fr_glist;
        p.fr_gchg = part->fr_gchg;
        p.fr_sparse = plan->fr_sparse_warp;
        DAG_CUDA(cudaMemsetAsync(part->fr_act, 0, (size_t)std::max(part->tiles, 1) * sizeof(int), s));
    }
    p.nblocks = nb;
    p.delta = (variant == DAG_DELAYED) ? delta : 0;
    p.buf_cap = cap;
    p.buf_clamped = clamped;
    p.cta_row = part->cta_row;
    p.cta_tile = part->cta_tile;
    p.tile_row = part->tile_row;
    p.tile_nz = part->tile_nz;
    p.wpub = kind == WARP_ORDERED ? part->tpub : part->wpub;
    p.ntiles = part->tiles;
    p.m = (int)plan->m;
    p.sync = plan->sync;
    p.timeout_ns = plan->timeout_ns;
    p.skip_barrier_cta0 = 0;
    p.stall_fill = 0;
    if (plan->skip_barrier_once) {
        p.skip_barrier_cta0 = 1;
        p.timeout_ns = plan->skip_timeout_ns;
        plan->skip_barrier_once = 0;
    }
    rc = reset_sync(plan, s);
    if (rc) return rc;
    // stamps of an earlier solve must not pass for this one's
    DAG_CUDA(cudaMemsetAsync(p.wpub, 0,
                             (size_t)(kind == WARP_ORDERED ? part->tiles : part->nblocks) * sizeof(unsigned long long),
                             s));
    const void* k = warp_kernel(kind, mode, variant, plan->warp_ipt, ordered);
    const size_t dyn = (size_t)WWARPS * (size_t)cap * 4;
    DAG_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn));
    rc = launch_sweep_grid(k, nb, dyn, p, s);
    if (rc) return rc;
    *out_nblocks = nb * WWARPS;
    return DAG_OK;
}

// One synchronous sweep over rows [lo, hi) of the plan's graph (row sharding
// across GPUs, rowshard.py): x_in is the whole previous iterate, the new
// values of the range go to x_out[lo, hi), and d_sums receives {sum |r' - r|
// over the range (PageRank; Bellman-Ford: rows lowered), sum of r' over the
// range's vertices with out-edges (PageRank)} in FP64. The range's merge path
// is cut into warp tiles and warp runs as in a whole sweep.
__global__ void k_copy_sums(const SyncBlock* sb, double* out)
{
    out[0] = sb->acc_res[0];
    out[1] = sb->acc_g[0];
}

int sweep_rows(dag_plan* plan, int mode, int lo, int hi, SweepParams& p, double* d_sums, cudaStream_t s)
{
    const int WTILE = 32 * plan->warp_ipt;
    const void* k = sweep_warp_kernel_ptr(mode, DAG_SYNC, plan->warp_ipt);
    cudaFuncAttributes fa{};
    DAG_CUDA(cudaFuncGetAttributes(&fa, k));
    DAG_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 0));
    int per_sm = 0;
    DAG_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, NT, 0));
    if (per_sm < 1) return set_error(DAG_ERR_INVALID, "row sweep cannot be resident");
    int nb = per_sm * plan->num_sms;
    if (plan->worker_cap > 0) nb = std::min(nb, plan->worker_cap);
    Partition* part = nullptr;
    int rc = get_warp_partition_range(plan, nb * WWARPS, WTILE, warp_row_weight(WARP_RUNS, mode), lo, hi, &part, s);
    if (rc) return rc;
    p.nblocks = nb;
    p.m = (int)plan->m;
    p.max_iters = 1;
    p.tol = 0.0;
    p.delta = 0;
    p.buf_cap = 0;
    p.buf_clamped = 0;
    p.shard = 1;
    p.cta_row = part->cta_row;
    p.cta_tile = part->cta_tile;
    p.tile_row = part->tile_row;
    p.tile_nz = part->tile_nz;
    p.wpub = part->wpub;
    p.sync = plan->sync;
    p.timeout_ns = plan->timeout_ns;
    DAG_CUDA(cudaMemsetAsync(plan->sync, 0, sizeof(SyncBlock), s));
    DAG_CUDA(cudaMemsetAsync(part->wpub, 0, (size_t)part->nblocks * sizeof(unsigned long long), s));
    void* args[] = {(void*)&p};
    DAG_CUDA(cudaLaunchCooperativeKernel(k, dim3(nb), dim3(NT), args, 0, s));
    k_copy_sums<<<1, 1, 0, s>>>(plan->sync, d_sums);
    DAG_CUDA(cudaGetLastError());
    return DAG_OK;
}

}  // namespace dag

extern "C" int dag_plan_set_warp_tile(dag_plan* plan, int32_t items_per_lane)
{
    if (!plan) return dag::set_error(DAG_ERR_INVALID, "null plan");
    if (!dag::sweep_warp_kernel_ptr(dag::MODE_PR, DAG_SYNC, items_per_lane))
        return dag::set_error(DAG_ERR_INVALID, "items per lane must be 5, 7 or 11");
    plan->warp_ipt = items_per_lane;
    return DAG_OK;
}

extern "C" int32_t dag_warp_tile_items(const dag_plan* plan)
{
    return 32 * (plan ? plan->warp_ipt : dag::WIPT_DEFAULT);
}

extern "C" int dag_plan_set_warp_frontier_marks(dag_plan* plan, float marks_per_tile)
{
    if (!plan) return dag::set_error(DAG_ERR_INVALID, "null plan");
    if (!(marks_per_tile >= 0.0f) || !(marks_per_tile <= 1.0e6f))
        return dag::set_error(DAG_ERR_INVALID, "marks per tile must lie in [0, 1e6]");
    plan->fr_sparse_warp = marks_per_tile;
    return DAG_OK;
}
