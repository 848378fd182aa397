// Batched personalized PageRank and batched Bellman-Ford in one persistent
// launch (no counterpart in the paper: each column is an independent problem
// solved with the paper's sweep, Sec. III; columns stop on their own): the
// launch logic, and the kernel of the delayed form (and of the other forms when
// dag_plan_set_batched_wide is off; else they run batched_runs.cu).
//
// State X is row-major [n][B]: the B values of a vertex are contiguous, so an
// in-edge gathers one contiguous slice of B values. A CTA owns a vertex block
// (Sec. III-A partition) and holds one warp per 32-column chunk; every warp
// walks the CTA's merge-path tiles in vertex order, one lane per column. A
// column that met its stopping rule is frozen (not read, not written) for the
// rest of the launch, and a warp whose 32 columns are all frozen skips the
// tile. In the delayed form the "worker" of Sec. III-B is a (CTA, column
// chunk) pair: each warp buffers delta rows of its 32 columns in shared
// memory and copies them out when the buffer is full or its block is done.
#include <algorithm>
#include <climits>
#include <map>
#include <mutex>
#include <string>
#include <tuple>
#include <vector>

#include "batched.cuh"
#include "devmem.cuh"

namespace dag {

constexpr int BU = 8;  // edges gathered per warp before accumulating

template <bool BF>
__device__ __forceinline__ uint32_t b_ident()
{
    return BF ? INF : 0u;
}

template <bool BF>
__device__ __forceinline__ uint32_t b_comb(uint32_t a, uint32_t b)
{
    if constexpr (BF) return a < b ? a : b;
    else return __float_as_uint(__uint_as_float(a) + __uint_as_float(b));
}

__device__ __forceinline__ uint32_t b_relax(uint32_t du, uint32_t w)
{
    if (du == INF) return INF;
    uint32_t s = du + w;
    return (s < du || s == INF) ? INF - 1u : s;
}

template <bool BF, int VAR, bool W8 = false>
__global__ void batched_kernel(const BatchParams p)
{
    constexpr bool SYNC = VAR == DAG_SYNC;
    constexpr bool DELAYED = VAR == DAG_DELAYED;
    constexpr bool LIVE = !SYNC && !BF;
    extern __shared__ __align__(16) uint32_t smem[];
    int* s_col = (int*)smem;
    int* s_end = s_col + TILE;
    uint32_t* s_w = (uint32_t*)(s_end + TILE + 1);
    uint32_t* s_buf = s_w + (BF ? TILE : 0);  // per warp: delta rows x 32 columns

    const int B = p.B;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int col = warp * 32 + lane;
    const bool colok = col < B;
    const int cb = blockIdx.x;
    const int row_lo = p.cta_row[cb], row_hi = p.cta_row[cb + 1];
    const int tile_lo = p.cta_tile[cb], tile_hi = p.cta_tile[cb + 1];
    unsigned long long bar = 0;
    uint32_t* mybuf = s_buf + (size_t)warp * (DELAYED ? p.delta : 0) * 32;

    // ---------------- initial values ----------------
    {
        float gpart = 0.0f, tpart = 0.0f;  // per-lane partials over the block; FP64 in the atomics
        uint32_t s0 = BF && colok ? p.src[col] : 0u;
        // four rows' inputs loaded before any is stored (the stores could alias the inputs, so the
        // compiler would not overlap them itself)
        for (int v0 = row_lo; colok && v0 < row_hi; v0 += 4) {
            if constexpr (BF) {
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int v = v0 + q;
                    if (v < row_hi) p.X0[(size_t)v * B + col] = ((uint32_t)v == s0) ? 0u : INF;
                }
            } else {
                float t[4], dg[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int v = v0 + q;
                    t[q] = v < row_hi ? p.V[(size_t)v * B + col] : 0.0f;
                    dg[q] = v < row_hi ? p.degf[v] : 0.0f;
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int v = v0 + q;
                    if (v >= row_hi) continue;
                    p.X0[(size_t)v * B + col] = __float_as_uint(dg[q] > 0.0f ? t[q] / dg[q] : t[q]);
                    if (dg[q] > 0.0f) gpart += t[q];
                    tpart += t[q];
                }
            }
        }
        if (!BF && colok) {
            if (tpart != 0.0f) atomicAdd(&p.T[col], (double)tpart);
            if (gpart != 0.0f) {
                atomicAdd(&p.acc_g[2 * B + col], (double)gpart);
                if (LIVE) atomicAdd(&p.gl[col], (double)gpart);
            }
        }
    }
    if (!grid_barrier(p.sb, p.nblocks, bar, p.timeout_ns)) return;
    double Tc = 0.0, gprev = 0.0;
    if (!BF && colok) {
        Tc = ld_relaxed_f64(&p.T[col]);
        gprev = ld_relaxed_f64(&p.acc_g[2 * B + col]);
    }
    bool active = colok;
    int last_it = 0;  // sweeps this column ran (same value in every CTA)
    int it = 0;
    for (; it < p.max_iters; ++it) {
        const int slot = it % 3;
        const uint32_t* xin = SYNC ? ((it & 1) ? p.X1 : p.X0) : p.X0;
        uint32_t* xout = SYNC ? ((it & 1) ? p.X0 : p.X1) : p.X0;
        float res = 0.0f, gsum = 0.0f, dg_acc = 0.0f;  // per-lane partials; FP64 in the atomics
        uint32_t carry = b_ident<BF>();
        int buf_first = row_lo, buf_cnt = 0;
        const bool warp_active = __any_sync(0xffffffffu, active);
        float gt = 0.0f;
        if (SYNC && !BF) gt = (float)((double)p.g_coef * (Tc - gprev));

        for (int t = tile_lo; t < tile_hi; ++t) {
            const int a0 = p.tile_row[t], b0 = p.tile_nz[t];
            const int NA = p.tile_row[t + 1] - a0, NB = p.tile_nz[t + 1] - b0;
            __syncthreads();  // previous tile's staging no longer read
            for (int i = threadIdx.x; i < NA; i += blockDim.x) s_end[i] = ld_stream_i32(p.rowptr + a0 + i + 1) - b0;
            if (threadIdx.x == 0) s_end[NA] = INT_MAX;
            for (int j = threadIdx.x; j < NB; j += blockDim.x) {
                s_col[j] = ld_stream_i32(p.colidx + b0 + j);
                if constexpr (BF && W8) s_w[j] = (uint32_t)p.w8[b0 + j];
                else if constexpr (BF) s_w[j] = ld_stream_u32(p.w + b0 + j);
            }
            __syncthreads();
            if (!warp_active) continue;
            if constexpr (LIVE) {
                if (active) gt = (float)((double)p.g_coef * (Tc - ld_relaxed_f64(&p.gl[col])));
            }
            uint32_t acc = carry;
            int i = 0;
            int re = s_end[0];
            // the inputs of the row being accumulated (old value, teleport entry, out-degree), loaded when
            // the row starts so that they arrive while its edges are gathered; only this lane writes the
            // row's value in this column, so a value loaded early is still the current one
            uint32_t pre_old = 0u;
            float pre_v = 0.0f, pre_dg = 0.0f;
            auto preload = [&](int r) {
                if (r >= NA || !active) return;
                const int v = a0 + r;
                const size_t k = (size_t)v * B + col;
                pre_old = SYNC ? ld_weak_b32(xin + k) : ld_relaxed_b32(xin + k);
                if constexpr (!BF) {
                    pre_v = ld_stream_f32(p.V + k);
                    pre_dg = p.degf[v];
                }
            };
            preload(0);
            auto finish_row = [&](int r, uint32_t sum) {
                const int v = a0 + r;
                if (!active) return;
                const size_t k = (size_t)v * B + col;
                uint32_t xnew;
                if constexpr (BF) {
                    const uint32_t old = pre_old;
                    xnew = sum < old ? sum : old;
                    if (xnew < old) res += 1.0f;
                } else {
                    const float xo = __uint_as_float(pre_old);
                    const float dg = pre_dg;
                    const float rold = dg > 0.0f ? xo * dg : xo;
                    const float rnew = (1.0f - p.d) * pre_v + p.d * __uint_as_float(sum) + gt;
                    res += fabsf(rnew - rold);
                    if (dg > 0.0f) {
                        gsum += rnew;
                        dg_acc += rnew - rold;
                    }
                    xnew = __float_as_uint(dg > 0.0f ? __fdividef(rnew, dg) : rnew);  // 2 ulp, no special-value path
                }
                if constexpr (SYNC) st_weak_b32(xout + k, xnew);
                else if constexpr (DELAYED) mybuf[(v - buf_first) * 32 + lane] = xnew;
                else st_relaxed_b32(xout + k, xnew);
            };
            auto maybe_flush = [&](bool force) {
                if constexpr (DELAYED) {
                    if (buf_cnt > 0 && (buf_cnt >= p.delta || force)) {
                        __syncwarp();
                        if (active)
                            for (int q = 0; q < buf_cnt; ++q)
                                st_relaxed_b32(p.X0 + (size_t)(buf_first + q) * B + col, mybuf[q * 32 + lane]);
                        if (LIVE && active && dg_acc != 0.0f) {
                            atomicAdd(&p.gl[col], (double)dg_acc);
                            dg_acc = 0.0f;
                        }
                        buf_first += buf_cnt;
                        buf_cnt = 0;
                        __syncwarp();
                        if (LIVE && active) gt = (float)((double)p.g_coef * (Tc - ld_relaxed_f64(&p.gl[col])));
                    }
                }
            };
            for (int j0 = 0; j0 < NB; j0 += BU) {
                uint32_t xv[BU];
#pragma unroll
                for (int u = 0; u < BU; ++u) {
                    const int j = j0 + u;
                    xv[u] = 0u;
                    if (j < NB && active) {
                        const size_t k = (size_t)s_col[j] * B + col;
                        xv[u] = SYNC ? ld_weak_b32(xin + k) : ld_relaxed_b32(xin + k);
                    }
                }
#pragma unroll
                for (int u = 0; u < BU; ++u) {
                    const int j = j0 + u;
                    if (j < NB) {
                        while (re <= j) {
                            finish_row(i, acc);
                            if constexpr (DELAYED) { ++buf_cnt; maybe_flush(false); }
                            acc = b_ident<BF>();
                            ++i;
                            re = s_end[i];
                            preload(i);
                        }
                        uint32_t term;
                        if constexpr (BF) term = b_relax(xv[u], s_w[j]);
                        else term = xv[u];
                        acc = b_comb<BF>(acc, term);
                    }
                }
            }
            while (i < NA) {
                finish_row(i, acc);
                if constexpr (DELAYED) { ++buf_cnt; maybe_flush(false); }
                acc = b_ident<BF>();
                ++i;
                preload(i);
            }
            carry = acc;
            if constexpr (DELAYED) maybe_flush(t == tile_hi - 1);
            if constexpr (VAR == DAG_ASYNC && !BF) {
                if (active && dg_acc != 0.0f) {
                    atomicAdd(&p.gl[col], (double)dg_acc);
                    dg_acc = 0.0f;
                }
            }
        }
        // ---- end of sweep ----
        if (active) {
            if (res != 0.0f) atomicAdd(&p.acc_res[slot * B + col], (double)res);
            if (SYNC && !BF && gsum != 0.0f) atomicAdd(&p.acc_g[slot * B + col], (double)gsum);
        }
        if (!grid_barrier(p.sb, p.nblocks, bar, p.timeout_ns)) return;
        int still = 0;
        if (active) {
            const double r = ld_relaxed_f64(&p.acc_res[slot * B + col]);
            if (SYNC && !BF) gprev = ld_relaxed_f64(&p.acc_g[slot * B + col]);
            if (r <= p.tol) {
                active = false;
                last_it = it + 1;
                if (cb == 0) p.iters[col] = it + 1;
            } else {
                still = 1;
            }
        }
        if (cb == 0 && colok) {
            const int dead = (it + 2) % 3;
            p.acc_res[dead * B + col] = 0.0;
            p.acc_g[dead * B + col] = 0.0;
        }
        if (!__syncthreads_or(still)) { ++it; break; }
    }
    if (cb == 0 && active) p.iters[col] = it;  // not converged: ran them all
    if (active) last_it = it;
    {
        // every CTA holds all B columns and reads the same sums, so CTA 0 sees the outcome
        const int any_active = __syncthreads_or(active ? 1 : 0);
        if (cb == 0 && threadIdx.x == 0) {
            p.sb->iters = it;
            p.sb->converged = any_active ? 0 : 1;
        }
    }

    // ---------------- output: r = x * outdeg, from the buffer of each column's last sweep ----------------
    if (!colok) return;
    const uint32_t* xf = (SYNC && (last_it & 1)) ? p.X1 : p.X0;
    for (int v0 = row_lo; v0 < row_hi; v0 += 4) {  // four rows in flight
        uint32_t x[4];
        float dg[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int v = v0 + q;
            x[q] = v < row_hi ? ld_relaxed_b32(xf + (size_t)v * B + col) : 0u;
            dg[q] = (!BF && v < row_hi) ? p.degf[v] : 0.0f;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int v = v0 + q;
            if (v >= row_hi) continue;
            if constexpr (BF) p.X0[(size_t)v * B + col] = x[q];
            else p.X0[(size_t)v * B + col] =
                __float_as_uint(dg[q] > 0.0f ? __uint_as_float(x[q]) * dg[q] : __uint_as_float(x[q]));
        }
    }
}

// is_bf: 0 PPR, 1 Bellman-Ford with four-byte weights, 2 with one-byte weights
static BKernel bkernel_for(int is_bf, int variant)
{
    static const BKernel table[3][3] = {
        {batched_kernel<false, DAG_SYNC>, batched_kernel<false, DAG_ASYNC>, batched_kernel<false, DAG_DELAYED>},
        {batched_kernel<true, DAG_SYNC>, batched_kernel<true, DAG_ASYNC>, batched_kernel<true, DAG_DELAYED>},
        {batched_kernel<true, DAG_SYNC, true>, batched_kernel<true, DAG_ASYNC, true>,
         batched_kernel<true, DAG_DELAYED, true>},
    };
    return table[is_bf][variant];
}

// ---------------------------------------------------------------------------
// CUDA graphs of batched launches (dag_plan_set_batched_graph). A launch shape
// (kernel, grid, block, shared memory, control block) is captured once into a
// graph of two nodes: the reset of the control block and the cooperative
// kernel. Every call replays it with its own kernel arguments. Capture runs on
// a private stream (the caller's may be the legacy default stream, which
// cannot be captured); when capture or instantiation fails, the shape is
// marked and its calls launch directly. The cache sits here, keyed by plan,
// and is released by dag_plan_destroy.
// ---------------------------------------------------------------------------
struct BatchGraph {
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    cudaGraphNode_t knode = nullptr;  // the kernel node, whose arguments each call sets
    bool failed = false;              // capture or instantiation failed: launch directly
};
using ShapeKey = std::tuple<const void*, int, int, size_t, size_t, const void*>;
struct PlanGraphs {
    bool on = true;  // graphs are the default for every plan
    std::map<ShapeKey, BatchGraph> shapes;
};
static std::mutex g_graph_mu;
static std::map<const dag_plan*, PlanGraphs> g_graphs;

static bool batched_graph_on(const dag_plan* plan)
{
    std::lock_guard<std::mutex> lk(g_graph_mu);
    auto it = g_graphs.find(plan);
    return it == g_graphs.end() || it->second.on;  // on unless the plan turned it off
}

// Records the reset and the kernel launch into bg (nothing runs); on any
// failure bg.failed is set and the error state cleared.
static void capture_shape(BatchGraph& bg, const void* k, int nb, int threads, size_t dyn, void* bsync,
                          size_t cbytes, void** args)
{
    cudaStream_t cs = nullptr;
    if (cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking) != cudaSuccess) {
        cudaGetLastError();
        bg.failed = true;
        return;
    }
    cudaGraph_t g = nullptr;
    cudaGraphExec_t ex = nullptr;
    cudaGraphNode_t kn = nullptr;
    const cudaError_t e0 = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
    if (e0 != cudaSuccess) set_error(DAG_OK, std::string("batched graph: begin capture: ") + cudaGetErrorString(e0));
    if (e0 == cudaSuccess) {
        const cudaError_t e1 = cudaMemsetAsync(bsync, 0, cbytes, cs);
        const cudaError_t e2 = cudaLaunchCooperativeKernel(k, dim3(nb), dim3(threads), args, dyn, cs);
        const cudaError_t e3 = cudaStreamEndCapture(cs, &g);  // ends capture mode whatever happened
        cudaError_t e4 = cudaErrorUnknown;
        if (e1 == cudaSuccess && e2 == cudaSuccess && e3 == cudaSuccess && g) e4 = cudaGraphInstantiate(&ex, g, 0);
        const cudaError_t bad = e1 != cudaSuccess ? e1 : e2 != cudaSuccess ? e2 : e3 != cudaSuccess ? e3 : e4;
        if (bad != cudaSuccess)  // recorded for dag_last_error_message; the call itself launches directly
            set_error(DAG_OK, std::string("batched graph: capture (memset, launch, end, instantiate ") +
                                  std::to_string((int)e1) + " " + std::to_string((int)e2) + " " +
                                  std::to_string((int)e3) + " " + std::to_string((int)e4) + "): " +
                                  cudaGetErrorString(bad));
        if (e4 == cudaSuccess) {
            size_t cnt = 0;
            if (cudaGraphGetNodes(g, nullptr, &cnt) == cudaSuccess && cnt > 0) {
                std::vector<cudaGraphNode_t> nodes(cnt);
                if (cudaGraphGetNodes(g, nodes.data(), &cnt) == cudaSuccess) {
                    for (size_t i = 0; i < cnt; ++i) {
                        cudaGraphNodeType t;
                        if (cudaGraphNodeGetType(nodes[i], &t) == cudaSuccess && t == cudaGraphNodeTypeKernel)
                            kn = nodes[i];
                    }
                }
            }
        }
    }
    cudaStreamDestroy(cs);
    if (!kn && ex) {
        size_t cnt = 0;
        cudaGraphGetNodes(g, nullptr, &cnt);
        std::string types;
        std::vector<cudaGraphNode_t> nodes(cnt);
        if (cnt) cudaGraphGetNodes(g, nodes.data(), &cnt);
        for (size_t i = 0; i < cnt; ++i) {
            cudaGraphNodeType t;
            cudaGraphNodeGetType(nodes[i], &t);
            types += " " + std::to_string((int)t);
        }
        set_error(DAG_OK, "batched graph: no kernel node among " + std::to_string(cnt) + " nodes:" + types);
    }
    if (!kn) {
        if (ex) cudaGraphExecDestroy(ex);
        if (g) cudaGraphDestroy(g);
        cudaGetLastError();
        bg.failed = true;
        return;
    }
    bg.graph = g;
    bg.exec = ex;
    bg.knode = kn;
}

// One batched launch on stream s through the plan's graph of this shape
// (captured on first use), or directly when the shape cannot be captured.
static cudaError_t graph_launch(dag_plan* plan, const void* k, int nb, int threads, size_t dyn, size_t cbytes,
                                void** args, cudaStream_t s, bool* replayed)
{
    *replayed = false;
    std::lock_guard<std::mutex> lk(g_graph_mu);
    BatchGraph& bg = g_graphs[plan].shapes[ShapeKey(k, nb, threads, dyn, cbytes, plan->bsync)];
    if (!bg.exec && !bg.failed) capture_shape(bg, k, nb, threads, dyn, plan->bsync, cbytes, args);
    if (!bg.failed) {
        cudaKernelNodeParams kp{};
        kp.func = const_cast<void*>(k);
        kp.gridDim = dim3(nb);
        kp.blockDim = dim3(threads);
        kp.sharedMemBytes = (unsigned)dyn;
        kp.kernelParams = args;
        kp.extra = nullptr;
        // the replay must run with this call's arguments: if they cannot be set, or the graph
        // cannot be launched, nothing was enqueued, and the shape launches directly from now on
        const cudaError_t ep = cudaGraphExecKernelNodeSetParams(bg.exec, bg.knode, &kp);
        const cudaError_t el = ep == cudaSuccess ? cudaGraphLaunch(bg.exec, s) : ep;
        if (el == cudaSuccess) {
            *replayed = true;
            return cudaSuccess;
        }
        set_error(DAG_OK, std::string("batched graph: replay: ") + cudaGetErrorString(el));
        cudaGetLastError();
        bg.failed = true;
    }
    const cudaError_t e = cudaMemsetAsync(plan->bsync, 0, cbytes, s);
    if (e != cudaSuccess) return e;
    return cudaLaunchCooperativeKernel(k, dim3(nb), dim3(threads), args, dyn, s);
}

void release_batched_graphs(const dag_plan* plan)
{
    std::lock_guard<std::mutex> lk(g_graph_mu);
    auto it = g_graphs.find(plan);
    if (it == g_graphs.end()) return;
    for (auto& kv : it->second.shapes) {
        if (kv.second.exec) cudaGraphExecDestroy(kv.second.exec);
        if (kv.second.graph) cudaGraphDestroy(kv.second.graph);
    }
    g_graphs.erase(it);
}

// Items (rows + in-edges) per warp of a small graph, and the weight of a run of a large one. Short runs keep the
// sweep in vertex order (fewer sweeps) and even out the warps; a run's fixed cost (its partials, the pipeline's
// start) is worth more columns' work the fewer columns there are. Measured for 128, 256, 512, 1024, 4096: PPR of 256
// columns (RMAT, 1 M vertices) 27.4, 27.1, 28-30, 29.7, 34.6 ms; of 64 columns (uniform, 262 K) 6.0, 4.9, 4.3, 4.1,
// 3.9 ms; of 20 columns (RMAT, 100 K) 2.0, 1.4, 1.3, 1.3, 1.3 ms; Bellman-Ford of 64 columns (RMAT, 1 M) 7.1, 6.9,
// 7.1, 7.1, 7.1 ms.
constexpr int RUN_MIN_ITEMS = 16;
constexpr int RUN_ITEMS = 1024;
constexpr int RUN_ITEMS_WIDE = 256;

static int launch_on(bool runs, dag_plan* plan, int is_bf, int variant, int delta, int max_iters, int B, float d,
                     double tol, const void* V_or_src, const uint32_t* w, void* out, int* iters, dag_batch_stats* st,
                     cudaStream_t s)
{
    const int n = plan->n;
    const int W = (B + 31) / 32;
    const int threads = W * 32;
    if (is_bf) {
        // sources must be vertices of the graph
        std::vector<uint32_t> hs(B);
        DAG_CUDA(cudaMemcpyAsync(hs.data(), V_or_src, (size_t)B * 4, cudaMemcpyDeviceToHost, s));
        DAG_CUDA(cudaStreamSynchronize(s));
        for (int c = 0; c < B; ++c)
            if (hs[c] >= (uint32_t)n) return set_error(DAG_ERR_INVALID, "source outside [0, n)");
    }
    const int dl = (variant == DAG_DELAYED) ? delta : 0;
    size_t dyn = (size_t)(2 * TILE + 1 + (is_bf ? TILE : 0)) * 4 + (size_t)W * dl * 32 * 4;
    BKernel k = bkernel_for(is_bf, variant);
    int threads_launch = threads;
    if (runs) {
        k = run_kernel_for(is_bf != 0, B);
        threads_launch = NT;
        dyn = run_smem_bytes(is_bf != 0, B);
    }
    int per_sm = 0;
    const auto fit_key = std::make_tuple((const void*)k, threads_launch, dyn);
    const auto fit = plan->batched_fit.find(fit_key);
    if (fit != plan->batched_fit.end()) {
        per_sm = fit->second.first;
        Shape how;
        how.kernels[0] = (const void*)k;
        how.dyn = (int)dyn;
        how.carveout = fit->second.second;
        const int rc = apply_shape(how);
        if (rc) return rc;
    } else {
        int max_dyn = 0;
        DAG_CUDA(cudaDeviceGetAttribute(&max_dyn, cudaDevAttrMaxSharedMemoryPerBlockOptin, plan->device));
        if (dyn > (size_t)max_dyn)
            return set_error(DAG_ERR_INVALID, "delta too large for the batched delay buffers in shared memory");
        DAG_CUDA(cudaFuncSetAttribute((const void*)k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn));
        DAG_CUDA(cudaFuncSetAttribute((const void*)k, cudaFuncAttributePreferredSharedMemoryCarveout, 100));
        DAG_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, (const void*)k, threads_launch, dyn));
        if (per_sm < 1) return set_error(DAG_ERR_INVALID, "batched kernel cannot be resident");
        cudaFuncAttributes fa;
        DAG_CUDA(cudaFuncGetAttributes(&fa, (const void*)k));
        int pct = 0;
        const int rc =
            set_l1_carveout((const void*)k, plan->device, threads_launch, fa.sharedSizeBytes, dyn, per_sm, &pct);
        if (rc) return rc;
        plan->batched_fit[fit_key] = {per_sm, pct};
    }
    int nb = per_sm * plan->num_sms;
    if (plan->worker_cap > 0 && nb > plan->worker_cap) nb = plan->worker_cap;
    Partition* part = nullptr;
    int rc = DAG_OK, nruns = 0;
    if (runs) {
        // a warp's run holds at least RUN_MIN_ITEMS items, so a small graph's grid barrier stays small
        const long long warps = ((long long)n + plan->m + RUN_MIN_ITEMS - 1) / RUN_MIN_ITEMS;
        nb = (int)std::min((long long)nb, (warps + RUN_WARPS - 1) / RUN_WARPS);
        const int row_w = run_row_weight(is_bf != 0, B);
        const long long work = (long long)row_w * n + plan->m, W = nb * RUN_WARPS;
        // about `items` of weight per run, as many runs for every warp
        const int items = B > 128 ? RUN_ITEMS_WIDE : RUN_ITEMS;
        nruns = (int)(W * std::max(1LL, (work + items * W / 2) / (items * W)));
        rc = get_batch_runs(plan, nruns, row_w, &part, s);
    } else {
        rc = get_partition(plan, nb, &part, s, 0);
    }
    if (rc) return rc;
    // workspace: the second iterate (sync), a padded first one when the caller's rows are not whole aligned 16-byte
    // chunks (runs), and the per-column control block
    const int stride = runs ? (B + 3) & ~3 : B;
    const bool padded = runs && (stride != B || ((uintptr_t)out & 15u) != 0);
    const size_t xrows = (size_t)n * stride * 4;
    const size_t xbytes = xrows * ((variant == DAG_SYNC ? 1 : 0) + (padded ? 1 : 0));
    if (xbytes > plan->bx_bytes) {
        cudaFree(plan->bx);
        plan->bx = nullptr;
        plan->bx_bytes = 0;
        if (cudaMalloc(&plan->bx, xbytes) != cudaSuccess) {
            cudaGetLastError();
            return set_error(DAG_ERR_NOMEM, "batched workspace allocation failed");
        }
        plan->bx_bytes = xbytes;
    }
    const size_t cbytes = sizeof(SyncBlock) + (size_t)B * (3 + 3 + 1 + 1) * sizeof(double) +
                          (size_t)nruns * sizeof(unsigned long long);
    if (cbytes > plan->bsync_bytes) {
        cudaFree(plan->bsync);
        plan->bsync = nullptr;
        plan->bsync_bytes = 0;
        if (cudaMalloc(&plan->bsync, cbytes) != cudaSuccess) {
            cudaGetLastError();
            return set_error(DAG_ERR_NOMEM, "batched control allocation failed");
        }
        plan->bsync_bytes = cbytes;
    }
    // the runs' published partials, and (Bellman-Ford) each vertex's last change
    const size_t part_bytes = ((size_t)nruns + (size_t)nb * RUN_WARPS) * stride * 4;
    const size_t rbytes = runs ? part_bytes + (is_bf ? (size_t)n : 0) : 0;
    if (rbytes > plan->bruns_bytes) {
        if (plan->bruns) DAG_CUDA(cudaDeviceSynchronize());  // a solve in flight may still use the smaller one
        dev_free(plan->bruns);
        plan->bruns = nullptr;
        plan->bruns_bytes = 0;
        if (rbytes > plan->bruns_limit || dev_alloc(&plan->bruns, rbytes) != cudaSuccess) {
            cudaGetLastError();
            return set_error(DAG_ERR_NOMEM, "batched workspace allocation failed");
        }
        plan->bruns_bytes = rbytes;
    }
    const bool use_graph = batched_graph_on(plan);
    if (!use_graph) DAG_CUDA(cudaMemsetAsync(plan->bsync, 0, cbytes, s));  // the graph holds its own reset
    BatchParams p{};
    p.n = n;
    p.B = B;
    p.nblocks = nb;
    p.rowptr = plan->rowptr;
    p.colidx = plan->colidx;
    p.w = is_bf == 1 ? w : nullptr;
    p.w8 = is_bf == 2 ? (const uint8_t*)w : nullptr;
    p.degf = plan->degf;
    p.V = is_bf ? nullptr : (const float*)V_or_src;
    p.src = is_bf ? (const uint32_t*)V_or_src : nullptr;
    p.d = d;
    p.g_coef = d / (float)n;
    p.tol = is_bf ? 0.0 : tol;
    p.max_iters = max_iters;
    p.delta = dl;
    p.X0 = padded ? (uint32_t*)((char*)plan->bx + (variant == DAG_SYNC ? xrows : 0)) : (uint32_t*)out;
    p.X1 = (uint32_t*)plan->bx;
    p.cta_row = part->cta_row;
    p.cta_tile = part->cta_tile;
    p.tile_row = part->tile_row;
    p.tile_nz = part->tile_nz;
    p.sb = (SyncBlock*)plan->bsync;
    double* base = (double*)((char*)plan->bsync + sizeof(SyncBlock));
    p.acc_res = base;
    p.acc_g = base + 3 * B;
    p.gl = base + 6 * B;
    p.T = base + 7 * B;
    p.iters = iters;
    p.timeout_ns = plan->timeout_ns;
    if (runs) {
        p.nruns = nruns;
        p.sync = variant == DAG_SYNC ? 1 : 0;
        p.stride = stride;
        p.v16 = !is_bf && B % 4 == 0 && ((uintptr_t)V_or_src & 15u) == 0 ? 1 : 0;
        p.out = (uint32_t*)out;
        p.run_row = part->cta_row;
        p.run_nz = part->cta_tile;
        p.pub = (unsigned long long*)(base + 8 * B);
        p.part = (uint32_t*)plan->bruns;
        p.chg = (uint8_t*)plan->bruns + part_bytes;
    }
    if (st) {
        for (cudaEvent_t& e : plan->ev)
            if (!e) DAG_CUDA(cudaEventCreate(&e));
        cudaEventRecord(plan->ev[0], s);
    }
    void* args[] = {(void*)&p};
    bool replayed = false;
    cudaError_t le = use_graph ? graph_launch(plan, (const void*)k, nb, threads_launch, dyn, cbytes, args, s, &replayed)
                               : cudaLaunchCooperativeKernel((const void*)k, dim3(nb), dim3(threads_launch), args, dyn, s);
    if (le != cudaSuccess) return cuda_check(le, "batched cooperative launch");
    if (!st) return DAG_OK;
    cudaEventRecord(plan->ev[1], s);
    SyncBlock sb;
    DAG_CUDA(cudaMemcpyAsync(&sb, plan->bsync, SYNC_HEAD, cudaMemcpyDeviceToHost, s));
    std::vector<int> hit(B);
    DAG_CUDA(cudaMemcpyAsync(hit.data(), iters, (size_t)B * sizeof(int), cudaMemcpyDeviceToHost, s));
    DAG_CUDA(cudaStreamSynchronize(s));
    float ms = 0.0f;
    cudaEventElapsedTime(&ms, plan->ev[0], plan->ev[1]);
    int rc2 = DAG_OK;
    if (sb.err) rc2 = sb.err;
    else if (!sb.converged) rc2 = DAG_ERR_NOT_CONVERGED;
    long long colsw = 0;
    for (int c = 0; c < B; ++c) colsw += hit[c];
    st->sweeps = sb.iters;
    st->err = rc2;
    st->ms = ms;
    st->workers = nb;
    st->delta = dl;
    st->column_sweeps = colsw;
    st->graph = replayed ? 1 : 0;
    if (rc2 == DAG_ERR_BARRIER_TIMEOUT) set_error(rc2, "grid barrier wait ran out of time");
    return rc2;
}

// Runs of the merge path but for the delayed form; where their scratch (partials, a padded copy of rows that are not
// whole 16-byte chunks) does not fit on the device, the 32-column kernel, whose in-place forms take none: what the
// attempt allocated is given back first.
int launch_batched(dag_plan* plan, int is_bf, int variant, int delta, int max_iters, int B, float d, double tol,
                   const void* V_or_src, const uint32_t* w, void* out, int* iters, dag_batch_stats* st,
                   cudaStream_t s)
{
    const bool runs = plan->batched_wide && variant != DAG_DELAYED;
    const int rc = launch_on(runs, plan, is_bf, variant, delta, max_iters, B, d, tol, V_or_src, w, out, iters, st, s);
    if (!runs || rc != DAG_ERR_NOMEM) return rc;
    cudaGetLastError();  // the allocation's
    DAG_CUDA(cudaFree(plan->bx));  // (waits for the device; the kernel's second iterate is allocated afresh)
    plan->bx = nullptr;
    plan->bx_bytes = 0;
    return launch_on(false, plan, is_bf, variant, delta, max_iters, B, d, tol, V_or_src, w, out, iters, st, s);
}

}  // namespace dag

extern "C" int dag_debug_limit_batched_scratch(dag_plan* plan, int64_t bytes)
{
    if (!plan || bytes < 0) return dag::set_error(DAG_ERR_INVALID, "bad argument");
    if ((unsigned long long)bytes < plan->bruns_bytes) {
        DAG_CUDA(cudaDeviceSynchronize());  // a solve in flight may still use it
        dag::dev_free(plan->bruns);
        plan->bruns = nullptr;
        plan->bruns_bytes = 0;
    }
    plan->bruns_limit = (size_t)bytes;
    return DAG_OK;
}

extern "C" int dag_plan_set_batched_wide(dag_plan* plan, int32_t on)
{
    if (!plan) return dag::set_error(DAG_ERR_INVALID, "null plan");
    plan->batched_wide = on != 0;
    return DAG_OK;
}

extern "C" int dag_plan_set_batched_graph(dag_plan* plan, int32_t on)
{
    if (!plan) return dag::set_error(DAG_ERR_INVALID, "null plan");
    std::lock_guard<std::mutex> lk(dag::g_graph_mu);
    dag::g_graphs[plan].on = on != 0;
    return DAG_OK;
}
