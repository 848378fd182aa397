// Gradients of a loss through weighted PageRank, after the adjoint solve
// (no counterpart in the paper). With M_vu = w_uv / s_u, r the forward fixed
// point and lambda the adjoint (lambda = c + d M^T lambda + d g sum(lambda)/n):
//   dL/dw_uv = d r_u (lambda_v - (M^T lambda)_u) / s_u,   dL/dt_v = (1 - d) lambda_v.
// A pass over the vertices packs each source's two factors, d r_u / s_u and
// (M^T lambda)_u, into one 8-byte pair; then one pass over the in-edges in the
// caller's (in-CSR) order, one gather per edge: each CTA walks its vertex
// block tile by tile. An edge's row is the last one starting at or before it:
// rows leave their number at their first edge, and a running maximum over the
// warp's edges spreads it (a binary search over the tile's row ends per edge
// took 250 us for 33.5 M edges, this takes 216; one gather per SM clock would be
// 110).
#include <climits>

#include "dag_internal.cuh"
#include "devmem.cuh"

namespace dag {

__global__ void k_grad_coef(const float* s_norm, const float* rank, const float* mt, float d, int n, float2* coef)
{
    const int u = blockIdx.x * blockDim.x + threadIdx.x;
    if (u < n) coef[u] = make_float2(d * rank[u] / s_norm[u], mt[u]);  // s_u = 0: u is no edge's source
}

__global__ void __launch_bounds__(NT) k_edge_grad(const int* rowptr, const int* colidx, const int* cta_tile,
                                                  const int* tile_row, const int* tile_nz, const float2* coef,
                                                  const float* lambda, float* grad_w)
{
    __shared__ int s_row[TILE];       // 1 + the row (from a0) whose first edge in the tile this is, else 0
    __shared__ int s_last[NWARP];     // the last row started in each warp's part of the tile
    constexpr int PART = TILE / NWARP;  // edges per warp, IPT per lane, 32 at a time
    const int c = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int t = cta_tile[c]; t < cta_tile[c + 1]; ++t) {
        const int a0 = tile_row[t], b0 = tile_nz[t];
        const int NA = tile_row[t + 1] - a0, NB = tile_nz[t + 1] - b0;
        int col[IPT];
#pragma unroll
        for (int q = 0; q < IPT; ++q) {
            const int j = warp * PART + 32 * q + lane;
            col[q] = j < NB ? colidx[b0 + j] : -1;
        }
        __syncthreads();  // the previous tile's rows are read
        for (int j = tid; j < NB; j += NT) s_row[j] = 0;
        __syncthreads();
        // row i starts where row i - 1 ends (the first at the tile's first edge); row NA goes on past the tile
        for (int i = tid; i <= NA; i += NT) {
            const int b = i > 0 ? rowptr[a0 + i] - b0 : 0, e = i < NA ? rowptr[a0 + i + 1] - b0 : NB;
            if (b < e) s_row[b] = i + 1;
        }
        __syncthreads();
        int m[IPT], run = 0;
#pragma unroll
        for (int q = 0; q < IPT; ++q) {
            const int j = warp * PART + 32 * q + lane;
            int v = j < NB ? s_row[j] : 0;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) v = max(v, __shfl_up_sync(0xffffffffu, v, o));  // (below lane o: its own)
            m[q] = max(v, run);
            run = __shfl_sync(0xffffffffu, m[q], 31);
        }
        if (lane == 0) s_last[warp] = run;
        __syncthreads();
        int before = 0;
        for (int k = 0; k < warp; ++k) before = max(before, s_last[k]);
#pragma unroll
        for (int q = 0; q < IPT; ++q) {
            const int j = warp * PART + 32 * q + lane;
            if (col[q] < 0) continue;
            const float2 cf = coef[col[q]];
            grad_w[b0 + j] = cf.x * (lambda[a0 + max(m[q], before) - 1] - cf.y);
        }
    }
}

__global__ void k_teleport_grad(const float* lambda, float one_minus_d, float* grad_t, int n)
{
    int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v < n) grad_t[v] = one_minus_d * lambda[v];
}

int launch_edge_grad(dag_plan* plan, float d, const float* val, const float* s_norm, const float* rank,
                     const float* lambda, const float* mt, float* grad_w, float* grad_t, cudaStream_t st)
{
    (void)val;
    const int P = plan->num_sms * 4;
    Partition* part = nullptr;
    int rc = get_partition(plan, P, &part, st, 0);
    if (rc) return rc;
    if (grad_w && plan->m > 0) {
        if (!plan->grad_coef) DAG_CUDA(dev_alloc(&plan->grad_coef, (size_t)plan->n * sizeof(float2)));
        k_grad_coef<<<(plan->n + 255) / 256, 256, 0, st>>>(s_norm, rank, mt, d, plan->n, (float2*)plan->grad_coef);
        k_edge_grad<<<P, NT, 0, st>>>(plan->rowptr, plan->colidx, part->cta_tile, part->tile_row, part->tile_nz,
                                      (const float2*)plan->grad_coef, lambda, grad_w);
    }
    if (grad_t) k_teleport_grad<<<(plan->n + 255) / 256, 256, 0, st>>>(lambda, 1.0f - d, grad_t, plan->n);
    DAG_CUDA(cudaGetLastError());
    return DAG_OK;
}

}  // namespace dag
