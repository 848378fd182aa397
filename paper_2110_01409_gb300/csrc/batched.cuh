// Parameters and kernel tables of the batched solves, shared by the kernels over runs of the merge path
// (batched_runs.cu: synchronous and asynchronous forms) and by the 32-column kernel and the launch logic
// (batched.cu).
#pragma once

#include "dag_internal.cuh"

namespace dag {

struct BatchParams {
    int n;
    int B;
    int nblocks;
    const int* rowptr;
    const int* colidx;
    const uint32_t* w;
    const uint8_t* w8;     // one-byte weights, else nullptr
    const float* degf;
    const float* V;        // PPR teleports [n][B]
    const uint32_t* src;   // BF sources [B]
    float d;
    float g_coef;
    double tol;
    int max_iters;
    int delta;             // rows per warp buffer (delayed)
    uint32_t* X0;          // [n][B] (the caller's output array; runs: or a padded copy, rows of `stride` values)
    uint32_t* X1;          // [n][B] workspace (sync)
    const int* cta_row;
    const int* cta_tile;
    const int* tile_row;
    const int* tile_nz;
    SyncBlock* sb;
    double* acc_res;       // [3][B]
    double* acc_g;         // [3][B]
    double* gl;            // [B] live non-dangling mass (async / delayed PPR)
    double* T;             // [B] teleport totals
    int* iters;            // [B] sweeps of each column (output)
    long long timeout_ns;
    // runs of the merge path (batched_runs.cu)
    int nruns;             // warp w of W takes runs w, w + W, ...
    int sync;              // 1: synchronous form
    int stride;            // values per row of X0 / X1: B rounded up to a multiple of 4
    int v16;               // V's rows are 16-byte aligned and whole
    uint32_t* out;         // [n][B] the caller's output array
    const int* run_row;    // [nruns + 1] first row of each run (the row it starts in)
    const int* run_nz;     // [nruns + 1] first in-edge of each run
    unsigned long long* pub;  // [nruns] sweep stamp and flags of the partial each run published (zero at launch)
    uint32_t* part;        // [nruns + W][stride] the partial of the row each run leaves unfinished; each warp's
                           // pending run's partial of its first row
    uint8_t* chg;          // [n] BF: low byte of the last sweep that lowered a value of the vertex
};

using BKernel = void (*)(const BatchParams);

constexpr int RUN_WARPS = NT / 32;  // warps (runs) per CTA

// The run kernel for B columns (1 to 1024) of PPR (is_bf 0) or Bellman-Ford, and its dynamic shared memory per CTA.
BKernel run_kernel_for(bool is_bf, int B);
size_t run_smem_bytes(bool is_bf, int B);
// A row's weight in the runs beside its in-edges.
int run_row_weight(bool is_bf, int B);

}  // namespace dag
