// Batched personalized PageRank and batched Bellman-Ford, synchronous and asynchronous forms, one warp per run
// of the merge path (no counterpart in the paper: each column is an independent problem solved with its sweep,
// Sec. III; columns stop on their own).
//
// State X is row-major, a vertex's B values contiguous (rows padded to a multiple of four values), so an in-edge
// reads one contiguous row. The merge path of the whole graph (rows and in-edges in vertex order) is cut into runs of
// equal weight and the warps take the runs in turn: Sec. III-A's balance by in-degree, at warp granularity, so a hub
// row's in-edges are spread over as many warps as its length asks for, and a sweep moves through the vertex order as
// one stream. A row whose in-edges span runs is finished by the run that ends it, from the partials the earlier runs
// published (a bounded look-back, as in sweep_warp.cu), one run later.
//
// What bounds it: bytes in flight, then instructions. A row of B values is 4 B bytes from a random place, about a
// microsecond away. So a run is a stream of fetches in the order they are needed: the source rows of its in-edges,
// and at each row end the row's old values (PPR: and its teleport entries). Each warp copies them with 16-byte
// cp.async into its own shared-memory ring of two batches, one in flight while the other is added up; nothing waits
// for another warp inside a run. Lanes hold four columns each; a row of fewer than 32 such chunks takes a
// power-of-two group of lanes and the warp's groups take in-edges in turn, joined by shuffles where a row ends.
// Rings of four half-size batches ran the same loads with twice the instructions per in-edge (150 against 75 at 256
// columns) and were 5 to 30% slower.
//
// Measured (RMAT, against a CTA block of whole rows walked in tiles by eight warps with a barrier per tile, and a
// warp of 32 columns for other column counts): PPR of 256 columns at 1 M vertices 66.5 -> 26.3 ms, of 20 columns at
// 100 K vertices 7.06 -> 1.05 ms (a hub's row was one warp's), Bellman-Ford of 64 columns at 1 M vertices 24.4 -> 7.5;
// small uniform graphs the least: PPR of 32 columns at 3 K vertices 163 -> 146 us.
//
// Bellman-Ford reads only what can lower something: chg[u] is the last sweep that lowered any of u's columns, and
// a sweep skips an in-edge whose source changed neither in it nor in the one before (its value is already in the
// row), and a row with nothing left to read (the conditional updates of Sec. V, at vertex granularity). Distances
// and the synchronous trajectory are those of the full sweep.
#include <cfloat>
#include <climits>
#include <cstdint>

#include "batched.cuh"

namespace dag {

namespace {

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
// 16 bytes through L2 (never L1), so an asynchronous sweep sees other warps' latest stores
__device__ __forceinline__ void cp16(uint32_t dst, const void* src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp4(uint32_t dst, const void* src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// All groups have landed, or all but the latest.
__device__ __forceinline__ void cp_wait(bool but_one)
{
    if (but_one) asm volatile("cp.async.wait_group 1;" ::: "memory");
    else asm volatile("cp.async.wait_group 0;" ::: "memory");
}

template <bool BF>
__device__ __forceinline__ uint32_t ident()
{
    return BF ? INF : 0u;
}
template <bool BF>
__device__ __forceinline__ uint32_t comb(uint32_t a, uint32_t b)
{
    if constexpr (BF) return a < b ? a : b;
    else return __float_as_uint(__uint_as_float(a) + __uint_as_float(b));
}
// Adds b to the sum hi + lo, the rounding of hi's addition kept in lo (Knuth's two-sum): FP32 parts on their way to an
// FP64 sum, without FP64 additions, which issue at two lanes per clock and SM. (An infinite sum has no rounding.)
__device__ __forceinline__ void two_add(float& hi, float& lo, float b)
{
    const float s = hi + b, t = s - hi;
    if (fabsf(s) <= FLT_MAX) lo += (hi - (s - t)) + (b - t);
    hi = s;
}
// The same with the sum of lane ^ o.
__device__ __forceinline__ void two_join(float& hi, float& lo, int o)
{
    const float b = __shfl_xor_sync(0xffffffffu, hi, o), bl = __shfl_xor_sync(0xffffffffu, lo, o);
    two_add(hi, lo, b);
    lo += bl;
}
__device__ __forceinline__ uint32_t relax_w(uint32_t du, uint32_t w)
{
    const uint32_t s = du + w;
    return (du == INF) ? INF : (s < du || s == INF) ? INF - 1u : s;
}
__device__ __forceinline__ uint4 ld_relaxed_v4(const uint32_t* p)
{
    uint4 v;
    asm volatile("ld.relaxed.gpu.global.v4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_relaxed_v4(uint32_t* p, const uint32_t (&v)[4])
{
    asm volatile("st.relaxed.gpu.global.v4.b32 [%0], {%1, %2, %3, %4};"
                 ::"l"(p), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]) : "memory");
}
__device__ __forceinline__ void st_relaxed_u8(uint8_t* p, unsigned v)
{
    asm volatile("st.relaxed.gpu.global.u8 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ unsigned long long ld_pub(const unsigned long long* p)
{
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_pub(unsigned long long* p, unsigned long long v)
{
    asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

constexpr unsigned PUB_EMPTY = 1u;   // the published partial is the identity: its payload is not written
constexpr int FOLD_STAGES = 2;       // PPR: stages inside one row after which its sum is folded
constexpr int LIVE_STAGES = 16;      // asynchronous PPR: a warp adds to and reads the live mass every 16 stages

// Up to 32 items of a run, in order, as the fetches they need. Vertex and weight (PPR: the row's out-degree) of item k
// are in the warp's list; `old` marks the items that read a row's old values, `fin` the row's last item (PPR: its
// teleport entries; Bellman-Ford: the old values themselves).
struct RunStage {
    unsigned old, fin;
    int cnt;
};

__device__ __forceinline__ unsigned below(int k) { return k >= 32 ? 0xffffffffu : (1u << k) - 1u; }

}  // namespace

constexpr int run_min_blocks(bool BF, int CH) { return CH >= 4 ? 1 : CH == 2 || !BF ? 2 : 3; }
// CTAs per SM the registers are sized for: PPR at two (three spilled up to 64 bytes: 64 columns, uniform, 20 K vertices
// 483 -> 346 us; RMAT, 400 K, 7.1 -> 4.3 ms), Bellman-Ford, which waits for last-change bytes, at three.
// Ring slots per warp: two batches, 4 to 8 KB of rows (16 KB above 512 columns). 8 KB for 64 columns left three CTAs
// 28 KB of L1: Bellman-Ford uniform 20 K 615 -> 490 us with half of it (RMAT 1 M 7.1 -> 7.5 ms).
constexpr int run_depth(int LPR, int CH) { return CH >= 4 ? 4 : CH == 2 ? 8 : LPR >= 16 ? 16 : 32; }

// The ring's rows are as long as the lanes that hold them, so that a row that does not fill them is added up without a
// test per chunk and with constant addresses; columns past its end hold what is there and are never stored. PPR, RMAT
// 262 K and uniform 100 K vertices: 20 columns 2.32 -> 2.08 and 1.19 -> 1.05 ms, 68 columns 5.60 -> 5.01 and 2.12 ->
// 1.92 (both with EVERY, below, half of it), 200 columns 7.80 -> 7.29 and 3.03 -> 2.85; Bellman-Ford 500 columns 14.7
// -> 11.8 and 9.2 -> 7.5. Not Bellman-Ford of 65 to 128 columns, where the longer ring takes L1 from the last-change
// bytes (100 columns, RMAT: 3.71 -> 3.93). EVERY on rows of several chunks lost: 136 columns 7.0 -> 9.6 ms, as most
// lanes of the last chunk fetch one address.
constexpr bool run_padded(bool BF, int LPR, int CH) { return !BF || LPR < 32 || CH > 1; }

// LPR lanes hold a row (four columns per lane and chunk), CH chunks per lane (more than one only with LPR = 32);
// WHOLE: the row fills them all, so its length is a constant.
template <bool BF, int LPR, int CH, bool WHOLE>
__global__ void __launch_bounds__(NT, run_min_blocks(BF, CH)) batched_runs_kernel(const BatchParams p)
{
    constexpr unsigned FULL = 0xffffffffu;
    constexpr int GRP = 32 / LPR;          // in-edges a warp adds at a time
    constexpr int RW = BF ? 1 : 2;         // items at a row end
    constexpr int D = run_depth(LPR, CH), G = D / 2;
    constexpr bool PAD = run_padded(BF, LPR, CH), EVERY = !BF && CH == 1;
    extern __shared__ __align__(16) unsigned char smem_raw[];

    const int B = p.B, S = WHOLE ? 4 * LPR * CH : p.stride, NCH = S >> 2;
    const int SR = PAD ? 4 * LPR * CH : S;  // values between fetched rows
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int grp = lane / LPR, lr = lane % LPR;
    const bool sync = p.sync != 0;
    const int W = p.nblocks * RUN_WARPS, w = blockIdx.x * RUN_WARPS + warp;

    double* s_T = (double*)smem_raw;                              // [S] teleport totals (PPR; async: times g_coef)
    double* s_live = s_T + (BF ? 0 : S);                          // [S] the CTA's change of the live mass (async PPR)
    float* s_red = (float*)(s_live + (BF ? 0 : S));               // [RUN_WARPS][S] the warps' per-column sums
    uint32_t* s_head = (uint32_t*)(s_red + RUN_WARPS * S);        // [RUN_WARPS][S] partial of the run's first row
    int* s_last = (int*)(s_head + RUN_WARPS * S);                 // [S] sweeps each column ran
    int* s_run = s_last + S;                                      // [S] 1: the column still runs
    float* s_gt = (float*)(s_run + S);                            // [S] the dangling term at the start of a sweep (PPR)
    int* s_list = (int*)(s_gt + (BF ? 0 : S));                    // [RUN_WARPS][2][2][32] items: vertex, weight
    uint32_t* s_ring = (uint32_t*)(s_list + RUN_WARPS * 128);     // [RUN_WARPS][D][SR] fetched rows
    int* list = s_list + warp * 128;
    uint32_t* ring = s_ring + (size_t)warp * D * SR;
    uint32_t* head_sum = s_head + warp * S;
    uint32_t* fold = (uint32_t*)s_red + warp * S;  // PPR, during the sweep: the folded part of the row in progress
    const uint32_t ring_at = smem_addr(ring);

    uint32_t* const head_part = p.part + ((size_t)p.nruns + w) * S;  // the first row's partial of the run left pending
    unsigned long long bar = 0;

    // the columns of this lane's chunk q: 4 (lr + 32 q) .. + 3
    auto col0 = [&](int q) { return 4 * (lr + 32 * q); };
    auto has = [&](int q) { return WHOLE || lr + 32 * q < NCH; };
    // EVERY: a lane without columns copies the row's last four too (and never stores them), which saves the branch
    auto from = [&](int q) { return !EVERY || has(q) ? col0(q) : S - 4; };

    // a column's dangling term from its mass on linked vertices (FP64 issues slowly here: once per column where it can be)
    auto dangling = [&](double linked, double T) {
        return sync ? (float)((double)p.g_coef * (T - linked)) : (float)fma(-(double)p.g_coef, linked, T);
    };

    // per-column sums of the CTA's warps (group 0's lanes hold them), added in a fixed order, one FP64 atomic each
    // (Bellman-Ford's counts in FP32: only a zero matters, and no sum rounds to it)
    auto cta_sum = [&](const float (&part)[CH][4], double* dst, double* dst2) {
        __syncthreads();
#pragma unroll
        for (int q = 0; q < CH; ++q)
            if (grp == 0 && has(q))
#pragma unroll
                for (int e = 0; e < 4; ++e) s_red[warp * S + col0(q) + e] = part[q][e];
        __syncthreads();
        for (int c = tid; c < B; c += NT) {
            float v = s_red[c], low = 0.0f;
#pragma unroll
            for (int k = 1; k < RUN_WARPS; ++k) {
                if constexpr (BF) v += s_red[k * S + c];
                else two_add(v, low, s_red[k * S + c]);
            }
            if (v != 0.0f || low != 0.0f) {
                const double sum = (double)v + (double)low;
                atomicAdd(&dst[c], sum);
                if (dst2) atomicAdd(&dst2[c], sum);
            }
        }
    };

    // ---------------- initial values, rows in turn over the whole grid's groups ----------------
    {
        float gpart[CH][4], tpart[CH][4];
        uint32_t sv[CH][4];
#pragma unroll
        for (int q = 0; q < CH; ++q)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                gpart[q][e] = tpart[q][e] = 0.0f;
                sv[q][e] = (BF && has(q) && col0(q) + e < B) ? p.src[col0(q) + e] : INF;
            }
        for (int v0 = w * GRP; v0 < p.n; v0 += W * GRP) {  // warp-uniform: every lane takes part in the vote
            const int v = v0 + grp;
            const bool in = v < p.n;
            float dg = 0.0f;
            if constexpr (!BF) dg = in ? p.degf[v] : 0.0f;
            bool is_src = false;
#pragma unroll
            for (int q = 0; q < CH; ++q) {
                if (!in || !has(q)) continue;
                uint32_t x[4];
                if constexpr (BF) {
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        x[e] = (uint32_t)v == sv[q][e] ? 0u : INF;
                        is_src |= (uint32_t)v == sv[q][e];
                    }
                } else {
                    float t[4] = {0.0f, 0.0f, 0.0f, 0.0f};
                    const float* vp = p.V + (size_t)v * B + col0(q);
                    if (p.v16) {
                        const float4 f = *(const float4*)vp;
                        t[0] = f.x; t[1] = f.y; t[2] = f.z; t[3] = f.w;
                    } else {
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            if (col0(q) + e < B) t[e] = vp[e];
                    }
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        x[e] = __float_as_uint(dg > 0.0f ? t[e] / dg : t[e]);
                        if (dg > 0.0f) gpart[q][e] += t[e];
                        tpart[q][e] += t[e];
                    }
                }
                *(uint4*)(p.X0 + (size_t)v * S + col0(q)) = make_uint4(x[0], x[1], x[2], x[3]);
                if (BF && sync) *(uint4*)(p.X1 + (size_t)v * S + col0(q)) = make_uint4(x[0], x[1], x[2], x[3]);
            }
            if constexpr (BF) {  // a source counts as changed in the sweep before the first; the value elsewhere
                                 // only costs a needless read when a solve reaches sweep 128
                unsigned any = __ballot_sync(FULL, is_src);
                if (LPR < 32) any = (any >> (grp * LPR)) & below(LPR);
                if (in && lr == 0) p.chg[v] = any ? 255 : 128;
            }
        }
        if constexpr (!BF) {
            // the groups' FP32 parts, joined in two floats per column
            float glow[CH][4], tlow[CH][4];
#pragma unroll
            for (int q = 0; q < CH; ++q)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    glow[q][e] = tlow[q][e] = 0.0f;
#pragma unroll
                    for (int o = LPR; o < 32; o <<= 1) {
                        two_join(gpart[q][e], glow[q][e], o);
                        two_join(tpart[q][e], tlow[q][e], o);
                    }
                }
            cta_sum(tpart, p.T, nullptr);
            cta_sum(gpart, p.acc_g + 2 * B, sync ? nullptr : p.gl);
            if constexpr (GRP > 1) {
                cta_sum(tlow, p.T, nullptr);
                cta_sum(glow, p.acc_g + 2 * B, sync ? nullptr : p.gl);
            }
        }
    }
    if (!grid_barrier(p.sb, p.nblocks, bar, p.timeout_ns)) return;
    for (int c = tid; c < S; c += NT) {
        if constexpr (!BF) {
            s_T[c] = c < B ? (sync ? 1.0 : (double)p.g_coef) * ld_relaxed_f64(&p.T[c]) : 0.0;
            s_live[c] = 0.0;
            s_gt[c] = c < B ? dangling(ld_relaxed_f64(&p.acc_g[2 * B + c]), s_T[c]) : 0.0f;
        }
        s_last[c] = 0;
        s_run[c] = c < B ? 1 : 0;
    }
    __syncthreads();

    // the warp's first run is the same in every sweep
    const int first_i0 = p.run_row[w], first_ie = p.run_row[w + 1], first_j0 = p.run_nz[w], first_je = p.run_nz[w + 1];
    const bool first_head = first_j0 > p.rowptr[first_i0] && first_ie > first_i0;
    int it = 0;
    for (; it < p.max_iters; ++it) {
        const int slot = it % 3;
        const unsigned stamp = (unsigned)it + 1u;
        const uint32_t* xin = sync ? ((it & 1) ? p.X1 : p.X0) : p.X0;
        uint32_t* xout = sync ? ((it & 1) ? p.X0 : p.X1) : p.X0;
        const unsigned now = (unsigned)it & 255u, before = (unsigned)(it - 1) & 255u;
        float res[CH][4], mass[CH][4], gt[CH][4];  // mass: this sweep's (sync) or the change of the live (async)
        uint32_t acc[CH][4], xo[CH][4];
        unsigned act[CH];                          // columns of the lane that still run, four bits per chunk
#pragma unroll
        for (int q = 0; q < CH; ++q) {
            act[q] = 0u;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                res[q][e] = mass[q][e] = gt[q][e] = 0.0f;
                acc[q][e] = ident<BF>();
                xo[q][e] = 0u;
                if (has(q)) {
                    act[q] |= s_run[col0(q) + e] ? 1u << e : 0u;
                    if (!BF) gt[q][e] = s_gt[col0(q) + e];
                }
            }
        }
        // asynchronous PPR: this warp's change of the live mass goes to the CTA's, the CTA's to the grid's (by each
        // warp on its own turns: the columns' few L2 lines take one atomic at a time, and an atomic per warp and
        // column held up the whole sweep), and the global term comes in
        int turn = warp;
        auto give_mass = [&]() {
#pragma unroll
            for (int q = 0; q < CH; ++q)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    if (mass[q][e] != 0.0f) atomicAdd(&s_live[col0(q) + e], (double)mass[q][e]);
                    mass[q][e] = 0.0f;
                }
        };
        auto live = [&]() {
            give_mass();
            if ((++turn & (RUN_WARPS - 1)) == 0)
                for (int c = lane; c < B; c += 32) {
                    const double v = __longlong_as_double((long long)atomicExch((unsigned long long*)&s_live[c], 0ULL));
                    if (v != 0.0) atomicAdd(&p.gl[c], v);
                }
#pragma unroll
            for (int q = 0; q < CH; ++q)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    if (!((act[q] >> e) & 1u)) continue;
                    const int c = col0(q) + e;
                    gt[q][e] = dangling(ld_relaxed_f64(&p.gl[c]), s_T[c]);
                }
        };
        // row v's new values from its sum (every group holds it) and inputs; group 0 stores them
        auto update = [&](int v, const uint32_t (&sum)[CH][4], const uint32_t (&old)[CH][4], const float (&tv)[CH][4],
                          float dg) {
            bool lowered = false;
            const float inv = BF || dg == 0.0f ? 1.0f : 1.0f / dg;  // (a dangling row's x is r itself)
            const float mul = BF || dg == 0.0f ? 1.0f : dg;
#pragma unroll
            for (int q = 0; q < CH; ++q) {
                uint32_t xn[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const bool run = grp == 0 && ((act[q] >> e) & 1u);
                    if constexpr (BF) {
                        xn[e] = sum[q][e] < old[q][e] ? sum[q][e] : old[q][e];
                        if (run && xn[e] < old[q][e]) {
                            res[q][e] += 1.0f;
                            lowered = true;
                        }
                    } else {
                        const float rold = __uint_as_float(old[q][e]) * mul;
                        const float rnew = (1.0f - p.d) * tv[q][e] + p.d * __uint_as_float(sum[q][e]) + gt[q][e];
                        if (run) {
                            res[q][e] += fabsf(rnew - rold);
                            if (dg > 0.0f) mass[q][e] += sync ? rnew : rnew - rold;
                        }
                        xn[e] = __float_as_uint(rnew * inv);  // 1.5 ulp
                    }
                }
                if (grp == 0) {
                    uint32_t* o = xout + (size_t)v * S + col0(q);
                    if (act[q] == 15u) {
                        st_relaxed_v4(o, xn);
                    } else {
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            if ((act[q] >> e) & 1u) st_relaxed_b32(o + e, xn[e]);
                    }
                }
            }
            if constexpr (BF) {
                if (__any_sync(FULL, lowered) && lane == 0) st_relaxed_u8(p.chg + v, now);
            }
        };
        auto join_groups = [&](uint32_t (&a)[CH][4]) {
#pragma unroll
            for (int o = LPR; o < 32; o <<= 1)
#pragma unroll
                for (int q = 0; q < CH; ++q)
#pragma unroll
                    for (int e = 0; e < 4; ++e) a[q][e] = comb<BF>(a[q][e], __shfl_xor_sync(FULL, a[q][e], o));
        };

        // A run begun inside a row: the row's sum so far is in head_part; the partials of runs t - 1, t - 2, ... back to
        // the first that ends a row or starts at one are added (32 at a time, one flag per lane), and the row gets its
        // values. False when a wait ran out or another CTA recorded an error.
        auto resolve = [&](int t, int row) -> bool {
            uint32_t tot[CH][4];
#pragma unroll
            for (int q = 0; q < CH; ++q)
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    tot[q][e] = (grp == 0 && has(q)) ? head_part[col0(q) + e] : ident<BF>();
            bool ok = true;
            for (int hi = t - 1; hi >= 0; hi -= 32) {
                const int k = hi - lane;
                bool stop = false, got = true, full = false;
                if (k >= 0) {
                    const int r0 = p.run_row[k];
                    stop = p.run_row[k + 1] > r0 || p.run_nz[k] <= p.rowptr[r0];
                }
                const unsigned stops = __ballot_sync(FULL, stop);
                const int n_back = stops ? __ffs(stops) : 32;  // lanes below it hold the row's runs
                if (lane < n_back && k >= 0) {
                    const unsigned long long t0 = globaltimer_ns();
                    unsigned spins = 0;
                    for (;;) {
                        const unsigned long long v = ld_pub(p.pub + k);
                        if ((unsigned)(v >> 32) == stamp) {
                            full = !((unsigned)v & PUB_EMPTY);
                            break;
                        }
                        if (ld_relaxed_i32(&p.sb->err) != 0) { got = false; break; }
                        if ((++spins & 15u) == 0 && (long long)(globaltimer_ns() - t0) > p.timeout_ns) {
                            atomicCAS(&p.sb->err, 0, DAG_ERR_BARRIER_TIMEOUT);
                            got = false;
                            break;
                        }
                        __nanosleep(64);
                    }
                }
                ok = __all_sync(FULL, got) != 0;
                if (!ok) break;
                const unsigned have = __ballot_sync(FULL, full);
                fence_gpu();  // the flags before the partials
                for (int l = grp; l < n_back; l += GRP) {
                    if (!((have >> l) & 1u)) continue;
#pragma unroll
                    for (int q = 0; q < CH; ++q) {
                        if (!has(q)) continue;
                        const uint4 x = ld_relaxed_v4(p.part + (size_t)(hi - l) * S + col0(q));
                        tot[q][0] = comb<BF>(tot[q][0], x.x); tot[q][1] = comb<BF>(tot[q][1], x.y);
                        tot[q][2] = comb<BF>(tot[q][2], x.z); tot[q][3] = comb<BF>(tot[q][3], x.w);
                    }
                }
                __syncwarp();
                if (stops) break;
            }
            join_groups(tot);
            if (ok) {
                uint32_t old[CH][4];
                float tv[CH][4];
#pragma unroll
                for (int q = 0; q < CH; ++q) {
                    uint4 x = make_uint4(0u, 0u, 0u, 0u);
                    if (has(q)) x = ld_relaxed_v4(xin + (size_t)row * S + col0(q));
                    old[q][0] = x.x; old[q][1] = x.y; old[q][2] = x.z; old[q][3] = x.w;
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        tv[q][e] = (!BF && has(q) && col0(q) + e < B) ? p.V[(size_t)row * B + col0(q) + e] : 0.0f;
                }
                update(row, tot, old, tv, BF ? 0.0f : p.degf[row]);
            }
            return ok;
        };

        int stages = 0;
        int pend = -1, pend_row = 0;  // the run whose first row waits for earlier runs' partials
        bool ok = true;
        for (int t = w; t < p.nruns && ok; t += W) {
            // ---------------- run t, as a stream of fetches ----------------
            // rows [i0, i_end) end in this run; head: it starts inside row i0 and ends it
            const int i0 = t == w ? first_i0 : p.run_row[t], i_end = t == w ? first_ie : p.run_row[t + 1];
            const int j0 = t == w ? first_j0 : p.run_nz[t], j_end = t == w ? first_je : p.run_nz[t + 1];
            const bool head = t == w ? first_head : j0 > p.rowptr[i0] && i_end > i0;
            int i = i0, j = j0, ph = 0;   // next row end, next in-edge, 1: row i's old values are behind, its V ahead
            bool carry_need = false;      // BF: the row in progress has a kept in-edge in an earlier stage
            bool head_pending = head;
            int whole = 0;                // PPR: stages in a row that ended no row (a long row's sum is folded, below)
            bool folded = false;
            // the next stage's row ends and in-edges, loaded while the current one is walked
            int raw_end, raw_col;
            uint32_t raw_w = 0u;  // BF: the in-edges' weights; PPR: the rows' out-degrees (float bits)
            auto load_raw = [&]() {
                raw_end = i + lane < i_end ? ld_stream_i32(p.rowptr + i + lane + 1) : INT_MAX;
                raw_col = 0;
                if constexpr (!BF) raw_w = i + lane < i_end ? __float_as_uint(ld_stream_f32(p.degf + i + lane)) : 0u;
                if (j + lane < j_end) {
                    raw_col = ld_stream_i32(p.colidx + j + lane);
                    if constexpr (BF) raw_w = p.w8 ? (uint32_t)p.w8[j + lane] : ld_stream_u32(p.w + j + lane);
                }
            };
            load_raw();
            // The next items of the run into list half lb (all of them, or for Bellman-Ford the ones a sweep needs);
            // an empty stage means that the run is done.
            auto build = [&](int lb) -> RunStage {
                RunStage st{0u, 0u, 0};
                int* lv = list + lb * 64;
                for (;;) {
                    const int left = (j_end - j) + RW * (i_end - i) - ph;
                    const int cnt = min(32, left);
                    if (cnt <= 0) return st;
                    const int pos = raw_end == INT_MAX ? INT_MAX : (raw_end - j) + RW * lane - ph;  // of row i + lane's old
                    unsigned old = __reduce_or_sync(FULL, (pos >= 0 && pos < cnt) ? 1u << pos : 0u);
                    unsigned fin = old;
                    if constexpr (!BF)
                        fin = __reduce_or_sync(
                            FULL, (pos != INT_MAX && pos + 1 >= 0 && pos + 1 < cnt) ? 1u << (pos + 1) : 0u);
                    const unsigned special = old | fin;
                    const int eo = lane - __popc(special & below(lane));  // in-edge of item `lane`, from j
                    const int row = i + __popc(fin & below(lane));
                    const int src = __shfl_sync(FULL, raw_col, eo & 31);
                    const uint32_t wt = __shfl_sync(FULL, raw_w, (BF ? eo : row - i) & 31);
                    const bool sp = (special >> lane) & 1u;
                    const int vert = sp ? row : src;
                    int kept = cnt;
                    if constexpr (BF) {
                        // in-edges whose source changed in this sweep or the one before; rows that keep any, the run's
                        // first row while earlier runs hold a part of it, and (synchronous) rows whose other buffer is
                        // a sweep behind
                        const unsigned c = lane < cnt && (!sp || sync) ? p.chg[vert] : 128u;
                        const bool fresh = lane < cnt && !sp && (c == now || c == before);
                        const unsigned edges = __ballot_sync(FULL, fresh);
                        const unsigned prior = special & below(lane);
                        const int from = prior ? 32 - __clz(prior) : 0;
                        const bool any = (edges & below(lane) & ~below(from)) != 0u || (!prior && carry_need);
                        const bool keep_row = lane < cnt && sp && (any || (head && row == i0) || (sync && c == before));
                        const unsigned need = edges | __ballot_sync(FULL, keep_row);
                        const int last = special & below(cnt) ? 32 - __clz(special & below(cnt)) : 0;
                        carry_need = (edges & ~below(last)) != 0u || (last == 0 && carry_need);
                        kept = __popc(need);
                        const int at = __popc(need & below(lane));
                        old = fin = __reduce_or_sync(FULL, keep_row ? 1u << at : 0u);
                        if ((need >> lane) & 1u) {
                            lv[at] = vert;
                            lv[32 + at] = (int)wt;
                        }
                    } else {
                        if (lane < cnt) {
                            lv[lane] = vert;
                            lv[32 + lane] = (int)wt;
                        }
                    }
                    const unsigned all = special & below(cnt);
                    const int ended = __popc(BF ? all : fin);
                    ph = (!BF && ((old >> (cnt - 1)) & 1u)) ? 1 : 0;  // the old values were the stage's last item
                    i += ended;
                    j += cnt - __popc(all);
                    load_raw();
                    if (kept > 0) {
                        st.old = old;
                        st.fin = fin;
                        st.cnt = kept;
                        __syncwarp();
                        return st;
                    }
                }
            };
            auto fold_in = [&](uint32_t (&a)[CH][4]) {  // the groups' joined part of the row in progress
#pragma unroll
                for (int q = 0; q < CH; ++q)
                    if (has(q))
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            if (grp == 0) fold[col0(q) + e] = folded ? comb<BF>(fold[col0(q) + e], a[q][e]) : a[q][e];
                            a[q][e] = ident<BF>();
                        }
                folded = true;
                __syncwarp();
            };
            auto unfold = [&](uint32_t (&a)[CH][4]) {  // adds it back, in every group
#pragma unroll
                for (int q = 0; q < CH; ++q)
                    if (has(q))
#pragma unroll
                        for (int e = 0; e < 4; ++e) a[q][e] = comb<BF>(a[q][e], fold[col0(q) + e]);
                folded = false;
                __syncwarp();
            };
            auto batches = [&](const RunStage& st) { return (st.cnt + G - 1) / G; };
            constexpr int STEPS = G >= GRP ? G / GRP : 1;  // groups' turns in a batch
            // copies of batch b of a stage into ring half `half`
            auto fetch = [&](const RunStage& st, int lb, int b, int half) {
                const int* lv = list + lb * 64 + b * G;
                const uint32_t at = ring_at + (uint32_t)(half * G * SR + 4 * lr) * 4u;
                const int have = st.cnt - b * G;
                const unsigned tele = BF ? 0u : st.fin >> (b * G);
#pragma unroll
                for (int u = 0; u < STEPS; ++u) {
                    const int k = u * GRP + grp;
                    if (k >= have || (G < GRP && k >= G)) continue;
                    const int v = lv[k];
                    const uint32_t dst = at + (uint32_t)(k * SR) * 4u;
                    if (BF || !((tele >> k) & 1u)) {
                        const uint32_t* x = xin + (size_t)v * S;
#pragma unroll
                        for (int q = 0; q < CH; ++q)
                            if (EVERY || has(q)) cp16(dst + 512u * q, x + from(q));
                    } else if (p.v16) {
                        const float* x = p.V + (size_t)v * B;
#pragma unroll
                        for (int q = 0; q < CH; ++q)
                            if (EVERY || has(q)) cp16(dst + 512u * q, x + from(q));
                    } else {
#pragma unroll
                        for (int q = 0; q < CH; ++q)
#pragma unroll
                            for (int e = 0; e < 4; ++e)
                                if (has(q) && col0(q) + e < B)
                                    cp4(dst + 512u * q + 4u * e, p.V + (size_t)v * B + col0(q) + e);
                    }
                }
            };
            // batch b of a stage from ring half `half`
            auto consume = [&](const RunStage& st, int lb, int b, int half) {
                const int* lv = list + lb * 64 + b * G;
                const uint32_t* rows = ring + half * G * SR + 4 * lr;
                auto add = [&](int k) {
                    const uint32_t wt = BF ? (uint32_t)lv[32 + k] : 0u;
#pragma unroll
                    for (int q = 0; q < CH; ++q) {
                        if (!PAD && !has(q)) continue;
                        const uint4 x = *(const uint4*)(rows + k * SR + 128 * q);
                        acc[q][0] = comb<BF>(acc[q][0], BF ? relax_w(x.x, wt) : x.x);
                        acc[q][1] = comb<BF>(acc[q][1], BF ? relax_w(x.y, wt) : x.y);
                        acc[q][2] = comb<BF>(acc[q][2], BF ? relax_w(x.z, wt) : x.z);
                        acc[q][3] = comb<BF>(acc[q][3], BF ? relax_w(x.w, wt) : x.w);
                    }
                };
                const int have = min(G, st.cnt - b * G);
                unsigned rem = ((st.old | st.fin) >> (b * G)) & below(have);
                if (rem == 0u) {  // in-edges only
#pragma unroll
                    for (int u = 0; u < STEPS; ++u) {
                        const int k = u * GRP + grp;
                        if (k < have) add(k);
                    }
                    return;
                }
                const unsigned old = BF ? 0u : st.old >> (b * G);
                int a = 0;
                for (;;) {
                    const int e1 = rem ? __ffs(rem) - 1 : have;
                    for (int k = a + grp; k < e1; k += GRP) add(k);
                    if (!rem) break;
                    rem &= rem - 1u;
                    a = e1 + 1;
                    uint4 x[CH];
#pragma unroll
                    for (int q = 0; q < CH; ++q) {
                        x[q] = make_uint4(0u, 0u, 0u, 0u);
                        if (PAD || has(q)) x[q] = *(const uint4*)(rows + e1 * SR + 128 * q);
                    }
                    if (!BF && ((old >> e1) & 1u)) {
#pragma unroll
                        for (int q = 0; q < CH; ++q) {
                            xo[q][0] = x[q].x; xo[q][1] = x[q].y; xo[q][2] = x[q].z; xo[q][3] = x[q].w;
                        }
                        continue;
                    }
                    join_groups(acc);
                    if (!BF && folded) unfold(acc);
                    if (head_pending) {  // begun in an earlier run: finished after this one
#pragma unroll
                        for (int q = 0; q < CH; ++q)
                            if (grp == 0 && has(q))
                                *(uint4*)(head_sum + col0(q)) = make_uint4(acc[q][0], acc[q][1], acc[q][2], acc[q][3]);
                        head_pending = false;
                    } else {
                        float tv[CH][4];
#pragma unroll
                        for (int q = 0; q < CH; ++q) {
                            if constexpr (BF) {
                                xo[q][0] = x[q].x; xo[q][1] = x[q].y; xo[q][2] = x[q].z; xo[q][3] = x[q].w;
                            } else {
                                tv[q][0] = __uint_as_float(x[q].x); tv[q][1] = __uint_as_float(x[q].y);
                                tv[q][2] = __uint_as_float(x[q].z); tv[q][3] = __uint_as_float(x[q].w);
                            }
                        }
                        update(lv[e1], acc, xo, tv, BF ? 0.0f : __int_as_float(lv[32 + e1]));
                    }
#pragma unroll
                    for (int q = 0; q < CH; ++q)
#pragma unroll
                        for (int e = 0; e < 4; ++e) acc[q][e] = ident<BF>();
                }
            };

            int lb = 0, half = 0, fb = 0;  // list half and first ring half of `cur`; batches fetched, from cur's first
            RunStage cur = build(0), nxt{0u, 0u, 0};
            bool ahead = false;            // nxt is built
            while (cur.cnt > 0) {
                const int ncb = batches(cur);
                for (int b = 0; b < ncb; ++b) {
                    while (fb < b + 2) {  // batch fb goes where batch fb - 2 (added up already) was
                        if (fb < ncb) {
                            fetch(cur, lb, fb, (half + fb) & 1);
                        } else {
                            if (!ahead) {
                                nxt = build(lb ^ 1);
                                ahead = true;
                            }
                            if (fb - ncb >= batches(nxt)) break;
                            fetch(nxt, lb ^ 1, fb - ncb, (half + fb) & 1);
                        }
                        cp_commit();
                        ++fb;
                    }
                    cp_wait(fb - b == 2);
                    __syncwarp();
                    consume(cur, lb, b, (half + b) & 1);
                    __syncwarp();
                }
                if constexpr (!BF) {
                    // a long row's FP32 sum in two levels: every FOLD_STAGES stages its part moves to shared memory,
                    // so a hub's thousands of terms are not one chain of additions
                    whole = cur.fin ? 0 : whole + 1;
                    if (whole >= FOLD_STAGES) {
                        join_groups(acc);
                        fold_in(acc);
                        whole = 0;
                    }
                }
                if (!ahead) nxt = build(lb ^ 1);
                cur = nxt;
                ahead = false;
                half = (half + ncb) & 1;
                lb ^= 1;
                fb -= ncb;
                if (!BF && !sync && (++stages & (LIVE_STAGES - 1)) == 0) live();
            }

            // ---------------- the row this run leaves unfinished, and the one it started inside ----------------
            join_groups(acc);
            if (!BF && folded) unfold(acc);
            bool some = false;
#pragma unroll
            for (int q = 0; q < CH; ++q)
                if (has(q))
#pragma unroll
                    for (int e = 0; e < 4; ++e) some |= acc[q][e] != ident<BF>();
            some = __any_sync(FULL, some);
            if (some && grp == 0) {
#pragma unroll
                for (int q = 0; q < CH; ++q)
                    if (has(q)) st_relaxed_v4(p.part + (size_t)t * S + col0(q), acc[q]);
            }
            if (some) fence_gpu();
            __syncwarp();
            if (lane == 0) st_pub(p.pub + t, ((unsigned long long)stamp << 32) | (some ? 0u : PUB_EMPTY));
            // the pending row is finished a run later, by when the runs before it have published theirs (a run publishes
            // before its warp waits for an older one, so the lowest pending run can always finish)
            if (pend >= 0) ok = resolve(pend, pend_row);
            pend = head ? t : -1;
            pend_row = i0;
            if (head && grp == 0) {
#pragma unroll
                for (int q = 0; q < CH; ++q)
                    if (has(q)) *(uint4*)(head_part + col0(q)) = *(const uint4*)(head_sum + col0(q));
            }
#pragma unroll
            for (int q = 0; q < CH; ++q)
#pragma unroll
                for (int e = 0; e < 4; ++e) acc[q][e] = ident<BF>();
        }  // runs
        if (ok && pend >= 0) resolve(pend, pend_row);
        // ---------------- end of sweep: per-column sums, barrier, stopping rules ----------------
        cta_sum(res, p.acc_res + slot * B, nullptr);
        if (!BF) cta_sum(mass, sync ? p.acc_g + slot * B : p.gl, nullptr);
        if (!BF && !sync)  // what the warps gave during the sweep (cta_sum's barriers stand before and after)
            for (int c = tid; c < B; c += NT) {
                const double v = s_live[c];
                if (v != 0.0) atomicAdd(&p.gl[c], v);
                s_live[c] = 0.0;
            }
        if (!grid_barrier(p.sb, p.nblocks, bar, p.timeout_ns)) return;
        int still = 0;
        for (int c = tid; c < B; c += NT) {
            // the sweep's first dangling term for the whole CTA: while every warp read the live mass at its first run, the
            // columns' few lines in L2 held up small graphs (PPR of 32 columns, uniform, 3 K vertices 200 -> 146 us, 30 K
            // 395 -> 342; synchronous, formed per lane before, 169 -> 146; 256 columns at 1 M vertices the same)
            const double res = ld_relaxed_f64(&p.acc_res[slot * B + c]);
            if (!BF) s_gt[c] = dangling(ld_relaxed_f64(sync ? &p.acc_g[slot * B + c] : &p.gl[c]), s_T[c]);
            if (s_run[c]) {
                if (res <= p.tol) {
                    s_run[c] = 0;
                    s_last[c] = it + 1;
                    if (blockIdx.x == 0) p.iters[c] = it + 1;
                } else {
                    still = 1;
                }
            }
            if (blockIdx.x == 0) {
                const int dead = (it + 2) % 3;  // read by everyone before this barrier
                p.acc_res[dead * B + c] = 0.0;
                p.acc_g[dead * B + c] = 0.0;
            }
        }
        if (!__syncthreads_or(still)) {
            ++it;
            break;
        }
    }
    int any = 0;
    for (int c = tid; c < B; c += NT)
        if (s_run[c]) {  // not converged: ran them all
            any = 1;
            s_last[c] = it;
            if (blockIdx.x == 0) p.iters[c] = it;
        }
    any = __syncthreads_or(any);
    if (blockIdx.x == 0 && tid == 0) {
        p.sb->iters = it;
        p.sb->converged = any ? 0 : 1;
    }

    // ---------------- output: r = x * outdeg, from the buffer of each column's last sweep ----------------
    const bool packed = S == B && ((uintptr_t)p.out & 15u) == 0;
    for (int v = w * GRP + grp; v < p.n; v += W * GRP) {
        float dg = 0.0f;
        if constexpr (!BF) dg = p.degf[v];
#pragma unroll
        for (int q = 0; q < CH; ++q) {
            if (!has(q)) continue;
            const size_t at = (size_t)v * S + col0(q);
            uint4 x = ld_relaxed_v4(p.X0 + at);
            if (sync) {
                const uint4 y = ld_relaxed_v4(p.X1 + at);
                if (s_last[col0(q)] & 1) x.x = y.x;
                if (s_last[col0(q) + 1] & 1) x.y = y.y;
                if (s_last[col0(q) + 2] & 1) x.z = y.z;
                if (s_last[col0(q) + 3] & 1) x.w = y.w;
            }
            uint32_t o[4] = {x.x, x.y, x.z, x.w};
            if constexpr (!BF) {
                if (dg > 0.0f)
#pragma unroll
                    for (int e = 0; e < 4; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * dg);
            }
            uint32_t* dst = p.out + (size_t)v * B + col0(q);
            if (packed) {
                *(uint4*)dst = make_uint4(o[0], o[1], o[2], o[3]);
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (col0(q) + e < B) dst[e] = o[e];
            }
        }
    }
}

// Lanes per row 1, 2, 4, 8, 16, 32 (k 0 to 5), then chunks per lane 2, 4, 8 (k 6 to 8).
static int run_shape(int B)
{
    int k = 0;
    while ((4 << k) < B) ++k;
    return k;
}

size_t run_smem_bytes(bool is_bf, int B)
{
    const size_t S = (size_t)((B + 3) & ~3);
    const int k = run_shape(B), depth = run_depth(k < 5 ? 1 << k : 32, k > 5 ? 1 << (k - 5) : 1);
    const size_t SR = run_padded(is_bf, k < 5 ? 1 << k : 32, k > 5 ? 1 << (k - 5) : 1) ? (size_t)4 << k : S;
    return (is_bf ? 0 : 2 * S * 8 + S * 4) + 2 * RUN_WARPS * S * 4 + 2 * S * 4 + RUN_WARPS * 128 * 4 +
           (size_t)RUN_WARPS * depth * SR * 4;
}

// PPR: two items to fetch, an update and a store, against an in-edge's one addition, which costs the less the fewer
// lanes hold a row. Measured (RMAT): 256 columns at 1 M vertices 94 ms with weight 1, 40 with 3, 33 with 5, 36 with 8
// and 42 with 20 (one run per warp); 20 columns at 100 K vertices 4.8, 2.1, 1.5, 1.3 and 1.3, 1.2 ms with 12.
// Bellman-Ford mostly skips rows: 7.1 to 7.4 ms for weights 1 to 8 (64 columns, 1 M vertices).
int run_row_weight(bool is_bf, int B)
{
    if (is_bf) return 2;
    return B > 128 ? 5 : B > 64 ? 6 : B > 32 ? 8 : 12;
}

BKernel run_kernel_for(bool is_bf, int B)
{
    const int k = run_shape(B);
#define DAG_RUNS(BFV, WH)                                                                                          \
    {batched_runs_kernel<BFV, 1, 1, WH>, batched_runs_kernel<BFV, 2, 1, WH>, batched_runs_kernel<BFV, 4, 1, WH>, \
     batched_runs_kernel<BFV, 8, 1, WH>, batched_runs_kernel<BFV, 16, 1, WH>, batched_runs_kernel<BFV, 32, 1, WH>, \
     batched_runs_kernel<BFV, 32, 2, WH>, batched_runs_kernel<BFV, 32, 4, WH>, batched_runs_kernel<BFV, 32, 8, WH>}
    static const BKernel table[2][2][9] = {{DAG_RUNS(false, false), DAG_RUNS(false, true)},
                                           {DAG_RUNS(true, false), DAG_RUNS(true, true)}};
#undef DAG_RUNS
    return table[is_bf ? 1 : 0][((B + 3) & ~3) == (4 << k) ? 1 : 0][k];
}

}  // namespace dag
