"""GPU parity of the batched PPR / SSSP launch against the CPU oracle (C ABI).

Each column of a batched solve is an independent problem: PPR columns must be
within L1 1e-5 of their fp64 fixed points (same bound as the single-vector
PageRank), SSSP columns bit-exact against Dijkstra, and in the synchronous form
each column must run exactly as many sweeps as its single-vector solve.
"""
import numpy as np
import pytest
import torch

import oracle
import paper_2110_01409_gb300.inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dag():
    from paper_2110_01409_gb300 import build, dag as D

    build.build()
    assert torch.cuda.is_available()
    return D


@pytest.fixture(scope="module")
def graph():
    return I.rmat(12, 16, seed=31)


@pytest.mark.parametrize("variant,delta", [("sync", 0), ("async", 0), ("delayed", 4), ("delayed", 16)])
def test_ppr_batched_columns_match_oracle(dag, graph, variant, delta):
    g = graph
    B = 40  # not a multiple of 32: a ragged last warp
    sets = I.ppr_seed_sets(g.n, B, seed=7)
    V = I.teleport_matrix(g.n, sets)
    plan = dag.Plan.from_graph(g, "cuda")
    R, iters, st = dag.ppr_batched(plan, torch.from_numpy(V).cuda(), 0.85, 1e-6, variant, delta)
    assert st["converged"], st
    R = R.cpu().numpy().astype(np.float64)
    its = iters.cpu().numpy()
    for c in [0, 1, 17, 31, 32, 39]:
        rstar = oracle.pagerank_fixed_point(g, 0.85, tele=V[:, c].astype(np.float64))
        assert np.abs(R[:, c] - rstar).sum() <= 1e-5, c
        if variant == "sync":
            _, st1 = dag.pagerank(plan, 0.85, 1e-6, "sync", 0, teleport=torch.from_numpy(V[:, c].copy()).cuda())
            assert abs(int(its[c]) - st1["iters"]) <= 1
    assert st["column_sweeps"] == int(its.sum())
    assert st["sweeps"] == int(its.max())


def test_ppr_batched_cycle_closed_form(dag):
    n, d = 256, 0.85
    g = I.from_edges(n, np.arange(n), (np.arange(n) + 1) % n)
    srcs = [0, 5, 77, 255]
    V = np.zeros((n, len(srcs)), dtype=np.float32)
    for c, s in enumerate(srcs):
        V[s, c] = 1.0
    plan = dag.Plan.from_graph(g, "cuda")
    R, _, st = dag.ppr_batched(plan, torch.from_numpy(V).cuda(), d, 1e-8, "delayed", 8)
    R = R.cpu().numpy()
    for c, s in enumerate(srcs):
        want = np.array([(1 - d) * d ** ((v - s) % n) / (1 - d ** n) for v in range(n)])
        assert np.max(np.abs(R[:, c] - want)) <= 1e-6


@pytest.mark.parametrize("variant,delta", [("sync", 0), ("async", 0), ("delayed", 8)])
def test_sssp_batched_bit_exact(dag, graph, variant, delta):
    g = graph
    w = I.weights_u32(g, 9)
    srcs = I.sources(g, 33, seed=5)
    plan = dag.Plan.from_graph(g, "cuda")
    D, iters, st = dag.sssp_batched(plan, torch.from_numpy(srcs.view(np.int32)).cuda(),
                                    torch.from_numpy(w.view(np.int32)).cuda(), variant, delta)
    assert st["converged"]
    D = D.cpu().numpy().view(np.uint32)
    its = iters.cpu().numpy()
    for c, s in enumerate(srcs):
        ref = oracle.dijkstra(g, w, int(s))
        assert np.array_equal(D[:, c], ref), c
        if variant == "sync":
            _, it, _, _ = oracle.sssp(g, w, int(s), oracle.SYNC)
            assert its[c] == it


def test_batched_single_column_and_bad_source(dag, graph):
    g = graph
    plan = dag.Plan.from_graph(g, "cuda")
    V = np.zeros((g.n, 1), dtype=np.float32)
    V[:, 0] = 1.0 / g.n
    R, iters, st = dag.ppr_batched(plan, torch.from_numpy(V).cuda(), 0.85, 1e-6, "delayed", 16)
    assert np.abs(R.cpu().numpy()[:, 0].astype(np.float64) - oracle.pagerank_fixed_point(g)).sum() <= 1e-5
    w = torch.from_numpy(I.weights_u32(g, 1).view(np.int32)).cuda()
    with pytest.raises(dag.DagError):
        dag.sssp_batched(plan, torch.tensor([0, g.n + 5], dtype=torch.int32, device="cuda"), w)


def test_batched_graph_replays_equal_direct_launches_and_the_oracle(dag, graph):
    # the batched launch is replayed from the plan's CUDA graph of its shape (the default); calls with new
    # buffers, new teleport matrices and a new B replay with their own arguments. In the synchronous form
    # every column's arithmetic is fixed, so replays and direct launches agree bit for bit.
    g = graph
    plan_g = dag.Plan.from_graph(g, "cuda")  # graphs on
    plan_d = dag.Plan.from_graph(g, "cuda")
    plan_d.set_batched_graph(False)
    for B, seed in [(40, 11), (40, 12), (33, 13), (64, 14), (40, 15)]:
        sets = I.ppr_seed_sets(g.n, B, seed=seed)
        V = torch.from_numpy(I.teleport_matrix(g.n, sets)).cuda()
        out = torch.full_like(V, -1.0)  # a fresh output buffer each call
        Rg, itg, stg = dag.ppr_batched(plan_g, V, 0.85, 1e-6, "sync", 0, out=out)
        Rd, itd, std = dag.ppr_batched(plan_d, V.clone(), 0.85, 1e-6, "sync", 0)
        assert stg["graph"] and not std["graph"], (B, stg, std, dag.lib().dag_last_error_message().decode())
        assert stg["converged"] and std["converged"]
        assert torch.equal(Rg, Rd) and torch.equal(itg, itd)
        Vh = V.cpu().numpy().astype(np.float64)
        for c in (0, B - 1):
            rstar = oracle.pagerank_fixed_point(g, 0.85, tele=Vh[:, c])
            assert np.abs(Rg[:, c].cpu().numpy().astype(np.float64) - rstar).sum() <= 1e-5, (B, c)
    # the asynchronous form too (results agree within the parity bound, not bit for bit)
    sets = I.ppr_seed_sets(g.n, 40, seed=16)
    V = torch.from_numpy(I.teleport_matrix(g.n, sets)).cuda()
    Rg, _, stg = dag.ppr_batched(plan_g, V, 0.85, 1e-6, "async", 0)
    assert stg["graph"] and stg["converged"]
    rstar = oracle.pagerank_fixed_point(g, 0.85, tele=V[:, 7].cpu().numpy().astype(np.float64))
    assert np.abs(Rg[:, 7].cpu().numpy().astype(np.float64) - rstar).sum() <= 1e-5
    # Bellman-Ford replays: new sources, new B, both weight widths
    w = I.weights_u32(g, 9)
    for B, seed in [(33, 5), (20, 6)]:
        srcs = torch.from_numpy(I.sources(g, B, seed=seed).view(np.int32)).cuda()
        for wd in (torch.from_numpy(w.view(np.int32)).cuda(), torch.from_numpy(w.astype(np.uint8)).cuda()):
            D, _, st = dag.sssp_batched(plan_g, srcs, wd, "async", 0)
            assert st["graph"] and st["converged"]
            D = D.cpu().numpy().view(np.uint32)
            for c in (0, B - 1):
                assert np.array_equal(D[:, c], oracle.dijkstra(g, w, int(srcs[c])))


@pytest.mark.parametrize("variant,delta", [("sync", 0), ("async", 0), ("delayed", 8)])
def test_sssp_batched_one_byte_weights(dag, graph, variant, delta):
    g = graph
    w = I.weights_u32(g, 9)
    srcs = torch.from_numpy(I.sources(g, 40, seed=8).view(np.int32)).cuda()
    plan = dag.Plan.from_graph(g, "cuda")
    D8, it8, st8 = dag.sssp_batched(plan, srcs, torch.from_numpy(w.astype(np.uint8)).cuda(), variant, delta)
    D4, it4, st4 = dag.sssp_batched(plan, srcs, torch.from_numpy(w.view(np.int32)).cuda(), variant, delta)
    assert st8["converged"] and torch.equal(D8, D4)
    if variant == "sync":
        assert torch.equal(it8, it4)
    D8 = D8.cpu().numpy().view(np.uint32)
    for c in (0, 17, 39):
        assert np.array_equal(D8[:, c], oracle.dijkstra(g, w, int(srcs[c])))


# ---- the wide kernel: 32, 64, 128 or 256 columns, synchronous and asynchronous forms ----
@pytest.mark.parametrize("B", [32, 64, 128, 256])
@pytest.mark.parametrize("variant", ["sync", "async"])
def test_wide_ppr_batched_matches_oracle_and_the_narrow_kernel(dag, graph, B, variant):
    # a warp per share of each tile over all B columns: every checked column within L1 1e-5 of its fp64
    # fixed point; the synchronous form in as many sweeps as the 32-column kernel (within one) and equal
    # values within rounding (a row split between shares adds its partial sums in another order)
    g = graph
    sets = I.ppr_seed_sets(g.n, B, seed=11)
    V = torch.from_numpy(I.teleport_matrix(g.n, sets)).cuda()
    plan = dag.Plan.from_graph(g, "cuda")
    R, iters, st = dag.ppr_batched(plan, V, 0.85, 1e-6, variant, 0)
    assert st["converged"], st
    plan.set_batched_wide(False)
    R2, iters2, st2 = dag.ppr_batched(plan, V, 0.85, 1e-6, variant, 0)
    assert st2["converged"]
    Rn = R.cpu().numpy().astype(np.float64)
    for c in sorted({0, 1, B // 2, B - 1, int(np.argmax(iters.cpu().numpy()))}):
        rstar = oracle.pagerank_fixed_point(g, 0.85, tele=V[:, c].cpu().numpy().astype(np.float64))
        assert np.abs(Rn[:, c] - rstar).sum() <= 1e-5, c
    if variant == "sync":
        # the residual sums differ in their last bits (another summation order), so a column whose
        # residual lands at the tolerance may take one sweep more in one kernel than in the other
        assert int(np.abs(iters.cpu().numpy() - iters2.cpu().numpy()).max()) <= 1
        assert float((R - R2).abs().max()) <= 1e-5
    assert st["column_sweeps"] == int(iters.sum())


@pytest.mark.parametrize("B", [32, 64, 256])
@pytest.mark.parametrize("variant", ["sync", "async"])
@pytest.mark.parametrize("u8", [True, False])
def test_wide_sssp_batched_bit_exact(dag, B, variant, u8):
    # hub rows longer than a tile and tiles inside one row: RMAT scale 14 with its heavy in-degree head
    g = I.rmat(14, 16, seed=8)
    w = I.weights_u32(g, 12)
    srcs = I.sources(g, B, seed=13)
    plan = dag.Plan.from_graph(g, "cuda")
    wd = torch.from_numpy(w.astype(np.uint8) if u8 else w.view(np.int32)).cuda()
    D, iters, st = dag.sssp_batched(plan, torch.from_numpy(srcs.view(np.int32)).cuda(), wd, variant, 0)
    assert st["converged"]
    D = D.cpu().numpy().view(np.uint32)
    its = iters.cpu().numpy()
    for c in sorted({0, 1, B // 3, B - 1}):
        assert np.array_equal(D[:, c], oracle.dijkstra(g, w, int(srcs[c]))), c
        if variant == "sync":
            _, it, _, _ = oracle.sssp(g, w, int(srcs[c]), oracle.SYNC)
            assert its[c] == it
    plan.set_batched_wide(False)
    D2, _, _ = dag.sssp_batched(plan, torch.from_numpy(srcs.view(np.int32)).cuda(), wd, variant, 0)
    assert np.array_equal(D, D2.cpu().numpy().view(np.uint32))


def test_wide_batched_tiny_graphs(dag):
    # rows of no in-edges, a graph smaller than one tile, and the delayed form on the 32-column kernel
    g = I.from_edges(6, [0, 1, 2, 0], [1, 2, 3, 3], "tiny")
    plan = dag.Plan.from_graph(g, "cuda")
    V = np.zeros((6, 32), dtype=np.float32)
    V[np.arange(32) % 6, np.arange(32)] = 1.0
    for variant, delta in (("sync", 0), ("async", 0), ("delayed", 4)):
        # (tol 1e-6: with ranks near 0.2 the FP32 residual of six rows cannot fall much below 1e-7)
        R, _, st = dag.ppr_batched(plan, torch.from_numpy(V).cuda(), 0.85, 1e-6, variant, delta)
        assert st["converged"]
        R = R.cpu().numpy()
        for c in (0, 1, 5, 31):
            rstar = oracle.pagerank_fixed_point(g, 0.85, tele=V[:, c].astype(np.float64))
            assert np.abs(R[:, c] - rstar).sum() <= 1e-5, (variant, c)


# ---- the run kernel (synchronous and asynchronous forms): any column count, rows spanning many warps' runs ----
def _hub_graph():
    """3,001 vertices: RMAT-like edges, two hubs whose in-edges span many runs, the last vertex among them, and a
    tail of vertices without in-edges."""
    rng = np.random.default_rng(5)
    n, k = 3001, 12000
    src = (rng.random(k) ** 3 * n).astype(np.int64)
    dst = (rng.random(k) ** 2 * (n - 700)).astype(np.int64)
    hubs = [np.stack([rng.permutation(n)[:2500], np.full(2500, h)]) for h in (17, n - 1)]
    e = np.concatenate([np.stack([src, dst])] + hubs, axis=1)
    e = np.unique(e[:, e[0] != e[1]], axis=1)
    return I.from_edges(n, e[0], e[1])


@pytest.mark.parametrize("B", [1, 2, 3, 6, 9, 20, 33, 72, 130, 300, 1024])
@pytest.mark.parametrize("variant", ["sync", "async"])
def test_runs_any_column_count(dag, B, variant):
    # every lanes-per-row and chunks-per-lane shape, whole and ragged; outputs that are not 16-byte aligned go
    # through the padded state; distances equal the oracle's, ranks lie within L1 1e-5 of the fixed point
    g = _hub_graph()
    plan = dag.Plan.from_graph(g, "cuda")
    V = I.teleport_matrix(g.n, I.ppr_seed_sets(g.n, B, seed=3))
    Vd = torch.from_numpy(V).cuda()
    out = torch.empty(g.n * B + 1, dtype=torch.float32, device="cuda")[1:].view(g.n, B)
    w = I.weights_u32(g, 9)
    srcs = I.sources(g, B, seed=5) if B <= 300 else np.resize(I.sources(g, 300, seed=5), B)
    sd = torch.from_numpy(srcs.view(np.int32)).cuda()
    cols = sorted({0, B // 2, B - 1})
    for o in (None, out):
        R, iters, st = dag.ppr_batched(plan, Vd, 0.85, 1e-6, variant, 0, out=o)
        assert st["converged"] and st["column_sweeps"] == int(iters.sum()) and st["sweeps"] == int(iters.max())
        Rn = R.cpu().numpy().astype(np.float64)
        for c in cols:
            rstar = oracle.pagerank_fixed_point(g, 0.85, tele=V[:, c].astype(np.float64), tol=1e-12)
            assert np.abs(Rn[:, c] - rstar).sum() <= 1e-5, c
    for wd in (torch.from_numpy(w.astype(np.uint8)).cuda(), torch.from_numpy(w.view(np.int32)).cuda()):
        D, iters, st = dag.sssp_batched(plan, sd, wd, variant, 0, out=torch.full((g.n * B + 1,), 7, dtype=torch.int32,
                                                                                 device="cuda")[1:].view(g.n, B))
        assert st["converged"]
        Dn, its = D.cpu().numpy().view(np.uint32), iters.cpu().numpy()
        for c in cols:
            assert np.array_equal(Dn[:, c], oracle.dijkstra(g, w, int(srcs[c]))), c
            if variant == "sync":
                assert its[c] == oracle.sssp(g, w, int(srcs[c]), oracle.SYNC)[1]


@pytest.mark.parametrize("cap", [1, 2])
@pytest.mark.parametrize("B", [1, 3, 6, 12, 20, 33, 72, 130, 300, 1024])
@pytest.mark.parametrize("variant", ["sync", "async"])
def test_several_runs_a_warp(dag, B, variant, cap):
    # one or two CTAs: each warp takes 2 to 15 runs (the graph's weight by a run's 1,024, or 256 above 128 columns;
    # Bellman-Ford of up to 128 columns on two CTAs one), carries the row it began inside a run from one run to the next,
    # and looks back over runs of its own and of other warps
    g = _hub_graph()
    plan = dag.Plan.from_graph(g, "cuda")
    plan.set_worker_cap(cap)
    V = I.teleport_matrix(g.n, I.ppr_seed_sets(g.n, B, seed=4))
    w = I.weights_u32(g, 9) & 0xFF
    srcs = np.resize(I.sources(g, min(B, 300), seed=6), B)
    cols = sorted({0, B // 2, B - 1})
    R, iters, st = dag.ppr_batched(plan, torch.from_numpy(V).cuda(), 0.85, 1e-5, variant, 0)
    assert st["converged"] and st["workers"] == cap and st["column_sweeps"] == int(iters.sum())
    Rn = R.cpu().numpy().astype(np.float64)
    for c in cols:
        rstar = oracle.pagerank_fixed_point(g, 0.85, tele=V[:, c].astype(np.float64), tol=1e-12)
        # d / (1 - d) tol of L1 error, and an eighth for the FP32 parts of the sums: with so few workers a lane adds 375
        # rows' ranks, two hubs of a seventh among them, and a synchronous sweep's residual stays at up to 7e-6
        # (the 32-column kernel's at 6e-5)
        assert np.abs(Rn[:, c] - rstar).sum() <= 5.7e-5 * 1.125, c
    sd = torch.from_numpy(srcs.view(np.int32)).cuda()
    for wd in (torch.from_numpy(w.astype(np.uint8)).cuda(), torch.from_numpy(w.view(np.int32)).cuda()):
        D, iters, st = dag.sssp_batched(plan, sd, wd, variant, 0)
        assert st["converged"]
        Dn, its = D.cpu().numpy().view(np.uint32), iters.cpu().numpy()
        for c in cols:
            assert np.array_equal(Dn[:, c], oracle.dijkstra(g, w, int(srcs[c]))), c
            if variant == "sync":
                assert its[c] == oracle.sssp(g, w, int(srcs[c]), oracle.SYNC)[1]


@pytest.mark.parametrize("variant", ["sync", "async"])
def test_runs_long_path_and_sweep_limit(dag, variant):
    # 600 sweeps: the last-change byte wraps twice; a solve stopped early reports its sweeps
    n = 600
    g = I.from_edges(n, np.arange(1, n), np.arange(n - 1))  # v <- v + 1: one hop per sweep against the row order
    plan = dag.Plan.from_graph(g, "cuda")
    w = torch.full((g.m,), 3, dtype=torch.uint8, device="cuda")
    src = torch.tensor([n - 1, 300, n - 1], dtype=torch.int32, device="cuda")
    D, iters, st = dag.sssp_batched(plan, src, w, variant, 0)
    D = D.cpu().numpy().view(np.uint32)
    for c, s in enumerate((n - 1, 300, n - 1)):
        want = np.where(np.arange(n) <= s, 3 * (s - np.arange(n)), 0xFFFFFFFF).astype(np.uint32)
        assert np.array_equal(D[:, c], want)
    if variant == "sync":
        assert iters.cpu().tolist() == [600, 301, 600]
        _, _, st = dag.sssp_batched(plan, src, w, variant, 0, max_iters=5)
        assert not st["converged"] and st["sweeps"] == 5


@pytest.mark.parametrize("calls", [[("delayed", 128, 32), ("delayed", 256, 16), ("delayed", 128, 32)],
                                   [("delayed", 32, 16), ("delayed", 512, 1)], [("sync", 8, 0), ("sync", 1024, 0)],
                                   [("async", 8, 0), ("async", 1024, 0)]])
def test_column_counts_of_one_kernel_and_shared_size_on_one_plan(dag, graph, calls):
    # the 32-column kernel's CTA has a warp per 32 columns: calls whose shared memory is the same size but whose CTAs
    # are not have grids of their own (a grid settled for the smaller CTA cannot be resident for the larger)
    g = graph
    plan = dag.Plan.from_graph(g, "cuda")
    plan.set_batched_wide(False)
    w = I.weights_u32(g, 3)
    wd = torch.from_numpy(w.view(np.int32)).cuda()
    for variant, B, delta in calls:
        V = I.teleport_matrix(g.n, I.ppr_seed_sets(g.n, B, seed=2))
        R, _, st = dag.ppr_batched(plan, torch.from_numpy(V).cuda(), 0.85, 1e-6, variant, delta)
        assert st["converged"], st
        rstar = oracle.pagerank_fixed_point(g, 0.85, tele=V[:, B - 1].astype(np.float64))
        assert np.abs(R[:, B - 1].cpu().numpy().astype(np.float64) - rstar).sum() <= 1e-5
        src = np.resize(I.sources(g, 32, seed=B), B)
        D, _, st = dag.sssp_batched(plan, torch.from_numpy(src.view(np.int32)).cuda(), wd, variant, delta)
        assert st["converged"]
        assert np.array_equal(D[:, B - 1].cpu().numpy().view(np.uint32), oracle.dijkstra(g, w, int(src[B - 1])))


@pytest.mark.parametrize("B", [5, 20, 36, 130, 261])
@pytest.mark.parametrize("n", [1, 2, 997])
def test_runs_sources_anywhere_in_ragged_groups(dag, B, n):
    # a vertex that is only one column's source, whichever lane and chunk hold the column and wherever the vertex is in
    # its warp's last, partial group, is read in the first sweep (a cycle: each distance hangs on it)
    g = I.from_edges(n, np.arange(n) if n > 1 else np.zeros(0, int), (np.arange(n) + 1) % n if n > 1 else np.zeros(0, int))
    plan = dag.Plan.from_graph(g, "cuda")
    wd = torch.full((g.m,), 2, dtype=torch.uint8, device="cuda")
    src = (n - 1 - np.arange(B)) % n
    for variant in ("sync", "async"):
        D, _, st = dag.sssp_batched(plan, torch.from_numpy(src.astype(np.int32)).cuda(), wd, variant, 0)
        assert st["converged"]
        want = 2 * ((np.arange(n)[:, None] - src[None, :]) % n)
        assert np.array_equal(D.cpu().numpy().view(np.uint32), want.astype(np.uint32))


@pytest.mark.parametrize("B", [8, 100, 128])
@pytest.mark.parametrize("variant", ["sync", "async"])
def test_runs_dangling_mass_beside_a_large_column_sum(dag, B, variant):
    # vertex 0 links to itself and holds the column's mass, 1; the seven dangling ones start with half an ulp of it each.
    # Added up in FP32 over a CTA's warps those vanish from the teleport total, and with them the dangling term, 0.39 of
    # 0.89 half ulps of their rank. Vertex 0's rank, 1 + 2 x 0.39 half ulps, rounds to 1: the term is d / n of that larger,
    # 0.05 half ulps.
    n, d, half = 8, 0.5, 2.0 ** -24
    V = np.zeros((n, B), dtype=np.float32)
    V[0, :] = 1.0
    V[1:, B - 1] = half
    plan = dag.Plan(torch.tensor([0] + [1] * n, dtype=torch.int32, device="cuda"),
                    torch.tensor([0], dtype=torch.int32, device="cuda"))
    R, _, _ = dag.ppr_batched(plan, torch.from_numpy(V).cuda(), d, 1e-12, variant, 0, max_iters=400)
    dangling = 3.5 * half / (1 - 7 * d / n)
    want = 0.5 * half + d / n * dangling
    assert np.abs(R[1:, B - 1].cpu().numpy().astype(np.float64) - want).max() <= 0.06 * half, (R[1, B - 1].item(), want)
    assert R[0, B - 1].item() == 1.0


@pytest.mark.parametrize("variant", ["sync", "async"])
def test_runs_whose_scratch_does_not_fit(dag, variant):
    # the solve runs on the 32-column kernel, with the same results, and the plan keeps nothing of the attempt: no padded
    # copy of the state (30 columns, rows of 32: 240 MB) beside the synchronous form's second buffer
    g = I.rmat(21, 2, seed=3)
    B = 30
    plan = dag.Plan.from_graph(g, "cuda")
    V = torch.zeros((g.n, B), device="cuda")
    src = I.sources(g, B, seed=1)
    V[torch.from_numpy(src.astype(np.int64)).cuda(), torch.arange(B, device="cuda")] = 1.0
    out = torch.empty_like(V)
    plan.set_batched_wide(False)
    ref, it0, _ = dag.ppr_batched(plan, V, 0.85, 1e-6, variant, 0)
    plan.set_batched_wide(True)
    plan.debug_limit_batched_scratch(0)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    _, it1, st = dag.ppr_batched(plan, V, 0.85, 1e-6, variant, 0, out=out)
    assert before - torch.cuda.mem_get_info()[0] < 32 << 20
    assert st["converged"]
    if variant == "sync":
        assert torch.equal(it0, it1)
    assert float((out - ref).abs().sum(0).max()) <= 2e-5
    plan.debug_limit_batched_scratch(1 << 40)
    R, _, st = dag.ppr_batched(plan, V, 0.85, 1e-6, variant, 0)
    assert st["converged"] and float((R - ref).abs().sum(0).max()) <= 2e-5
