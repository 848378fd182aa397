"""GPU parity of the PageRank adjoint (gradients through weighted PageRank).

Loss L = sum_i w_i r_i over target vertices; the GPU gives dL/dw per edge and
dL/dt per vertex from one adjoint sweep solve. Checked on an n = 512 subgraph
against the dense fp64 adjoint (norm-wise rel <= 1e-4) and fp64 central finite
differences (rel <= 1e-3), and on a larger graph against the oracle's Jacobi
adjoint. Norm-wise relative error: ||g - g_ref||_2 / ||g_ref||_2.
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


def _rel(a, b):
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / np.linalg.norm(b))


def _subgraph512():
    # induced subgraph of the scale-22 RMAT on vertex ids 0..511 (its densest corner)
    big = I.rmat(22, 16, seed=2)
    end = big.rowptr[512]
    src = big.colidx[:end]
    dst = np.repeat(np.arange(512, dtype=np.int32), np.diff(big.rowptr[:513]))
    keep = src < 512
    return I.from_edges(512, src[keep], dst[keep], "rmat22_sub512")


def _problem(g, seed, k):
    w = I.weights_f32(g, seed)
    targets, wt = I.adjoint_targets(g.n, k, seed)
    c = np.zeros(g.n)
    c[targets] = wt
    t = np.zeros(g.n)
    t[I.distinct_choice(np.arange(g.n), 8, seed, 77)] = 1.0 / 8
    return w, t, c


FORMS = [("sync", 0, "refresh"), ("delayed", 64, "refresh"), ("async", 0, "refresh"), ("sync", 0, "warp"),
         ("async", 0, "warp+cached"), ("delayed", 64, "warp"), ("async", 0, "ordered+cached")]


@pytest.mark.parametrize("variant,delta,reads", FORMS)
def test_adjoint_subgraph512_vs_dense_and_fd(dag, variant, delta, reads):
    g = _subgraph512()
    w, t, c = _problem(g, 5, 64)
    plan = dag.Plan.from_graph(g, "cuda")
    model = dag.WeightedPageRank(plan, d=0.85, tol=1e-6, variant=variant, delta=delta, reads=reads)
    wt = torch.from_numpy(w).cuda().requires_grad_(True)
    tt = torch.from_numpy(t.astype(np.float32)).cuda().requires_grad_(True)
    r = dag.PageRankFn.apply(wt, tt, model)
    loss = (r.double() * torch.from_numpy(c).cuda()).sum()
    loss.backward()
    gw_ref, gt_ref, r_ref, _ = oracle.dense_grads(g, w.astype(np.float64), t, c)
    assert np.abs(r.detach().cpu().numpy() - r_ref).sum() <= 1e-5
    assert _rel(wt.grad.cpu().numpy(), gw_ref) <= 1e-4
    assert _rel(tt.grad.cpu().numpy(), gt_ref) <= 1e-4
    # finite differences on a sample of edges and all of t
    edges = np.arange(0, g.m, max(1, g.m // 64))
    fw, ft = oracle.fd_grads(g, w.astype(np.float64), t, c, edges=edges)
    assert _rel(wt.grad.cpu().numpy()[edges], fw) <= 1e-3
    assert _rel(tt.grad.cpu().numpy(), ft) <= 1e-3


def test_adjoint_larger_graph_vs_jacobi_oracle(dag):
    g = I.rmat(14, 16, seed=12)
    w, t, c = _problem(g, 6, 512)
    plan = dag.Plan.from_graph(g, "cuda")
    model = dag.WeightedPageRank(plan, tol=1e-7, variant="delayed", delta=64)
    r, val, s, st = model.forward(torch.from_numpy(w).cuda(), torch.from_numpy(t.astype(np.float32)).cuda())
    assert st["converged"]
    gw, gt, _, st2 = model.backward(val, s, r, torch.from_numpy(c.astype(np.float32)).cuda())
    assert st2["converged"]
    val64, s64 = oracle.normalize(g, w.astype(np.float64))
    rr = oracle.pagerank_fixed_point(g, 0.85, t, val64)
    lam, _ = oracle.pagerank_adjoint(g, val64, c, 0.85, tol=1e-14)
    gw_ref, gt_ref = oracle.pagerank_grads(g, val64, s64, 0.85, rr, lam)
    assert _rel(gw.cpu().numpy(), gw_ref) <= 1e-4
    assert _rel(gt.cpu().numpy(), gt_ref) <= 1e-4


@pytest.fixture(scope="module")
def scaled_case(dag):
    g = I.rmat(14, 16, seed=12)
    w, t, c = _problem(g, 6, 512)
    val64, s64 = oracle.normalize(g, w.astype(np.float64))
    rr = oracle.pagerank_fixed_point(g, 0.85, t, val64)
    lam, _ = oracle.pagerank_adjoint(g, val64, c, 0.85, tol=1e-14)
    gw_ref, gt_ref = oracle.pagerank_grads(g, val64, s64, 0.85, rr, lam)
    return g, w, t, c, gw_ref, gt_ref


@pytest.mark.parametrize("alpha", [1e-6, 1e6])
@pytest.mark.parametrize("variant,delta,reads", [("async", 0, "refresh"), ("delayed", 64, "refresh"),
                                                 ("async", 0, "warp+cached"), ("async", 0, "ordered+cached")])
def test_adjoint_gradients_scale_with_c(dag, scaled_case, variant, delta, reads, alpha):
    # The adjoint is linear in c and stops relative to ||c||_1, so c -> alpha c scales both
    # gradients by alpha. The asynchronous and delayed sweeps keep the live sum of lambda in
    # fixed point with a unit set from ||c||_1; this checks that unit far from ||c||_1 ~ 1.
    g, w, t, c, gw_ref, gt_ref = scaled_case
    plan = dag.Plan.from_graph(g, "cuda")
    model = dag.WeightedPageRank(plan, tol=1e-7, variant=variant, delta=delta, reads=reads)
    r, val, s, st = model.forward(torch.from_numpy(w).cuda(), torch.from_numpy(t.astype(np.float32)).cuda())
    assert st["converged"]
    gw, gt, _, st2 = model.backward(val, s, r, torch.from_numpy((c * alpha).astype(np.float32)).cuda())
    assert st2["converged"]
    assert _rel(gw.double().cpu().numpy() / alpha, gw_ref) <= 1e-4
    assert _rel(gt.double().cpu().numpy() / alpha, gt_ref) <= 1e-4


def test_adjoint_refuses_flags_it_does_not_take(dag):
    g = I.rmat(10, 16, seed=1)
    plan = dag.Plan.from_graph(g, "cuda")
    model = dag.WeightedPageRank(plan, tol=1e-6, variant="async", delta=0)
    w, t, c = _problem(g, 2, 16)
    r, val, s, _ = model.forward(torch.from_numpy(w).cuda())
    for reads in ("frontier", "local"):
        model.adjoint_reads = reads
        with pytest.raises(dag.DagError):
            model.backward(val, s, r, torch.from_numpy(c.astype(np.float32)).cuda())


def test_transpose_and_normalize_match_definitions(dag):
    g = I.rmat(12, 16, seed=14)
    plan = dag.Plan.from_graph(g, "cuda")
    orow, ocol, perm = dag.transpose(plan)
    src, dst = g.edges()
    order = np.lexsort((dst, src))
    assert np.array_equal(perm.cpu().numpy(), order)
    assert np.array_equal(ocol.cpu().numpy(), dst[order])
    assert np.array_equal(orow.cpu().numpy(), np.concatenate([[0], np.cumsum(np.bincount(src, minlength=g.n))]))
    w = I.weights_f32(g, 3)
    val, s = dag.normalize_weights(plan, torch.from_numpy(w).cuda())
    v64, s64 = oracle.normalize(g, w.astype(np.float64))
    assert np.max(np.abs(val.cpu().numpy() - v64)) <= 1e-6
    has = s64 > 0
    assert np.max(np.abs(s.cpu().numpy()[has] - s64[has]) / s64[has]) <= 1e-5



def test_normalize_hubs_and_repeat(dag):
    # Sources past the warp-sized sum (one of 6000 out-edges, one of exactly 2048 and one of 2049)
    # beside ordinary ones: every s[u] within FP32 rounding of the fp64 definition, and a second
    # call on the same weights gives the same bits (a fixed summation order).
    rng = np.random.default_rng(21)
    n = 8000
    src = [np.zeros(6000, np.int64), np.full(2048, 1), np.full(2049, 2), rng.integers(3, n, 40000)]
    dst = [rng.choice(np.arange(1, n), 6000, replace=False), rng.choice(np.arange(3, n), 2048, replace=False),
           rng.choice(np.arange(3, n), 2049, replace=False), rng.integers(0, n, 40000)]
    src, dst = np.concatenate(src), np.concatenate(dst)
    keep = src != dst
    g = I.from_edges(n, src[keep], dst[keep], "hubs8000")
    plan = dag.Plan.from_graph(g, "cuda")
    w = I.weights_f32(g, 9)
    wd = torch.from_numpy(w).cuda()
    val, s = dag.normalize_weights(plan, wd)
    v64, s64 = oracle.normalize(g, w.astype(np.float64))
    has = s64 > 0
    assert np.max(np.abs(s.cpu().numpy()[has] - s64[has]) / s64[has]) <= 1e-5
    assert np.max(np.abs(val.cpu().numpy() - v64)) <= 1e-6
    val2, s2 = dag.normalize_weights(plan, wd)
    assert torch.equal(s, s2) and torch.equal(val, val2)
    # new weights on the kept order
    w3 = I.weights_f32(g, 10)
    val3, s3 = dag.normalize_weights(plan, torch.from_numpy(w3).cuda())
    v64, s64 = oracle.normalize(g, w3.astype(np.float64))
    assert np.max(np.abs(val3.cpu().numpy() - v64)) <= 1e-6

@pytest.mark.parametrize("variant,delta,reads", FORMS)
def test_adjoint_deflation_cuts_the_slow_mode(dag, scaled_case, variant, delta, reads):
    # The adjoint's slow error mode along 1 (B 1 = d 1) is deflated after every sweep, so the
    # adjoint solve needs far fewer sweeps than the plain Jacobi adjoint at the same tolerance
    # (the oracle, which does not deflate), and its gradients stay within the dense bound.
    g, w, t, c, gw_ref, gt_ref = scaled_case
    plan = dag.Plan.from_graph(g, "cuda")
    model = dag.WeightedPageRank(plan, tol=1e-6, variant=variant, delta=delta, reads=reads)
    r, val, s, st = model.forward(torch.from_numpy(w).cuda(), torch.from_numpy(t.astype(np.float32)).cuda())
    gw, gt, _, st2 = model.backward(val, s, r, torch.from_numpy(c.astype(np.float32)).cuda())
    assert st2["converged"]
    val64, _ = oracle.normalize(g, w.astype(np.float64))
    _, jacobi_sweeps = oracle.pagerank_adjoint(g, val64, c, 0.85, tol=1e-6)
    assert st2["iters"] <= jacobi_sweeps // 2, (st2["iters"], jacobi_sweeps)
    assert st2["iters"] <= 2 * st["iters"]
    assert _rel(gw.cpu().numpy(), gw_ref) <= 1e-4
    assert _rel(gt.cpu().numpy(), gt_ref) <= 1e-4


def test_normalisation_and_edge_gradients_at_the_kernels_edges(dag):
    # sources of 0, 1, 8, 63 .. 65, 2047 .. 2049 and 5000 out-edges (eight lanes, a warp, a block per source); in-edge
    # tiles inside one row, with runs of empty rows, and ending at a row's end
    n = 6000
    degs = {0: 1, 1: 8, 2: 63, 3: 64, 4: 65, 5: 2047, 6: 2048, 7: 2049, 8: 5000}
    rng = np.random.default_rng(4)
    src = np.concatenate([np.full(k, u) for u, k in degs.items()] + [np.arange(9, 5400)])
    dst = np.concatenate([rng.permutation(np.arange(9, n))[:k] for k in degs.values()] + [np.full(5391, 5999)])
    keep = src != dst
    g = I.from_edges(n, src[keep], dst[keep])
    plan = dag.Plan.from_graph(g, "cuda")
    w = torch.rand(g.m, generator=torch.Generator().manual_seed(1)).add_(0.1).cuda()
    val, s = dag.normalize_weights(plan, w)
    col = plan.colidx.long()
    ref = torch.zeros(n, dtype=torch.float64, device="cuda").index_add_(0, col, w.double())
    # a source's FP32 sum of k terms: at most 160 additions in a row, 160 * 2^-24 < 1e-5
    assert torch.allclose(s.double(), ref, rtol=1e-5, atol=0)
    assert torch.allclose(val.double(), w.double() / ref[col], rtol=2e-5, atol=0)
    val2, s2 = dag.normalize_weights(plan, w)
    assert torch.equal(s, s2) and torch.equal(val, val2)
    orow, ocol, perm = dag.transpose(plan)
    out_plan = dag.Plan(orow, ocol)
    r, _ = dag.pagerank(plan, 0.85, 1e-6, "sync", 0, val=val)
    c = torch.rand(n, generator=torch.Generator().manual_seed(2)).cuda()
    gw, gt, lam, _ = dag.pagerank_adjoint(plan, out_plan, val, val[perm.long()].contiguous(), s, r, c, 0.85, 1e-7, "sync",
                                          0, want_lambda=True)
    dst_of = torch.repeat_interleave(torch.arange(n, device="cuda"), (plan.rowptr[1:] - plan.rowptr[:-1]).long())
    lam64, val64 = lam.double(), val.double()
    mt = torch.zeros(n, dtype=torch.float64, device="cuda").index_add_(0, col, val64 * lam64[dst_of])
    want = 0.85 * (r.double() / s.double())[col] * (lam64[dst_of] - mt[col])
    # lambda and M^T lambda are FP32 values of size max|lambda|: their difference is good to a few of their roundings,
    # and the sweep's M^T lambda is of the iterate before, 1e-7 of |c|_1 = n / 2 away at most
    scale = float((r / s).nan_to_num(0, 0, 0)[col].abs().max()) * float(lam.abs().max())
    assert float((gw.double() - want).abs().max()) <= 2e-4 * scale
    assert torch.allclose(gt, 0.15 * lam, rtol=1e-6, atol=0)
