"""What a program does with this framework, as cases that can be timed and compared.

Each case is one call (or one forward and backward pass) through the public entry points of
paper_2110_01409_gb300.dag on a synthetic graph: RMAT (a = .57, b = c = .19; a social or web graph's skew),
uniform random ("er") or banded (15 in-edges within +-1024 and one uniform; a clustered graph), 16 in-edges per
vertex before duplicates go. The graph, the weights and the plan are what a program holds before the call; the
plan's own per-shape tables are built by its first solve, as in a user's program.
"""
import torch

from paper_2110_01409_gb300 import dag

D, TOL, DEG = 0.85, 1e-6, 16

# (variant, delta, reads): the forms a program runs, the library's default first.
PR_FORMS = (("delayed", 256, "refresh"), ("delayed", 32, "cached"), ("async", 0, "refresh"), ("async", 0, "ordered+cached"),
            ("async", 0, "warp+cached"), ("sync", 0, "refresh"), ("sync", 0, "warp"), ("delayed", 256, "warp"))
BF_FORMS = (("delayed", 32, "refresh"), ("async", 0, "refresh"), ("async", 0, "own_l1+frontier"), ("async", 0, "warp+frontier"),
            ("async", 0, "ordered+cached+frontier"), ("sync", 0, "frontier"), ("sync", 0, "warp"), ("delayed", 256, "warp+cached"))
FIELDS = ("op", "graph", "n", "variant", "delta", "reads", "tile", "weights", "teleport", "columns")


def _case(op, graph, n, form=("async", 0, "refresh"), tile=7, weights="", teleport=False, columns=0, name=None):
    c = dict(zip(FIELDS, (op, graph, n) + tuple(form) + (tile, weights, teleport, columns)))
    return c if name is None else dict(c, name=name)


def listed():
    big, mid = 1 << 22, 1 << 21
    return [
        # the smallest calls: a service ranking or routing over a small graph on every request; latency counts
        _case("pagerank", "rmat", 1024, PR_FORMS[0], name="pagerank_small"),
        _case("sssp", "rmat", 1000, BF_FORMS[0], weights="u32", name="sssp_small"),
        # ordinary calls with the library's default form, and with the tile frontier, on odd sizes
        _case("pagerank", "rmat", 200_003, PR_FORMS[0], name="pagerank_default"),
        _case("sssp", "er", 300_007, BF_FORMS[2], weights="u32", name="sssp_frontier"),
        # the synchronous baseline with a personalised teleport, on a graph without skew
        _case("pagerank", "er", mid, PR_FORMS[6], teleport=True, name="pagerank_sync"),
        # large graphs with the forms the tuner picks: one in-order stream; the warp-tile frontier; warp runs
        _case("pagerank", "rmat", big, PR_FORMS[3], tile=11, name="pagerank_ordered"),
        _case("sssp", "rmat", big, BF_FORMS[4], weights="u8", name="sssp_ordered_frontier"),
        _case("pagerank", "banded", big, PR_FORMS[4], name="pagerank_banded"),
        # many personalised rankings or sources in one call: the largest states; a ragged batch
        _case("ppr_batched", "rmat", 1 << 20, columns=256, name="ppr_batched_256"),
        _case("sssp_batched", "rmat", 1 << 20, weights="u8", columns=64, name="sssp_batched_64"),
        _case("ppr_batched", "rmat", 100_003, columns=20, name="ppr_batched_20"),
        # learning edge weights: forward and backward of weighted PageRank
        _case("weighted", "rmat", mid, PR_FORMS[4], name="weighted_forward_backward"),
    ]


def draw(rng):
    op = rng.choice(("pagerank", "pagerank", "sssp", "sssp", "ppr_batched", "sssp_batched", "weighted"))
    batched = op.endswith("batched")
    graph = rng.choice(("rmat", "er") if batched else ("rmat", "rmat", "er", "banded"))
    n = int(2 ** rng.uniform(13 if graph == "banded" else 12 if op == "weighted" else 9, 21 if op == "weighted" else 22 if not batched else 19))
    if batched:
        columns = int(2 ** rng.uniform(0, 8.02))
        columns = max(1, min(columns, (1 << 26) // n))
        return _case(op, graph, n, rng.choice((("async", 0, "refresh"), ("async", 0, "refresh"), ("sync", 0, "refresh"), ("delayed", 16, "refresh"))),
                     weights=rng.choice(("u8", "u32")) if op == "sssp_batched" else "", columns=columns)
    if op == "sssp":
        return _case(op, graph, n, rng.choice(BF_FORMS), tile=rng.choice((5, 7, 11)), weights=rng.choice(("u8", "u32")))
    if op == "weighted":
        return _case(op, graph, n, rng.choice((("delayed", 256, "refresh"), ("async", 0, "refresh"), ("async", 0, "warp+cached"), ("sync", 0, "warp"))))
    return _case(op, graph, n, rng.choice(PR_FORMS), tile=rng.choice((5, 7, 11)), teleport=rng.random() < 0.5)


def _graph(kind, n, gen, edges=0):
    """In-edge CSR (rowptr, colidx, int32, sorted within a row) without loops and duplicates; `edges`: exactly
    so many, picked at random from three times DEG draws per vertex."""
    deg, dev = 3 * DEG if edges else DEG, "cuda"
    m = n * deg
    if kind == "rmat":
        bits = max(1, (n - 1).bit_length())
        src = torch.zeros(m, dtype=torch.int32, device=dev)
        dst = torch.zeros(m, dtype=torch.int32, device=dev)
        for _ in range(bits):
            r = torch.rand(m, generator=gen, device=dev)
            src.mul_(2).add_(r >= 0.76)
            dst.mul_(2).add_(((r >= 0.57) & (r < 0.76)) | (r >= 0.95))
        src, dst = src.long(), dst.long()
        keep = (src < n) & (dst < n) & (src != dst)
        key = (dst * n + src)[keep]
    elif kind == "er":
        src = torch.randint(0, n, (m,), generator=gen, device=dev)
        dst = torch.randint(0, n, (m,), generator=gen, device=dev)
        key = (dst * n + src)[src != dst]
    else:
        dst = torch.arange(n, device=dev).repeat_interleave(deg)
        off = torch.randint(1, 1025, (m,), generator=gen, device=dev) * (torch.randint(0, 2, (m,), generator=gen, device=dev) * 2 - 1)
        src = torch.remainder(dst + off, n)
        src[::deg] = torch.randint(0, n, (n,), generator=gen, device=dev)
        key = (dst * n + src)[src != dst]
    key = torch.unique(key)
    if edges:
        if key.numel() < edges:
            raise ValueError("too few distinct edges")
        key = key[torch.randperm(key.numel(), generator=gen, device=dev)[:edges]].sort().values
    dst = torch.div(key, n, rounding_mode="floor")
    rowptr = torch.zeros(n + 1, dtype=torch.int32, device=dev)
    rowptr[1:] = torch.cumsum(torch.bincount(dst, minlength=n), 0).int()
    return rowptr, (key - dst * n).int()


def _inputs(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    n = case["n"]
    # per-edge outputs (gradients) have one shape for every seed, so the weighted graphs have exactly n DEG edges
    rowptr, colidx = _graph(case["graph"], n, gen, n * DEG if case["op"] == "weighted" else 0)
    m = colidx.numel()
    x = {"rowptr": rowptr, "colidx": colidx}
    if case["weights"]:  # uniform in [1, 255]
        x["w"] = torch.randint(1, 256, (m,), generator=gen, device="cuda", dtype=torch.int32).to(
            torch.uint8 if case["weights"] == "u8" else torch.int32)
        pick = torch.randint(0, m, (max(1, case["columns"]),), generator=gen, device="cuda")
        x["src"] = colidx[pick].contiguous()  # vertices with an out-edge
    if case["teleport"] or case["op"] == "weighted":
        t = torch.rand(n, generator=gen, device="cuda", dtype=torch.float64) + 0.1
        x["t"] = (t / t.sum()).float()
    if case["op"] == "weighted":  # weights in (0, 1]; the loss looks at 4,096 vertices
        x["w"] = 1.0 - torch.rand(m, generator=gen, device="cuda")
        c = torch.zeros(n, device="cuda")
        at = torch.randperm(n, generator=gen, device="cuda")[:4096]
        c[at] = torch.randn(at.numel(), generator=gen, device="cuda")
        x["c"] = c
    if case["op"] == "ppr_batched":  # 1 to 64 seed vertices per column, equal shares
        B = case["columns"]
        k = torch.randint(1, 65, (B,), generator=gen, device="cuda")
        V = torch.zeros(n, B, device="cuda")
        for j in range(64):
            v = torch.randint(0, n, (B,), generator=gen, device="cuda")
            V[v, torch.arange(B, device="cuda")] += torch.where(k > j, 1.0 / k, torch.zeros_like(k, dtype=torch.float32))
        x["V"] = V
    return x


def prepare(case, seed):
    x = _inputs(case, seed)
    s = dict(x, case=case, plan=dag.Plan(x["rowptr"], x["colidx"]))
    s["plan"].set_warp_tile(case["tile"])
    s["form"] = dict(variant=case["variant"], delta=case["delta"])
    if case["op"] == "sssp":
        s["src"] = int(x["src"][0])
    if case["op"] == "weighted":
        s["model"] = dag.WeightedPageRank(s["plan"], D, TOL, reads=case["reads"], **s["form"])
        s["w"].requires_grad_(True)
        s["t"].requires_grad_(True)
    return s


def run(s):
    op, plan, form = s["case"]["op"], s["plan"], s["form"]
    if op == "pagerank":
        return dag.pagerank(plan, D, TOL, teleport=s.get("t"), reads=s["case"]["reads"], **form)[0]
    if op == "sssp":
        return dag.sssp(plan, s["src"], s["w"], reads=s["case"]["reads"], **form)[0]
    if op == "ppr_batched":
        return dag.ppr_batched(plan, s["V"], D, TOL, **form)[0]
    if op == "sssp_batched":
        return dag.sssp_batched(plan, s["src"], s["w"], **form)[0]
    r = dag.PageRankFn.apply(s["w"], s["t"], s["model"])
    gw, gt = torch.autograd.grad(r, (s["w"], s["t"]), s["c"])
    return {"rank": r.detach(), "grad_w": gw, "grad_t": gt}


def work(case):
    n, B = case["n"], max(1, case["columns"])
    m = n * DEG
    csr = 4 * (n + 1) + 4 * m
    if case["op"] == "weighted":  # weights, teleport and loss gradient in; ranks and both gradients out
        return {"bytes": csr + 4 * m + 8 * n + 8 * n + 4 * m, "flops": 8 * m}
    w = {"": 0, "u8": 1, "u32": 4}[case["weights"]] * m
    dense = 4 * n * B * (2 if case["op"] == "ppr_batched" else 1)
    return {"bytes": csr + w + dense + (4 * n if case["teleport"] else 0), "flops": 2 * m * B}


def tolerance(case):
    if case["op"].startswith("sssp"):
        return "exact"
    # The stopping rule leaves up to d / (1 - d) tol of L1 error: against 64 bits the forms end 1e-7 to 3e-6 off in
    # the 2-norm (banded graphs furthest). Edge gradients are differences of nearly equal adjoint values: 1e-5.
    if case["op"] == "weighted":
        return {"rel": 4e-5, "max": 1e-2}
    return {"rel": 1.5e-5, "max": 5e-4}


def _fixed_point(mat, dangling, base, n):
    """x = base + D (mat x + dangling mass / n) in 64 bits, to a change of 1e-13 of the largest column."""
    x = base.clone()
    for _ in range(400):
        y = base + D * (mat @ x + x[dangling].sum(0, keepdim=True) / n)
        change = float((y - x).abs().sum(0).max() / base.abs().sum(0).max())
        x = y
        if change < 1e-13:
            break
    return x


def exact(case, seed):
    if case["op"].startswith("sssp"):
        return None
    x = _inputs(case, seed)
    n, rowptr, col = case["n"], x["rowptr"].long(), x["colidx"].long()
    m = col.numel()
    dst = torch.repeat_interleave(torch.arange(n, device="cuda"), rowptr[1:] - rowptr[:-1])
    deg = torch.bincount(col, minlength=n)
    w = x["w"].double() if case["op"] == "weighted" else torch.ones(m, dtype=torch.float64, device="cuda")
    s = torch.zeros(n, dtype=torch.float64, device="cuda").index_add_(0, col, w)
    val = w / s[col]
    mat = torch.sparse_csr_tensor(rowptr, col, val, (n, n))
    t = x["V"].double() if "V" in x else x["t"].double()[:, None] if "t" in x else torch.full((n, 1), 1.0 / n, dtype=torch.float64, device="cuda")
    r = _fixed_point(mat, deg == 0, (1 - D) * t, n)
    if case["op"] == "ppr_batched":
        return r
    r = r[:, 0]
    if case["op"] == "pagerank":
        return r
    # the adjoint: lam = c + D M^T lam + D [dangling] (sum lam) / n, over the out-edges
    order = torch.argsort(col, stable=True)
    orow = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    orow[1:] = torch.cumsum(deg, 0)
    mt = torch.sparse_csr_tensor(orow, dst[order], val[order], (n, n))
    c, hang = x["c"].double(), (deg == 0).double()
    lam = c.clone()
    for _ in range(400):
        new = c + D * ((mt @ lam[:, None])[:, 0] + hang * (lam.sum() / n))
        change = float((new - lam).abs().sum() / c.abs().sum())
        lam = new
        if change < 1e-13:
            break
    back = (mt @ lam[:, None])[:, 0]
    return {"rank": r, "grad_w": D * (r / s)[col] * (lam[dst] - back[col]), "grad_t": (1 - D) * lam}
