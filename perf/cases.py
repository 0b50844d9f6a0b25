"""The work that a user of this framework has it do, as measurable cases.

A case names a graph family and size, a layout (C, sigma, split width) and one
public call on it:

  bfs            SlimSellGraph.bfs: distances and parents of one root (and, for
                 the real semiring, SlimSellGraph.values: the path counts)
  multi          SlimSellGraph.bfs_multi: k bit-packed sources, distances
  multi_parents  SlimSellGraph.bfs_multi_parents: k sources, distances and parents
  bc             SlimSellGraph.bc: betweenness centrality over k sources
  batch          slimsell_batch_run: one BFS on each of `graphs` graphs, one launch
  build          SlimSellGraph(...) from a CSR on the device, the layout's tables
                 (slimsell_export_layout), one BFS, close

Graphs are the families of the benchmark and the tests (Graph500 Kronecker with
edge factor 16, G(n, 8n), L x L lattices with 5 % of the edges deleted), drawn
on the GPU from the seed.  A BFS case keeps what a user's program keeps between
roots: the built handle and the output buffers.

Left out: the learned policy (it runs the heuristic policy's kernels, chosen by
a network that has to be trained first), the Sell-C-sigma format (a comparison
against SlimSell), and the statistics and profiling calls.
"""
import math

import torch

import paper_2010_09913_gb300 as ss

DEV = "cuda"


def listed():
    kron = dict(family="kron", C=32, sigma=0, split_w=256)  # sigma 0: a global sort
    return [
        # the smallest call: a graph of a thousand vertices, all launches and latency
        dict(kron, name="bfs kron10 tropical", call="bfs", scale=10, semiring="tropical", policy="slimwork",
             split_w=64),
        # the paper's method on the benchmark graph, one root (the benchmark repeats it)
        dict(kron, name="bfs kron22 tropical", call="bfs", scale=22, semiring="tropical", policy="slimwork"),
        # the same over the real semiring, whose path counts the user reads as well
        dict(kron, name="bfs kron22 real", call="bfs", scale=22, semiring="real", policy="slimwork"),
        # a graph whose bitmap and vectors are well past shared memory: the roofline point
        dict(kron, name="bfs kron24 selmax", call="bfs", scale=24, semiring="selmax", policy="slimwork"),
        # a user who only wants the BFS, as fast as it goes: the per-level choice of variant
        dict(kron, name="bfs kron22 adaptive", call="bfs", scale=22, semiring="boolean", policy="heuristic"),
        # no hubs, an odd number of vertices, a sorting window and a narrower chunk
        dict(name="bfs er4M adaptive", call="bfs", family="er", n=4000037, C=16, sigma=4096, split_w=256,
             semiring="selmax", policy="heuristic"),
        # a road-network-like graph: thousands of small levels
        dict(name="bfs lattice4096 adaptive", call="bfs", family="lattice", L=4096, C=32, sigma=0, split_w=256,
             semiring="tropical", policy="heuristic"),
        # many sources at once: one 64-source word per vertex
        dict(kron, name="multi64 kron22", call="multi", scale=22, k=64),
        # two words, the second one ragged, and every source's parents
        dict(kron, name="multi100 parents kron20", call="multi_parents", scale=20, k=100),
        # betweenness centrality, one full batch of sources
        dict(kron, name="bc64 kron22", call="bc", scale=22, k=64),
        # many small graphs in one launch
        dict(kron, name="batch64 kron10-17", call="batch", lo=10, hi=17, graphs=64, semiring="tropical",
             policy="slimwork"),
        # a new graph arrives: the layout is built, its tables read, one BFS run, all given back
        dict(kron, name="build kron22", call="build", scale=22),
    ]


def draw(rng):
    """One more case of the same ranges."""
    call = rng.choice(["bfs", "bfs", "bfs", "bfs", "multi", "multi_parents", "bc", "batch", "build"])
    case = dict(call=call, C=rng.choice([8, 16, 32, 32, 64]), sigma=rng.choice([0, 0, 4096, 1 << 16]),
                split_w=rng.choice([64, 256, 256, 1024, 4096]))
    if call == "batch":
        lo = rng.randint(9, 13)
        case.update(family="kron", lo=lo, hi=lo + rng.randint(1, 4), graphs=rng.randint(8, 96), sigma=0,
                    semiring=rng.choice(["tropical", "real", "boolean", "selmax"]),
                    policy=rng.choice(["slimwork", "heuristic"]))
        return case
    if call == "bfs":
        case["family"] = rng.choice(["kron", "kron", "er", "lattice"])
        case.update(semiring=rng.choice(["tropical", "real", "boolean", "selmax"]),
                    policy=rng.choice(["slimwork", "slimwork", "heuristic", "heuristic", "full", "push",
                                       "pull_filtered"]))
    else:
        case["family"] = rng.choice(["kron", "er"])
    if call in ("multi", "multi_parents"):
        case["k"] = int(round(2 ** rng.uniform(0, 10)))
        # n * k entries an output
        top = min(22, int((28 if call == "multi" else 27) - math.log2(case["k"])))
    elif call == "bc":
        case["k"] = int(round(2 ** rng.uniform(0, 6)))
        top = 21
    else:
        top = 23
    if case["family"] == "kron":
        case["scale"] = rng.randint(10, top)
    elif case["family"] == "er":
        case["n"] = int(2 ** rng.uniform(10, top)) | 1
    else:  # lattices: the grid-wide policies take tens of microseconds a level
        adaptive = case["policy"] in ("heuristic", "push")
        if case["semiring"] == "real":  # its path counts leave the range of fp32
            case["semiring"] = "tropical"
        case["L"] = int(2 ** rng.uniform(6, 11.9 if adaptive else 9))
    return case


# ---- inputs ------------------------------------------------------------------------------

def _csr(n, u, v):
    """Symmetric CSR without self-loops and duplicates, rows ascending."""
    keep = u != v
    u, v = u[keep], v[keep]
    key = torch.unique(torch.cat([u * n + v, v * n + u]))
    rows = torch.div(key, n, rounding_mode="floor")
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    row_ptr[1:] = torch.bincount(rows, minlength=n).cumsum(0)
    return row_ptr, (key - rows * n).to(torch.int32)


def _kron(scale, g):
    """Kronecker graph, initiator (0.57, 0.19, 0.19, 0.05), 16 edges a vertex, permuted labels."""
    n, m = 1 << scale, 16 << scale
    u = torch.zeros(m, dtype=torch.int64, device=DEV)
    v = torch.zeros(m, dtype=torch.int64, device=DEV)
    for level in range(scale):
        r = torch.rand(m, generator=g, device=DEV)
        u |= (r >= 0.76).to(torch.int64) << level
        v |= (((r >= 0.57) & (r < 0.76)) | (r >= 0.95)).to(torch.int64) << level
    label = torch.randperm(n, generator=g, device=DEV)
    return _csr(n, label[u], label[v])


def _er(n, g):
    return _csr(n, torch.randint(n, (8 * n,), generator=g, device=DEV),
                torch.randint(n, (8 * n,), generator=g, device=DEV))


def _lattice(L, g):
    at = torch.arange(L * L, device=DEV).view(L, L)
    u = torch.cat([at[:, :-1].reshape(-1), at[:-1, :].reshape(-1)])
    v = torch.cat([at[:, 1:].reshape(-1), at[1:, :].reshape(-1)])
    keep = torch.rand(u.numel(), generator=g, device=DEV) >= 0.05
    return _csr(L * L, u[keep], v[keep])


def _graph(case, g):
    if case["family"] == "kron":
        return _kron(case["scale"], g)
    return _er(case["n"], g) if case["family"] == "er" else _lattice(case["L"], g)


def _roots(row_ptr, k, g):
    """k vertices drawn among those with an edge."""
    live = torch.nonzero(row_ptr[1:] > row_ptr[:-1]).view(-1)
    return live[torch.randint(live.numel(), (k,), generator=g, device=DEV)].to(torch.int32)


def _inputs(case, seed):
    """(row_ptr, col, roots) from the seed: what prepare and exact share."""
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    row_ptr, col = _graph(case, g)
    return row_ptr, col, _roots(row_ptr, case.get("k", 1), g)


def _build(case, row_ptr, col):
    return ss.SlimSellGraph(row_ptr, col, C=case["C"], sigma=case["sigma"] or None, split_w=case["split_w"])


def _ints(*shape):
    return torch.empty(shape, dtype=torch.int32, device=DEV)


class _Batch:
    """The graphs of a batch, their outputs side by side in two buffers, and the batch handle."""

    def __init__(self, case, seed):
        g = torch.Generator(device=DEV)
        g.manual_seed(int(seed))
        span = case["hi"] - case["lo"] + 1
        self.graphs, roots = [], []
        for i in range(case["graphs"]):
            row_ptr, col = _kron(case["lo"] + i % span, g)
            roots.append(_roots(row_ptr, 1, g))
            self.graphs.append(_build(case, row_ptr, col))
        self.roots = torch.cat(roots)
        sizes = [G.n for G in self.graphs]
        self.dist, self.parent = _ints(sum(sizes)), _ints(sum(sizes))
        self.dists, self.parents = list(self.dist.split(sizes)), list(self.parent.split(sizes))
        self.b = ss.slimsell_batch_create([G.h for G in self.graphs], ss.SEMIRINGS[case["semiring"]],
                                          ss.POLICIES[case["policy"]])

    def __del__(self):
        ss.slimsell_batch_destroy(getattr(self, "b", None))  # before the handles that it runs on
        for G in getattr(self, "graphs", ()):
            G.close()


def prepare(case, seed):
    call = case["call"]
    if call == "batch":
        return {"case": case, "batch": _Batch(case, seed)}
    row_ptr, col, roots = _inputs(case, seed)
    n = row_ptr.numel() - 1
    if call == "build":
        return {"case": case, "row_ptr": row_ptr, "col": col, "root": int(roots[0])}
    state = {"case": case, "G": _build(case, row_ptr, col)}
    if call == "bfs":
        state.update(root=int(roots[0]), dist=_ints(n), parent=_ints(n))
        if case["semiring"] == "real":
            state["values"] = torch.empty(n, dtype=torch.float32, device=DEV)
    else:
        state["roots"] = roots
        if call != "bc":
            state["dist"] = _ints(n, case["k"])
        if call == "multi_parents":
            state["parent"] = _ints(n, case["k"])
    return state


# ---- one pass ----------------------------------------------------------------------------

def run(state):
    case = state["case"]
    call = case["call"]
    if call == "bfs":
        G = state["G"]
        out = list(G.bfs(state["root"], case["semiring"], case["policy"], state["dist"], state["parent"]))
        if case["semiring"] == "real":
            out.append(G.values(state["values"]))
        return out
    if call == "multi":
        return state["G"].bfs_multi(state["roots"], "slimwork", state["dist"])
    if call == "multi_parents":
        return list(state["G"].bfs_multi_parents(state["roots"], "slimwork", state["dist"], state["parent"]))
    if call == "bc":
        return state["G"].bc(state["roots"])
    if call == "batch":
        b = state["batch"]
        ss.slimsell_batch_run(b.b, b.roots, b.dists, b.parents)
        return [b.dist, b.parent]
    # build: what the new graph gives (col is read through the BFS; the order of the
    # work list is a schedule, not a result, and is not read)
    G = _build(case, state["row_ptr"], state["col"])
    inf = G.info()
    perm, cl = _ints(inf.n_chunks * inf.C), _ints(inf.n_chunks)
    cs = torch.empty(inf.n_chunks + 1, dtype=torch.int64, device=DEV)
    ss.slimsell_export_layout(G.h, perm, cl, cs, None, None)
    dist, parent = G.bfs(state["root"], "tropical", "slimwork")
    out = [dist, parent, perm, cl, cs, inf.slots, inf.padding, inf.n_items, inf.n_split_chunks, inf.max_degree]
    G.close()
    return out


# ---- the work of one pass ----------------------------------------------------------------

def _kron_edges(scale):
    """Directed edges left of 32 a vertex once loops and duplicates are gone (measured, scales 10 .. 22)."""
    return (1 - 0.357 * 0.842 ** (scale - 10)) * (32 << scale)


def _sizes(case):
    """(vertices, directed edges), expected."""
    if case["family"] == "kron":
        return 1 << case["scale"], _kron_edges(case["scale"])
    if case["family"] == "er":
        return case["n"], 16.0 * case["n"]
    return case["L"] ** 2, 4 * 0.95 * case["L"] * (case["L"] - 1)


def work(case):
    """Every neighbour read once, every output written once; centrality adds each
    path count and each dependency over each edge for every source once."""
    call = case["call"]
    if call == "batch":
        scales = [case["lo"] + i % (case["hi"] - case["lo"] + 1) for i in range(case["graphs"])]
        return {"bytes": sum(4 * _kron_edges(s) + 8 * (1 << s) for s in scales), "flops": 0.0}
    n, nnz = _sizes(case)
    k = case.get("k", 1)
    if call == "bfs":
        return {"bytes": 4 * nnz + (12 if case["semiring"] == "real" else 8) * n, "flops": 0.0}
    if call == "multi":
        return {"bytes": 4 * nnz + 4.0 * n * k, "flops": 0.0}
    if call == "multi_parents":
        return {"bytes": 4 * nnz + 8.0 * n * k, "flops": 0.0}
    if call == "bc":
        return {"bytes": 4 * nnz + 8 * n, "flops": nnz * k}
    return {"bytes": 4 * nnz + 8 * n + 4 * nnz + 4 * n + 8 * n, "flops": 0.0}  # the CSR, the layout, dist and parent


# ---- the same in 64 bits -----------------------------------------------------------------

def _adjacency(row_ptr, col):
    one = torch.ones(col.numel(), dtype=torch.float64, device=DEV)
    n = row_ptr.numel() - 1
    return torch.sparse_csr_tensor(row_ptr.to(torch.int32), col, one, (n, n), dtype=torch.float64)


def _levels(A, roots):
    """sigma (shortest-path counts) and level of every vertex from every root, both [n][k]."""
    n, k = A.shape[0], roots.numel()
    at = (roots.long(), torch.arange(k, device=DEV))
    sigma = torch.zeros(n, k, dtype=torch.float64, device=DEV)
    level = torch.full((n, k), -1, dtype=torch.int16, device=DEV)
    sigma[at], level[at] = 1.0, 0
    front, depth = sigma.clone(), 0
    while True:
        x = A @ front
        new = (x > 0) & (level < 0)
        if not bool(new.any()):
            return sigma, level, depth
        depth += 1
        level[new] = depth
        front = torch.where(new, x, 0.0)
        sigma += front


def exact(case, seed):
    call = case["call"]
    if call not in ("bfs", "bc") or (call == "bfs" and case["semiring"] != "real"):
        return None  # whole numbers only
    if case["family"] == "lattice" and case["L"] > 1024:
        return None  # thousands of passes over all edges
    row_ptr, col, roots = _inputs(case, seed)
    A = _adjacency(row_ptr, col)
    if call == "bfs":
        sigma, _, _ = _levels(A, roots)
        return [None, None, sigma.view(-1)]
    sigma, level, depth = _levels(A, roots)
    delta = torch.zeros_like(sigma)
    for d in range(depth - 1, 0, -1):  # Brandes: delta(v) = sigma(v) * sum over w one level down of (1 + delta(w)) / sigma(w)
        t = torch.where(level == d + 1, (1.0 + delta) / sigma, 0.0)
        delta += torch.where(level == d, sigma * (A @ t), 0.0)
    return delta.sum(1)
