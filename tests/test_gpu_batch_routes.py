"""GPU: batches on both sides of the rule that runs a graph as one cluster or as a loop of
grid-wide launches: a larger graph alone, in company that leaves the GPU room, and in
company that fills it, with small graphs beside it, against the oracle."""
import numpy as np
import pytest
import torch

import graphgen as gg
import oracle
import paper_2010_09913_gb300 as ss

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    ss.build()


@pytest.mark.parametrize("large,C", [("uniform", 32), ("lattice", 16), ("items", 64)])
@pytest.mark.parametrize("copies,small", [(1, 0), (1, 30), (9, 3), (24, 2)])
def test_routes_match_oracle(large, C, copies, small):
    # past the sizes that are a cluster in any company: 1.3 M slots, 80,000 rows; 0.6 M, 160,000
    # and items of more than 16 K slots
    big = {"uniform": lambda: gg.erdos_renyi(80000, 16.0, seed=2), "lattice": lambda: gg.lattice(400, 0.05, seed=3),
           "items": lambda: gg.kronecker(13, seed=4)}[large]()
    w = 4096 if large == "items" else 256
    graphs = [big] * copies + [gg.kronecker(9, seed=40 + i) for i in range(small)]
    Gs = [ss.SlimSellGraph.from_host(g.row_ptr, g.col, C=C, sigma=g.n, split_w=w) for g in graphs]
    for sr in ("tropical", "selmax"):
        b = ss.slimsell_batch_create([G.h for G in Gs], ss.SEMIRINGS[sr], ss.V_SLIMWORK)
        roots = [int(gg.roots(g, copies + 1, seed=7)[i % copies]) for i, g in enumerate(graphs)]
        dists = [torch.empty(g.n, dtype=torch.int32, device="cuda") for g in graphs]
        pars = [torch.empty(g.n, dtype=torch.int32, device="cuda") for g in graphs]
        ss.slimsell_batch_run(b, torch.tensor(roots, dtype=torch.int32, device="cuda"), dists, pars)
        for g, r, dd, pp, st in zip(graphs, roots, dists, pars, ss.slimsell_batch_get_stats(b, len(graphs))):
            d = oracle.bfs_queue(g.row_ptr, g.col, r)
            np.testing.assert_array_equal(dd.cpu().numpy(), d, err_msg=g.name)
            np.testing.assert_array_equal(pp.cpu().numpy(), oracle.dp(g.row_ptr, g.col, d, r), err_msg=g.name)
            assert st.reached == int((d >= 0).sum())
        ss.slimsell_batch_destroy(b)
    for G in Gs:
        G.close()
