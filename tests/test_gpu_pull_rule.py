"""GPU: which pull the frontier-size rule takes: the filtered pass for frontiers that hold a
fifth of the edges, where rows stop early; for the real semiring, whose rows never do, on
graphs that fill the GPU, once seven eighths of the rows are reached.  Results equal the
oracle's either way."""
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


@pytest.mark.parametrize("make,C,w", [(lambda: gg.kronecker(17, seed=2), 8, 64), (lambda: gg.kronecker(17, seed=2), 64, 0),
                                      (lambda: gg.erdos_renyi(200000, 16.0, seed=3), 8, 64)])
def test_rule_by_semiring(make, C, w):
    g = make()
    live = int((np.diff(g.row_ptr) > 0).sum())
    G = ss.SlimSellGraph.from_host(g.row_ptr, g.col, C=C, sigma=g.n, split_w=w)
    full = G.info().n_items >= 128 * 152
    pulls = 0
    for r in gg.roots(g, 3, seed=5):
        d = oracle.bfs_queue(g.row_ptr, g.col, int(r))
        p = oracle.dp(g.row_ptr, g.col, d, int(r))
        for sr in ("real", "boolean"):
            dist, parent = G.bfs(int(r), sr, "heuristic")
            torch.cuda.synchronize()
            np.testing.assert_array_equal(dist.cpu().numpy(), d)
            np.testing.assert_array_equal(parent.cpu().numpy(), p)
            st, its = G.run_stats(cap=64)
            reached = 0
            for i in range(1, st.iterations + 1):
                reached += its[i - 1].frontier
                if its[i].variant not in (ss.V_SLIMWORK, ss.V_PULL_FILTERED):
                    continue
                pulls += 1
                filtered = 8 * reached >= 7 * live if sr == "real" and full else 5 * its[i - 1].frontier_degree >= g.nnz
                assert (its[i].variant == ss.V_PULL_FILTERED) == filtered, (sr, i, reached, its[i - 1].frontier_degree)
    assert pulls >= 3
    G.close()
