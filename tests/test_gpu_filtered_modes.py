"""GPU: the filtered pull on both sides of the share of edges (a fifth) from which its chunks go
in groups of lanes, with chunks of every kind (short, long, split), rows that stop early and
rows that never do, against the oracle and the SlimWork pass's levels."""
import numpy as np
import pytest
import torch

import graphgen as gg
import oracle
import paper_2010_09913_gb300 as ss

pytestmark = pytest.mark.gpu

GRAPHS = [gg.kronecker(12, seed=3), gg.lattice(60, 0.1, seed=4), gg.erdos_renyi(4000, 30.0, seed=5),
          gg.from_edges(1200, [(0, i) for i in range(1, 900)] + [(i, i + 1) for i in range(1, 1199)])]


@pytest.fixture(scope="module", autouse=True)
def _build():
    ss.build()


@pytest.mark.parametrize("C,sigma,w", [(8, None, 4), (16, 64, 64), (32, None, 256), (64, 1, 0)])
@pytest.mark.parametrize("sr", ["tropical", "real", "selmax"])
def test_levels_with_few_and_many_hits(C, sigma, w, sr):
    shares = []
    for g in GRAPHS:
        G = ss.SlimSellGraph.from_host(g.row_ptr, g.col, C=C, sigma=sigma or g.n, split_w=w)
        for r in sorted({0, g.n - 1, int(gg.roots(g, 1, seed=6)[0])}):
            d = oracle.bfs_queue(g.row_ptr, g.col, r)
            p = oracle.dp(g.row_ptr, g.col, d, r)
            dist, parent = G.bfs(r, sr, "pull_filtered")
            torch.cuda.synchronize()
            np.testing.assert_array_equal(dist.cpu().numpy(), d, err_msg=g.name)
            np.testing.assert_array_equal(parent.cpu().numpy(), p, err_msg=g.name)
            if sr == "real":
                _, _, val, _, _ = oracle.bfs_semiring(g.row_ptr, g.col, r, "real")
                ok = (d >= 0) & (val < 2.0 ** 24)
                np.testing.assert_array_equal(G.values().cpu().numpy()[ok], val[ok])
            st, its = G.run_stats(cap=2048)
            levels = [(its[i].frontier, its[i].frontier_degree, its[i].active_chunks, its[i].slots)
                      for i in range(st.iterations + 1)]
            shares += [lv[1] / g.nnz for lv in levels]
            G.set_option(ss.OPT_SMEM_BYTES, 0)  # (grid-wide, nothing staged)
            G.bfs(r, sr, "slimwork")
            st, its = G.run_stats(cap=2048)
            for i, lv in enumerate(levels):
                assert lv[:3] == (its[i].frontier, its[i].frontier_degree, its[i].active_chunks), (g.name, i)
                assert lv[3] <= its[i].slots  # rows that stop read no more than the whole chunks
            G.set_option(ss.OPT_SMEM_BYTES, 212992)
        G.close()
    assert min(shares) < 0.2 < max(shares)
