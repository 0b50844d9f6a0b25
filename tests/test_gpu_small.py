"""GPU: whole runs in one launch (small graphs, fixed policies), at the sizes where
the cluster changes, against the oracle and against the grid-wide path (which the
staged-prefix option forces)."""
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


def graphs():
    return [gg.from_edges(2, [(0, 1)]), gg.from_edges(9, [(i, i + 1) for i in range(7)]),  # 8 is isolated
            gg.from_edges(700, [(0, i) for i in range(1, 600)]), gg.lattice(40, 0.05, seed=3),
            gg.erdos_renyi(1800, 16.0, seed=4), gg.kronecker(10, seed=5)]


@pytest.mark.parametrize("C,sigma,w", [(8, 16, 4), (16, 1, 0), (32, None, 64), (64, 128, 16)])
@pytest.mark.parametrize("sr", ["tropical", "real", "boolean", "selmax"])
def test_whole_run_matches_oracle_and_grid(C, sigma, w, sr):
    for g in graphs():
        G = ss.SlimSellGraph.from_host(g.row_ptr, g.col, C=C, sigma=sigma or g.n, split_w=w)
        for r in sorted({0, g.n - 1, g.n // 2}):
            d = oracle.bfs_queue(g.row_ptr, g.col, r)
            p = oracle.dp(g.row_ptr, g.col, d, r)
            seen = []
            for policy, smem in [("slimwork", 212992), ("full", 212992), ("slimwork", 0)]:
                G.set_option(ss.OPT_SMEM_BYTES, smem)  # 0: nothing staged, so the grid-wide path
                dist, parent = G.bfs(r, sr, policy)
                st, it = G.run_stats(64)
                np.testing.assert_array_equal(dist.cpu().numpy(), d, err_msg=g.name)
                np.testing.assert_array_equal(parent.cpu().numpy(), p, err_msg=g.name)
                if sr == "real":
                    _, _, val, _, _ = oracle.bfs_semiring(g.row_ptr, g.col, r, "real")
                    ok = (d >= 0) & (val < 2.0 ** 24)
                    np.testing.assert_array_equal(G.values().cpu().numpy()[ok], val[ok])
                seen.append((st.iterations, st.reached, st.reached_degree,
                             [it[i].frontier for i in range(min(st.iterations + 1, 64))]))
                if policy == "slimwork":
                    slots = [it[i].slots for i in range(min(st.iterations + 1, 64))]
                    assert smem or slots == ref_slots
                    ref_slots = slots
            assert seen[0] == seen[1] == seen[2]
        G.close()


def test_batch_over_cluster_sizes():
    """Graphs of one to eight CTAs' worth and one that runs grid-wide, side by side."""
    gs = [gg.kronecker(s, seed=20 + s) for s in (6, 9, 11, 13, 15, 18)]
    Gs = [ss.SlimSellGraph.from_host(g.row_ptr, g.col, C=32, sigma=g.n, split_w=256) for g in gs]
    b = ss.slimsell_batch_create([G.h for G in Gs], ss.TROPICAL, ss.V_SLIMWORK)
    for rep in range(2):
        roots = [int(gg.roots(g, 2, seed=rep)[rep]) for g in gs]
        dists = [torch.empty(g.n, dtype=torch.int32, device="cuda") for g in gs]
        pars = [torch.empty(g.n, dtype=torch.int32, device="cuda") for g in gs]
        ss.slimsell_batch_run(b, torch.tensor(roots, dtype=torch.int32, device="cuda"), dists, pars)
        stats = ss.slimsell_batch_get_stats(b, len(gs))
        for g, r, dd, pp, st in zip(gs, roots, dists, pars, stats):
            d = oracle.bfs_queue(g.row_ptr, g.col, r)
            np.testing.assert_array_equal(dd.cpu().numpy(), d, err_msg=g.name)
            np.testing.assert_array_equal(pp.cpu().numpy(), oracle.dp(g.row_ptr, g.col, d, r))
            assert st.reached == int((d >= 0).sum()) and st.iterations == int(d.max()) + 1
    ss.slimsell_batch_destroy(b)
    for G in Gs:
        G.close()
