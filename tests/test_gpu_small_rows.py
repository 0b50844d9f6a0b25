"""GPU: runs in one launch by the number of rows, on both sides of the limits (8,192 rows with
a neighbour, 512 K slots, items of 16 K, 32 K slots), against the oracle and the
grid-wide path (which the staged-prefix option forces)."""
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


def with_isolated(g, extra):
    """g and `extra` rows without neighbours after it."""
    row_ptr = np.concatenate([g.row_ptr, np.full(extra, g.row_ptr[-1])])
    return type(g)(g.n + extra, row_ptr, g.col, g.name + "+isolated")


GRAPHS = [gg.kronecker(10, seed=1), gg.kronecker(13, seed=2), gg.erdos_renyi(8192, 16.0, seed=3),
          gg.erdos_renyi(8200, 16.0, seed=4), gg.erdos_renyi(8000, 68.0, seed=5),  # 544 K slots
          gg.lattice(90, 0.0, seed=6), gg.lattice(91, 0.0, seed=7),  # 8,100 and 8,281 rows
          gg.from_edges(16000, [(i, i + 1) for i in range(60)] + [(i, i + 1) for i in range(100, 15999, 2)]),
          with_isolated(gg.kronecker(11, seed=8), 3001)]


@pytest.mark.parametrize("C,sigma,w", [(8, None, 64), (32, None, 256), (32, 256, 256), (64, 1, 4096), (64, None, 256)])
@pytest.mark.parametrize("sr,policy", [("tropical", "slimwork"), ("real", "slimwork"), ("selmax", "full")])
def test_runs_by_rows_match_oracle_and_grid(C, sigma, w, sr, policy):
    for g in GRAPHS:
        G = ss.SlimSellGraph.from_host(g.row_ptr, g.col, C=C, sigma=sigma or g.n, split_w=w)
        live = np.flatnonzero(np.diff(g.row_ptr))
        for r in (int(live[0]), int(live[-1]), g.n - 1):
            d = oracle.bfs_queue(g.row_ptr, g.col, r)
            p = oracle.dp(g.row_ptr, g.col, d, r)
            seen = []
            for smem in (212992, 0):
                G.set_option(ss.OPT_SMEM_BYTES, smem)
                dist, parent = G.bfs(r, sr, policy)
                st, it = G.run_stats(256)
                np.testing.assert_array_equal(dist.cpu().numpy(), d, err_msg=g.name)
                np.testing.assert_array_equal(parent.cpu().numpy(), p, err_msg=g.name)
                if sr == "real":
                    _, _, val, _, _ = oracle.bfs_semiring(g.row_ptr, g.col, r, "real")
                    ok = (d >= 0) & (val < 2.0 ** 24)
                    np.testing.assert_array_equal(G.values().cpu().numpy()[ok], val[ok])
                seen.append((st.iterations, st.reached, st.reached_degree, st.slots,
                             [(it[i].frontier, it[i].active_chunks) for i in range(min(st.iterations + 1, 256))]))
            assert seen[0] == seen[1], g.name
        G.close()
