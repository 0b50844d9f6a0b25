"""GPU: levels that the grid-wide push takes (more than 131,072 edges), where the rows of a
frontier fold into a neighbour's claim word: parents of every id from 0 on, neighbours that
one, several or all of the frontier's rows reach, neighbours of earlier levels that must
keep theirs, and the real values, for vertex units, block units and both."""
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


def folds(c, leaves, seed):
    """A clique of c rows with ids 0 .. c-1, row c the root next to all of it, and `leaves`
    rows that each hang on row 0 alone, on a few rows of the clique, or on all of it."""
    rng = np.random.default_rng(seed)
    i, j = np.triu_indices(c, 1)
    src, dst = [i, np.arange(c)], [j, np.full(c, c)]
    for leaf in range(c + 1, c + 1 + leaves):
        kind = leaf % 16
        on = [0] if kind < 6 else rng.choice(c, rng.integers(1, 9), replace=False) if kind < 15 else np.arange(c)
        src.append(np.full(len(on), leaf))
        dst.append(np.asarray(on))
    return gg.edges_to_csr(c + 1 + leaves, np.concatenate(src), np.concatenate(dst), None, name=f"folds{c}-{leaves}")


@pytest.mark.parametrize("sr", ["tropical", "real", "selmax"])
@pytest.mark.parametrize("C,sigma", [(8, 1), (16, None), (32, 1), (64, None)])
def test_folds_match_oracle(sr, C, sigma):
    for g, r in [(folds(420, 900, 1), 420), (folds(380, 40, 2), 380)]:
        d = oracle.bfs_queue(g.row_ptr, g.col, r)
        p = oracle.dp(g.row_ptr, g.col, d, r)
        G = ss.SlimSellGraph.from_host(g.row_ptr, g.col, C=C, sigma=sigma or g.n, split_w=64)
        for blocks in (0, 1, 2):
            G.set_option(ss.OPT_PUSH_BLOCKS, blocks)
            dist, parent = G.bfs(r, sr, "push")
            torch.cuda.synchronize()
            np.testing.assert_array_equal(dist.cpu().numpy(), d)
            np.testing.assert_array_equal(parent.cpu().numpy(), p)
            if sr == "real":
                _, _, val, _, _ = oracle.bfs_semiring(g.row_ptr, g.col, r, "real")
                assert val.max() < 2.0 ** 24  # exact in fp32
                np.testing.assert_array_equal(G.values().cpu().numpy()[d >= 0], val[d >= 0])
            st, its = G.run_stats(cap=8)
            assert its[2].variant == ss.V_PUSH, [its[i].variant for i in range(1, st.iterations + 1)]
        G.close()
