"""GPU: the cluster push takes its first frontier from the bitmap that a grid-wide level
left.  On graphs of up to 131,072 rows the lanes of a warp share its words (2, 4 .. 32
lanes a word), so no word may be cleared before all of them have read it: frontiers
that fill whole words, at every sharing factor, against the oracle."""
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


def clique_and_fringe(fringe, pad):
    """Root, a clique of 400 (159,600 edges, more than the cluster takes), `fringe` rows on the
    clique with consecutive ids, each with one row more behind it, and `pad` isolated rows."""
    c = 400
    i, j = np.triu_indices(c, 1)
    f = np.arange(fringe)
    src = np.concatenate([np.zeros(c, np.int64), 1 + i, 1 + f % c, 1 + c + f])
    dst = np.concatenate([1 + np.arange(c), 1 + j, 1 + c + f, 1 + c + fringe + f])
    return gg.edges_to_csr(1 + c + 2 * fringe + pad, src, dst, None, name=f"fringe{fringe}-{pad}")


@pytest.mark.parametrize("fringe,pad", [(1, 0), (33, 0), (3800, 0), (3800, 8000), (8000, 16000), (16000, 32000),
                                        (40000, 50000), (40000, 200000)])
@pytest.mark.parametrize("sr,C", [("tropical", 32), ("real", 8), ("selmax", 64)])
def test_first_frontier_of_shared_words(fringe, pad, sr, C):
    g = clique_and_fringe(fringe, pad)
    G = ss.SlimSellGraph.from_host(g.row_ptr, g.col, C=C, sigma=1, split_w=256)
    d = oracle.bfs_queue(g.row_ptr, g.col, 0)
    p = oracle.dp(g.row_ptr, g.col, d, 0)
    for loop in (1, 0):
        G.set_option(ss.OPT_DEVICE_LOOP, loop)
        for _ in range(3):
            dist, parent = G.bfs(0, sr, "push")
            torch.cuda.synchronize()
            np.testing.assert_array_equal(dist.cpu().numpy(), d)
            np.testing.assert_array_equal(parent.cpu().numpy(), p)
        st, its = G.run_stats(cap=16)
        seq = [its[i].variant for i in range(1, st.iterations + 1)]
        # the clique's level runs grid-wide and leaves the fringe as a bitmap
        assert seq[1] == ss.V_PUSH and seq[2] == ss.VARIANT_PUSH_LOCAL, seq
    G.close()
