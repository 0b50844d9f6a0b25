"""GPU: cluster-push levels around the sizes where their handling changes with the edges
they hold (8,192: row data of new rows only, no columns asked for ahead) and with the
entries of a segment (32: one list for all warps), against the oracle."""
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


def comb(width, teeth, seed):
    """A root, `width` neighbours, and behind each a chain of `teeth` rows with cross links to
    the next chain: `teeth` levels of about 4 * width edges each."""
    ids = 1 + np.arange(width * teeth).reshape(teeth, width)
    src = [np.zeros(width, np.int64), ids[:-1].ravel(), ids[:-1].ravel()]
    dst = [ids[0], ids[1:].ravel(), np.roll(ids[1:], 1, axis=1).ravel()]
    n = 1 + width * teeth
    return gg.edges_to_csr(n, np.concatenate(src), np.concatenate(dst), gg.permutation(n, seed), name=f"comb{width}")


@pytest.mark.parametrize("width", [2047, 2048, 2049, 5000, 8191, 8192, 8193, 12000])
def test_wide_levels_match_oracle(width):
    g = comb(width, 6, seed=width)
    root = int(gg.permutation(g.n, width)[0])
    d = oracle.bfs_queue(g.row_ptr, g.col, root)
    p = oracle.dp(g.row_ptr, g.col, d, root)
    for C, sr in [(32, "tropical"), (8, "real")]:
        G = ss.SlimSellGraph.from_host(g.row_ptr, g.col, C=C, sigma=g.n, split_w=256)
        dist, parent = G.bfs(root, sr, "push")
        torch.cuda.synchronize()
        np.testing.assert_array_equal(dist.cpu().numpy(), d)
        np.testing.assert_array_equal(parent.cpu().numpy(), p)
        if sr == "real":
            _, _, val, _, _ = oracle.bfs_semiring(g.row_ptr, g.col, root, "real")
            np.testing.assert_array_equal(G.values().cpu().numpy(), val)
        st, its = G.run_stats(cap=16)
        assert all(its[i].variant == ss.VARIANT_PUSH_LOCAL for i in range(1, 7)), [its[i].variant for i in range(8)]
        G.close()
