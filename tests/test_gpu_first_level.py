"""GPU: the first level, where only the root is in the frontier, is a stream of the column
array on layouts of at least 4 M slots: against the oracle, and its counters against the
real semiring's, which takes the general pass.  Repeated edges, a self-loop at the root,
a root alone in the last chunk, split chunks, and chunks of every height."""
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


def with_repeats(n, seed):
    """A symmetric CSR with every edge at the root twice, a self-loop there, and rows
    ascending; the root is vertex n - 1 (alone in its chunk for n = 1 mod C and sigma 1)."""
    g = gg.erdos_renyi(n, 10.0, seed=seed)
    u = np.repeat(np.arange(n), np.diff(g.row_ptr))
    v = np.asarray(g.col, dtype=np.int64)
    r = n - 1
    more = np.array([5, 7, 1 << 10, n // 2, n - 2])
    u = np.concatenate([u, u[(u == r) | (v == r)], np.full(5, r), more, [r]])
    v = np.concatenate([v, v[(np.repeat(np.arange(n), np.diff(g.row_ptr)) == r) | (v == r)], more, np.full(5, r), [r]])
    order = np.lexsort((v, u))
    u, v = u[order], v[order]
    row_ptr = np.zeros(n + 1, dtype=np.int64)
    np.add.at(row_ptr, u + 1, 1)
    return np.cumsum(row_ptr).astype(g.row_ptr.dtype), v.astype(np.int32), r


@pytest.mark.parametrize("C,sigma,w", [(8, 1, 4), (16, 4096, 64), (32, 1, 8), (64, 0, 256)])
def test_first_level(C, sigma, w):
    n = 420000 // 64 * 64 + 1
    row_ptr, col, root = with_repeats(n, seed=3)
    assert len(col) >= 4 << 20
    G = ss.SlimSellGraph.from_host(row_ptr, col, C=C, sigma=sigma or n, split_w=w)
    for r in (root, 0):
        want = oracle.bfs_queue(row_ptr, col, r)
        par = oracle.dp(row_ptr, col, want, r)
        for policy in ("slimwork", "full"):
            first = {}
            for sr in ("tropical", "boolean", "selmax", "real"):
                dist, parent = G.bfs(r, sr, policy)
                torch.cuda.synchronize()
                np.testing.assert_array_equal(dist.cpu().numpy(), want)
                np.testing.assert_array_equal(parent.cpu().numpy(), par)
                _, it = G.run_stats(64)
                first[sr] = (it[1].frontier, it[1].frontier_degree, it[1].slots, it[1].active_chunks)
            assert len(set(first.values())) == 1, first
    G.close()
