"""GPU: multi-source distances from level planes, where their handling changes: runs of
more than one epoch of 15 levels, k not a multiple of 4 or 64, outputs off 16-byte
alignment, rows without neighbours, repeated roots, and both one-word kernels (sparse
and dense levels)."""
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


def path(n, extra=0):  # n - 1 levels; `extra` isolated vertices
    return gg.from_edges(n + extra, [(i, i + 1) for i in range(n - 1)], name=f"path{n}")


GRAPHS = [path(15), path(16), path(17, 3), path(31), path(46, 40), gg.lattice(24, 0.05, seed=2),
          gg.kronecker(12, seed=8), gg.erdos_renyi(3001, 3.0, seed=5)]


@pytest.mark.parametrize("C,k", [(32, 1), (32, 64), (64, 63), (32, 65), (8, 30), (16, 100), (64, 260)])
def test_levels_match_oracle(C, k):
    for g in GRAPHS:
        G = ss.SlimSellGraph.from_host(g.row_ptr, g.col, C=C, sigma=g.n, split_w=16)
        rng = np.random.default_rng(k)
        roots = rng.integers(0, g.n, k).astype(np.int32)
        roots[0] = 0
        want = {int(r): oracle.bfs_queue(g.row_ptr, g.col, int(r)) for r in set(roots.tolist())}
        buf = torch.empty(g.n * k + 1, dtype=torch.int32, device="cuda")
        for off in (0, 1):  # the second output starts off a 16-byte boundary
            for policy in ("slimwork", "full"):
                buf.fill_(77)
                dist = buf[off:off + g.n * k].view(g.n, k)
                G.bfs_multi(roots, policy, dist)
                torch.cuda.synchronize()
                got = dist.cpu().numpy()
                for s, r in enumerate(roots):
                    np.testing.assert_array_equal(got[:, s], want[int(r)], err_msg=f"{g.name} source {s}")
        G.close()
