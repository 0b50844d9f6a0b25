"""GPU: the cluster push's entries at the sizes where their handling changes (rows of
more than 4, 64 and 128 edges, levels of more than 256 and 512 edges, frontiers that
outgrow the cluster), against the oracle, for both loops and the real values."""
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


def broom(path, leaves, tail):
    """A path to a hub of `leaves` neighbours, each the start of a path of `tail` vertices."""
    e = [(i, i + 1) for i in range(path)]
    n = path + 1
    for _ in range(leaves):
        prev = path
        for _ in range(tail):
            e.append((prev, n))
            prev, n = n, n + 1
    return gg.from_edges(n, e, name=f"broom{path}-{leaves}-{tail}")


def caterpillar(path, leaves):
    e = [(i, i + 1) for i in range(path)] + [(i, path + 1 + i * leaves + j) for i in range(path + 1)
                                             for j in range(leaves)]
    return gg.from_edges(path + 1 + (path + 1) * leaves, e, name=f"caterpillar{path}-{leaves}")


GRAPHS = [broom(3, 5, 4), broom(3, 64, 6), broom(2, 65, 6), broom(2, 129, 5),  # unit boundaries of the hub row
          broom(4, 257, 8), broom(4, 600, 8),     # solo levels that are spread over the cluster and stay there
          broom(3, 9000, 2),                      # more entries than one CTA holds
          caterpillar(30, 3), caterpillar(40, 70), caterpillar(12, 140),  # shrinks back to one CTA level after level
          broom(2, 70000, 1),                     # more vertices than the cluster takes
          gg.lattice(60, 0.05, seed=9), gg.kronecker(13, seed=6)]


@pytest.mark.parametrize("sr,C,sigma", [("tropical", 32, None), ("real", 16, 64), ("real", 32, None), ("boolean", 8, 1),
                                        ("selmax", 64, None)])
def test_entries_match_oracle(sr, C, sigma):
    for g in GRAPHS:
        G = ss.SlimSellGraph.from_host(g.row_ptr, g.col, C=C, sigma=sigma or g.n, split_w=64)
        for r in sorted({0, g.n - 1}):
            d = oracle.bfs_queue(g.row_ptr, g.col, r)
            p = oracle.dp(g.row_ptr, g.col, d, r)
            for loop in (1, 0):
                G.set_option(ss.OPT_DEVICE_LOOP, loop)
                for policy in ("push", "heuristic"):
                    dist, parent = G.bfs(r, sr, policy)
                    torch.cuda.synchronize()
                    np.testing.assert_array_equal(dist.cpu().numpy(), d, err_msg=f"{g.name} {policy} {loop}")
                    np.testing.assert_array_equal(parent.cpu().numpy(), p, err_msg=f"{g.name} {policy} {loop}")
                    if sr == "real":
                        _, _, val, _, _ = oracle.bfs_semiring(g.row_ptr, g.col, r, "real")
                        ok = (d >= 0) & (val < 2.0 ** 24)
                        np.testing.assert_array_equal(G.values().cpu().numpy()[ok], val[ok], err_msg=g.name)
        G.close()
