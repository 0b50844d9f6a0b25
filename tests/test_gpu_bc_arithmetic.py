"""GPU: the number formats of betweenness centrality.  Path counts run as 64-bit
integers and dependencies as 128-bit fixed point; counts past the fixed point's
range (2^(66 - bits(n))) or past 2^63 make the batch go on in fp64, during the
backward or already during the forward pass.  Tolerance as for the other
centrality tests: 1e-9 relative (fp64 sums in another order on either side)."""
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


# L x L lattices without deletions: a corner's counts reach binomial(2 L - 2, L - 1)
@pytest.mark.parametrize("L", [12,   # 2^19: integers and fixed point throughout
                               31,   # 2^57: integer counts, fp64 dependencies
                               45])  # 2^84: counts leave the integers halfway
def test_formats_by_path_count(L):
    g = gg.lattice(L, 0.0, seed=1)
    G = ss.SlimSellGraph.from_host(g.row_ptr, g.col, C=16, sigma=g.n, split_w=64)
    src = np.array([0, L * L - 1, (L // 2) * L, 7], dtype=np.int32)
    for _ in range(2):  # the second run starts from the first one's scratch
        got = G.bc(src)
        torch.cuda.synchronize()
        want = oracle.bc(g.row_ptr, g.col, src)
        np.testing.assert_allclose(got.cpu().numpy(), want, rtol=1e-9, atol=1e-9 * want.max())
    G.close()


def test_rows_of_several_units_and_batches():
    # a hub of 700 neighbours (three units) two levels from the sources, and 70
    # sources (two batches over the same scratch)
    edges = [(0, i) for i in range(1, 701)] + [(i, 701 + i) for i in range(1, 701)]
    edges += [(1, i) for i in range(1500, 1900)]
    g = gg.from_edges(2000, edges)
    G = ss.SlimSellGraph.from_host(g.row_ptr, g.col, C=32, sigma=g.n, split_w=16)
    src = np.array([701 + 10 * i + 1 for i in range(70)], dtype=np.int32)
    got = G.bc(src)
    torch.cuda.synchronize()
    want = oracle.bc(g.row_ptr, g.col, src)
    np.testing.assert_allclose(got.cpu().numpy(), want, rtol=1e-9, atol=1e-9 * want.max())
    G.close()
