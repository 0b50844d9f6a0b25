"""GPU: chunks that the filtered pull starts in a group of lanes and finishes in a whole
warp.  Such a chunk stores its frontier and visited bits twice, from two lanes; the
second store (with the rows of both) must be the one that stays.  Every chunk of these
graphs has rows found in its first 8 columns and rows found after its 40th."""
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


def two_levels(n, deg, seed):
    """Root 0 with 64 neighbours (ids 1 .. 64); the other rows have `deg` neighbours among the
    rest, and one frontier neighbour: half of them a row of the highest ids (met first, as
    neighbours are stored in descending id), half one of the lowest (met last)."""
    rng = np.random.default_rng(seed)
    rest = np.arange(129, n)
    half = rest % 2 == 0
    src = [np.zeros(128, np.int64), rest]
    dst = [np.arange(1, 129), np.where(half, 1 + rest % 64, 65 + rest % 64)]
    for _ in range(deg // 2):
        src.append(rest)
        dst.append(rng.permutation(rest))
    relabel = np.arange(n)  # frontier rows 1 .. 64 keep low ids, 65 .. 128 get the highest
    relabel[65:129] = np.arange(n - 64, n)
    relabel[129:] = np.arange(65, n - 64)
    return gg.edges_to_csr(n, np.concatenate(src), np.concatenate(dst), relabel, name=f"twolevels{n}-{deg}")


@pytest.mark.parametrize("C", [8, 16, 32, 64])
@pytest.mark.parametrize("sr", ["tropical", "boolean", "selmax"])
def test_chunks_left_by_their_group(C, sr):
    for n, deg in [(1500, 60), (9000, 110)]:
        g = two_levels(n, deg, seed=C)
        d = oracle.bfs_queue(g.row_ptr, g.col, 0)
        p = oracle.dp(g.row_ptr, g.col, d, 0)
        G = ss.SlimSellGraph.from_host(g.row_ptr, g.col, C=C, sigma=1, split_w=0)
        for loop in (1, 0):
            G.set_option(ss.OPT_DEVICE_LOOP, loop)
            for _ in range(3):
                dist, parent = G.bfs(0, sr, "pull_filtered")
                torch.cuda.synchronize()
                np.testing.assert_array_equal(dist.cpu().numpy(), d)
                np.testing.assert_array_equal(parent.cpu().numpy(), p)
            st, its = G.run_stats(cap=8)
            assert [its[i].frontier for i in range(st.iterations + 1)] == np.bincount(d[d >= 0]).tolist() + [0]
        G.close()
