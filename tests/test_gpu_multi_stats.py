"""GPU: the level statistics of a profiled multi-source run hold the time of the kernels that
write its distances, also where these are kept as level planes and written at the end:
on a graph with a few edges and 4 M vertices the writes are nearly all of the work, and
cannot take less than the output's bytes take at 8 TB/s."""
import numpy as np
import pytest
import torch

import graphgen as gg
import paper_2010_09913_gb300 as ss

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    ss.build()


@pytest.mark.parametrize("k", [64, 63])
def test_distance_writes_are_counted(k):
    n = 1 << 22
    g = gg.from_edges(n, [(0, 1), (1, 2), (2, 3)])
    G = ss.SlimSellGraph.from_host(g.row_ptr, g.col, C=32, sigma=n, split_w=256)
    roots = torch.arange(k, dtype=torch.int32, device="cuda") % 5
    before = G.info().device_bytes
    ss.slimsell_set_profiling(G.h, True)
    dist = G.bfs_multi(roots, "slimwork")
    torch.cuda.synchronize()
    assert G.info().device_bytes - before >= 32 * n  # the planes were used
    st, its = G.run_stats(cap=16)
    per_level = [its[i].kernel_ns for i in range(1, st.iterations + 1)]
    assert abs(sum(per_level) / 1e6 - st.iter_kernel_ms) < 1e-3 * len(per_level)
    assert st.iter_kernel_ms >= 4.0 * n * k / 8e12 * 1e3
    assert st.iter_kernel_ms <= st.total_ms
    want = np.full((n, 5), -1, np.int32)
    for s in range(5):
        for v in range(4):
            if s < 4:
                want[v, s] = abs(v - s)
    want[4, 4] = 0
    np.testing.assert_array_equal(dist.cpu().numpy(), want[:, np.arange(k) % 5])
    G.close()
