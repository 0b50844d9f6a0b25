"""GPU: calls on a device that is nearly full: a build for which the device holds the layout with
the build's temporaries, and the layout with the BFS state, but not all three; a build that
does not fit; and a handle whose multi-source scratch must make room for other scratch."""
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


class Device:
    """A graph of 2^25 vertices, a build and run of it, and the device filled beside them."""

    def __init__(self):
        n = self.n = 1 << 25  # about 28 bytes a vertex of temporaries, 24 of state, 12 of tables
        row_ptr = np.zeros(n + 1, np.int64)
        row_ptr[1:5] = [1, 3, 5, 6]
        row_ptr[5:] = 6
        self.rp = torch.from_numpy(row_ptr).cuda()
        self.col = torch.tensor([1, 0, 2, 1, 3, 2], dtype=torch.int32, device="cuda")
        self.out = torch.empty((2, n), dtype=torch.int32, device="cuda")
        self.keep = []

    def build(self):
        return ss.SlimSellGraph(self.rp, self.col, C=32, sigma=None, split_w=256)

    def run(self):
        G, out = self.build(), self.out
        G.bfs(0, "tropical", "slimwork", out[0], out[1])
        torch.cuda.synchronize()
        assert out[:, :5].cpu().tolist() == [[0, 1, 2, 3, -1], [0, 0, 1, 2, -1]] and int((out[0] >= 0).sum()) == 4
        held = G.info().device_bytes
        G.close()
        torch.cuda.empty_cache()
        return held

    def leave(self, size):
        """Fill the device up to `size` free bytes; what is free then."""
        while True:
            free = torch.cuda.mem_get_info()[0]
            if free < size + (64 << 20):
                return free
            self.keep.append(torch.empty(min(free - size, 64 << 30) - (32 << 20), dtype=torch.uint8, device="cuda"))


@pytest.fixture
def device():
    d = Device()
    yield d
    d.keep.clear()
    torch.cuda.empty_cache()


def test_state_waits_for_the_temporaries(device):
    held = device.run()
    free = device.leave(held + device.n * 12)  # the handle, and less than half of the temporaries
    assert free < held + device.n * 24, (free, held)
    assert device.run() == held
    assert torch.cuda.mem_get_info()[0] >= free - (8 << 20)


def test_out_of_memory_is_reported_once(device):
    """A build that does not fit leaves nothing behind: no memory, and no error for the next."""
    held = device.run()
    free = device.leave(held // 2)
    with pytest.raises(ss.SlimSellError):
        device.build()
    assert torch.cuda.mem_get_info()[0] >= free - (8 << 20)
    device.keep.clear()
    torch.cuda.empty_cache()
    assert device.run() == held


def test_level_planes_make_room_for_centrality(device):
    """A multi-source run leaves its level planes with the handle; a centrality call whose scratch
    does not fit beside them gets their memory, and the next multi-source run does without."""
    g = gg.erdos_renyi(1 << 18, 12.0, seed=3)
    G = ss.SlimSellGraph.from_host(g.row_ptr, g.col, C=32, sigma=g.n, split_w=256)
    roots = torch.from_numpy(gg.roots(g, 1000, seed=4).astype(np.int32)).cuda()
    src = gg.roots(g, 3, seed=5).astype(np.int32)
    d_src = torch.from_numpy(src).cuda()
    dist = torch.empty((g.n, 1000), dtype=torch.int32, device="cuda")
    G.bfs_multi(roots, "slimwork", dist)
    want = dist.clone()
    planes = 32 * 16 * g.n  # 134 MB; the centrality scratch takes 1,536 bytes a row, 403 MB
    torch.cuda.empty_cache()
    held = G.info().device_bytes
    free = device.leave(1536 * g.n - planes // 2)
    assert free < 1536 * g.n
    got = G.bc(d_src).cpu().numpy()
    np.testing.assert_allclose(got, oracle.bc(g.row_ptr, g.col, src), rtol=1e-9, atol=1e-9 * got.max())
    assert G.info().device_bytes < held + 1536 * g.n
    dist.fill_(7)
    G.bfs_multi(roots, "slimwork", dist)
    device.keep.clear()
    torch.cuda.empty_cache()
    assert torch.equal(dist, want)
    d = oracle.bfs_queue(g.row_ptr, g.col, int(roots[0]))
    np.testing.assert_array_equal(dist[:, 0].cpu().numpy(), d)
    G.close()
