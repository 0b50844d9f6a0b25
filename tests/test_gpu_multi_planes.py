"""GPU: the level planes of multi-source distances and the one-word level kernel, on graphs that
meet their gates (an output of 16 M entries, more than half of the words' sources, 12,160
work items): runs that end in the first epoch of 15 levels, in the long epochs of 255 after
it and past those, one word and several, ragged k, outputs off 16-byte alignment, isolated
rows and roots, both policies, and chunks of 8 to 64, against the oracle.  That the planes
ran is seen in the memory that the handle takes for them: 32 bytes a row and word, and 64
more once a run goes on past 15 levels."""
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


def strip(width, length, extra, seed, isolated=0):
    """A lattice of length x width with 3 % of its edges gone, `extra` random ones that shorten
    it, shuffled ids, and isolated rows after it."""
    rng = np.random.default_rng(seed)
    at = np.arange(width * length).reshape(length, width)
    src = np.concatenate([at[:, :-1].ravel(), at[:-1].ravel()])
    dst = np.concatenate([at[:, 1:].ravel(), at[1:].ravel()])
    keep = rng.random(len(src)) >= 0.03
    u, v = rng.integers(0, width * length, (2, extra))
    n = width * length + isolated
    return gg.edges_to_csr(n, np.concatenate([src[keep], u]), np.concatenate([dst[keep], v]), gg.permutation(n, seed))


# (graph, chunk, split width, k, words, offset of the output in ints)
SHORT = dict(width=600, length=700, extra=900000, seed=1, isolated=1001)  # 421,001 rows, 9 levels
MIDDLE = dict(width=600, length=700, extra=3000, seed=2, isolated=37)     # 420,037 rows, 16 to 255
LONG = dict(width=650, length=650, extra=20, seed=3)                      # 422,500 rows, over 300
CASES = [(SHORT, 32, 256, 64, 1, 0), (SHORT, 32, 256, 63, 1, 0), (SHORT, 64, 2, 40, 1, 1), (SHORT, 16, 64, 125, 2, 0),
         (SHORT, 8, 256, 250, 4, 2), (MIDDLE, 32, 256, 64, 1, 0), (MIDDLE, 64, 1, 61, 1, 3), (MIDDLE, 32, 256, 100, 2, 0),
         (MIDDLE, 64, 256, 101, 2, 1), (LONG, 32, 256, 48, 1, 0), (LONG, 16, 256, 70, 2, 0)]


@pytest.mark.parametrize("spec,C,w,k,W,off", CASES)
def test_planes_match_oracle(spec, C, w, k, W, off):
    g = strip(**spec)
    assert g.n * k >= 16 << 20 and k > 32 * W
    G = ss.SlimSellGraph.from_host(g.row_ptr, g.col, C=C, sigma=g.n, split_w=w)
    inf = G.info()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    if W == 1:
        assert inf.n_items >= 80 * sms  # the one-word kernel's gate
    roots = np.concatenate([gg.roots(g, k - 3, seed=4), np.flatnonzero(np.diff(g.row_ptr) == 0)[:1], [0, 0]])[:k]
    roots = np.concatenate([roots, np.zeros(k - len(roots), roots.dtype)]).astype(np.int32)
    want = np.stack([oracle.bfs_queue(g.row_ptr, g.col, int(r)) for r in roots], axis=1)
    assert {id(SHORT): 1, id(MIDDLE): 16, id(LONG): 300}[id(spec)] <= want.max() < {id(SHORT): 16, id(MIDDLE): 256}.get(id(spec), 4096)
    buf = torch.full((g.n * k + 8,), -7, dtype=torch.int32, device="cuda")
    dist = buf[off:off + g.n * k].view(g.n, k)
    d_roots = torch.from_numpy(roots).cuda()
    for policy in ("slimwork", "full", "slimwork"):
        before = G.info().device_bytes
        G.bfs_multi(d_roots, policy, dist)
        torch.cuda.synchronize()
        if before == inf.device_bytes:  # the first run: state words, planes and long planes
            planes = 32 * inf.n_chunks * C * W
            took = G.info().device_bytes - before - 3 * 8 * inf.n_chunks * C * W
            assert took >= planes * (3 if want.max() > 15 else 1), (took, planes)
        np.testing.assert_array_equal(dist.cpu().numpy(), want, err_msg=policy)
        assert (buf[:off] == -7).all() and (buf[off + g.n * k:] == -7).all()
        dist.fill_(5)
        if want.max() > 255:
            break  # (a few hundred levels are enough once)
    if k <= 64:
        parent = torch.empty((g.n, k), dtype=torch.int32, device="cuda")
        G.bfs_multi_parents(d_roots, "slimwork", dist, parent)
        torch.cuda.synchronize()
        np.testing.assert_array_equal(dist.cpu().numpy(), want)
        got = parent.cpu().numpy()
        for s in (0, k // 2, k - 1):
            np.testing.assert_array_equal(got[:, s], oracle.dp(g.row_ptr, g.col, want[:, s], int(roots[s])))
    G.close()


def test_one_word_kernel_under_centrality():
    """Betweenness over level words made by the one-word kernel (no distances asked for)."""
    g = gg.lattice(640, 0.05, seed=5)
    G = ss.SlimSellGraph.from_host(g.row_ptr, g.col, C=32, sigma=g.n, split_w=256)
    assert G.info().n_items >= 80 * torch.cuda.get_device_properties(0).multi_processor_count
    src = gg.roots(g, 4, seed=6).astype(np.int32)
    got = G.bc(torch.from_numpy(src).cuda()).cpu().numpy()
    np.testing.assert_allclose(got, oracle.bc(g.row_ptr, g.col, src), rtol=1e-9, atol=1e-9 * got.max())
    G.close()
