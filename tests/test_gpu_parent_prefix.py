"""Shortest-path parents in long rows: the prefix of a row that can hold the
parent ends at, before and behind the edges of what one warp takes and of the
pieces that the rest is cut into, with the only parent anywhere in it."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2506_19349_gb300 as eic  # noqa: E402

PREFIX = (0, 1, 31, 32, 127, 128, 129, 255, 256, 511, 512, 513, 544, 545, 640, 767, 768, 769, 1023, 1024, 1025, 3000)


@pytest.mark.parametrize("tail", [0, 1, 33, 700])  # heavier entries behind the prefix
@pytest.mark.parametrize("tied", [0.0, 0.3, 1.0])  # of a prefix's neighbours, how many are as short a way
def test_parent_prefixes(tail, tied):
    rng = np.random.default_rng(tail + int(10 * tied))
    src, dst, w, at = [], [], [], 1
    for p in PREFIX:  # a hub at distance 1000: its prefix is the edge to the source and p neighbours
        hub, leaf = at, np.arange(at + 1, at + 1 + p + tail, dtype=np.uint32)
        wl = np.concatenate([rng.integers(1, 1000, p), rng.integers(1001, 5000, tail)]).astype(np.uint32)
        ways = rng.random(p) < tied
        if p and not ways.any():
            ways[rng.integers(0, p)] = tied > 0
        first = rng.permutation(p + tail)  # ids in no order of weight
        leaf = leaf[first]
        src += [np.full(leaf.size, hub, np.uint32), np.zeros(p, np.uint32), np.zeros(1, np.uint32)]
        dst += [leaf, leaf[:p], np.full(1, hub, np.uint32)]
        w += [wl, np.where(ways, 1000 - wl[:p], 1000 + wl[:p]).astype(np.uint32), np.full(1, 1000, np.uint32)]
        at += 1 + p + tail
    src, dst, w = (np.concatenate(x).astype(np.uint32) for x in (src, dst, w))
    g, og = eic.Graph(at, src, dst, w), O.Graph(at, src, dst, w)
    for s in (0, 1, at - 1):
        par = torch.empty(at, dtype=torch.int32, device="cuda")
        d, rc, _ = eic.sssp(g, s, parent=par)
        want = og.dijkstra(s)[0]
        assert rc == 0 and np.array_equal(eic.to_host_u32(d), want)
        assert np.array_equal(eic.to_host_u32(par), og.parent(s, want))


def test_parent_in_pieces_without_a_wide_weight():
    """Unit weights: every row is its own prefix, most of it in pieces."""
    n, k = 9000, 6
    hubs = np.repeat(np.arange(k, dtype=np.uint32), n - k)
    leaves = np.tile(np.arange(k, n, dtype=np.uint32), k)
    g, og = eic.Graph(n, hubs, leaves, np.ones(hubs.size, np.uint32)), O.Graph(n, hubs, leaves, np.ones(hubs.size, np.uint32))
    for s in (3, n - 1):
        par = torch.empty(n, dtype=torch.int32, device="cuda")
        d, rc, _ = eic.sssp(g, s, parent=par)
        want = og.dijkstra(s)[0]
        assert rc == 0 and np.array_equal(eic.to_host_u32(par), og.parent(s, want))
