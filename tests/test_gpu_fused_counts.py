"""Statistics of fused rounds. On a tree a vertex has one path, so it is reached
and relaxed from exactly once in its step whatever the order: the counts of a
query are those of plain rounds, also for vertices whose windows are empty, cut
into tasks, or left to the next round."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2506_19349_gb300 as eic  # noqa: E402


def _tree(name):
    """(n, the parents of vertices 1 .. n - 1)"""
    rng = np.random.default_rng(len(name))
    if name == "recursive":  # every degree small: road-like
        n = 20000
        return n, (rng.random(n - 1) * np.arange(1, n)).astype(np.uint32)
    if name == "preferential":  # hubs of some hundreds
        n = 20000
        p = np.zeros(n - 1, np.uint32)
        for v in range(2, n):
            j = int(rng.integers(1, v))
            p[v - 1] = j if rng.random() < 0.4 else p[j - 1]
        return n, p
    if name == "hubs":  # a chain of hubs: 70 children each, each child a short path
        p, at, prev = [], 1, 0
        for _ in range(60):
            hub = at
            p += [prev] + [hub] * 70 + list(range(hub + 1, hub + 71))
            at += 141
            prev = hub + 1
        return at, np.array(p, np.uint32)
    n = 30000  # path
    return n, np.arange(n - 1, dtype=np.uint32)


@pytest.mark.parametrize("gap_shift", [0, 4, 9])
@pytest.mark.parametrize("wmax", [1, 7, 255])
@pytest.mark.parametrize("name", ["recursive", "preferential", "hubs", "path"])
def test_counts_on_trees(name, wmax, gap_shift):
    if name == "path" and gap_shift == 0:
        pytest.skip("a step per vertex")
    n, par = _tree(name)
    rng = np.random.default_rng(wmax)
    v = np.arange(1, n, dtype=np.uint32)
    w = rng.integers(1, wmax + 1, n - 1).astype(np.uint32)
    g, og = eic.Graph(n, par, v, w), O.Graph(n, par, v, w)
    for s in (0, n // 2):
        want = og.dijkstra(s)[0]
        for pull in (0, eic.FLAG_NO_PULL):
            got = []
            for fuse in (0, eic.FLAG_NO_FUSE):
                d, rc, info = eic.sssp(g, s, params=eic.default_params(gap_shift=gap_shift, flags=pull | fuse), stats=True)
                assert rc == 0 and np.array_equal(eic.to_host_u32(d), want)
                got.append((info["frontier"], info["improved"]))
            assert got[0] == got[1]
