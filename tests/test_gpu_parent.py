"""Shortest-path parents where rows are shared out: degrees on both sides of the
limit, rows that end inside and at the end of a chunk, ties, unreachable hubs."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2506_19349_gb300 as eic  # noqa: E402


@pytest.mark.parametrize("degrees", [(512,), (513,), (511, 512, 513, 514), (1024, 768, 513), (5000, 600, 600, 40, 1)])
@pytest.mark.parametrize("wmax", [1, 3, 70000])
def test_parent_big_rows(degrees, wmax):
    rng = np.random.default_rng(sum(degrees) + wmax)
    k = len(degrees)
    n = 6000 + k + 600  # the last vertices: a hub with 550 leaves of its own, unreachable
    src, dst = [], []
    for h, d in enumerate(degrees):
        src.append(np.full(d, h, np.uint32))
        dst.append(k + rng.choice(6000, d, replace=False).astype(np.uint32))
    a = rng.integers(k, k + 6000, (2, 4000)).astype(np.uint32)
    src += [a[0], np.full(550, n - 1, np.uint32)]
    dst += [a[1], np.arange(n - 551, n - 1, dtype=np.uint32)]
    src, dst = np.concatenate(src), np.concatenate(dst)
    w = rng.integers(1, wmax + 1, src.size).astype(np.uint32)
    g, og = eic.Graph(n, src, dst, w), O.Graph(n, src, dst, w)
    for s in (0, k + 17, n - 1):
        par = torch.empty(n, dtype=torch.int32, device="cuda")
        d, rc, _ = eic.sssp(g, s, parent=par)
        want = og.dijkstra(s)[0]
        assert rc == 0 and np.array_equal(eic.to_host_u32(d), want)
        assert np.array_equal(eic.to_host_u32(par), og.parent(s, want))
