"""Fused rounds by warp groups: block sizes that leave a short last group,
local queues that overflow, rows that keep a cursor and long chains of waves,
against the oracle's Dijkstra (bit for bit) with the same step trace."""
import numpy as np
import pytest

import oracle as O
from paper_2506_19349_gb300 import graphgen as G

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2506_19349_gb300 as eic  # noqa: E402


def _matchings(n, k, wmax, seed):
    """Union of k random perfect matchings: every degree at most k."""
    rng = np.random.default_rng(seed)
    src, dst = [], []
    for _ in range(k):
        p = rng.permutation(n).astype(np.uint32)
        src.append(p[0::2])
        dst.append(p[1::2])
    src, dst = np.concatenate(src), np.concatenate(dst)
    return n, src, dst, rng.integers(1, wmax + 1, src.size).astype(np.uint32)


def _graphs():
    wl = G.road(67, seed=41, wmax=255, nsources=1)
    yield "grid67", wl.n, wl.src, wl.dst, wl.w
    n = 2049  # one long chain: one vertex a wave
    a = np.arange(n - 1, dtype=np.uint32)
    yield "path", n, a, a + 1, (a % 9 + 1).astype(np.uint32)
    yield ("matchings17", *_matchings(4096, 17, 3, 42))   # rows of 17: cursors
    yield ("matchings32", *_matchings(16384, 32, 2, 43))  # full local queues


GRAPHS = list(_graphs())


@pytest.mark.parametrize("block", [128, 160, 288, 512])
@pytest.mark.parametrize("gap_shift", [0, 6])
@pytest.mark.parametrize("graph", GRAPHS, ids=[g[0] for g in GRAPHS])
def test_fused_groups(graph, gap_shift, block):
    _, n, src, dst, w = graph
    g, og = eic.Graph(n, src, dst, w), O.Graph(n, src, dst, w)
    assert g.max_deg <= 32
    for s in (0, n - 1):
        d, rc, info = eic.sssp(g, s, params=eic.default_params(block_threads=block, gap_shift=gap_shift), trace_cap=4096)
        assert rc == 0 and np.array_equal(eic.to_host_u32(d), og.dijkstra(s)[0])
        if gap_shift == 0:
            keys = ("lb", "ub", "st", "gap_lb", "sumd_lb", "highd_lb", "settled")
            _, _, trace, _ = og.eic(s)
            assert [{k: r[k] for k in keys} for r in info["trace"]] == [{k: r[k] for k in keys} for r in trace]
    d = eic.new_dist(n)
    st = eic.sssp_batch([g], [n // 2], [d], params=eic.default_params(block_threads=block, gap_shift=gap_shift))
    assert st.tolist() == [0] and np.array_equal(eic.to_host_u32(d), og.dijkstra(n // 2)[0])
