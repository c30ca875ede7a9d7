"""The step boundary over the forms that its phases distinguish: candidate
grids of several sizes, rings below and above the shared-memory window, wide
weights, many and few distinct degrees, small blocks. Step traces equal the
oracle's Algorithm 1 and distances its Dijkstra."""
import numpy as np
import pytest

import oracle as O
from paper_2506_19349_gb300 import graphgen as G

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2506_19349_gb300 as eic  # noqa: E402

KEYS = ("lb", "ub", "st", "gap_lb", "sumd_lb", "highd_lb", "settled")


def _wide_grid():
    wl = G.road(80, seed=51, wmax=9001, nsources=2)  # a window of 9001 slots: three to a chunk
    return wl


GRAPHS = {
    "kron13_w255": lambda: G.kron(13, seed=52, nsources=2),
    "kron13_lognormal": lambda: G.kron(13, seed=53, weights="lognormal", nsources=2),
    "kron12_power24": lambda: G.kron(12, seed=54, weights="power:24", nsources=2),
    "grid80_w9001": _wide_grid,
    "grid60_w4096": lambda: G.road(60, seed=55, wmax=4096, nsources=2),
    "urand12": lambda: G.urand(12, 15, seed=56, nsources=2),
}


@pytest.mark.parametrize("st_num", [1, 7, 1024, 5000, 65536])
@pytest.mark.parametrize("block", [128, 512])
@pytest.mark.parametrize("name", list(GRAPHS))
def test_boundary_trace(name, block, st_num):
    wl = GRAPHS[name]()
    g, og = eic.Graph(wl.n, wl.src, wl.dst, wl.w), O.Graph(wl.n, wl.src, wl.dst, wl.w)
    for s in wl.sources:
        s = int(s)
        p = eic.default_params(st_num=st_num, block_threads=block)
        d, rc, info = eic.sssp(g, s, params=p, trace_cap=8192)
        assert rc == 0 and np.array_equal(eic.to_host_u32(d), og.dijkstra(s)[0])
        _, _, trace, _ = og.eic(s, st_num=st_num)
        assert [{k: r[k] for k in KEYS} for r in info["trace"]] == [{k: r[k] for k in KEYS} for r in trace]


def test_highd0_many_degrees():
    """highD(0) with more distinct degrees than threads: a union of stars."""
    src, dst, at = [], [], 0
    for k in range(1, 1400):
        src.append(np.full(k, at, np.uint32))
        dst.append(np.arange(at + 1, at + 1 + k, dtype=np.uint32))
        at += k + 1
    src, dst = np.concatenate(src), np.concatenate(dst)
    g = eic.Graph(at, src, dst, np.ones(src.size, np.uint32))
    deg = np.bincount(np.concatenate([src, dst]), minlength=at).astype(np.uint32)
    assert g.highd0 == O.highd(deg)
