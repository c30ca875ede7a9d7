"""Fused rounds on graphs with long rows: hubs reached within a fused round
(deferred to a plain round), items with long windows (grid tasks), rounds cut
short at the iteration limit, against Dijkstra and the oracle's step trace,
with and without fusion."""
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


def _hub_chain(k, leaves, hop, wmax, seed):
    """k hubs in a chain, `hop` path vertices between neighbours, `leaves`
    leaves each, shared by the next hub: hubs come up wave after wave."""
    rng = np.random.default_rng(seed)
    src, dst, at, prev = [], [], 0, None
    for _ in range(k):
        hub = at
        lv = np.arange(at + 1, at + 1 + leaves, dtype=np.uint32)
        src.append(np.full(leaves, hub, np.uint32))
        dst.append(lv)
        at += 1 + leaves
        if prev is not None:
            chain = np.concatenate([[prev[0]], np.arange(at, at + hop), [hub]]).astype(np.uint32)
            at += hop
            src += [chain[:-1], prev[1][: leaves // 2]]
            dst += [chain[1:], lv[: leaves // 2]]
        prev = (hub, lv)
    src, dst = np.concatenate(src), np.concatenate(dst)
    return at, src, dst, rng.integers(1, wmax + 1, src.size).astype(np.uint32)


def _graphs():
    yield ("hubs65", *_hub_chain(40, 65, 3, 4, 61))     # windows just above the longest of a wave
    yield ("hubs64", *_hub_chain(40, 63, 0, 4, 62))
    yield ("hubs900", *_hub_chain(12, 900, 5, 255, 63))
    for name, wl in (("kron13", G.kron(13, seed=64, nsources=1)), ("urand12", G.urand(12, 16, seed=65)),
                     ("kron12_power24", G.kron(12, seed=66, weights="power:24", nsources=1))):
        yield name, wl.n, wl.src, wl.dst, wl.w


GRAPHS = list(_graphs())


@pytest.mark.parametrize("gap_shift", [0, 3, 8])
@pytest.mark.parametrize("graph", GRAPHS, ids=[g[0] for g in GRAPHS])
def test_fused_general(graph, gap_shift):
    _, n, src, dst, w = graph
    g, og = eic.Graph(n, src, dst, w), O.Graph(n, src, dst, w)
    assert g.max_deg > 32
    deg = og.degrees()
    for s in (int(np.flatnonzero(deg)[0]), int(np.flatnonzero(deg)[-1]), int(np.argmax(deg))):
        want = og.dijkstra(s)[0]
        for flags in (0, eic.FLAG_NO_FUSE, eic.FLAG_NO_PULL):
            for block in (512, 160):
                p = eic.default_params(gap_shift=gap_shift, flags=flags, block_threads=block)
                d, rc, info = eic.sssp(g, s, params=p, trace_cap=4096)
                assert rc == 0 and np.array_equal(eic.to_host_u32(d), want)
            if gap_shift == 0 and flags != eic.FLAG_NO_PULL:
                _, _, trace, _ = og.eic(s)
                assert [{k: r[k] for k in KEYS} for r in info["trace"]] == [{k: r[k] for k in KEYS} for r in trace]
        ds = [eic.new_dist(n) for _ in range(3)]
        st = eic.sssp_batch([g] * 3, [s] * 3, ds, params=eic.default_params(gap_shift=gap_shift))
        assert st.tolist() == [0, 0, 0] and all(np.array_equal(eic.to_host_u32(d), want) for d in ds)
