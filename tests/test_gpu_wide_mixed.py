"""Graphs with weights of 2^20 and above (Function 2's bins, filled by every
block of a group between two more barriers) beside narrow ones: one group runs
them in turn with the same scratch, in batches and in a server, whose launches
wait for the end of a burst."""
import time

import numpy as np
import pytest

import oracle as O
from paper_2506_19349_gb300 import graphgen as G

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2506_19349_gb300 as eic  # noqa: E402


@pytest.fixture(scope="module")
def mixed():
    wls = [G.kron(12, seed=131, weights=f"uniform:{1 << 24}", nsources=4), G.kron(12, seed=132, nsources=4),
           G.kron(10, seed=133, weights=f"uniform:{(1 << 20) + 5}", nsources=4), G.road(60, seed=134, wmax=9001, nsources=4)]
    graphs = [eic.Graph(w.n, w.src, w.dst, w.w) for w in wls]
    queries = [(k, int(w.sources[j])) for j in range(4) for k, w in enumerate(wls)]
    oracles = [O.Graph(w.n, w.src, w.dst, w.w) for w in wls]
    return graphs, queries, [oracles[k].dijkstra(s)[0] for k, s in queries]


@pytest.mark.parametrize("st_num", [1024, 5000])  # the bins in shared memory, and too many for it
@pytest.mark.parametrize("groups", [1, 3])
def test_batch_of_wide_and_narrow_graphs(mixed, groups, st_num):
    graphs, queries, want = mixed
    params = eic.default_params(batch_groups=groups, st_num=st_num)
    dists = [eic.new_dist(graphs[k].n) for k, _ in queries]
    gs, ss = [graphs[k] for k, _ in queries], [s for _, s in queries]
    assert eic.sssp_batch(gs, ss, dists, params=params).tolist() == [0] * len(queries)
    for d, x in zip(dists, want):
        assert np.array_equal(eic.to_host_u32(d), x)
    b = eic.Batch(gs, ss, dists, params=params)
    for _ in range(2):
        for d in dists:
            d.zero_()
        b.run()
        assert b.wait().tolist() == [0] * len(queries)
        for d, x in zip(dists, want):
            assert np.array_equal(eic.to_host_u32(d), x)
    b.close()


@pytest.mark.parametrize("groups", [1, 4, 16])
def test_server_of_wide_and_narrow_graphs(mixed, groups):
    graphs, queries, want = mixed
    srv = eic.Server(graphs, groups=groups, idle_us=300)
    for _ in range(3):  # a burst, then one request to an idle server
        tickets = [srv.submit(k, s) for k, s in queries]
        for t, (k, _), x in zip(tickets, queries, want):
            assert srv.wait(t) == 0
            assert np.array_equal(srv.result(t, graphs[k].n)[0], x)
            srv.release(t)
        time.sleep(0.1)
        before = srv.stats()
        assert before["in_flight"] == 0 and before["queued"] == 0
        t = srv.submit(*queries[0])
        assert srv.wait(t) == 0
        assert np.array_equal(srv.result(t, graphs[0].n)[0], want[0])
        srv.release(t)
        after = srv.stats()
        assert after["kernel_launches"] == before["kernel_launches"] + 1
        assert after["completed"] == before["completed"] + 1
        time.sleep(0.1)
    srv.close()
