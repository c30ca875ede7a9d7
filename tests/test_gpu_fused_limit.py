"""A fused round ends after a bounded number of waves: a step that spans a long
chain takes several rounds, so that the blocks that wait at the barrier
meanwhile (with a short limit here) do not give up."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2506_19349_gb300 as eic  # noqa: E402


@pytest.mark.parametrize("heavy_min", [16, 64])  # (with 16 the graph with a vertex of degree 40 is not road-like)
@pytest.mark.parametrize("chains", [1, 40])
def test_long_chains_in_one_step(chains, heavy_min):
    # unit-weight paths joined at vertex 0, the last edge of the first one as wide as all of them: highD is 2, so
    # Eq. 2 has no solution, the gap is the largest weight and the second step spans the paths
    per = 50000 if chains == 1 else 8000
    n = 1 + chains * per
    at = np.arange(1, n, dtype=np.uint32)
    src = np.where((at - 1) % per == 0, 0, at - 1).astype(np.uint32)
    w = np.ones(n - 1, np.uint32)
    w[per - 1] = 65535
    g, og = eic.Graph(n, src, at, w), O.Graph(n, src, at, w)
    for s in (1 + per // 2, n - 1 if chains == 1 else 7):
        want = og.dijkstra(s)[0]
        p = eic.default_params(max_spin_log2=14, heavy_min=heavy_min, flags=eic.FLAG_NO_PULL)
        d, rc, info = eic.sssp(g, s, params=p, trace_cap=64, raise_on_error=False)
        assert rc == 0 and np.array_equal(eic.to_host_u32(d), want)
        long_steps = [r for r in info["trace"] if r["settled"] > per // 3]
        assert long_steps and all(r["rounds"] > 1 for r in long_steps)
        d = eic.new_dist(n)
        assert eic.sssp_batch([g], [s], [d], params=p).tolist() == [0]
        assert np.array_equal(eic.to_host_u32(d), want)


@pytest.mark.parametrize("degree", [2, 10, 12, 14])  # (the larger, the fewer waves to a round)
def test_wait_of_the_stated_length(degree):
    """A wait shorter than max_spin_log2 states (2^max_spin_log2 times 0.5 us) does not run out."""
    per, leaves = 40000, max(0, degree - 2)
    n = 1 + per + leaves  # a path, and leaves on a vertex near its end
    at = np.arange(1, n, dtype=np.uint32)
    src = np.where(at > per, per - 10, at - 1).astype(np.uint32)
    w = np.ones(n - 1, np.uint32)
    w[per - 1] = 65535
    g, og = eic.Graph(n, src, at, w), O.Graph(n, src, at, w)
    assert g.max_deg == degree
    s = per - 20
    want = og.dijkstra(s)[0]
    flags = eic.FLAG_NO_PULL
    eic.sssp(g, s, params=eic.default_params(flags=flags))
    _, _, info = eic.sssp(g, s, params=eic.default_params(flags=flags), trace_cap=64)
    rounds = max(r["rounds"] for r in info["trace"])
    assert rounds > 10
    wait_us = 1e3 * info["kernel_ms"] / rounds  # the other blocks' wait in each of them
    log2 = int(np.ceil(np.log2(1.2 * wait_us / 0.5)))
    d, rc, _ = eic.sssp(g, s, params=eic.default_params(flags=flags, max_spin_log2=log2), raise_on_error=False)
    assert rc == 0 and np.array_equal(eic.to_host_u32(d), want)
