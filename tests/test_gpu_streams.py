"""First calls on a non-blocking stream while the legacy default stream is
busy: what a call sets up on the device is in place before its own kernels,
and nothing of it lands later, during a query."""
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

BUSY_CYCLES = 60_000_000  # about 30 ms


def _setup():
    wl = G.urand(13, 16, seed=91, nsources=2)
    g, og = eic.Graph(wl.n, wl.src, wl.dst, wl.w), O.Graph(wl.n, wl.src, wl.dst, wl.w)
    want = [og.dijkstra(int(s))[0] for s in wl.sources]
    return wl, g, want, torch.cuda.Stream()


def _check(outs, want):
    for out in outs:
        for k, d in enumerate(out):
            assert np.array_equal(eic.to_host_u32(d), want[k])


def test_first_query_beside_a_busy_default_stream():
    wl, g, want, side = _setup()
    outs = [[eic.new_dist(wl.n) for _ in want] for _ in range(100)]
    torch.cuda.synchronize()
    torch.cuda._sleep(BUSY_CYCLES)
    t0 = time.perf_counter()
    for out in outs:  # (the first makes the graph's workspace; the last come after the busy time)
        for s, d in zip(wl.sources, out):
            eic.sssp(g, int(s), dist=d, stream=side)
    assert time.perf_counter() - t0 < 10
    torch.cuda.synchronize()
    _check(outs, want)


def test_first_batch_beside_a_busy_default_stream():
    wl, g, want, side = _setup()
    outs = [[eic.new_dist(wl.n) for _ in want] for _ in range(60)]
    torch.cuda.synchronize()
    torch.cuda._sleep(BUSY_CYCLES)
    for k, out in enumerate(outs):
        if k % 2:
            assert eic.sssp_batch([g] * len(out), wl.sources, out, stream=side).tolist() == [0] * len(out)
        else:
            b = eic.Batch([g] * len(out), wl.sources, out)
            b.run(stream=side)
            assert b.wait(stream=side).tolist() == [0] * len(out)
    torch.cuda.synchronize()
    _check(outs, want)


def test_new_server_beside_a_busy_default_stream():
    wl, g, want, _ = _setup()
    torch.cuda.synchronize()
    for _ in range(4):
        torch.cuda._sleep(BUSY_CYCLES)
        with_server = eic.Server([g])
        t0 = time.perf_counter()
        while time.perf_counter() - t0 < 0.05:  # before and after the default stream is idle again
            tickets = [with_server.submit(0, int(s)) for s in wl.sources]
            for k, t in enumerate(tickets):
                assert with_server.wait(t, 5000) == 0
                assert np.array_equal(with_server.result(t, wl.n)[0], want[k])
                with_server.release(t)
        with_server.close()
        torch.cuda.synchronize()
