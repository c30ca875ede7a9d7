"""A dense graph of unit weights, whose every entry falls into one step: enough
entries of one weight that the query takes all blocks, and just too few."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2506_19349_gb300 as eic  # noqa: E402


@pytest.mark.parametrize("n", [6800, 7000])  # 2m of 46.2 M and 49.0 M on both sides of 45 * 2^20
def test_complete_graph_without_one_matching(n):
    i = torch.triu_indices(n, n, 1, device="cuda").to(torch.int32)
    keep = ~((i[0] % 2 == 0) & (i[1] == i[0] + 1))  # 2k and 2k + 1 are two hops apart
    src, dst = i[0][keep].contiguous(), i[1][keep].contiguous()
    g = eic.Graph(n, src, dst, torch.ones_like(src))
    assert g.m == n * (n - 1) // 2 - n // 2
    for s in (0, 4711):
        want = np.ones(n, np.uint32)
        want[s] = 0
        want[s ^ 1] = 2
        par = torch.empty(n, dtype=torch.int32, device="cuda")
        d, rc, _ = eic.sssp(g, s, parent=par)
        assert rc == 0 and np.array_equal(eic.to_host_u32(d), want)
        parents = np.full(n, s, np.uint32)
        parents[s ^ 1] = min(set(range(4)) - {s, s ^ 1})
        assert np.array_equal(eic.to_host_u32(par), parents)
