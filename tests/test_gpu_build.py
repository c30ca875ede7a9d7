"""The device CSR builder over its forms: tuple counts at the edges of the sort
and compaction tiles, keys that hold the weight and keys that do not, RtoW from
the histogram and from sorted weights, duplicates, loops and isolated vertices.
Rows, weights and RtoW equal the oracle's byte for byte."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2506_19349_gb300 as eic  # noqa: E402


def _check(n, src, dst, w, on_device=False):
    if on_device:
        g = eic.Graph(n, *[torch.from_numpy(x.view(np.int32)).cuda() for x in (src, dst, w)])
    else:
        g = eic.Graph(n, src, dst, w)
    og = O.Graph(n, src, dst, w)
    row, nbr, ww, rt = g.export()
    orow, onbr, ow = og.csr()
    assert np.array_equal(row, orow) and np.array_equal(nbr, onbr) and np.array_equal(ww, ow)
    assert (g.m, g.max_w, g.max_deg) == (og.m, og.maxw, og.maxdeg)
    if og.m:
        assert np.array_equal(rt, og.rtow()) and g.min_w == int(ow.min())
        assert g.highd0 == O.highd(og.degrees())
    deg = np.diff(orow).astype(np.int64)
    i2o, irow, inbr, iw = g.export_internal()
    assert np.array_equal(i2o, np.lexsort((np.arange(n), -deg))[: int((deg > 0).sum())].astype(np.uint32))
    assert np.array_equal(np.diff(irow.astype(np.int64)), deg[i2o])
    key = (iw.astype(np.uint64) << np.uint64(32)) | i2o[inbr].astype(np.uint64)
    same = np.ones(max(inbr.size - 1, 0), dtype=bool)
    same[irow[1:-1].astype(np.int64) - 1] = False
    assert np.all(key[1:][same] > key[:-1][same])
    g.close()


@pytest.mark.parametrize("T", [1, 2, 31, 2047, 2048, 2049, 4095, 4096, 4097, 12289, 300001])
@pytest.mark.parametrize("n,wmax", [(3, 5), (1000, 4095), (1000, 4096), (50000, 65535), (50000, 65536),
                                    (1 << 20, (1 << 24) + 5), ((1 << 20) + 1, 1 << 23), (70000, 4294967295)])
def test_csr(T, n, wmax):
    # (2 vbits + wbits: 7, 32, 33, 48, 49, 65 (no weight in the key), 66, 66)
    rng = np.random.default_rng(T * 7 + n)
    src = rng.integers(0, n, T).astype(np.uint32)
    dst = rng.integers(0, n, T).astype(np.uint32)
    w = np.where(rng.random(T) < 0.5, rng.integers(1, wmax + 1, T), wmax).astype(np.uint32)
    _check(n, src, dst, w, on_device=bool(T & 1))


def test_duplicates_and_loops():
    rng = np.random.default_rng(5)
    T = 30000  # long runs of equal pairs across tiles, in both orientations
    src = rng.integers(0, 3, T).astype(np.uint32)
    dst = rng.integers(0, 3, T).astype(np.uint32)
    _check(5, src, dst, rng.integers(9, 1 << 20, T).astype(np.uint32))
    _check(40000, src + np.uint32(20000), dst + np.uint32(20000), rng.integers(1, 300, T).astype(np.uint32))
    x = np.arange(5000, dtype=np.uint32)
    _check(5000, x, x, x + np.uint32(1))  # loops only


def test_hub_and_sparse():
    n = 1 << 21  # few edges on many vertices, one long row
    leaves = (np.arange(1, 9000, dtype=np.uint32) * np.uint32(233)) % np.uint32(n)
    _check(n, np.full(leaves.size, n - 1, np.uint32), leaves, leaves % np.uint32(7) + np.uint32(1))
