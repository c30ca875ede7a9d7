"""The single-precision filters of the step boundary, restated in numpy
float32, against the double-precision formulas of the oracle: wherever a filter
decides, it decides as they do."""
import numpy as np
import pytest

import oracle as O

f32 = np.float32


@pytest.mark.parametrize("beta", [0.9, 0.5, 0.05, 0.951])
def test_gap_estimate(beta):
    """Eq. 2's RtoW position in float32 is within the guard of 0.02 of the double one."""
    rng = np.random.default_rng(71)
    n = 200000
    two_m = np.exp(rng.uniform(np.log(8), np.log(2.0**32 - 2), n)).astype(np.uint64)
    sumd = (rng.random(n) * two_m).astype(np.uint64)
    highd = np.minimum(np.exp(rng.uniform(np.log(4), np.log(1e6), n)), two_m).astype(np.uint64)
    highd = np.where(rng.random(n) < 0.5, rng.integers(4, 40, n).astype(np.uint64), highd)
    big = np.maximum(sumd, two_m - sumd)
    prob = np.minimum(big / two_m, beta)
    pos = -np.expm1(np.log1p(-prob) / (prob * highd)) * 4095.0
    p = np.minimum(big.astype(f32) / two_m.astype(f32), f32(beta))
    with np.errstate(divide="ignore"):
        q = -np.expm1(np.log1p(-p) / (p * highd.astype(f32))) * f32(4095)
    use = p <= f32(0.95)
    assert use.any() and np.abs(q.astype(np.float64) - pos)[use].max() < 0.01
    frac = q - np.floor(q)
    decided = use & (frac > f32(0.02)) & (frac < f32(0.98))
    assert (np.floor(q)[decided] == np.floor(pos)[decided]).all()
    table = np.arange(4096, dtype=np.uint32)
    for i in np.flatnonzero(decided)[:500]:
        assert O.gap(int(sumd[i]), int(highd[i]), int(two_m[i]), table, beta=beta)[0] == int(np.floor(q[i]))


@pytest.mark.parametrize("maxw,st_num", [(2, 7), (255, 1024), (4095, 1024), (65535, 4000), ((1 << 20) - 1, 1024)])
def test_profit_filter(maxw, st_num):
    """The candidates that pass the integer test and the float32 estimate hold
    the first largest positive profit."""
    rng = np.random.default_rng(maxw)
    kept = positive = 0
    for _ in range(150):
        two_m = int(np.exp(rng.uniform(np.log(64), np.log(2.0**32 - 2))))
        sumd = int(rng.random() * two_m * rng.choice([0.5, 0.05, 1e-3]))
        ub = int(rng.integers(1, 3 * maxw + 2))
        y = ub + int(rng.integers(1, maxw + 1))
        st0 = int(rng.integers(0, ub))
        st1 = int(rng.integers(st0, ub + 1))
        lo = max(ub - maxw, 0)
        # degree sums of the distances [lo, ub), at most two_m - sumd in all
        share = rng.random(min(ub - lo, 4096)) ** rng.integers(1, 6)
        dens = np.zeros(ub - lo)
        dens[np.sort(rng.choice(ub - lo, share.size, replace=False))] = share
        deg = np.floor(dens / max(dens.sum(), 1e-9) * (two_m - sumd) * rng.random()).astype(np.int64)
        suffix = np.concatenate([np.cumsum(deg[::-1])[::-1], [0]])
        push_w = min(y, ub + maxw) - ub
        inv, inv2m = f32(1) / f32(maxw), f32(1) / f32(two_m)
        e = f32(push_w) * f32(suffix[0]) * inv * f32(2.0**-19)
        xs, vs, ps = [], [], []
        for k in range(st_num + 1):
            x = st0 + k * (st1 - st0) // st_num
            if x >= ub:
                continue
            xc = max(x, ub - maxw)
            d = int(suffix[xc - lo])
            ps.append(O.profit(x, ub, y, d, sumd, maxw, two_m))
            pull_w = min(y, xc + maxw) - xc
            if push_w * d <= pull_w * sumd:
                assert ps[-1] <= 0.0
                vs.append(f32(-1))
            else:
                pulled = f32(pull_w) * f32(sumd) * inv
                vs.append(f32(push_w) * f32(d) * inv - pulled * f32(d) * inv2m - pulled + e)
            xs.append(k)
        if not ps or max(ps) <= 0.0:
            continue
        positive += 1
        best, top = int(np.argmax(ps)), max(vs)
        assert vs[best] > 0 and vs[best] >= top - f32(2) * e
        kept += sum(v > 0 and v >= top - f32(2) * e for v in vs)
    assert positive > 5 and kept >= positive


def test_highd_crossing():
    """The last present rank with 2 low <= total, or the next present one,
    whichever splits more evenly (ties: the former), is the oracle's highD."""
    rng = np.random.default_rng(72)
    for _ in range(400):
        dv = np.sort(rng.choice(np.arange(1, 200), rng.integers(1, 40), replace=False))
        cnt = rng.integers(0, 5, dv.size) * (rng.random(dv.size) < 0.7)
        degrees = np.repeat(dv, cnt).astype(np.uint32)
        total, low, got, prev = int((dv * cnt).sum()), 0, 0, None
        for d, c in zip(dv.tolist(), cnt.tolist()):
            if not c:
                continue
            if 2 * low <= total:
                got, prev = d, total - 2 * low
            else:
                if 2 * low - total < prev:
                    got = d
                break
            low += d * c
        assert got == (O.highd(degrees) if total else 0)
