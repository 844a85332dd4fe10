"""The plan that a tensor-core exact search runs (esg_bruteforce_search_plan, no
GPU work): its order and coverage are the inspected plan's, its dense rows fit
their buffer, a work item's tiles are a rotation, and the shares balance the
costs it is made by."""
import numpy as np
import pytest

import synthetic

E = pytest.importorskip("paper_2504_04018_gb300")

TM = TN = 128


def _costs(d, k, l, r, order, tiles, items, cta_first, dense):
    """Cost of each CTA's share by the header's formula."""
    nk = -(-d // 64)
    f = 2.0 / nk
    g = f if nk <= 2 else f ** 3
    c = min(k + 12, 128) / 24.0 if k > 20 else 1.0
    lt, rt = l[order] // TN, r[order] // TN
    cost = np.empty(len(items))
    for i, (qt, off, cnt, _) in enumerate(items):
        a, b = tiles[off:off + cnt].min(), tiles[off:off + cnt].max()
        q = slice(qt * TM, min(len(order), (qt + 1) * TM))
        lo, hi = np.maximum(lt[q], a), np.minimum(rt[q], b)
        over, dn = lo <= hi, dense[q] >= 0
        begin = over & (lt[q] > a) & ~dn
        cost[i] = (cnt + 16.0 * c * g * begin.sum() + 0.5 * c * g * (over & ~dn & ~begin).sum() +
                   0.0104 * g * (hi - lo + 1)[over & dn].sum())
    return np.array([cost[cta_first[c]:cta_first[c + 1]].sum() for c in range(len(cta_first) - 1)])


def check(n, d, k, l, r, ctas=152):
    l, r = np.asarray(l, np.int64), np.asarray(r, np.int64)
    order, tiles, items, cta_first, dense, floats, period = plan = E.esg_bruteforce_search_plan(n, d, k, l, r, ctas)
    order0, tiles0, _, _ = E.esg_bruteforce_plan(n, d, l, r, ctas)
    assert np.array_equal(order, order0)
    # the items: consecutive pieces of the sequence, at most one per CTA and query tile
    T = len(tiles)
    assert T == len(tiles0)
    G = len(cta_first) - 1
    assert G == max(1, min(ctas, T)) and cta_first[0] == 0 and cta_first[-1] == len(items)
    if T:
        assert items[0, 1] == 0 and np.all(items[:, 2] >= 1) and items[-1, 1] + items[-1, 2] == T
        assert np.array_equal(items[1:, 1], items[:-1, 1] + items[:-1, 2]) and np.all(np.diff(items[:, 0]) >= 0)
        assert np.all(np.diff(cta_first) >= 1)
    for c in range(G):
        qt = items[cta_first[c]:cta_first[c + 1], 0]
        assert len(np.unique(qt)) == len(qt)
    # an item's tiles: its piece of the ascending sequence, rotated to the first
    # one at or after a multiple of the period
    for _, off, cnt, _ in items:
        asc, got = tiles0[off:off + cnt], tiles[off:off + cnt]
        lead = int(np.searchsorted(asc, -(-int(asc[0]) // period) * period))
        assert np.array_equal(got, np.roll(asc, -lead))
    # dense rows: the ranges up to a width that is the widest or a power of two
    # below it, none past 128 dimensions, one after the other in their buffer
    widest, most = (131_072, 1 << 28) if k <= 20 else (262_144, 1 << 29)
    w = (r - l + 1)[order]
    on = dense >= 0
    room = (r[order] | 3) - (l[order] & ~3) + 1
    assert floats <= most and floats == room[on].sum()
    if d > 128:
        assert not on.any()
    else:
        W = widest
        while W >= 64 and room[w <= W].sum() > most:
            W //= 2
        assert np.array_equal(on, w <= W if W >= 64 else np.zeros(len(w), bool))
    at = np.argsort(dense[on], kind="stable")
    off, size = dense[on][at], room[on][at]
    assert np.all(off % 4 == 0) and np.all(off + size <= floats)
    assert np.all(off[1:] == off[:-1] + size[:-1]) and (len(off) == 0 or off[0] == 0)
    return plan


@pytest.mark.parametrize("seed,nq,ctas,d,k", [(0, 1000, 152, 128, 10), (1, 1300, 37, 768, 10), (2, 129, 152, 64, 100),
                                              (3, 5000, 152, 96, 21), (4, 700, 152, 129, 120), (5, 300, 9, 100, 1)])
def test_search_plan_random(seed, nq, ctas, d, k):
    n = 200_003
    rng = np.random.default_rng(seed)
    l, r = synthetic.ranges_from_fractions(n, 2.0 ** -rng.integers(0, 14, nq), seed + 10)
    l = np.where(rng.random(nq) < 0.05, r + 1, l)   # some invalid ranges
    check(n, d, k, l, r, ctas)


def test_search_plan_edges():
    check(1000, 128, 10, [5, -1, 10], [4, 3, 1000])            # no valid range
    check(1000, 128, 10, [0], [999])                           # fewer tiles than CTAs
    l = np.array([0, 999] * 64 + [17])
    check(1000, 64, 100, l, l)                                 # one-point ranges, a partial query tile
    n = 400_000                                                # at and just past the widest dense row
    for k, w in ((20, 131_072), (21, 262_144)):
        check(n, 128, k, [0, 1, 2, 3, 5], np.array([0, 1, 2, 3, 5]) + w - 1 + np.array([0, 0, 0, 0, 1]))


@pytest.mark.parametrize("k,nq", [(10, 3000), (100, 6000)])
def test_search_plan_halves_the_dense_width(k, nq):
    """More points in narrow ranges than the buffer holds: the widest ones keep lists."""
    n = 1_000_000
    rng = np.random.default_rng(k)
    w = np.exp(rng.uniform(np.log(60_000), np.log(131_072), nq)).astype(np.int64)
    l = (rng.random(nq) * (n - w)).astype(np.int64)
    dense = check(n, 96, k, l, l + w - 1)[4]
    assert (dense >= 0).any() and (dense < 0).any()


def test_search_plan_balances_its_cost():
    """Widths 2^-j N (j = 0..10) over 1M points: the largest share stays within
    15 % of the mean, as in the inspected plan."""
    n = 1_000_000
    for nq, d, k in ((10_000, 128, 10), (10_000, 768, 10), (10_000, 96, 100), (1000, 128, 10)):
        l, r = synthetic.ranges_from_fractions(n, 2.0 ** -(np.arange(nq) % 11).astype(np.float64), 77)
        order, tiles, items, cta_first, dense, _, _ = check(n, d, k, l, r)
        cost = _costs(d, k, l, r, order, tiles, items, cta_first, dense)
        assert cost.max() <= 1.15 * cost.mean(), (nq, d, k, cost.max() / cost.mean())
