"""Kernels at the sizes where their tiling can go wrong: edges of tiles and
chunks, remainders, the smallest and largest of each range."""
import os
import subprocess
import sys

import numpy as np
import pytest

import oracle as O
from oracle import mlp as OM

torch = pytest.importorskip("torch")
E = pytest.importorskip("paper_2504_04018_gb300")

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _t(a):
    return torch.as_tensor(np.ascontiguousarray(a), device=DEV)


@pytest.mark.parametrize("B", [1, 7, 8, 9, 2431, 2432, 2433, 5000])
def test_mlp_batch_edges(B):
    """Chunks of 8 rows on at most 304 blocks: part chunks, one chunk per
    block, blocks with one and two chunks. Sums of float32 terms grouped by
    8 rows and then by block: well within 1e-4 of the largest gradient, and
    the same bits when repeated."""
    rng = np.random.default_rng(B)
    F = E.esg_mlp_num_features()
    p = (rng.standard_normal(OM.n_params(F)) * 0.2).astype(np.float32)
    X = (rng.standard_normal((B, F)) * 2 + 0.5).astype(np.float32)
    T = rng.standard_normal((B, 2)).astype(np.float32)
    mu, sigma = rng.standard_normal(F).astype(np.float32), (rng.random(F) + 0.5).astype(np.float32)
    a = (_t(p), _t(X), _t(T), _t(mu), _t(sigma))
    y = E.esg_mlp_forward(a[0], a[1], a[3], a[4]).cpu().numpy()
    ref, _ = OM.forward(p, X, mu, sigma)
    assert np.allclose(y, ref, rtol=1e-5, atol=1e-5)
    loss, g = E.esg_mlp_loss_grad(*a, 0.9)
    again, g2 = E.esg_mlp_loss_grad(*a, 0.9)
    ref_loss, ref_g = OM.loss_and_grad(p, X, T, mu, sigma, 0.9)
    assert abs(loss - ref_loss) <= 1e-5 * max(1.0, abs(ref_loss))
    assert np.max(np.abs(g.cpu().numpy() - ref_g)) <= 1e-4 * np.max(np.abs(ref_g)) + 1e-8
    assert loss == again and torch.equal(g, g2)


def _check_exact(X, Q, l, r, k, metric, ids, dist, count):
    """Exact answers against float64: counts, distances within 1e-5 relative
    or the forward error bound of the FP32 sum, and every row that float64
    puts below the k-th distance by more than four times that."""
    X64, Q64 = torch.as_tensor(X).double(), torch.as_tensor(Q).double()
    for i in range(len(Q)):
        a, b = int(l[i]), int(r[i]) + 1
        terms = (X64[a:b] - Q64[i]) ** 2 if metric == "l2" else -X64[a:b] * Q64[i]
        d = terms.sum(1)
        c = min(k, b - a)
        want, order = torch.sort(d)
        assert count[i] == c and np.all(ids[i, c:] == -1) and np.all(np.isinf(dist[i, c:]))
        got = ids[i, :c]
        assert len(set(got.tolist())) == c and got.min() >= a and got.max() < b
        bound = X.shape[1] * 2.0 ** -24 * terms.abs().sum(1)
        tol = np.maximum(1e-5 * np.abs(d.numpy()), bound.numpy())
        assert np.all(np.abs(dist[i, :c] - d.numpy()[got - a]) <= tol[got - a])
        assert np.all(np.diff(dist[i, :c]) >= 0)
        sure = order[:c][want[:c] < want[c - 1] - 4 * tol.max()] + a
        assert set(sure.tolist()) <= set(got.tolist())


@pytest.mark.parametrize("d", [32, 64, 100, 128, 132, 192, 256, 260])
@pytest.mark.parametrize("metric", ["l2", "ip"])
@pytest.mark.parametrize("k", [1, 12, 13, 20, 21, 50])
def test_exact_lists_and_dense_rows(d, metric, k):
    """Lists of 24 and 32 in registers and of up to 62 in memory, dense rows
    up to 131,072 points wide and lists above, query tiles in tensor memory
    (d <= 256, one or two issuers) and streamed; ranges at tile edges, one
    point, the whole set, and a second, partial query tile."""
    n, nq = 131_072 + 777, 131
    g = torch.Generator(device=DEV).manual_seed(d * 100 + k)
    cen = torch.randn(64, d, generator=g, device=DEV)
    X = cen[torch.randint(0, 64, (n,), generator=g, device=DEV)] + 0.5 * torch.randn(n, d, generator=g, device=DEV)
    Q = cen[torch.randint(0, 64, (nq,), generator=g, device=DEV)] + 0.5 * torch.randn(nq, d, generator=g, device=DEV)
    rng = np.random.default_rng(d + k)
    w = np.exp(rng.uniform(0, np.log(n), nq)).astype(np.int64)
    l = (rng.random(nq) * (n - w + 1)).astype(np.int64)
    r = l + w - 1
    edge = [(0, n - 1), (0, 131_071), (0, 131_072), (1, n - 1), (0, 0), (n - 1, n - 1), (127, 128), (128, 255),
            (127, 256), (n - 777, n - 1), (700, 131_771), (500, n - 3)]
    l[:len(edge)], r[:len(edge)] = zip(*edge)
    ids, dist, count = E.esg_bruteforce_filtered_knn(X, Q, _t(l), _t(r), k, metric)
    torch.cuda.synchronize()
    pick = list(range(len(edge))) + rng.choice(np.arange(len(edge), nq), 12, replace=False).tolist()
    _check_exact(X.cpu().numpy(), Q.cpu().numpy()[pick], l[pick], r[pick], k, metric, ids.cpu().numpy()[pick],
                 dist.cpu().numpy()[pick], count.cpu().numpy()[pick])


@pytest.mark.parametrize("d", [32, 64, 128, 192, 260])
@pytest.mark.parametrize("metric", ["l2", "ip"])
@pytest.mark.parametrize("k", [51, 56, 57, 100, 116, 120, 121])
def test_exact_long_lists(d, metric, k):
    """Lists of up to 128 (k up to 120, summed in dimension order where the
    SIMT kernel used to answer) and the SIMT kernel above, over ranges that are
    dense rows and lists, shorter than k, one point, and at tile edges."""
    n, nq = 9_001, 140
    g = torch.Generator(device=DEV).manual_seed(d * 1000 + k)
    X = torch.randn(n, d, generator=g, device=DEV)
    Q = torch.randn(nq, d, generator=g, device=DEV)
    rng = np.random.default_rng(d + k)
    w = np.exp(rng.uniform(0, np.log(n), nq)).astype(np.int64)
    l = (rng.random(nq) * (n - w + 1)).astype(np.int64)
    r = l + w - 1
    edge = [(0, n - 1), (0, 0), (n - 1, n - 1), (127, 128), (128, 128 + k - 1), (100, 100 + k), (0, 255)]
    l[:len(edge)], r[:len(edge)] = zip(*edge)
    ids, dist, count = E.esg_bruteforce_filtered_knn(X, Q, _t(l), _t(r), k, metric)
    torch.cuda.synchronize()
    pick = list(range(len(edge))) + rng.choice(np.arange(len(edge), nq), 20, replace=False).tolist()
    _check_exact(X.cpu().numpy(), Q.cpu().numpy()[pick], l[pick], r[pick], k, metric, ids.cpu().numpy()[pick],
                 dist.cpu().numpy()[pick], count.cpu().numpy()[pick])


@pytest.mark.parametrize("k,d", [(100, 96), (57, 64), (51, 128)])
def test_exact_long_lists_equal_simt(k, d, monkeypatch):
    """Where the SIMT kernel used to answer, the lists' answers are its, bit
    for bit: ids, distances, counts (ranges of list and dense rows)."""
    n, nq = 300_000, 40
    g = torch.Generator(device=DEV).manual_seed(k)
    cen = torch.randn(200, d, generator=g, device=DEV)
    X = cen[torch.randint(0, 200, (n,), generator=g, device=DEV)] + 0.3 * torch.randn(n, d, generator=g, device=DEV)
    Q = X[torch.randint(0, n, (nq,), generator=g, device=DEV)] + 0.1 * torch.randn(nq, d, generator=g, device=DEV)
    rng = np.random.default_rng(k)
    w = np.exp(rng.uniform(np.log(50), np.log(n), nq)).astype(np.int64)
    w[:2] = n, n - 1
    l = (rng.random(nq) * (n - w + 1)).astype(np.int64)
    a = E.esg_bruteforce_filtered_knn(X, Q, _t(l), _t(l + w - 1), k)
    monkeypatch.setenv("ESG_BF_SIMT", "1")
    b = E.esg_bruteforce_filtered_knn(X, Q, _t(l), _t(l + w - 1), k)
    torch.cuda.synchronize()
    assert all(torch.equal(x, y) for x, y in zip(a, b))


@pytest.mark.parametrize("d,M,efc,n", [(8, 1, 3, 200), (32, 4, 40, 400), (128, 16, 200, 500), (768, 8, 300, 400)])
@pytest.mark.parametrize("metric", ["l2", "ip"])
def test_build_one_at_a_time_is_the_oracles(d, M, efc, n, metric):
    """With rounds of one point the build is the oracle's: the same rows (as
    sets) on small integer coordinates, whose distances are exact in float32
    (pools of one and several steps, of rows staged in shared memory wholly
    and in part; full rows re-selected)."""
    rng = np.random.default_rng(d + M)
    X = rng.integers(-20, 21, (n, d)).astype(np.float32)
    ix = E.esg_build(X, None, M=M, leaf_size=64, n_entries=8, ef_construction=efc, batch_div=1 << 20, metric=metric)
    adj, _, _ = E.esg_index_export(ix)
    want = O.build_index(X, np.arange(n, dtype=np.float64), metric, 64, M, efc=efc, n_entries=8).adj
    assert adj.shape == want.shape
    for lev in range(ix.L):
        for p in range(n):
            got = adj[lev, p]
            assert np.all(np.diff((got == 0xFFFFFFFF).astype(int)) >= 0)
            assert set(got.tolist()) == set(np.asarray(want[lev, p], dtype=np.uint32).tolist()), (lev, p)


def _long_list_case(nq=70, n=20_000, d=64, k=100):
    g = torch.Generator(device=DEV).manual_seed(5)
    X = torch.randn(n, d, generator=g, device=DEV)
    Q = torch.randn(nq, d, generator=g, device=DEV)
    rng = np.random.default_rng(5)
    w = np.exp(rng.uniform(0, np.log(n), nq)).astype(np.int64)
    l = (rng.random(nq) * (n - w + 1)).astype(np.int64)
    return X, Q, _t(l), _t(l + w - 1), k


@pytest.mark.parametrize("k", [10, 60])
def test_exact_short_range_keeps_points_without_bf16_parts(k, monkeypatch):
    """A finite element above the largest BF16 leaves its row without an
    approximate distance; a range shorter than the list still holds the row."""
    X, Q, _, _, _ = _long_list_case(nq=4, n=300)
    X[7, 0] = 3.4e38
    Q[:, 0] = 1e-30
    l, r = _t(np.array([0, 7, 3, 100])), _t(np.array([7, 7, 20, 111]))
    a = E.esg_bruteforce_filtered_knn(X, Q, l, r, k, "ip")
    monkeypatch.setenv("ESG_BF_SIMT", "1")
    b = E.esg_bruteforce_filtered_knn(X, Q, l, r, k, "ip")
    assert a[2].tolist()[:2] == [8, 1] and torch.equal(a[2], b[2]) and torch.equal(a[0], b[0])


def test_exact_long_lists_under_capture():
    """A call the SIMT kernel can answer too is captured like any launch."""
    X, Q, l, r, k = _long_list_case()
    want = E.esg_bruteforce_filtered_knn(X, Q, l, r, k)
    out = tuple(torch.empty_like(t) for t in want)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        E.esg_bruteforce_filtered_knn(X, Q, l, r, k, out=out)
    for t in out:
        t.zero_()
    g.replay()
    torch.cuda.synchronize()
    assert all(torch.equal(x, y) for x, y in zip(want, out))


@pytest.mark.parametrize("k,kth", [(100, 1), (100, 2), (10, 2)])
def test_exact_without_memory_for_scratch(k, kth, monkeypatch):
    """Short of memory for the point blocks, lists of k = 100 come from the SIMT
    kernel; short of it for the dense rows, every range keeps lists."""
    X, Q, l, r, _ = _long_list_case()
    want = E.esg_bruteforce_filtered_knn(X, Q, l, r, k)
    monkeypatch.setenv("ESG_FAULT_ALLOC", str(kth))
    got = E.esg_bruteforce_filtered_knn(X, Q, l, r, k)
    torch.cuda.synchronize()
    assert all(torch.equal(x, y) for x, y in zip(want, got))


@pytest.mark.parametrize("M", [8, 16, 32])
@pytest.mark.parametrize("width", [1, 2])
@pytest.mark.parametrize("rows", ["f32", "bf16"])
def test_search_merges_every_batch_size(M, width, rows):
    """Rows of 16, 32 and 64 neighbours, one or two expanded at a time: admitted
    batches from one candidate to 128, merged 32 at a time. With a beam that holds
    the whole set, answers are the exact ones (of the reachable points: recall
    0.99), each once, ascending, at its float64 distance."""
    n, nq, k = 700, 40, 100
    rng = np.random.default_rng(M)
    X = rng.standard_normal((n, 32)).astype(np.float32)
    ix = E.esg_build(X, None, M=M, leaf_size=64, n_entries=16, storage=rows)
    q = rng.standard_normal((nq, 32)).astype(np.float32)
    w = np.exp(rng.uniform(np.log(k), np.log(n), nq)).astype(np.int64)
    l = (rng.random(nq) * (n - w + 1)).astype(np.int64)
    ids, dist, count, status = (t.cpu().numpy() for t in E.esg_search_batch(
        ix, _t(q), _t(l), _t(l + w - 1), None, k,
        params=E.search_params(704, traversal=rows, width=width))[:4])
    hit = 0
    for i in range(nq):
        got = ids[i, :count[i]]
        assert len(set(got.tolist())) == len(got) and got.min() >= l[i] and got.max() < l[i] + w[i]
        d = ((X.astype(np.float64) - q[i]) ** 2).sum(1)
        assert np.allclose(dist[i, :count[i]], d[got], rtol=1e-5) and np.all(np.diff(dist[i, :count[i]]) >= 0)
        want = np.argsort(d[l[i]:l[i] + w[i]], kind="stable")[:k] + l[i]
        hit += len(set(want.tolist()) & set(got.tolist()))
    assert hit >= 0.99 * nq * k


@pytest.mark.parametrize("k", [10, 60])
def test_exact_equal_zeros_order_by_row(k):
    """Inner products that underflow from either side are 0, a tie of all rows:
    the answer is the first rows, in order."""
    X, Q, _, _, _ = _long_list_case(nq=3, d=32)
    X[:] = 1e-30
    X[::3] = -1e-30
    Q[:] = 1e-30
    l = np.array([0, 5, 0])
    r = np.array([19, 24, len(X) - 1])
    ids, dist, count = E.esg_bruteforce_filtered_knn(X, Q, _t(l), _t(r), k, "ip")
    for i, c in enumerate((min(k, 20), min(k, 20), k)):
        assert count[i] == c and torch.all(dist[i, :c] == 0)
        assert ids[i, :c].tolist() == list(range(l[i], l[i] + c))


@pytest.mark.parametrize("k", [10, 60])
def test_exact_inner_products_near_the_largest_float(k, monkeypatch):
    """A product that FP32 holds, of elements whose BF16 parts' product does not."""
    X, Q, _, _, _ = _long_list_case(nq=3)
    X[3] = 0
    Q[0] = 0
    X[3, 0], Q[0, 0] = -1.843e19, 1.843e19
    l, r = _t(np.array([0, 0, 0])), _t(np.array([9, 299, len(X) - 1]))
    a = E.esg_bruteforce_filtered_knn(X, Q, l, r, k, "ip")
    assert a[2].tolist() == [10, k, k] and 3 in a[0][0].tolist()
    monkeypatch.setenv("ESG_BF_SIMT", "1")
    b = E.esg_bruteforce_filtered_knn(X, Q, l, r, k, "ip")
    assert torch.equal(a[2], b[2]) and torch.equal(a[0], b[0])


_HOST_FAILURE = """
import os, torch
import paper_2504_04018_gb300 as E
g = torch.Generator(device="cuda").manual_seed(1)
X = torch.randn(200_000, 128, generator=g, device="cuda")
Q = torch.randn(300, 128, generator=g, device="cuda")
l = torch.zeros(300, dtype=torch.int64, device="cuda")
r = l + 199_999
want = {k: E.esg_bruteforce_filtered_knn(X, Q, l, r, k) for k in (10, 100)}
def used():
    torch.cuda.synchronize()
    free, total = torch.cuda.mem_get_info()
    return total - free
before = used()
for k in (10, 100):
    for kth in ("1", "2"):
        os.environ["ESG_FAULT_HOST_ALLOC"] = kth
        try:
            got = E.esg_bruteforce_filtered_knn(X, Q, l, r, k)
            assert k == 100 and all(torch.equal(a, b) for a, b in zip(got, want[k]))
        except E.EsgError as e:
            assert k == 10 and "out of memory" in str(e), str(e)
        del os.environ["ESG_FAULT_HOST_ALLOC"]
        E.esg_bruteforce_filtered_knn(X, Q, l, r, k)
after = used()
assert after <= before + (8 << 20), (before, after)
print("ok")
"""


def test_exact_host_failure_gives_scratch_back():
    """A host allocation that fails with device scratch held and work queued: the
    call fails (or answers through the SIMT kernel) and its scratch, 0.1 GB, is
    given back. In a process whose pool keeps nothing mapped."""
    env = dict(os.environ, ESG_POOL_KEEP_MB="0")
    out = subprocess.run([sys.executable, "-c", _HOST_FAILURE], env=env, capture_output=True, text=True, timeout=300,
                         cwd=os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
    assert out.returncode == 0 and out.stdout.strip().endswith("ok"), out.stderr[-2000:]


@pytest.mark.parametrize("n,nq,w,tensor", [(1_000_000, 1, 1000, False), (1_000_000, 1, 100_000, True),
                                           (1_000_000, 64, 1000, True), (700, 1, 700, False), (60, 500, 60, False),
                                           (2_000_000, 3, 100, False)])
@pytest.mark.parametrize("k", [57, 100])
def test_exact_long_lists_take_the_shorter_path(n, nq, w, tensor, k, monkeypatch):
    """A few narrow ranges, and small sets, are answered by the SIMT kernel without
    preparing the points; the answers do not depend on the path."""
    g = torch.Generator(device=DEV).manual_seed(n + nq)
    X = torch.randn(n, 32, generator=g, device=DEV)
    Q = torch.randn(nq, 32, generator=g, device=DEV)
    l = np.random.default_rng(n).integers(n // 2, n // 2 + 200 + 1, nq) if n > 1000 else np.zeros(nq, np.int64)
    r = l + w - 1
    E.esg_profile_enable(True)
    try:
        a = E.esg_bruteforce_filtered_knn(X, Q, _t(l), _t(r), k)
        torch.cuda.synchronize()
        assert (E.esg_profile_tensor_work() > 0) == tensor
    finally:
        E.esg_profile_enable(False)
    monkeypatch.setenv("ESG_BF_SIMT", "1")
    b = E.esg_bruteforce_filtered_knn(X, Q, _t(l), _t(r), k)
    torch.cuda.synchronize()
    assert all(torch.equal(x, y) for x, y in zip(a, b))


@pytest.mark.parametrize("d,M,efc,n", [(32, 4, 40, 6000), (128, 16, 200, 5000), (768, 8, 100, 3000)])
@pytest.mark.parametrize("metric", ["l2", "ip"])
def test_build_by_warps_is_the_build_by_blocks(d, M, efc, n, metric, monkeypatch):
    """Rounds of one to half of the points, every round's edges by blocks, by warps,
    and by the rule's choice: the same rows (as sets)."""
    rng = np.random.default_rng(d)
    X = rng.standard_normal((n, d)).astype(np.float32)
    rows = []
    for points in (str(1 << 30), "1", None):
        if points is None:
            monkeypatch.delenv("ESG_BUILD_WARP_ROUND")
        else:
            monkeypatch.setenv("ESG_BUILD_WARP_ROUND", points)
        ix = E.esg_build(X, None, M=M, leaf_size=64, n_entries=8, ef_construction=efc, batch_div=1, metric=metric)
        adj, _, _ = E.esg_index_export(ix)
        assert np.all(np.diff((adj == 0xFFFFFFFF).astype(np.int8), axis=-1) >= 0)
        rows.append(np.sort(adj, axis=-1))
    assert np.array_equal(rows[0], rows[1]) and np.array_equal(rows[0], rows[2])


@pytest.mark.parametrize("B", [9727, 9728, 9729, 30_001])
def test_mlp_forward_block_edges(B):
    """Chunks of 8 rows on at most 1,216 blocks: blocks with one and several."""
    rng = np.random.default_rng(B)
    F = E.esg_mlp_num_features()
    p = (rng.standard_normal(OM.n_params(F)) * 0.2).astype(np.float32)
    X = (rng.standard_normal((B, F)) * 2 + 0.5).astype(np.float32)
    mu, sigma = rng.standard_normal(F).astype(np.float32), (rng.random(F) + 0.5).astype(np.float32)
    y = E.esg_mlp_forward(_t(p), _t(X), _t(mu), _t(sigma)).cpu().numpy()
    assert np.allclose(y, OM.forward(p, X, mu, sigma)[0], rtol=1e-5, atol=1e-5)


@pytest.mark.parametrize("metric", ["l2", "ip"])
@pytest.mark.parametrize("rows", ["f32", "bf16", "fp8"])
def test_search_orders_nan_distances(metric, rows):
    """NaN elements in points and queries, and inner products of infinite terms:
    such points are at +inf, each point comes at most once and from its range,
    and queries without them are answered as without them."""
    n, d, k, nq = 3000, 32, 20, 64
    rng = np.random.default_rng(7)
    X = rng.standard_normal((n, d)).astype(np.float32)
    bad = rng.choice(n, 90, replace=False)
    X[bad[:30], 0] = np.nan
    X[bad[30:60]] = np.nan
    X[bad[60:]] = np.where(np.arange(d) % 2, np.float32(3e37), np.float32(-3e37))
    q = rng.standard_normal((nq, d)).astype(np.float32)
    q[::4, 1] = np.nan
    q[1::8] *= 100
    w = np.where(np.arange(nq) % 2, 40, 2500)   # scanned leaf pieces and graph pieces
    l = (rng.random(nq) * (n - w + 1)).astype(np.int64)
    ix = E.esg_build(X, None, M=16, leaf_size=64, n_entries=16, ef_construction=100, metric=metric, storage=rows)
    ids, dist, count, _ = (t.cpu().numpy() for t in E.esg_search_batch(
        ix, _t(q), _t(l), _t(l + w - 1), None, k, params=E.search_params(256, traversal=rows))[:4])
    is_bad = np.zeros(n, bool)
    is_bad[bad] = True
    for i in range(nq):
        got, dd = ids[i, :count[i]], dist[i, :count[i]]
        assert len(set(got.tolist())) == len(got) and np.all((got >= l[i]) & (got < l[i] + w[i]))
        assert not np.isnan(dd).any() and np.all(dd[:-1] <= dd[1:])
        if i % 4 == 0:
            assert np.all(dd == np.inf)
            continue
        good = np.flatnonzero(~is_bad[l[i]:l[i] + w[i]]) + l[i]
        got = got[dd < np.inf]
        assert len(got) == k and (metric == "ip" or not is_bad[got].any())
        if metric == "l2":
            d64 = ((X[good].astype(np.float64) - q[i]) ** 2).sum(1)
            want = good[np.argsort(d64)[:k]]
            assert len(set(want.tolist()) & set(got.tolist())) >= 0.9 * k
