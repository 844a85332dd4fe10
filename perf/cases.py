"""Performance cases of the library: the calls its users make, through the
Python binding of the C ABI, over the sizes they are made at.

Kinds of a case:
  search      range-filtered search of one batch on an index that is kept
              (one esg_search_batch call, or a CUDA-graph batch that is given
              its queries and replayed);
  bruteforce  exact range-filtered k-NN of one batch over a point matrix (the
              ground truth of an evaluation, the dense baseline);
  mlp         one training step of the search-budget network: loss, gradients
              and the Adam update;
  build       an index built from host vectors and then asked once.

Points and queries come from the distributions of synthetic.py, drawn on the
GPU: a Gaussian mixture (unit vectors for the inner product), or a power-law
spectrum for the 768-dimensional embeddings. An index stands for the deployed
one: it is made from the case alone and kept while batches of other seeds ask
it; queries, ranges and everything else come from the seed.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2504_04018_gb300 as E

N_COMP = 1024
SIGMA = 0.1
LEAF = 256
MIXED_K = (1, 10, 100)


def _search(name, n, d, metric, nq, k, ef, rows="f32", width=1, learned=False, graph=False, widths="log",
            M=32, data="mixture"):
    """k = 0: drawn from {1, 10, 100} per query. widths: "pow2" 2^-j of n, "log" log-uniform 0.1 % - 100 %,
    "log4" log-uniform 0.01 % - 100 %."""
    return dict(name=name, kind="search", n=n, d=d, metric=metric, nq=nq, k=k, ef=ef, rows=rows, width=width,
                learned=learned, graph=graph, widths=widths, M=M, data=data)


def _bruteforce(name, n, d, metric, nq, k, widths="log", data="mixture"):
    return dict(name=name, kind="bruteforce", n=n, d=d, metric=metric, nq=nq, k=k, widths=widths, data=data)


def listed():
    return [
        # one user waiting for one answer
        _search("search-1-query", 1_000_000, 128, "l2", 1, 10, 64, widths="pow2"),
        # a small batch of an online service, an odd number of queries
        _search("search-61-queries", 1_000_000, 128, "l2", 61, 10, 64, widths="pow2"),
        # the scale workload: plain FP32 rows at the beam its recall target needs
        _search("search-scale-10k", 1_000_000, 128, "l2", 10_000, 10, 24, widths="pow2"),
        # the offline batch: uneven widths and k, a learned budget, BF16 rows, one CUDA graph
        _search("search-batch-100k", 1_000_000, 96, "ip", 100_000, 0, 64, rows="bf16", width=2, learned=True,
                graph=True, widths="log4"),
        # the smallest rows: FP8 traversal at the wider beam it needs
        _search("search-fp8-10k", 1_000_000, 96, "ip", 10_000, 10, 96, rows="fp8"),
        # 768-dimensional embeddings, BF16 rows; a ragged index size
        _search("search-768d-10k", 200_003, 768, "ip", 10_000, 10, 64, rows="bf16", data="spectrum"),
        # exact answers of the scale workload
        _bruteforce("exact-scale-10k", 1_000_000, 128, "l2", 10_000, 10, widths="pow2"),
        # exact answers for k = 100, as the batching workload's ground truth needs
        _bruteforce("exact-k100-10k", 1_000_000, 96, "ip", 10_000, 100),
        # exact answers over wide embeddings, ragged sizes
        _bruteforce("exact-768d-2k", 200_003, 768, "ip", 1_999, 10, data="spectrum"),
        # a few exact answers over a small set whose dimension is no multiple of the tile's
        _bruteforce("exact-small-61", 99_991, 100, "l2", 61, 10),
        # one minibatch of the budget network's training
        dict(name="mlp-step-1024", kind="mlp", batch=1024),
        # the tiny workload's index, built and asked
        dict(name="build-10k", kind="build", n=10_000, d=128, metric="l2", M=16, ef_construction=200, nq=200, k=10,
             ef=64),
    ]


def _log_int(rng: random.Random, lo: int, hi: int) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choices(["search", "bruteforce", "mlp", "build"], weights=[5, 4, 1, 2])[0]
    metric = rng.choice(["l2", "ip"])
    if kind == "search":
        rows = rng.choice(["f32", "f32", "bf16", "bf16", "fp8"])
        d = rng.choice({"f32": [32, 48, 64, 96, 128, 192, 256, 768], "bf16": [32, 48, 64, 96, 128, 192, 768],
                        "fp8": [32, 48, 64, 96, 128, 192]}[rows])
        n = _log_int(rng, 20_000, min(500_000, 100_000_000 // d))
        c = _search("", n, d, metric, _log_int(rng, 1, 20_000), rng.choice([1, 10, 10, 20, 50, 100, 0]),
                    _log_int(rng, 16, 256), rows=rows, width=rng.choice([1, 1, 2]),
                    learned=rng.random() < 0.3, graph=rng.random() < 0.4, widths=rng.choice(["pow2", "log", "log4"]),
                    M=rng.choice([16, 32]), data="spectrum" if d == 768 else "mixture")
    elif kind == "bruteforce":
        d = rng.choice([32, 52, 64, 96, 100, 128, 200, 256, 300, 768])
        n = _log_int(rng, 20_000, min(1_000_000, 200_000_000 // d))
        k = rng.choice([1, 10, 10, 20, 50, 100])
        nq = _log_int(rng, 1, min(10_000, max(64, 900_000_000_000 // (n * d))))
        c = _bruteforce("", n, d, metric, nq, k, widths=rng.choice(["pow2", "log", "log4"]),
                        data="spectrum" if d == 768 else "mixture")
    elif kind == "mlp":
        c = dict(kind="mlp", batch=_log_int(rng, 64, 8192))
    else:
        c = dict(kind="build", n=_log_int(rng, 1_500, 12_000), d=rng.choice([32, 64, 96, 128]), metric=metric,
                 M=rng.choice([8, 16, 16]), ef_construction=rng.choice([100, 200]), nq=_log_int(rng, 32, 512), k=10,
                 ef=64)
    c.pop("name", None)
    return c


# ------------------------------------------------------------------ inputs

def _gen(seed: int) -> torch.Generator:
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _points(case, count: int, seed: int) -> torch.Tensor:
    """`count` points of the case's distribution (its centers or axes depend on the dimension alone)."""
    d, g = case["d"], _gen(seed)
    out = torch.empty(count, d, device="cuda")
    if case.get("data") == "spectrum":
        axes = torch.linalg.qr(torch.randn(d, d, generator=_gen(1005), device="cuda"))[0]
        scale = torch.arange(1, d + 1, device="cuda", dtype=torch.float32).rsqrt()
    else:
        centers = torch.rand(N_COMP, d, generator=_gen(1000), device="cuda") * 2 - 1
    for s in range(0, count, 1 << 17):
        m = min(count - s, 1 << 17)
        z = torch.randn(m, d, generator=g, device="cuda")
        if case.get("data") == "spectrum":
            x = (z * scale) @ axes.T
        else:
            x = centers[torch.randint(0, N_COMP, (m,), generator=g, device="cuda")] + SIGMA * z
        out[s:s + m] = torch.nn.functional.normalize(x, dim=1) if case["metric"] == "ip" else x
    return out


def _ranges(case, seed: int):
    """Inclusive rank ranges: width max(1, round(share n)), the left end uniform where it fits."""
    n, nq, g = case["n"], case["nq"], _gen(seed + 500_009)
    if case.get("widths", "log") == "pow2":
        share = 2.0 ** -((torch.arange(nq, device="cuda") + seed) % 11).double()
    else:
        lo = math.log(1e-4 if case.get("widths") == "log4" else 1e-3)
        share = torch.exp(lo * (1 - torch.rand(nq, generator=g, device="cuda", dtype=torch.float64)))
    w = torch.clamp(torch.round(share * n).long(), 1, n)
    left = torch.rand(nq, generator=g, device="cuda", dtype=torch.float64)
    l = torch.minimum((left * (n - w + 1).double()).long(), n - w)
    return l.contiguous(), (l + w - 1).contiguous()


def _per_query_k(case, seed: int):
    if case["k"] != 0:
        return None
    pick = torch.randint(0, 3, (case["nq"],), generator=_gen(seed + 700_001), device="cuda")
    return torch.tensor(MIXED_K, dtype=torch.int32, device="cuda")[pick].contiguous()


def _k_max(case) -> int:
    return case["k"] if case["k"] else max(MIXED_K)


def _predictor() -> np.ndarray:
    """A search-budget network like a trained one: log2 ef rises with log2 width and log2 k, with an expansion
    budget of about four times ef (layer 1 passes features 0 and 5 on, layer 2 copies, the head weighs them)."""
    F, H = E.esg_mlp_num_features(), 64
    W1, W2, W3 = np.zeros((F, H), np.float32), np.eye(H, dtype=np.float32), np.zeros((H, 2), np.float32)
    W1[0, 0] = W1[5, 1] = 1.0
    W3[0], W3[1] = (0.12, 0.12), (0.25, 0.25)
    b3 = np.array([2.5, 4.5], np.float32)
    blob = np.zeros(E.esg_mlp_blob_size(), np.float32)
    params = np.concatenate([W1.ravel(), np.zeros(H, np.float32), W2.ravel(), np.zeros(H, np.float32), W3.ravel(), b3])
    blob[:len(params)] = params
    blob[len(params) + F:len(params) + 2 * F] = 1.0   # sigma; mu, margins and offsets stay 0
    return blob


_kept = {}   # the index in use (one at a time)


def _index(case):
    key = tuple((f, case[f]) for f in ("n", "d", "metric", "M", "data"))
    if _kept.get("key") != key:
        _kept.clear()
        base = _points(case, case["n"], 77).cpu().numpy()
        ix = E.esg_build(base, None, M=case["M"], leaf_size=LEAF, n_entries=16, metric=case["metric"])
        E.esg_predictor_set(ix, _predictor(), 8, 256)
        _kept.update(key=key, index=ix)
    ix = _kept["index"]
    if case["rows"] != "f32":
        E.esg_index_add_storage(ix, case["rows"])   # kept if it is there
    return ix


def _prepare_search(case, seed):
    ix = _index(case)
    s = dict(index=ix, q=_points(case, case["nq"], seed + 1), k=_per_query_k(case, seed), k_max=_k_max(case),
             params=E.search_params(case["ef"], use_learned=int(case["learned"]), traversal=case["rows"],
                                    width=case["width"]))
    s["l"], s["r"] = _ranges(case, seed)
    if case["graph"]:
        nq, km = case["nq"], s["k_max"]
        b = E.Batch(ix, nq, km, s["params"], use_k=s["k"] is not None)
        s["batch"] = b
        s["in"] = [(b.view("queries", (nq, case["d"]), torch.float32), s["q"]),
                   (b.view("l", (nq,), torch.int64), s["l"]), (b.view("r", (nq,), torch.int64), s["r"])]
        if s["k"] is not None:
            s["in"].append((b.view("k", (nq,), torch.int32), s["k"]))
        s["out"] = (b.view("ids", (nq, km), torch.int64), b.view("dist", (nq, km), torch.float32),
                    b.view("count", (nq,), torch.int32), b.view("status", (nq,), torch.int32))
        for t in s["out"]:
            t.batch = b   # the views alias the batch's buffers: whoever holds one holds the batch
    return s


def _prepare_mlp(case, seed):
    g, B, F, P = _gen(seed), case["batch"], E.esg_mlp_num_features(), E.esg_mlp_num_params()
    # a network in the middle of its training: weights, moments and features of the usual size
    shape = [(F * 64, F), (64, 0), (64 * 64, 64), (64, 0), (64 * 2, 64), (2, 0)]
    params = torch.cat([(torch.rand(c, generator=g, device="cuda") * 2 - 1) * (math.sqrt(6 / f) if f else 0.1)
                        for c, f in shape])
    mu = torch.rand(F, generator=g, device="cuda") * 10
    sigma = torch.rand(F, generator=g, device="cuda") * 3 + 0.5
    X = mu + sigma * torch.randn(B, F, generator=g, device="cuda")
    T = torch.rand(B, 2, generator=g, device="cuda") * 5 + 3
    return dict(params=params, X=X.contiguous(), T=T, mu=mu, sigma=sigma, step=500,
                m=1e-2 * torch.randn(P, generator=g, device="cuda"),
                v=1e-4 * torch.rand(P, generator=g, device="cuda") + 1e-6)


def prepare(case, seed):
    if case["kind"] == "search":
        return dict(_prepare_search(case, seed), kind="search")
    if case["kind"] == "mlp":
        return dict(_prepare_mlp(case, seed), kind="mlp")
    l, r = _ranges(case, seed)
    q = _points(case, case["nq"], seed + 1)
    base = _points(case, case["n"], seed + 2)
    if case["kind"] == "bruteforce":
        return dict(kind="bruteforce", base=base, q=q, l=l, r=r, k=case["k"], metric=case["metric"])
    return dict(kind="build", base=base.cpu().numpy(), q=q, l=l, r=r, case=dict(case))


# -------------------------------------------------------------------- runs

def run(state):
    kind = state["kind"]
    if kind == "search":
        if "batch" in state:
            for dst, src in state["in"]:
                dst.copy_(src)
            state["batch"].run(state["q"].shape[0])
            return state["out"]
        return E.esg_search_batch(state["index"], state["q"], state["l"], state["r"], state["k"], state["k_max"],
                                  params=state["params"])[:4]
    if kind == "bruteforce":
        return E.esg_bruteforce_filtered_knn(state["base"], state["q"], state["l"], state["r"], state["k"],
                                             state["metric"])
    if kind == "mlp":
        state["step"] += 1
        loss, grad = E.esg_mlp_loss_grad(state["params"], state["X"], state["T"], state["mu"], state["sigma"], 0.9)
        E.esg_mlp_adam_step(state["params"], grad, state["m"], state["v"], state["step"], 1e-3)
        return loss, grad, state["params"], state["m"], state["v"]
    c = state["case"]
    ix = E.esg_build(state["base"], None, M=c["M"], leaf_size=LEAF, n_entries=16,
                     ef_construction=c["ef_construction"], metric=c["metric"])
    return E.esg_search_batch(ix, state["q"], state["l"], state["r"], None, c["k"], ef=c["ef"])[:4]


def _mean_share(case) -> float:
    """Mean range width over n."""
    w = case.get("widths", "log")
    if w == "pow2":
        return sum(2.0 ** -j for j in range(11)) / 11
    lo = 1e-4 if w == "log4" else 1e-3
    return (1 - lo) / math.log(1 / lo)


def work(case):
    """Search: the expansions and evaluations that beams of this width cannot do without, about 1.2 ef
    expansions per query and 10 new rows each, no more rows than the ranges hold. Brute force: one product
    per (query, point in range). Build: an insertion search per point and level, half the points of each."""
    if case["kind"] == "mlp":
        B, F, H = case["batch"], 9, 64
        P = F * H + H + H * H + H + H * 2 + 2
        return {"bytes": 4.0 * (B * (F + 2) + 2 * F + 8 * P), "flops": 6.0 * B * P}
    n, d, nq = case["n"], case["d"], case["nq"]
    if case["kind"] == "bruteforce":
        return {"bytes": 4.0 * n * d + nq * (4.0 * d + 16 + 12.0 * case["k"] + 4),
                "flops": 2.0 * d * nq * n * _mean_share(case)}
    km = _k_max(case)
    rows = {"f32": 4, "bf16": 2, "fp8": 1}[case.get("rows", "f32")]
    expansions = min(1.2 * max(case["ef"], km if case["k"] else 37), 0.1 * _mean_share(case) * n) * nq
    io = nq * (4.0 * d + 16 + 12.0 * km + 8)
    if case["kind"] == "build":
        levels = math.ceil(math.log2(max(2.0, n / LEAF))) + 1
        expansions += case["ef_construction"] * n * (1 + levels / 2)
        io += 4.0 * n * d + 8.0 * levels * n * case["M"]
    return {"bytes": io + expansions * (8.0 * case["M"] + 10.0 * d * rows), "flops": expansions * 10.0 * 2.0 * d}


# ----------------------------------------------------------- in 64 bits

def _exact_distances(base, q, l, r, k, metric):
    """The k smallest in-range distances of each query, ascending, +inf padded (float64)."""
    X, n = base.double(), base.shape[0]
    xn = (X * X).sum(1) if metric == "l2" else None
    out = torch.full((q.shape[0], k), math.inf, dtype=torch.float64, device="cuda")
    rows = torch.arange(n, device="cuda")
    step = max(1, (1 << 27) // n)
    for s in range(0, q.shape[0], step):
        Q = q[s:s + step].double()
        D = Q @ X.T
        D = (Q * Q).sum(1, keepdim=True) + xn - 2 * D if metric == "l2" else -D
        D.masked_fill_((rows < l[s:s + step, None]) | (rows > r[s:s + step, None]), math.inf)
        kk = min(k, n)
        out[s:s + step, :kk] = torch.topk(D, kk, dim=1, largest=False, sorted=True)[0]
    return out


def _exact_mlp(s):
    P64 = s["params"].double()
    F, H = 9, 64
    parts = torch.split(P64, [F * H, H, H * H, H, H * 2, 2])
    W1, b1, W2, b2, W3, b3 = (p.clone().requires_grad_() for p in parts)
    xh = (s["X"].double() - s["mu"].double()) / s["sigma"].double()
    h1 = torch.relu(xh @ W1.view(F, H) + b1)
    h2 = torch.relu(h1 @ W2.view(H, H) + b2)
    u = s["T"].double() - (h2 @ W3.view(H, 2) + b3)
    loss = torch.maximum(0.9 * u, (0.9 - 1) * u).mean()
    loss.backward()
    g = torch.cat([p.grad for p in (W1, b1, W2, b2, W3, b3)])
    m = 0.9 * s["m"].double() + 0.1 * g
    v = 0.999 * s["v"].double() + 0.001 * g * g
    t = s["step"] + 1
    p = P64 - 1e-3 * (m / (1 - 0.9 ** t)) / ((v / (1 - 0.999 ** t)).sqrt() + 1e-8)
    return loss.item(), g, p, m, v


def exact(case, seed):
    """None for the searches: which points they find is the graph's doing, and a missed neighbour changes the
    distances in its place (by more than half in the L2 mixture, where it can be another cluster's)."""
    if case["kind"] == "mlp":
        return _exact_mlp(_prepare_mlp(case, seed))
    if case["kind"] != "bruteforce" or 2.0 * case["nq"] * case["n"] * case["d"] > 6e12:
        return None
    l, r = _ranges(case, seed)
    return None, _exact_distances(_points(case, case["n"], seed + 2), _points(case, case["nq"], seed + 1), l, r,
                                  case["k"], case["metric"]), None
