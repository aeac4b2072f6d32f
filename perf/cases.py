"""The workloads that the library's speed is judged by.

Each case is a call (or a few calls) that a program makes through the public entry points of
``paper_2304_04015_gb300``: single-source SimRank queries from the smallest graph to one beyond the L2 cache,
batches of sources, sparse top-k batches, the query server, a cold start from host arrays, and the forward and
backward pass of the linearised form.  Graphs are seeded R-MAT or Erdos-Renyi graphs drawn on the device; all
weights, sources and seeds come from ``seed`` alone.
"""
import math

import numpy as np
import torch

import paper_2304_04015_gb300 as srk

C = 0.6  # the decay factor of every workload


def listed():
    return [
        # The small configuration of the tests: 1,000 nodes, 2,000 walk pairs per target, 32 steps.  All of it is latency.
        dict(name="er1000_query", kind="query", graph="er", n=1000, deg=5, eps=0.1, z=2000, L=32),
        # An interactive query on a small social graph (the small graph of the serving mix), tight enough to fill the GPU.
        dict(name="rmat16_query", kind="query", graph="rmat", n=65536, deg=16, eps=0.02, z=0, L=-1),
        # A graph without hubs and with a ragged number of nodes: uniform in-neighbours, as in a k-nearest-neighbour graph.
        dict(name="er_ragged_query", kind="query", graph="er", n=100003, deg=12, eps=0.03, z=0, L=-1),
        # The headline: 1,048,576 nodes, eps = 0.02, one query per launch; the graph fits the L2 cache.
        dict(name="rmat20_query", kind="query", graph="rmat", n=1048576, deg=16, eps=0.02, z=0, L=-1),
        # The same on a graph far larger than the L2 cache.
        dict(name="rmat22_query", kind="query", graph="rmat", n=4194304, deg=16, eps=0.05, z=0, L=-1),
        # A batch of sources of mixed degree and mixed error targets, dense scores out.
        dict(name="rmat16_multi", kind="multi", graph="rmat", n=65536, deg=16, eps=0.0, k=24, shared=False),
        # A batch with equal error targets that shares its target walks.
        dict(name="rmat18_shared", kind="multi", graph="rmat", n=262144, deg=16, eps=0.05, k=48, shared=True),
        # Recommendation lists: the 100 nearest targets of each of 64 sources.
        dict(name="rmat17_topk", kind="topk", graph="rmat", n=131072, deg=16, eps=0.05, k=64, top=100, shared=True),
        # Serving: a burst of requests with host results, four workers.
        dict(name="rmat16_serve", kind="serve", graph="rmat", n=65536, deg=16, eps=0.05, k=32),
        # A cold start: host arrays in, one query, host scores out.
        dict(name="rmat18_cold", kind="cold", graph="rmat", n=262144, deg=16, eps=0.1, z=0, L=-1),
        # Training through the linearised form: forward and gradient of every edge weight.
        dict(name="rmat18_linear", kind="linear", graph="rmat", n=262144, deg=16, L=10),
        # The same on a small ragged graph, where launches count.
        dict(name="er_small_linear", kind="linear", graph="er", n=5003, deg=6, L=6),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["query", "query", "query", "multi", "topk", "serve", "cold", "linear"])
    graph = rng.choice(["rmat", "rmat", "er"])
    deg = rng.randint(3, 20)
    if kind == "linear":
        return dict(kind=kind, graph=graph, n=_log_int(rng, 1000, 262144), deg=deg, L=rng.randint(1, 12))
    eps = rng.choice([0.1, 0.05, 0.04, 0.03, 0.02])
    if kind == "query":
        n = _log_int(rng, 1000, 1 << 20)
        return dict(kind=kind, graph=graph, n=n, deg=deg, eps=eps, z=0, L=-1)
    if kind == "cold":
        return dict(kind=kind, graph=graph, n=_log_int(rng, 1000, 262144), deg=deg, eps=max(eps, 0.04), z=0, L=-1)
    n = _log_int(rng, 1000, 65536)
    if kind == "serve":
        return dict(kind=kind, graph=graph, n=n, deg=deg, eps=max(eps, 0.03), k=rng.randint(4, 40))
    shared = rng.random() < 0.5
    eps = max(eps, 0.04)
    k = rng.randint(3, 70)
    if kind == "multi":
        return dict(kind=kind, graph=graph, n=n, deg=deg, eps=eps, k=k, shared=shared)
    return dict(kind=kind, graph=graph, n=n, deg=deg, eps=eps, k=k, top=_log_int(rng, 1, 1000), shared=shared)


# ------------------------------------------------------------------ inputs --

def _csr(n, src, dst):
    """In-neighbour CSR (int32) of the edges src -> dst: no self-loops, no duplicates, lists ascending."""
    keep = src != dst
    key = torch.unique(dst[keep] * n + src[keep])
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device=key.device)
    row_ptr[1:] = torch.cumsum(torch.bincount(key // n, minlength=n), 0)
    return row_ptr.to(torch.int32), (key % n).to(torch.int32)


def _graph(case, seed):
    n, m = case["n"], case["n"] * case["deg"]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1000003 * seed + 17)
    src = torch.zeros(m, dtype=torch.int64, device="cuda")
    dst = torch.zeros(m, dtype=torch.int64, device="cuda")
    if case["graph"] == "rmat":  # (a, b, c, d) = (0.57, 0.19, 0.19, 0.05), ids not permuted, nodes past n dropped
        for _ in range(max(1, (n - 1).bit_length())):
            r = torch.rand(m, generator=gen, device="cuda")
            src = 2 * src + (r >= 0.76)
            dst = 2 * dst + (((r >= 0.57) & (r < 0.76)) | (r >= 0.95))
        keep = (src < n) & (dst < n)
        src, dst = src[keep], dst[keep]
    else:  # m uniform edges: in-degrees are Poisson in the limit
        src = torch.randint(0, n, (m,), generator=gen, device="cuda")
        dst = torch.randint(0, n, (m,), generator=gen, device="cuda")
    return _csr(n, src, dst)


def _sources(case, row_ptr, seed):
    """k sources: all with in-neighbours, or, for a batch, a third each of top and median in-degree and the rest without
    in-neighbours (any node where a graph has none)."""
    rng = np.random.default_rng(seed + 7)
    deg = np.diff(row_ptr.cpu().numpy().astype(np.int64))
    k = case.get("k", 1)
    some = np.flatnonzero(deg > 0)
    if case["kind"] in ("query", "cold", "serve"):
        return rng.choice(some, k).astype(np.int32)
    order = np.argsort(-deg, kind="stable")
    median = np.flatnonzero(deg == int(np.median(deg[some])))
    none = np.flatnonzero(deg == 0)
    if none.size == 0:
        none = np.arange(deg.size)
    third = max(1, k // 3)
    parts = [rng.choice(order[:4 * third], third), rng.choice(median, third), rng.choice(none, max(1, k - 2 * third))]
    return np.concatenate(parts)[:k].astype(np.int32)


def _errors(case, seed):
    """One error target per source: mixed, where the case names none."""
    k = case["k"]
    if case["eps"]:
        return np.full(k, case["eps"])
    return np.random.default_rng(seed + 11).choice(np.array([0.05, 0.02, 0.01]), k)


def prepare(case, seed):
    row_ptr, col = _graph(case, seed)
    n, kind = case["n"], case["kind"]
    st = dict(case=case, seed=0x9E3779B97F4A7C15 * (seed + 1) % (1 << 64))
    if kind == "linear":
        rng = torch.Generator(device="cuda")
        rng.manual_seed(seed + 5)
        st["graph"] = srk.srk_graph_load(row_ptr, col)
        st["s"] = int(_sources(dict(kind="query"), row_ptr, seed)[0])
        st["w"] = torch.exp(0.5 * torch.randn(col.numel(), generator=rng, device="cuda"))
        st["grad"] = torch.randn(n, generator=rng, device="cuda")
        st["out"] = torch.empty(n, device="cuda")
        st["grad_w"] = torch.zeros(n * case["deg"], device="cuda")  # one slot per drawn edge; duplicates leave some over
        return st
    st["sources"] = _sources(case, row_ptr, seed)
    if kind == "cold":
        st["row_ptr"], st["col"] = row_ptr.cpu().numpy(), col.cpu().numpy()
        st["scores"], st["counts"] = np.zeros(n), np.zeros(n, dtype=np.uint32)
        return st
    st["graph"] = srk.srk_graph_load(row_ptr, col)
    k = case.get("k", 1)
    if kind == "serve":
        st["scores"] = np.zeros((k, n))
        st["server"] = srk.srk_server_create([st["graph"]], 16 << 30, 4)
        return st
    if kind == "topk":
        top = case["top"]
        st["eps"] = _errors(case, seed)
        st["out"] = [torch.empty((k, top), dtype=torch.int32, device="cuda"),
                     torch.empty((k, top), dtype=torch.float64, device="cuda"),
                     torch.empty(k, dtype=torch.int32, device="cuda"), torch.empty(k, dtype=torch.int64, device="cuda")]
        return st
    if kind == "multi":
        st["eps"] = _errors(case, seed)
        st["scores"] = torch.empty((k, n), dtype=torch.float64, device="cuda")
        st["counts"] = torch.empty((k, n), dtype=torch.int32, device="cuda")
        return st
    st["scores"] = torch.empty(n, dtype=torch.float64, device="cuda")
    st["counts"] = torch.empty(n, dtype=torch.int32, device="cuda")
    st["sums"] = torch.empty(n, dtype=torch.int64, device="cuda")
    return st


# ------------------------------------------------------------------- calls --

def run(state):
    case, seed = state["case"], state["seed"]
    kind = case["kind"]
    if kind == "linear":
        ctx = srk.srk_linear_fwd(state["graph"], state["w"], state["s"], C, case["L"], state["out"])
        srk.srk_linear_bwd(ctx, state["grad"], state["grad_w"][:state["w"].numel()])
        srk.srk_linear_ctx_free(ctx)
        return state["out"], state["grad_w"]
    if kind == "topk":
        nodes, scores, count, nnz = state["out"]
        srk.srk_multi_source_topk(state["graph"], state["sources"], C, state["eps"], seed, case["top"], nodes, scores,
                                  count, nnz, shared_walks=case["shared"])
        return nodes, scores, count, nnz
    if kind == "multi":
        srk.srk_multi_source(state["graph"], state["sources"], C, state["eps"], seed, state["scores"], state["counts"],
                             shared_walks=case["shared"])
        return state["scores"], state["counts"]
    if kind == "serve":
        for i, s in enumerate(state["sources"]):
            srk.srk_server_submit(state["server"], 0, int(s), C, case["eps"], seed + i, state["scores"][i], i)
        srk.srk_server_drain(state["server"])
        return state["scores"]
    s = int(state["sources"][0])
    over = dict(z_override=case["z"] or None, L_override=case["L"] if case["L"] >= 0 else None)
    if kind == "cold":
        with srk.srk_graph_load(state["row_ptr"], state["col"]) as g:
            srk.srk_single_source(g, s, C, case["eps"], seed, state["scores"], state["counts"], **over)
        return state["scores"], state["counts"]
    srk.srk_single_source(state["graph"], s, C, case["eps"], seed, state["scores"], state["counts"], state["sums"], **over)
    return state["scores"], state["counts"], state["sums"]


# ------------------------------------------------- what a pass has to move --

def _table(case, eps):
    """(z, walk counts by length) of one query (the sample-count rules of include/srk.h)."""
    n = case["n"]
    z = case.get("z") or math.log(2.0 * n) / (2.0 * (eps - 3.0 / n) ** 2)
    r = math.sqrt(C)
    L = case["L"] if case.get("L", -1) >= 0 else int(math.floor(math.log(n) / -math.log(r)))
    return z, [math.ceil(z * (r ** l * (1.0 - r))) for l in range(L + 1)]


def work(case):
    """The graph read once and the results written once; for walks, one decision per walk pair and target."""
    n, m, k = case["n"], case["n"] * case["deg"], case.get("k", 1)
    if case["kind"] == "linear":
        L = case["L"]
        return dict(bytes=4 * (n + 1 + 2 * m) + 4 * (2 * n + m), flops=2 * m * 4 * L + 4 * m * L)
    out = {"query": 20 * n, "cold": 12 * n, "multi": 12 * n * k, "serve": 8 * n * k}.get(case["kind"], 0)
    if case["kind"] == "topk":
        out = k * (12 * case["top"] + 12)
    pairs = sum(_table(case, case["eps"] or 0.02)[1])
    return dict(bytes=4 * (n + 1 + m) + out, flops=pairs * n * (1 if case.get("shared") else k))


# ------------------------------------------------------- plain 64-bit values --

def _u32(x):
    return x & 0xFFFFFFFF


def _mulhilo(a, x):
    """High and low words of the 32x32-bit product a x (a below 2^32, x int64 tensors holding words)."""
    lo = a * (x & 0xFFFF)
    hi = a * (x >> 16) + (lo >> 16)
    return hi >> 16, _u32((hi << 16) | (lo & 0xFFFF))


def _philox2(key, c0, c1):
    for r in range(10):
        hi, lo = _mulhilo(0xD256D193, c0)
        c0, c1 = hi ^ c1 ^ _u32(key + r * 0x9E3779B9), lo
    return c0, c1


def _philox4(seed, t, s):
    x = [t >> 1, torch.full_like(t, 0xFFFFFFFF), torch.full_like(t, 0xFFFFFFFF), torch.full_like(t, s)]
    for r in range(10):
        k0, k1 = _u32(seed + r * 0x9E3779B9), _u32((seed >> 32) + r * 0xBB67AE85)
        h0, l0 = _mulhilo(0xD2511F53, x[0])
        h1, l1 = _mulhilo(0xCD9E8D57, x[2])
        x = [h1 ^ x[1] ^ k0, l1, h0 ^ x[3] ^ k1, l0]
    return x


def _scale64(hi, lo, d):
    """floor((hi 2^32 + lo) d / 2^64) for words hi, lo and d below 2^31."""
    h1, l1 = _mulhilo2(hi, d)
    h0, _ = _mulhilo2(lo, d)
    return h1 + ((l1 + h0) >> 32)


def _mulhilo2(x, d):
    p = (x & 0xFFFF) * d  # below 2^47
    q = (x >> 16) * d + (p >> 16)
    return q >> 16, _u32((q << 16) | (p & 0xFFFF))


def _key(seed, q):
    z, M = seed, (1 << 64) - 1
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & M
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & M
    x = _u32(q ^ (z ^ (z >> 31)))
    x = _u32((x ^ (x >> 16)) * 0x7FEB352D)
    x = _u32((x ^ (x >> 15)) * 0x846CA68B)
    return x ^ (x >> 16)


class _Walker:
    """Walks one step at a time, all of them at once: node, replica and start node per walk."""

    def __init__(self, row_ptr, col, key):
        self.row_ptr, self.col, self.key = row_ptr, col, key

    def step(self, i, at, r, start, words):
        """Nodes after step i of the walks at `at` (in-degree above 0); `words` are the block's two words."""
        d = self.row_ptr[at + 1] - self.row_ptr[at]
        w = words[(i - 1) & 1]
        idx, low = _mulhilo2(w, d)
        bad = low < (1 << 32) % d
        if bool(bad.any()):
            top = 0x80000000
            c0 = (((i - 1) >> 1) << 24 | r[bad]) | (top if i & 1 else 0)
            y0, y1 = _philox2(self.key, c0, start[bad] | (0 if i & 1 else top))
            idx[bad] = _scale64(y0, y1, d[bad])
        return self.col[self.row_ptr[at] + idx].long()

    def words(self, i, r, start):
        return _philox2(self.key, ((i - 1) >> 1) << 24 | r, start)


def _scores(row_ptr, col, case, s, eps, seed, shared=False):
    """Scores of one query in plain 64-bit arithmetic, all targets."""
    dev = row_ptr.device
    n = case["n"]
    z, counts = _table(case, eps)
    N = sum(counts)
    length = torch.repeat_interleave(torch.arange(len(counts)), torch.tensor(counts)).to(dev)
    weight = torch.tensor([z * (math.sqrt(C) ** l * (1.0 - math.sqrt(C))) / c for l, c in enumerate(counts)],
                          dtype=torch.float64, device=dev)
    # the source's walks: node after every step, -1 past the end
    walk = _Walker(row_ptr, col, _key(seed, s))
    r = torch.arange(N, device=dev)
    at, alive = torch.full((N,), s, device=dev), torch.ones(N, dtype=torch.bool, device=dev)
    nodes = []
    words = None
    for i in range(1, len(counts)):
        alive = alive & (length >= i) & (row_ptr[at + 1] > row_ptr[at])
        if not bool(alive.any()):
            break
        if i & 1:
            words = walk.words(i, r, torch.full_like(r, s))
        a = alive.nonzero()[:, 0]
        at = at.clone()
        at[a] = walk.step(i, at[a], r[a], torch.full_like(a, s), [w[a] for w in words])
        nodes.append(torch.where(alive, at, torch.full_like(at, -1)))
    # the Fisher-Yates shuffle
    x = _philox4(seed, r, s)
    odd = (r & 1) == 1
    k = _scale64(torch.where(odd, x[2], x[0]), torch.where(odd, x[3], x[1]), r + 1).tolist()
    sigma = list(range(N))
    for t in range(N - 1, 0, -1):
        sigma[t], sigma[k[t]] = sigma[k[t]], sigma[t]
    sigma = torch.tensor(sigma, device=dev)
    steps = torch.zeros(N, dtype=torch.long, device=dev)
    for v in nodes:
        steps += v >= 0
    cap = torch.minimum(length, steps[sigma])
    w = torch.round(weight[length[sigma]] * weight[length] * 4294967296.0).long()
    pairs = (cap >= 1).nonzero()[:, 0]
    # every target's walks, some targets at a time
    walk = _Walker(row_ptr, col, _key(seed, 0xFFFFFFFE if shared else s))
    targets = (row_ptr[1:] > row_ptr[:-1]).nonzero()[:, 0]
    sums = torch.zeros(n, dtype=torch.long, device=dev)
    chunk = max(1, (1 << 25) // max(1, pairs.numel()))
    for t0 in range(0, targets.numel(), chunk):
        u = targets[t0:t0 + chunk]
        start = u.repeat_interleave(pairs.numel())
        j = pairs.repeat(u.numel())
        at, i, words = start, 1, None
        while j.numel():
            if i & 1:
                words = walk.words(i, j, start)
            at = walk.step(i, at, j, start, words)
            met = at == nodes[i - 1][sigma[j]]
            sums.index_add_(0, start[met], w[j[met]])
            go = ~met & (cap[j] > i) & (row_ptr[at + 1] > row_ptr[at])
            at, j, start, words = at[go], j[go], start[go], [v[go] for v in words]
            i += 1
    out = sums.double() * 2.0 ** -32 / z
    out[s] = 1.0
    return out


def _linear(row_ptr, col, w, s, grad, L):
    """Scores and weight gradients of the linearised form."""
    n = row_ptr.numel() - 1
    a = torch.repeat_interleave(torch.arange(n, device=col.device), row_ptr[1:] - row_ptr[:-1])  # edge col -> a
    w = w.double().requires_grad_(True)
    zero = torch.zeros(n, dtype=torch.float64, device=col.device)
    p = w / zero.index_add(0, a, w)[a]
    y = zero.clone()
    y[s] = 1.0
    ys = [y]
    for _ in range(L):
        ys.append(zero.index_add(0, col, p * ys[-1][a]))
    h = (1.0 - C) * ys[L]
    for t in range(L - 1, -1, -1):
        h = (1.0 - C) * ys[t] + C * zero.index_add(0, a, p * h[col])
    h.backward(grad.double())
    return h.detach(), w.grad


def exact(case, seed):
    kind = case["kind"]
    if kind != "linear":
        sets = 1 if kind in ("query", "cold") else case["k"]
        errs = [case["eps"]] if kind not in ("multi", "topk") else _errors(case, seed)
        cost = sum(sum(_table(case, e)[1]) for e in errs) * case["n"] * (sets if kind == "serve" else 1)
        if cost > 6e9:
            return None  # more than a few seconds
    row_ptr, col = _graph(case, seed)
    row_ptr, col = row_ptr.long(), col.long()
    if kind == "linear":
        rng = torch.Generator(device="cuda")
        rng.manual_seed(seed + 5)
        s = int(_sources(dict(kind="query"), row_ptr, seed)[0])
        w = torch.exp(0.5 * torch.randn(col.numel(), generator=rng, device="cuda"))
        grad = torch.randn(case["n"], generator=rng, device="cuda")
        out, grad_w = _linear(row_ptr, col, w, s, grad, case["L"])
        return out, torch.cat([grad_w, grad_w.new_zeros(case["n"] * case["deg"] - grad_w.numel())])
    src = _sources(case, row_ptr, seed)
    key = 0x9E3779B97F4A7C15 * (seed + 1) % (1 << 64)
    if kind == "serve":
        return torch.stack([_scores(row_ptr, col, case, int(s), case["eps"], key + i) for i, s in enumerate(src)])
    if kind in ("query", "cold"):
        out = _scores(row_ptr, col, case, int(src[0]), case["eps"], key)
        return (out, None, None) if kind == "query" else (out, None)
    rows = torch.stack([_scores(row_ptr, col, case, int(s), float(e), key, case["shared"]) for s, e in zip(src, errs)])
    if kind == "multi":
        return rows, None
    rows[torch.arange(len(src), device=rows.device), torch.from_numpy(src).long().to(rows.device)] = 0.0
    top = min(case["top"], case["n"])
    best = torch.zeros((len(src), case["top"]), dtype=torch.float64, device=rows.device)
    best[:, :top] = torch.sort(rows, dim=1, descending=True).values[:, :top]
    return None, best, None, None
