"""Workloads whose time is followed: calls of the public API (paper_1403_3005_gb300.nk) as a
user's program makes them, over the graph families and sizes of the tests, the benchmark and
the serving mix (Erdos-Renyi, Barabasi-Albert and R-MAT graphs, from a thousand vertices to
R-MAT scale 24).

A case names a call ("call"), a graph family with its size ("graph", "size": vertices, or the
R-MAT scale; "deg": average degree, attachments per vertex, or edge factor), the number of
sources ("k") and how the call's options come about ("opts"):
  default   no options, the library's own choice
  tuned     nk.autotune once per graph, its options kept (the documented way for repeated calls)
  128, 256  that many sources per launch
  wide      128 sources per launch, switch threshold 16: options kept from an earlier tuning
Inputs are edge lists drawn from the seed with torch, so that exact() has the same graph
without the library.
"""
import math

import numpy as np
import torch

WEIGHT_MAX = 16      # weighted case: integer weights 1..16
EXACT_COLUMNS = 64   # sources swept together in exact()


def listed():
    return [
        # Distances and path counts from one vertex of a small graph, results on the host: an
        # interactive query, all latency.
        {"name": "sssp_er2000", "call": "sssp", "graph": "er", "size": 2000, "deg": 8, "k": 1, "opts": "default"},
        # Exact betweenness of a small graph, the benchmark's exact configuration.
        {"name": "exact_er2000", "call": "exact", "graph": "er", "size": 2000, "deg": 8, "k": 2000, "opts": "default"},
        # A handful of chosen vertices on a million-vertex power-law graph: below 16 sources the
        # library sweeps one source at a time.
        {"name": "sources_rmat20_k8", "call": "sources", "graph": "rmat", "size": 20, "deg": 16, "k": 8, "opts": "default"},
        # A one-off sampled estimate on a graph of odd size without any tuning.
        {"name": "sampled_er200003_k300", "call": "sampled", "graph": "er", "size": 200003, "deg": 8, "k": 300, "opts": "default"},
        # The benchmark's sampled estimate on R-MAT 18, repeated on one graph with tuned options.
        {"name": "sampled_rmat18_k1024", "call": "sampled", "graph": "rmat", "size": 18, "deg": 16, "k": 1024, "opts": "tuned"},
        # The same on the benchmark's Barabasi-Albert graph: a million vertices of degree 8 and more.
        {"name": "sampled_ba1000000_k512", "call": "sampled", "graph": "ba", "size": 1000000, "deg": 8, "k": 512, "opts": "tuned"},
        # The largest graph: R-MAT 24, a slice of the headline's 8192 sources.
        {"name": "sampled_rmat24_k512", "call": "sampled", "graph": "rmat", "size": 24, "deg": 16, "k": 512, "opts": "wide"},
        # A graph seen for the first time: edge list to canonical CSR to one estimate.
        {"name": "new_graph_rmat18_k128", "call": "new_graph", "graph": "rmat", "size": 18, "deg": 16, "k": 128, "opts": "default"},
        # Edge betweenness, one score per arc.
        {"name": "edges_rmat18_k256", "call": "edges", "graph": "rmat", "size": 18, "deg": 16, "k": 256, "opts": "128"},
        # Closeness: distance sums and reach counts.
        {"name": "closeness_rmat18_k1024", "call": "closeness", "graph": "rmat", "size": 18, "deg": 16, "k": 1024, "opts": "256"},
        # Weighted betweenness, weights 1..16.
        {"name": "weighted_rmat18_k64", "call": "weighted", "graph": "rmat", "size": 18, "deg": 16, "k": 64, "opts": "default"},
        # A server under a burst of mixed requests, 16 graphs of 1e3 to 1e5 vertices, scores on the host.
        {"name": "serve_16", "call": "serve", "graph": "mix", "size": 100000, "deg": 8, "k": 1024, "opts": "default", "requests": 16},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["sssp", "exact", "sources", "sampled", "sampled", "sampled", "new_graph", "edges", "closeness",
                       "weighted", "serve"])
    if call == "serve":
        return {"call": call, "graph": "mix", "size": _log_int(rng, 5000, 100000), "deg": 8, "k": _log_int(rng, 128, 1024),
                "opts": "default", "requests": rng.randint(4, 16)}
    graph = rng.choice(["er", "ba", "rmat"])
    top = {"sssp": 300000, "exact": 4000, "sources": 1000000, "sampled": 1000000, "new_graph": 300000, "edges": 300000,
           "closeness": 300000, "weighted": 300000}[call]
    size = _log_int(rng, 1000, top)
    if graph == "rmat":
        size = max(10, int(round(math.log2(size))))
        if call == "sampled":
            size += rng.randint(0, 2)
    deg = {"er": rng.randint(4, 24), "ba": rng.randint(2, 12), "rmat": rng.choice([8, 16])}[graph]
    n = 1 << size if graph == "rmat" else size
    if call == "sssp":
        k = 1
    elif call == "exact":
        k = n
    elif call == "sources":
        k = rng.randint(1, 15)
    elif call == "weighted":
        k = _log_int(rng, 3, 64)
    else:
        k = _log_int(rng, 17, 1000)
    opts = "default"
    if call == "sampled":
        opts = rng.choice(["default", "tuned", "128", "wide"])
    elif call in ("edges", "closeness"):
        opts = rng.choice(["default", "128", "256"])
    return {"call": call, "graph": graph, "size": size, "deg": deg, "k": min(k, n), "opts": opts}


# ---------------------------------------------------------------- inputs
def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _edges(graph, size, deg, seed):
    """(n, u, v): an undirected edge list (int32, may hold loops and duplicates, which the
    canonical graph has not)."""
    dev = _device()
    gen = torch.Generator(device=dev).manual_seed(seed)
    if graph == "er":
        m = size * deg // 2
        u = torch.randint(size, (m,), generator=gen, device=dev, dtype=torch.int32)
        v = torch.randint(size, (m,), generator=gen, device=dev, dtype=torch.int32)
        return size, u, v
    if graph == "ba":
        # every edge of vertex x joins x to an end, drawn uniformly, of the edges so far
        # (Batagelj and Brandes): odd slots of the list of ends refer to an earlier slot
        m = size * deg
        e = torch.arange(m, device=dev)
        ref = (torch.rand(m, generator=gen, device=dev, dtype=torch.float64) * (2 * e + 1)).long().clamp_(max=2 * m - 1)
        ref = torch.minimum(ref, 2 * e)
        end = ref.clone()
        while True:
            odd = (end & 1) == 1
            if not bool(odd.any()):
                break
            end = torch.where(odd, ref[end >> 1], end)
        return size, torch.div(e, deg, rounding_mode="floor").int(), torch.div(end >> 1, deg, rounding_mode="floor").int()
    n, m = 1 << size, deg << size  # R-MAT with the quadrants 0.57, 0.19, 0.19, 0.05
    u = torch.zeros(m, device=dev, dtype=torch.int32)
    v = torch.zeros(m, device=dev, dtype=torch.int32)
    for _ in range(size):
        r = torch.rand(m, generator=gen, device=dev)
        low = r >= 0.76
        right = torch.where(low, r >= 0.95, r >= 0.57)
        u.mul_(2).add_(low)
        v.mul_(2).add_(right)
    return n, u, v


def _graph_seed(case, seed):
    """The graph follows the seed; edge betweenness, whose output has one entry per arc, keeps
    one graph, and its seed draws the sources."""
    return 1 if case["call"] == "edges" else seed


def _mix_graphs(case):
    """The serving mix: (graph, size, deg, k) per request, the three families in turn, sizes
    and source counts spread evenly over their logarithms."""
    c = case["requests"]
    out = []
    for i in range(c):
        graph = ("er", "ba", "rmat")[i % 3]
        n = 1000 * (case["size"] / 1000) ** (i / max(c - 1, 1))
        size = int(round(math.log2(n))) if graph == "rmat" else int(round(n))
        k = int(round(64 * (case["k"] / 64) ** (((7 * i) % c) / max(c - 1, 1))))
        out.append((graph, size, {"er": 8, "ba": 4, "rmat": 16}[graph], min(k, 1 << size if graph == "rmat" else size)))
    return out


def _mixed(x):
    """SplitMix64's finaliser on uint64 arrays."""
    x = (x ^ (x >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    x = (x ^ (x >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return x ^ (x >> np.uint64(31))


def _sampled(n, seed, k):
    """The sampled set of nk.h: the k vertices of the smallest SplitMix64 outputs."""
    with np.errstate(over="ignore"):
        keys = _mixed(np.uint64(seed) + np.arange(1, n + 1, dtype=np.uint64) * np.uint64(0x9E3779B97F4A7C15))
    return np.sort(np.argsort(keys, kind="stable")[:k]).astype(np.int32)


def _chosen(n, seed, k):
    return np.random.default_rng(seed).choice(n, size=k, replace=False).astype(np.int32)


# ---------------------------------------------------------------- the call
class State:
    def __init__(self, case, seed):
        self.call, self.k, self.seed = case["call"], case["k"], seed + 1
        self.opts = self.out = self.graph = None


def prepare(case, seed):
    from paper_1403_3005_gb300 import nk
    st = State(case, seed)
    st.nk = nk
    if st.call == "serve":
        st.work = []
        for i, (graph, size, deg, k) in enumerate(_mix_graphs(case)):
            n, u, v = _edges(graph, size, deg, seed * 1000 + i)
            st.work.append((nk.graph_from_edges(n, u, v), st.seed + i, k))
        st.server = nk.Server()
        return st
    n, u, v = _edges(case["graph"], case["size"], case["deg"], _graph_seed(case, seed))
    dev = u.device
    if st.call == "new_graph":
        st.n, st.u, st.v = n, u, v
        st.out = torch.empty(n, dtype=torch.float64, device=dev)
        return st
    g = st.graph = nk.graph_from_edges(n, u, v)
    if st.call in ("sssp", "sources"):
        st.src = _chosen(n, seed, st.k)
        if st.call == "sources":
            st.src = torch.from_numpy(st.src).to(dev)
            st.out = torch.empty(n, dtype=torch.float64, device=dev)
    elif st.call == "closeness":
        st.out = tuple(torch.empty(n, dtype=torch.float64, device=dev) for _ in range(2))
    elif st.call == "edges":
        st.out = torch.empty(g.n_arcs, dtype=torch.float64, device=dev)
    elif st.call != "exact":
        st.out = torch.empty(n, dtype=torch.float64, device=dev)
    if st.call == "weighted":
        nk.random_weights(g, st.seed, WEIGHT_MAX)
    if case["opts"] == "tuned":
        st.opts = nk.autotune(g, st.seed, st.k)
    elif case["opts"] == "wide":
        st.opts = nk.run_opts(batch=128, alpha=16.0)
    elif case["opts"] != "default":
        st.opts = nk.run_opts(batch=int(case["opts"]))
    return st


def run(st):
    nk, g = st.nk, st.graph
    if st.call == "sssp":
        return nk.sssp(g, int(st.src[0]))
    if st.call == "exact":
        return nk.betweenness_exact(g)
    if st.call == "sources":
        return nk.betweenness_sources(g, st.src, 1.0, st.opts, out=st.out)
    if st.call == "sampled":
        return nk.betweenness_sampled(g, st.seed, st.k, st.opts, out=st.out)
    if st.call == "new_graph":
        return nk.betweenness_sampled(nk.graph_from_edges(st.n, st.u, st.v), st.seed, st.k, out=st.out)
    if st.call == "edges":
        return nk.edge_betweenness_sampled(g, st.seed, st.k, st.opts, out=st.out)
    if st.call == "closeness":
        return nk.closeness_sampled(g, st.seed, st.k, st.opts, out=st.out)
    if st.call == "weighted":
        return nk.betweenness_weighted_sampled(g, st.seed, st.k, st.opts, out=st.out)
    sent = [st.server.submit(sg, s, k) for sg, s, k in st.work]
    for rid, _ in sent:
        rc = st.server.wait(rid)
        if rc != nk.OK:
            raise RuntimeError("request %d ended with status %d" % (rid, rc))
    return [scores for _, scores in sent]


# ---------------------------------------------------------------- work
def _work(call, graph, size, deg, k):
    n = 1 << size if graph == "rmat" else size
    arcs = deg * n * (1 if graph == "er" else 2)
    graph_bytes = 4 * n + 4 * arcs
    if call == "new_graph":
        graph_bytes = 4 * arcs  # the edge list: two 4-byte ids per edge
    if call == "weighted":
        graph_bytes += 4 * arcs
    out = {"sssp": 12 * n, "closeness": 16 * n, "edges": 8 * arcs}.get(call, 8 * n)
    # per source and edge: one addition of path counts; betweenness adds one dependency, edge
    # betweenness also the share; per source and vertex: the dependency's product and quotient
    per_edge = {"sssp": 1, "closeness": 1, "edges": 4}.get(call, 2)
    per_vertex = {"sssp": 0, "closeness": 1}.get(call, 4)
    return graph_bytes + out, k * (per_edge * arcs // 2 + per_vertex * n)


def work(case):
    if case["call"] == "serve":
        parts = [_work("sampled", *g) for g in _mix_graphs(case)]
    else:
        parts = [_work(case["call"], case["graph"], case["size"], case["deg"], case["k"])]
    return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}


# ---------------------------------------------------------------- exact values
def _canonical(n, u, v):
    """(row_ptr, col) of the symmetric graph without loops and duplicates."""
    u, v = u.long(), v.long()
    keep = u != v
    u, v = u[keep], v[keep]
    key = torch.unique(torch.cat([u * n + v, v * n + u]))
    row, col = torch.div(key, n, rounding_mode="floor"), key % n
    rp = torch.zeros(n + 1, dtype=torch.int64, device=u.device)
    rp[1:] = torch.cumsum(torch.bincount(row, minlength=n), 0)
    return rp, row, col


def _matrix(rp, col, n, val=None):
    val = torch.ones(col.numel(), dtype=torch.float64, device=col.device) if val is None else val
    return torch.sparse_csr_tensor(rp, col, val, size=(n, n))


def _forward(adj, n, src):
    """Levels and path counts from each source of src, one column each."""
    b, dev = len(src), adj.device
    cols = torch.arange(b, device=dev)
    dist = torch.full((n, b), -1, dtype=torch.int32, device=dev)
    sigma = torch.zeros((n, b), dtype=torch.float64, device=dev)
    dist[src, cols] = 0
    sigma[src, cols] = 1.0
    front, d = sigma.clone(), 0
    while True:
        front = adj @ front
        front[dist >= 0] = 0.0
        new = front > 0
        if not bool(new.any()):
            return dist, sigma, d
        d += 1
        dist[new] = d
        sigma += front


def _batches(src):
    for i in range(0, len(src), EXACT_COLUMNS):
        yield src[i:i + EXACT_COLUMNS]


def _betweenness(n, u, v, src, scale, edges=False):
    rp, row, col = _canonical(n, u, v)
    adj = _matrix(rp, col, n)
    scores = torch.zeros(n, dtype=torch.float64, device=u.device)
    arcs = torch.zeros(col.numel(), dtype=torch.float64, device=u.device)
    for part in _batches(src):
        dist, sigma, depth = _forward(adj, n, torch.as_tensor(part, device=u.device).long())
        delta = torch.zeros_like(sigma)
        for level in range(depth, 0, -1):
            psi = torch.where(dist == level, (1.0 + delta) / sigma, 0.0)
            up = torch.where(dist == level - 1, sigma, 0.0)
            if edges:
                for i in range(0, col.numel(), 1 << 21):
                    r, c = row[i:i + (1 << 21)], col[i:i + (1 << 21)]
                    arcs[i:i + (1 << 21)] += (up[r] * psi[c]).sum(1)
            if level > 1:
                delta += up * (adj @ psi)
        scores += delta.sum(1)
    if not edges:
        return scores * scale
    # an edge's score is that of its two directions; the arc (x, y) has its reverse where the
    # keys (y, x) sort
    return scale * (arcs + arcs[torch.argsort(torch.argsort(col * n + row))])


def _weighted(n, u, v, seed, src, scale):
    rp, row, col = _canonical(n, u, v)
    key = torch.minimum(row, col) << 32 | torch.maximum(row, col)
    with np.errstate(over="ignore"):
        x = _mixed(np.uint64(seed) + (key.cpu().numpy().astype(np.uint64) + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15))
    # floor(x * 16 / 2^64): the top bits of x
    w = 1 + torch.as_tensor((x >> np.uint64(60)).astype(np.int64), device=u.device)
    by_weight = []
    for i in range(1, WEIGHT_MAX + 1):
        sel = w == i
        p = torch.zeros(n + 1, dtype=torch.int64, device=u.device)
        p[1:] = torch.cumsum(torch.bincount(row[sel], minlength=n), 0)
        by_weight.append(_matrix(p, col[sel], n))
    scores = torch.zeros(n, dtype=torch.float64, device=u.device)
    for part in _batches(src):
        b = len(part)
        s, cols = torch.as_tensor(part, device=u.device).long(), torch.arange(b, device=u.device)
        dist = torch.full((n, b), -1, dtype=torch.int32, device=u.device)
        sigma = torch.zeros((n, b), dtype=torch.float64, device=u.device)
        dist[s, cols] = 0
        sigma[s, cols] = 1.0
        last, d = 0, 0  # distances are settled in increasing order
        while d - last < WEIGHT_MAX:
            d += 1
            count = torch.zeros_like(sigma)
            for i in range(1, min(d, WEIGHT_MAX) + 1):
                count += by_weight[i - 1] @ torch.where(dist == d - i, sigma, 0.0)
            new = (count > 0) & (dist < 0)
            if bool(new.any()):
                last = d
                dist[new] = d
                sigma = torch.where(new, count, sigma)
        delta = torch.zeros_like(sigma)
        psi = torch.zeros_like(sigma)
        for d in range(last, 0, -1):
            at, acc = dist == d, torch.zeros_like(sigma)
            for i in range(1, min(last - d, WEIGHT_MAX) + 1):
                acc += by_weight[i - 1] @ torch.where(dist == d + i, psi, 0.0)
            delta = torch.where(at, sigma * acc, delta)
            psi = torch.where(at, (1.0 + delta) / sigma, psi)
        scores += delta.sum(1)
    return scores * scale


def exact(case, seed):
    call, k = case["call"], case["k"]
    if case["graph"] == "rmat" and case["size"] > 21:
        return None  # minutes
    if call == "serve":
        out = []
        for i, (graph, size, deg, kk) in enumerate(_mix_graphs(case)):
            n, u, v = _edges(graph, size, deg, seed * 1000 + i)
            out.append(_betweenness(n, u, v, _sampled(n, seed + 1 + i, kk), n / (2.0 * kk)).cpu().numpy())
        return out
    n, u, v = _edges(case["graph"], case["size"], case["deg"], _graph_seed(case, seed))
    if call == "exact":
        return _betweenness(n, u, v, np.arange(n, dtype=np.int32), 0.5).cpu().numpy()
    if call == "sources":
        return _betweenness(n, u, v, _chosen(n, seed, k), 1.0)
    if call == "sssp":
        rp, _, col = _canonical(n, u, v)
        dist, sigma, _ = _forward(_matrix(rp, col, n), n, torch.as_tensor(_chosen(n, seed, 1), device=u.device).long())
        if float(sigma.max()) >= 2.0 ** 53:
            return None
        return dist[:, 0].cpu().numpy(), sigma[:, 0].cpu().numpy().astype(np.uint64)
    src = _sampled(n, seed + 1, k)
    if call == "weighted":
        return _weighted(n, u, v, seed + 1, src, n / (2.0 * k))
    if call == "closeness":
        rp, _, col = _canonical(n, u, v)
        adj = _matrix(rp, col, n)
        far = torch.zeros(n, dtype=torch.float64, device=u.device)
        reach = torch.zeros_like(far)
        for part in _batches(src):
            dist, _, _ = _forward(adj, n, torch.as_tensor(part, device=u.device).long())
            far += dist.clamp(min=0).sum(1)
            reach += (dist > 0).sum(1)
        return far * (n / k), reach * (n / k)
    return _betweenness(n, u, v, src, n / (2.0 * k), edges=call == "edges")
