"""Workloads for timing the framework through its public entry points.

Each case is betweenness centrality of one weighted graph (or, for serving, a
burst of requests on several) over a source list: the smallest graphs, where a
call is a handful of launches, up to R-MAT scale 20 with 4096 sources.  The
graph families, weights and source counts are those of the benchmark and the
tests: Erdos-Renyi (8 edges per vertex), Barabasi-Albert (4 per vertex), R-MAT
(.57, .19, .19; 16 per vertex) and the perturbed grid (5% of edges removed).
Graphs are drawn on the GPU from the seed alone.
"""
import math

import numpy as np
import torch

import paper_1701_05975_gb300 as bc
from paper_1701_05975_gb300 import gen

INF = 1 << 62


def listed():
    return [
        # an application's own small network, exact BC, one blocking call from
        # host arrays: launches and latency
        dict(name="er300_compute", entry="compute", kind="er", n=300, per=5, wmax=20, k=300),
        # exact BC of a 1024-vertex graph inside a simulation loop: a captured
        # step replayed with a single launch
        dict(name="er1k_step", entry="step", kind="er", n=1024, per=8, wmax=100, k=1024),
        # a caller that may not allocate on the device while it runs
        dict(name="er1k_noalloc", entry="noalloc", kind="er", n=1024, per=8, wmax=100, k=1024),
        # an ordinary scale-free network, exact BC from host arrays
        dict(name="ba12k_compute", entry="compute", kind="ba", n=12345, per=4, wmax=1000, k=12345),
        # a larger scale-free network, BC estimated from a sample of sources
        dict(name="ba65k_async", entry="async", kind="ba", n=65536, per=4, wmax=1000, k=2048),
        # a large graph without hubs, 256 sampled sources (a serving request's size)
        dict(name="er262k_async", entry="async", kind="er", n=262144, per=8, wmax=1000, k=256),
        # a road-like network (high diameter, low degree), lengths up to 10^4
        dict(name="grid512_step", entry="step", kind="grid", n=512 * 512, per=2, wmax=10000, k=512),
        # the same kind of network with fine length units: 64-bit distances
        dict(name="grid200_wide", entry="compute", kind="grid", n=200 * 200, per=2, wmax=1 << 24, k=304),
        # a directed web-like graph: distances over out-edges, ordered pairs
        dict(name="rmat16_directed", entry="async", kind="digraph", n=1 << 16, per=16, wmax=255, k=1024),
        # edge and vertex BC in one run
        dict(name="rmat16_edges", entry="edges", kind="rmat", n=1 << 16, per=16, wmax=255, k=1024),
        # requests of mixed sizes and kinds in flight at once on the serving loop
        dict(name="serving_burst", entry="serving", kind="pool", n=65536, per=8, wmax=1000, k=256),
        # the benchmark's workload: R-MAT scale 20, 4096 sampled sources
        dict(name="rmat20_step", entry="step", kind="rmat", n=1 << 20, per=16, wmax=255, k=4096),
    ]


def draw(rng):
    kind = rng.choice(["er", "ba", "grid", "rmat", "digraph"])
    # sizes over the logarithm of their range, odd ones among them; R-MAT has
    # a power of two of vertices
    n = int(round(2.0 ** rng.uniform(7.0, 17.0 if kind != "grid" else 18.0)))
    per = {"er": rng.choice([4, 8, 16]), "ba": rng.choice([2, 4, 6]), "grid": 2,
           "rmat": rng.choice([8, 16]), "digraph": rng.choice([8, 16])}[kind]
    if kind in ("rmat", "digraph"):
        n = 1 << max(8, int(math.log2(n)))
    elif kind == "grid":
        side = max(8, int(math.isqrt(n)))
        n = side * side
    wmax = int(round(2.0 ** rng.uniform(0.0, 14.0)))
    if kind in ("er", "grid") and rng.random() < 0.15:
        wmax = 1 << 26  # 64-bit distances
    # sources: exact BC on small graphs, else a sample
    most = max(1, min(n, int(3e9 / (2 * per * n + 4 * n))))
    k = n if n <= 4096 and n <= most else int(round(2.0 ** rng.uniform(0.0, math.log2(most))))
    entry = rng.choice(["compute", "async", "step", "edges", "serving1"])
    if kind != "digraph" and n <= 6000 and rng.random() < 0.2:
        entry = "noalloc"
    return dict(entry=entry, kind=kind, n=n, per=per, wmax=wmax, k=max(1, min(k, n)))


# ------------------------------------------------------------------ graphs


def _distinct(a, b, n, m, g, directed=False):
    """`m` of the distinct pairs without self-loops among (a, b), at random
    (fewer if there are fewer): a graph's entry count follows from its sizes
    alone.  The pairs come back sorted."""
    lo, hi = (a, b) if directed else (torch.minimum(a, b), torch.maximum(a, b))
    key = torch.unique((lo * n + hi)[a != b])
    key = key[torch.randperm(len(key), generator=g, device="cuda")[:m]]
    return key // n, key % n


def _pairs(kind, n, per, g):
    """Endpoint pairs (directed for "digraph", else each undirected edge once)."""
    dev = "cuda"
    if kind == "er":
        m = min(per * n, n * (n - 1) // 4)
        return _distinct(torch.randint(n, (2 * m + 64,), generator=g, device=dev),
                         torch.randint(n, (2 * m + 64,), generator=g, device=dev), n, m, g)
    if kind == "ba":
        # preferential attachment: a new edge's target is a uniformly drawn
        # endpoint of an earlier vertex's edge, resolved by pointer jumping;
        # repeated edges are replaced by uniform ones, up to 95% of the drawn
        m0 = per + 1
        iu = torch.triu_indices(m0, m0, 1, device=dev)
        seed_edges = iu.shape[1]
        src = torch.cat([iu[0], torch.arange(m0, n, device=dev).repeat_interleave(per)])
        first = torch.arange(len(src), device=dev)
        first[seed_edges:] -= (first[seed_edges:] - seed_edges) % per  # edges of earlier vertices only
        pick = (torch.rand(len(src), generator=g, device=dev, dtype=torch.float64) * (2 * first)).long()
        pos = pick.clone()
        pos[:seed_edges] = 2 * torch.arange(seed_edges, device=dev) + 1
        at = pos.clone()
        while True:
            follow = (at % 2 == 1) & (at // 2 >= seed_edges)
            if not bool(follow.any()):
                break
            at = torch.where(follow, pos[at // 2], at)
        dst = torch.where(at % 2 == 1, iu[1][torch.clamp(at // 2, max=seed_edges - 1)], src[at // 2])
        m = int(0.95 * len(src))
        u, v = _distinct(src, dst, n, m, g)
        while len(u) < m:
            u, v = _distinct(torch.cat([u, torch.randint(n, (m,), generator=g, device=dev)]),
                             torch.cat([v, torch.randint(n, (m,), generator=g, device=dev)]), n, m, g)
        return u, v
    if kind in ("rmat", "digraph"):
        # 85% of the drawn pairs are kept: about those that are distinct
        scale, m = int(math.log2(n)), int(0.85 * per * n)
        u = v = torch.zeros(0, dtype=torch.int64, device=dev)
        perm = torch.randperm(n, generator=g, device=dev)
        while len(u) < m:
            a = torch.zeros(per * n, dtype=torch.int64, device=dev)
            b = torch.zeros(per * n, dtype=torch.int64, device=dev)
            for bit in range(scale):
                r = torch.rand(per * n, generator=g, device=dev)
                down = r >= 0.76
                right = ((r >= 0.57) & ~down) | (r >= 0.95)
                a |= down.long() << bit
                b |= right.long() << bit
            u, v = _distinct(torch.cat([u, perm[a]]), torch.cat([v, perm[b]]), n, m, g, kind == "digraph")
        return u, v
    if kind == "grid":
        side = math.isqrt(n)
        ids = torch.arange(n, device=dev).reshape(side, side)
        u = torch.cat([ids[:, :-1].reshape(-1), ids[:-1].reshape(-1)])
        v = torch.cat([ids[:, 1:].reshape(-1), ids[1:].reshape(-1)])
        keep = torch.randperm(len(u), generator=g, device=dev)[: len(u) - round(0.05 * len(u))]
        return u[keep], v[keep]
    raise ValueError(kind)


def _csr(kind, n, per, wmax, seed):
    """row_ptr, col, weight on the GPU (int64), rows sorted by neighbour."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    u, v = _pairs(kind, n, per, g)
    w = torch.randint(1, wmax + 1, (len(u),), generator=g, device="cuda")
    if kind != "digraph":
        u, v, w = torch.cat([u, v]), torch.cat([v, u]), torch.cat([w, w])
    order = torch.argsort(u * n + v)
    u, v, w = u[order], v[order], w[order]
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    row_ptr[1:] = torch.cumsum(torch.bincount(u, minlength=n), 0)
    return row_ptr, v, w


def _sources(n, k, seed):
    if k >= n:
        return np.arange(n, dtype=np.uint32)
    rng = np.random.default_rng(seed + 1)
    return np.sort(rng.choice(n, size=k, replace=False)).astype(np.uint32)


def _scale(case, n, k):
    return (1.0 if case["kind"] == "digraph" else 0.5) * n / k


def _pool(case):
    """The burst's requests: exact BC on the smaller graphs, `k` sampled
    sources on the larger ones."""
    big, k = case["n"], case["k"]
    return [("er", 1024, 8, 1024), ("ba", 4096, 4, 4096), ("grid", 64 * 64, 2, 64 * 64), ("er", 4096, 8, 4096),
            ("ba", big // 4, 4, big // 8), ("er", big, 8, k), ("ba", big, 4, k), ("grid", big, 2, k)]


# ----------------------------------------------------------------- prepare


class State:
    """What the caller keeps between passes; closes its handles when dropped."""

    def __init__(self, case):
        self.case = case
        self.graphs = []
        self.step = None

    def __del__(self):
        if self.step is not None:
            self.step.close()
        for g in self.graphs:
            g.close()


def _graph(csr, n, directed=False):
    row_ptr, col, w = (x.cpu().numpy() for x in csr)
    host = gen.CSRGraph(n=n, row_ptr=row_ptr.astype(np.uint64), col=col.astype(np.uint32), w=w.astype(np.uint32))
    return bc.Graph(host, flags=bc.BC_DIRECTED if directed else 0)


def prepare(case, seed):
    st = State(case)
    entry = case["entry"]
    if entry == "serving":
        st.requests = []
        for i, (kind, n, per, k) in enumerate(_pool(case)):
            G = _graph(_csr(kind, n, per, case["wmax"], seed + i), n)
            st.graphs.append(G)
            st.requests.append((G, _sources(n, k, seed + i), 0.5 * n / k))
        return st
    n, k = case["n"], case["k"]
    csr = _csr(case["kind"], n, case["per"], case["wmax"], seed)
    src = _sources(n, k, seed)
    st.scale = _scale(case, n, k)
    st.sources = src
    st.d_sources = torch.from_numpy(src.astype(np.int32)).cuda()
    st.d_out = torch.empty(n, dtype=torch.float64, device="cuda")
    if entry == "noalloc":
        st.row_ptr, st.col, st.w = csr[0], csr[1].int(), csr[2].int()
        st.status = torch.empty(1, dtype=torch.int32, device="cuda")
        return st
    G = _graph(csr, n, case["kind"] == "digraph")
    st.graphs.append(G)
    if entry == "edges":
        st.d_edges = torch.empty(G.nnz, dtype=torch.float64, device="cuda")
    if entry == "step":
        st.step = G.step(st.d_sources, st.d_out, st.scale)
    return st


# --------------------------------------------------------------------- run


def run(st):
    entry = st.case["entry"]
    if entry == "serving":
        return [r.result() for r in [G.submit(src, scale) for G, src, scale in st.requests]]
    stream = torch.cuda.current_stream()
    if entry == "noalloc":
        bc.bc_compute_noalloc(st.row_ptr.data_ptr(), st.col.data_ptr(), st.w.data_ptr(), st.case["n"], len(st.col),
                              st.d_sources.data_ptr(), len(st.d_sources), st.scale, st.d_out.data_ptr(),
                              st.status.data_ptr(), stream.cuda_stream)
        return {"bc": st.d_out, "status": st.status}
    G = st.graphs[0]
    if entry == "compute":
        return G.compute(st.sources, st.scale)
    if entry == "serving1":
        return G.submit(st.sources, st.scale).result()
    if entry == "edges":
        G.edge_compute_async(st.d_sources, st.d_edges, st.d_out, st.scale, stream=stream)
        return {"edges": st.d_edges, "bc": st.d_out}
    if entry == "step":
        st.step.launch(stream)
    else:
        G.compute_async(st.d_sources, st.d_out, st.scale, stream=stream)
    return st.d_out


def _entries(kind, n, per):
    """CSR entries, about."""
    return n * per * (1 if kind == "digraph" else 2)


def work(case):
    """The graph and the sources read once, the result written once."""
    parts = _pool(case) if case["entry"] == "serving" else [(case["kind"], case["n"], case["per"], case["k"])]
    total = 0
    for kind, n, per, k in parts:
        nnz = _entries(kind, n, per)
        total += 8 * (n + 1) + 8 * nnz + 4 * k + 8 * n + (8 * nnz if case["entry"] == "edges" else 0)
    return {"bytes": total, "flops": 0}


# ------------------------------------------------------------------- exact


def _brandes(csr, n, sources, scale, edges):
    """Brandes' sums in 64-bit integers and doubles: relaxations, path counts
    and dependencies iterated over all entries until nothing changes."""
    row_ptr, col, w = csr
    rows = torch.repeat_interleave(torch.arange(n, device="cuda"), row_ptr[1:] - row_ptr[:-1])
    total = torch.zeros(n, dtype=torch.float64, device="cuda")
    total_e = torch.zeros(len(col), dtype=torch.float64, device="cuda")
    src = torch.from_numpy(sources.astype(np.int64)).cuda()
    step = max(1, min(256, (1 << 26) // max(1, len(col))))
    for b in range(0, len(src), step):
        s = src[b: b + step]
        lane = torch.arange(len(s), device="cuda")
        d = torch.full((n, len(s)), INF, dtype=torch.int64, device="cuda")
        d[s, lane] = 0
        while True:
            nd = d.clone().index_reduce_(0, col, d[rows] + w[:, None], "amin")
            if torch.equal(nd, d):
                break
            d = nd
        tight = ((d[rows] + w[:, None] == d[col]) & (d[rows] < INF)).double()
        sig = torch.zeros((n, len(s)), dtype=torch.float64, device="cuda")
        sig[s, lane] = 1.0
        one, depth = sig.clone(), 0
        while True:
            ns = one.clone().index_add_(0, col, tight * sig[rows])
            depth += 1
            if bool(((ns - sig).abs() <= 1e-14 * ns).all()):
                break
            sig = ns
        ratio = torch.where(tight > 0, sig[rows] / sig[col].clamp(min=1.0), 0.0)
        delta = torch.zeros_like(sig)
        for _ in range(depth):
            delta = torch.zeros_like(sig).index_add_(0, rows, ratio * (1.0 + delta[col]))
        if edges:
            total_e += (ratio * (1.0 + delta[col])).sum(1)
        delta[s, lane] = 0.0
        total += delta.sum(1)
    return scale * total, scale * total_e


def _affordable(kind, n, per, k):
    """Whether the sums above take well under 20 seconds."""
    depth = 3 * math.isqrt(n) if kind == "grid" else 25
    return 3.0 * depth * k * _entries(kind, n, per) < 2e11


def exact(case, seed):
    entry = case["entry"]
    if entry == "serving":
        out = []
        for i, (kind, n, per, k) in enumerate(_pool(case)):
            ok = _affordable(kind, n, per, 4 * k)
            out.append(_brandes(_csr(kind, n, per, case["wmax"], seed + i), n, _sources(n, k, seed + i),
                                0.5 * n / k, False)[0] if ok else None)
        return out
    n, k = case["n"], case["k"]
    if not _affordable(case["kind"], n, case["per"], k):
        return None
    b, e = _brandes(_csr(case["kind"], n, case["per"], case["wmax"], seed), n, _sources(n, k, seed),
                    _scale(case, n, k), entry == "edges")
    if entry == "noalloc":
        return {"bc": b, "status": None}
    return {"edges": e, "bc": b} if entry == "edges" else b
