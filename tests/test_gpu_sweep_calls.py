"""Calls around the sweep schedule: launches, workspaces, settings and counters.

Results are compared as in the other parity tests (distances and sigma exact,
BC within 1e-9 relative and zero where the oracle's is zero)."""
from __future__ import annotations

import os
import subprocess
import sys

import numpy as np
import pytest

import oracle
import paper_1701_05975_gb300 as bc
from paper_1701_05975_gb300 import gen
from test_gpu_parity import assert_bc_close

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(autouse=True)
def default_config():
    c0 = bc.bc_get_config()
    yield
    bc.bc_set_config(c0)


def fresh_process(code):
    """Run `code` in a new interpreter: no earlier call has prepared a kernel there."""
    head = "import numpy as np, oracle, paper_1701_05975_gb300 as bc\nfrom paper_1701_05975_gb300 import gen\n"
    r = subprocess.run([sys.executable, "-c", head + code], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr


@pytest.mark.parametrize("team", [0, 512, 1024])
def test_debug_hook_is_a_first_call_with_bits_past_48_kb(team):
    """2^18 vertices: 64 KB of vertex bits, above a kernel's default limit of dynamic shared memory."""
    fresh_process(f"""
g = gen.grid_graph(512, 512, wmin=1, wmax=10000, seed=5)
bc.bc_set_config(algorithm=bc.BC_ALGO_DELTA, team_threads={team})
with bc.Graph(g) as G:
    d, sig, _ = G.sssp_debug(77)
want = oracle.sssp(g, 77)
assert np.array_equal(d, want[0]) and np.array_equal(sig, want[1])
""")


def test_settings_may_change_while_requests_are_admitted():
    """The configuration flips between teams and schedules while the server admits
    requests: each runs with the settings it was planned with, none is refused."""
    fresh_process("""
import threading
graphs = [gen.ba_graph(1500, 5, 1, 100, seed=1), gen.grid_graph(470, 470, wmin=1, wmax=9, seed=2)]
src = [np.arange(0, g.n, g.n // 40, dtype=np.uint32) for g in graphs]
want = [oracle.bc(g, s, 0.5, nthreads=8) for g, s in zip(graphs, src)]
stop = threading.Event()
def flip():
    while not stop.is_set():
        for team in (32, 128, 256, 512, 1024):
            for algo in (bc.BC_ALGO_DELTA, bc.BC_ALGO_STRICT):
                bc.bc_set_config(team_threads=team, algorithm=algo)
t = threading.Thread(target=flip)
handles = [bc.Graph(g) for g in graphs]
t.start()
try:
    for _ in range(30):
        reqs = [(i, handles[i].submit(src[i], 0.5)) for i in (0, 1, 0, 0, 1, 0)]
        for i, r in reqs:
            got = r.result(60000)
            assert np.array_equal(got == 0, want[i] == 0)
            nz = want[i] != 0
            assert np.all(np.abs(got[nz] - want[i][nz]) <= 1e-9 * want[i][nz])
finally:
    stop.set()
    t.join()
for h in handles:
    h.close()
""")


def test_autotune_gives_the_other_candidates_workspaces_back():
    """Both schedules are timed at up to 1216 slabs; afterwards one workspace is left, not one per candidate."""
    torch = pytest.importorskip("torch")
    g = gen.ba_graph(30000, 4, 1, 1000, seed=41)
    src = np.arange(0, g.n, 12, dtype=np.uint32)
    with bc.Graph(g) as G:
        slab = G.info().slab_bytes
        most = 1216 * slab + (64 << 20)  # the largest workspace of one candidate
        free0 = torch.cuda.mem_get_info()[0]
        assert free0 > 4 * most  # no candidate is short of memory
        G.autotune(src)
        assert free0 - torch.cuda.mem_get_info()[0] <= most
        assert_bc_close(G.compute(src, 0.5), oracle.bc(g, src, 0.5, nthreads=8))
        assert free0 - torch.cuda.mem_get_info()[0] <= most
        # a workspace whose run has not been read yet is nobody's to free
        s = torch.cuda.Stream()
        d_src, out = torch.from_numpy(src.astype(np.int32)).cuda(), torch.empty(g.n, dtype=torch.float64, device="cuda")
        s.wait_stream(torch.cuda.current_stream())
        G.compute_async(d_src, out, 0.5, stream=s)
        G.autotune(src[:64])
        G.sync(s)
        assert_bc_close(out.cpu().numpy(), oracle.bc(g, src, 0.5, nthreads=8))


def test_tuned_settings_stay_with_the_row_order_they_were_timed_on():
    """The same CSR with and without landmarks (in its own order, past 32,768 vertices, it gets none):
    one unlimited bucket, right under landmark bounds, is not inherited by the other."""
    g0 = gen.ba_graph(33000, 4, 1, 1000, seed=43)
    u, v, w = (np.asarray(x) for x in g0.edges())
    deg = np.bincount(u, minlength=g0.n) + np.bincount(v, minlength=g0.n)
    new = np.empty(g0.n, np.int64)
    new[np.argsort(-deg, kind="stable")] = np.arange(g0.n)
    once = u < v
    g = gen.csr_from_undirected(g0.n, new[u[once]], new[v[once]], w[once])  # numbered by decreasing degree already
    src = np.arange(0, g.n, 330, dtype=np.uint32)
    unlimited = (1 << 64) - 1
    with bc.Graph(g) as A, bc.Graph(g, flags=bc.BC_KEEP_ORDER) as B:
        for G in (A, B):
            G.compute(src, 0.5)
        assert A.stats().bucket_width == unlimited and B.stats().bucket_width < unlimited
        A.autotune(src)
        A.compute(src, 0.5)
        with bc.Graph(g) as C, bc.Graph(g, flags=bc.BC_KEEP_ORDER) as D:
            for G in (C, D):
                G.compute(src, 0.5)
            assert C.stats().bucket_width == A.stats().bucket_width  # the same graph again: tuned
            assert D.stats().bucket_width == B.stats().bucket_width


@pytest.mark.parametrize("n", [1, 300, 1536, 1537, 5000])
def test_slab_bytes_hold_a_source(n):
    """Distances (4), records (16), list offsets (4) and queues of every vertex, in either kind of memory."""
    g = gen.er_graph(n, 4 * n, 1, 50, seed=n) if n > 1 else gen.csr_from_undirected(1, [], [], [])
    with bc.Graph(g) as G:
        assert 24 * n <= G.info().slab_bytes <= 120 * n + 16384


@pytest.mark.parametrize("spokes", [32768, 32769, 65537, 100001])
def test_hub_rows_are_in_landmark_order(spokes):
    """A hub's row at and past the length that is sorted by the whole GPU: spokes closer
    to the hub by another way than by their own edge give the row many different keys."""
    rng = np.random.default_rng(spokes)
    u = np.concatenate([np.zeros(spokes, np.int64), rng.integers(1, spokes + 1, 2 * spokes)])
    v = np.concatenate([np.arange(1, spokes + 1), rng.integers(1, spokes + 1, 2 * spokes)])
    w = np.concatenate([rng.integers(1, 4001, spokes), rng.integers(1, 401, 2 * spokes)])
    key = np.unique(np.minimum(u, v) * (spokes + 1) + np.maximum(u, v), return_index=True)[1]
    key = key[u[key] != v[key]]
    g = gen.csr_from_undirected(spokes + 1, u[key], v[key], w[key])
    src = np.concatenate([[0], rng.integers(1, spokes + 1, 11)]).astype(np.uint32)
    with bc.Graph(g) as G:
        assert_bc_close(G.compute(src, 0.5), oracle.bc(g, src, 0.5, nthreads=8))
        assert G.stats().bucket_width == (1 << 64) - 1  # landmarks are in use
        assert G.stats().entries_scanned < 1.5 * g.nnz * len(src)


@pytest.mark.parametrize("side,wmax,k", [(200, 1 << 24, 456), (200, 1 << 24, 457), (38, 50, 609), (38, 50, 1216)])
def test_sparse_graphs_have_their_sources_in_flight(side, wmax, k):
    """The team rule counts the teams an SM really holds: seven eighths with 64-bit words, few in shared memory."""
    g = gen.grid_graph(side, side, wmin=1, wmax=wmax, seed=3)
    src = np.arange(k, dtype=np.uint32)
    with bc.Graph(g) as G:
        assert_bc_close(G.compute(src, 0.5), oracle.bc(g, src, 0.5, nthreads=8))
        assert G.stats().algorithm == bc.BC_ALGO_DELTA
        assert G.stats().slots == k


@pytest.mark.parametrize("n,m", [(399, 4800), (400, 4799), (400, 4800), (1024, 16384), (1536, 18432), (1537, 18445),
                                 (600, 30000)])
def test_dense_rows_without_landmarks_run_in_slabs(n, m):
    """24 entries a row and more, weights so small that the prefix test keeps most entries."""
    g = gen.er_graph(n, m, 1, 2, seed=m)
    src = np.arange(0, n, 5, dtype=np.uint32)
    want, wante = oracle.bc(g, src, 0.5, nthreads=8), oracle.edge_bc(g, src, 0.5)
    bc.bc_set_config(algorithm=bc.BC_ALGO_DELTA)
    with bc.Graph(g) as G:
        G.compute(src, 0.5)
        assert G.stats().bucket_width < (1 << 64) - 1  # no landmarks
        in_slab = G.info().slab_bytes > 60 * n
        assert in_slab == (n > 1536 or (n >= 400 and g.nnz >= 24 * n))
        for team in (0, 32, 128, 512):
            bc.bc_set_config(team_threads=team)
            assert_bc_close(G.compute(src, 0.5), want)
            ebc, vbc = G.edge_compute(src, 0.5)
            assert_bc_close(ebc, wante)
            assert_bc_close(vbc, want)


@pytest.mark.parametrize("graph,k,strict", [
    (lambda: gen.er_graph(1024, 8192, 1, 3, seed=1), 1024, True),
    (lambda: gen.er_graph(1024, 8192, 1, 3, seed=1), 100, True),
    (lambda: gen.er_graph(1024, 8192, 1, 100, seed=1), 1024, False),
    (lambda: gen.er_graph(9000, 72000, 1, 8, seed=2), 305, True),
    (lambda: gen.er_graph(9000, 72000, 1, 8, seed=2), 304, False),
    (lambda: gen.er_graph(1400, 22400, 1, 16, seed=7), 100, True),  # landmarks
    (lambda: gen.er_graph(1400, 22400, 1, 16, seed=7), 1400, False),
    (lambda: gen.er_graph(2000, 32000, 1, 4, seed=3), 2000, False),
    (lambda: gen.er_graph(200, 1600, 1, 2, seed=4), 200, True),
    (lambda: gen.grid_graph(40, 40, wmin=1, wmax=2, seed=5), 1000, True),
    (lambda: gen.grid_graph(40, 40, wmin=1, wmax=2, seed=5), 100, False),
    (lambda: gen.ba_graph(3000, 4, 1, 2, seed=6), 3000, True),
    (lambda: gen.ba_graph(3000, 4, 1, 50, seed=6), 3000, False),
], ids=str)
def test_small_weights_take_the_strict_schedule(graph, k, strict):
    """AUTO's choice by tied paths and sources; edge output and a pinned schedule are not affected."""
    g = graph()
    src = np.arange(k, dtype=np.uint32)
    want = oracle.bc(g, src, 0.5, nthreads=8)
    with bc.Graph(g) as G:
        assert_bc_close(G.compute(src, 0.5), want)
        assert G.stats().algorithm == (bc.BC_ALGO_STRICT if strict else bc.BC_ALGO_DELTA)
        assert_bc_close(G.submit(src, 0.5).result(60000), want)
        ebc, vbc = G.edge_compute(src[:40], 0.5)
        assert G.stats().algorithm == bc.BC_ALGO_DELTA
        assert_bc_close(ebc, oracle.edge_bc(g, src[:40], 0.5))
        bc.bc_set_config(algorithm=bc.BC_ALGO_DELTA)
        assert_bc_close(G.compute(src, 0.5), want)
        assert G.stats().algorithm == bc.BC_ALGO_DELTA


def test_noalloc_schedule_by_the_largest_weight():
    """Weights on both sides of the lines where the call changes schedules, over all and over a few sources,
    one call after the other on the same scratch array."""
    torch = pytest.importorskip("torch")
    dev = lambda x, t: torch.from_numpy(np.ascontiguousarray(x).view(t)).cuda()  # noqa: E731
    calls = [(1024, 8, w, k) for w in (1, 15, 17, 31, 33, 100) for k in (1024, 50)]
    calls += [(400, 8, w, 400) for w in (16, 17)] + [(1537, 4, w, k) for w in (15, 16, 17) for k in (700, 90)]
    calls += [(2000, 16, w, 64) for w in (1, 126, 130)] + [(900, 2, w, 900) for w in (4, 5)] + [(5, 1, 1, 5)]
    for n, per, wmax, k in calls:
        g = gen.er_graph(n, per * n, 1, wmax, seed=n + wmax)
        g.w[g.w == g.w.max()] = wmax  # both entries of an edge
        src = np.arange(k, dtype=np.uint32)
        rp, col, w, d_src = dev(g.row_ptr, np.int64), dev(g.col, np.int32), dev(g.w, np.int32), dev(src, np.int32)
        out = torch.empty(n, dtype=torch.float64, device="cuda")
        status = torch.full((1,), 9, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        bc.bc_compute_noalloc(rp.data_ptr(), col.data_ptr(), w.data_ptr(), n, g.nnz, d_src.data_ptr(), k, 0.5,
                              out.data_ptr(), status.data_ptr(), 0)
        torch.cuda.synchronize()
        assert int(status.item()) == bc.BC_OK, (n, per, wmax, k)
        assert_bc_close(out.cpu().numpy(), oracle.bc(g, src, 0.5, nthreads=8))


@pytest.mark.parametrize("n,k", [(700, 700), (40000, 9), (250000, 2)])
def test_noalloc_pinned_strict_fills_its_slabs(n, k):
    """Many slabs with a block each, and few that several blocks share; the second call finds the first one's."""
    torch = pytest.importorskip("torch")
    g = gen.grid_graph(n // 50, 50, wmin=1, wmax=20, seed=n)
    src = np.arange(k, dtype=np.uint32)
    dev = lambda x, t: torch.from_numpy(np.ascontiguousarray(x).view(t)).cuda()  # noqa: E731
    rp, col, w, d_src = dev(g.row_ptr, np.int64), dev(g.col, np.int32), dev(g.w, np.int32), dev(src, np.int32)
    out, status = torch.empty(g.n, dtype=torch.float64, device="cuda"), torch.full((1,), 9, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    bc.bc_set_config(algorithm=bc.BC_ALGO_STRICT)
    want = oracle.bc(g, src, 0.5, nthreads=8)
    for _ in range(2):
        bc.bc_compute_noalloc(rp.data_ptr(), col.data_ptr(), w.data_ptr(), g.n, g.nnz, d_src.data_ptr(), k, 0.5,
                              out.data_ptr(), status.data_ptr(), 0)
        torch.cuda.synchronize()
        assert int(status.item()) == bc.BC_OK
        assert_bc_close(out.cpu().numpy(), want)


def csr(n, rows):
    """CSR from {vertex: [(neighbour, weight), ...]}, as given: nothing is made symmetric."""
    deg = np.zeros(n + 1, np.uint64)
    for v, r in rows.items():
        deg[v + 1] = len(r)
    ent = [e for v in sorted(rows) for e in rows[v]]
    return gen.CSRGraph(n=n, row_ptr=np.cumsum(deg).astype(np.uint64), col=np.array([e[0] for e in ent], np.uint32),
                        w=np.array([e[1] for e in ent], np.uint32), name="csr")


def one_way(base, extra, n=None):
    """The symmetric graph `base` with the one-directional entries (v, u, w) added."""
    rows = {}
    for u, v, w in zip(*(x.tolist() for x in base.edges())):
        rows.setdefault(u, []).append((v, w))
    for v, u, w in extra:
        rows[v] = sorted(rows.get(v, []) + [(u, w)])
    return csr(n or base.n, rows)


@pytest.mark.parametrize("team", [0, 32, 128, 512])
@pytest.mark.parametrize("bits", [32, 64])
def test_undirected_rows_without_their_reverses_are_an_error(team, bits):
    """An entry that lies on a shortest path from a source and has no reverse entry: BC_ERR_CUDA on every
    entry point.  Sources that it does not concern are computed, before and after, as is a graph whose
    one-directional entries lie on no shortest path."""
    torch = pytest.importorskip("torch")
    wmax = 1 << 27 if bits == 64 else 50
    base = gen.er_graph(300, 1200, 1, wmax, seed=5)
    whole = gen.csr_from_undirected(420, *(x[base.edges()[0] < base.edges()[1]] for x in base.edges()))
    free = np.arange(0, 300, 7, dtype=np.uint32)
    bc.bc_set_config(team_threads=team)
    # 310 -> 419: a target without a row and with the highest id; 320 -> 321 -> 322, one way each
    broken = one_way(whole, [(310, 419, 3), (320, 321, 2), (321, 322, 2), (330, 331, 5), (331, 330, 6)])
    heavy = one_way(whole, [(0, 1, 4_000_000_000 if bits == 64 else 1_000_000)])
    with bc.Graph(broken) as G, bc.Graph(heavy) as H:
        assert G.info().dist_bits == bits
        for pinned in (bc.BC_ALGO_AUTO, bc.BC_ALGO_DELTA):
            bc.bc_set_config(algorithm=pinned)
            for bad in (310, 320, 330):
                src = np.array([5, bad, 9], np.uint32)
                assert_bc_close(G.compute(free, 0.5), oracle.bc(whole, free, 0.5))
                calls = [lambda: G.compute(src, 0.5), lambda: G.edge_compute(src, 0.5), lambda: G.submit(src, 0.5).result(60000)]
                for call in calls:
                    with pytest.raises(bc.BCError) as ei:
                        call()
                    assert ei.value.code == bc.BC_ERR_CUDA
            d_src, out = torch.tensor([330], dtype=torch.int32, device="cuda"), torch.empty(420, dtype=torch.float64, device="cuda")
            s = torch.cuda.Stream()
            s.wait_stream(torch.cuda.current_stream())
            G.compute_async(d_src, out, 0.5, stream=s)
            with pytest.raises(bc.BCError) as ei:
                G.sync(s)
            assert ei.value.code == bc.BC_ERR_CUDA
            assert_bc_close(G.compute(free, 0.5), oracle.bc(whole, free, 0.5))
            assert G.stats().algorithm == bc.BC_ALGO_DELTA
            ebc, vbc = G.edge_compute(np.array([331 - 300, 6], np.uint32), 0.5)
            assert_bc_close(vbc, oracle.bc(whole, np.array([31, 6], np.uint32), 0.5))
            assert_bc_close(H.compute(free, 0.5), oracle.bc(whole, free, 0.5))
        with pytest.raises(bc.BCError) as ei:
            G.sssp_debug(320)
        assert ei.value.code == bc.BC_ERR_CUDA
        d, sig, _ = G.sssp_debug(8)
        want = oracle.sssp(whole, 8)
        assert np.array_equal(d, want[0]) and np.array_equal(sig, want[1])


@pytest.mark.parametrize("graph", [
    lambda: gen.er_graph(700, 5600, 1, 60, seed=1),
    lambda: gen.er_graph(700, 5600, 1, 1, seed=2),  # lists outgrow shared memory
    lambda: gen.er_graph(2000, 30000, 1, 40, seed=3),  # eight threads to a row
    lambda: gen.ba_graph(4000, 4, 1, 100, seed=4),
    lambda: gen.er_graph(3000, 1700, 1, 9, seed=5),  # most sources reach a few vertices
    lambda: gen.rmat_graph(12, 16, wmin=1, wmax=3, seed=6),
    lambda: gen.grid_graph(30, 30, wmin=1, wmax=1 << 27, seed=7),
], ids=str)
@pytest.mark.parametrize("team", [0, 32, 512])
def test_dag_edges_counts_the_edges(graph, team):
    """stats().dag_edges: the entries on shortest paths, in every form of the DAG build."""
    g = graph()
    src = np.arange(0, g.n, max(1, g.n // 60), dtype=np.uint32)
    rows, cols, ws = g.edges()
    edges = 0
    for s in src:
        d = oracle.sssp(g, int(s))[0]
        edges += int(np.sum((d[rows] != np.iinfo(np.uint64).max) & (d[rows] + ws.astype(np.uint64) == d[cols])))
    bc.bc_set_config(algorithm=bc.BC_ALGO_DELTA, team_threads=team)
    with bc.Graph(g) as G:
        G.compute(src, 0.5)
        assert G.stats().dag_edges == edges


@pytest.mark.parametrize("graph", [lambda: gen.er_graph(1024, 8192, 1, 3, seed=1), lambda: gen.ba_graph(3000, 4, 1, 50, seed=6)],
                         ids=["small-weights", "landmarks"])
def test_plain_form_keeps_its_split_width(graph):
    """The automatic schedule of the batched mode does not change the plain form's settings."""
    g = graph()
    src = np.arange(200, dtype=np.uint32)
    with bc.Graph(g) as G:
        bc.bc_set_config(algorithm=bc.BC_ALGO_DELTA)
        G.compute(src, 0.5)
        width = G.stats().bucket_width
        bc.bc_set_config(mode=bc.BC_MODE_PLAIN, algorithm=bc.BC_ALGO_AUTO)
        assert_bc_close(G.compute(src, 0.5), oracle.bc(g, src, 0.5))
        assert G.stats().bucket_width == width
