"""The sweep schedule at the edges of its tiers, against the CPU oracle.

Each graph sits on a boundary of the kernel: where per-source arrays move from
shared memory to slabs, where the vertex bits end in a word or past it, rows
and DAG lists one above or below a tier (one thread, eight lanes, a warp, the
whole team), lists that overflow, 16- and 32-bit landmark tables, entries that
do not pack, components and vertices the landmarks do not reach.  Same bar as
the other parity tests: BC zero exactly where the oracle's is zero, else a
relative error of at most 1e-9 per vertex (sums of at most ~10^4 non-negative
doubles: 10^4 x 2^-53 is 10^-12).
"""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import paper_1701_05975_gb300 as bc
from paper_1701_05975_gb300 import gen
from test_gpu_parity import assert_bc_close

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def default_config():
    c0 = bc.bc_get_config()
    yield
    bc.bc_set_config(c0)


def build(n, u, v, w, directed=False):
    if directed:
        key = np.unique(np.asarray(u, np.int64) * n + v, return_index=True)[1]
        return gen.csr_from_directed(n, np.asarray(u)[key], np.asarray(v)[key], np.asarray(w)[key])
    a, b = np.minimum(u, v).astype(np.int64), np.maximum(u, v).astype(np.int64)
    ok = a != b
    key = np.unique(a[ok] * n + b[ok], return_index=True)[1]
    return gen.csr_from_undirected(n, a[ok][key], b[ok][key], np.asarray(w)[ok][key])


def hubs(n, m, wmax, seed, isolated=0, directed=False, wmin=1):
    """Skewed degrees (endpoint density ~ x^-3/4), `isolated` vertices without entries."""
    rng = np.random.default_rng(seed)
    live = n - isolated
    u = (live * rng.random(m) ** 4).astype(np.int64)
    v = rng.integers(0, live, m)
    perm = rng.permutation(n)
    keep = u != v
    return build(n, perm[u[keep]], perm[v[keep]], rng.integers(wmin, wmax + 1, keep.sum()), directed)


def star(spokes, chords, seed, wmax=1000):
    """A hub with `spokes` neighbours (light spokes: a DAG list of that length) and a few heavy chords."""
    rng = np.random.default_rng(seed)
    u = np.concatenate([np.zeros(spokes, np.int64), rng.integers(1, spokes + 1, chords)])
    v = np.concatenate([np.arange(1, spokes + 1), rng.integers(1, spokes + 1, chords)])
    w = np.concatenate([rng.integers(1, 4, spokes), rng.integers(wmax // 2, wmax + 1, chords)])
    return build(spokes + 1, u, v, w)


def layers(width, count, wmax=1):
    """Complete bipartite layers of unit weight: many predecessors, DAG lists past their capacity."""
    u, v = [], []
    for a in range(count - 1):
        for i in range(width):
            u += [a * width + i] * width
            v += range((a + 1) * width, (a + 2) * width)
    return build(width * count, np.array(u), np.array(v), np.full(len(u), wmax))


def two_parts(seed):
    """Two skewed components and a path: sources the main landmark does not reach."""
    a, b = hubs(900, 5000, 50, seed), hubs(500, 2500, 50, seed + 1)
    ra, rb = a.edges(), b.edges()
    u = np.concatenate([ra[0], rb[0].astype(np.int64) + 900, np.arange(1400, 1440)])
    v = np.concatenate([ra[1], rb[1].astype(np.int64) + 900, np.arange(1401, 1441)])
    w = np.concatenate([ra[2], rb[2], np.full(40, 7)])
    return build(1441, u.astype(np.int64), v.astype(np.int64), w)


CASES = {
    "landmark-min-n": lambda: hubs(256, 1500, 60, 1),
    "below-landmark-n": lambda: hubs(255, 1500, 60, 2),
    "shared-memory-last": lambda: hubs(1536, 9000, 200, 3),
    "shared-memory-past": lambda: hubs(1537, 9000, 200, 4),
    "bits-word-edge": lambda: hubs(2080, 9000, 200, 5, isolated=0),
    "bits-isolated-tail": lambda: hubs(4000, 9000, 200, 6, isolated=1441),
    "row-of-4-5-20-21": lambda: build(2200, np.repeat([0, 1, 2, 3], [4, 5, 20, 21]), np.arange(10, 60),
                                      np.arange(1, 51)),
    "list-of-8": lambda: star(8, 2, 7),
    "list-of-9": lambda: star(9, 2, 8),
    "list-past-a-warp": lambda: star(2300, 60, 9),
    "rows-past-a-warp": lambda: hubs(6000, 60000, 255, 10),
    "lists-overflow": lambda: layers(20, 12),
    "lists-overflow-slab": lambda: layers(40, 60),
    "table-32-bit": lambda: hubs(3000, 15000, 200000, 11, wmin=1000),
    "entries-do-not-pack": lambda: hubs(3000, 24000, 3000000, 12, wmin=1000),
    "components": lambda: two_parts(13),
    "unit-weights": lambda: hubs(2500, 12000, 1, 14),
    "wide-rows-no-landmark": lambda: gen.er_graph(3000, 40000, 1, 500, seed=15),
    "deep": lambda: gen.grid_graph(60, 60, wmin=1, wmax=100, seed=16),
    "64-bit": lambda: gen.grid_graph(50, 50, wmin=1, wmax=1 << 26, seed=17),
}


@pytest.mark.parametrize("name", CASES)
@pytest.mark.parametrize("team", [0, 32, 128, 1024])
def test_tiers_match_oracle(name, team):
    g = CASES[name]()
    src = np.arange(0, g.n, max(1, g.n // 97), dtype=np.uint32)
    bc.bc_set_config(team_threads=team)
    want, wante = oracle.bc(g, src, 0.5, nthreads=8), oracle.edge_bc(g, src, 0.5)
    with bc.Graph(g) as G:
        for _ in range(2):  # the second run starts from what the first left in its slabs
            assert_bc_close(G.compute(src, 0.5), want)
        assert G.stats().algorithm == bc.BC_ALGO_DELTA
        assert G.stats().sources == len(src)
        ebc, vbc = G.edge_compute(src, 0.5)
        assert_bc_close(ebc, wante)
        assert_bc_close(vbc, want)
        assert_bc_close(G.compute(src[::-1].copy(), 0.5), want)


@pytest.mark.parametrize("isolated", [0, 700])
def test_directed_landmarks_and_unreached_parts(isolated):
    g = hubs(3000, 14000, 100, 21, isolated=isolated, directed=True)
    src = np.arange(0, g.n, 31, dtype=np.uint32)
    with bc.Graph(g, flags=bc.BC_DIRECTED) as G:
        for team in (0, 256):
            bc.bc_set_config(team_threads=team)
            assert_bc_close(G.compute(src, 1.0), oracle.bc_directed(g, src, 1.0))
            ebc, _ = G.edge_compute(src, 1.0)
            assert_bc_close(ebc, oracle.edge_bc(g, src, 1.0))


@pytest.mark.parametrize("n,per,wmax", [(1536, 4, 300), (1537, 12, 300), (6000, 2, 1), (3000, 8, 1 << 30)])
def test_noalloc_runs_the_sweep_schedule_with_64bit_words(n, per, wmax):
    """bc_compute_noalloc: arrays in shared memory up to 1536 vertices, slabs
    above, the bucket width from the largest weight on the device."""
    torch = pytest.importorskip("torch")
    g = gen.er_graph(n, per * n, 1, wmax, seed=n)
    src = np.arange(0, n, max(1, n // 61), dtype=np.uint32)
    dev = lambda x, t: torch.from_numpy(np.ascontiguousarray(x).view(t)).cuda()  # noqa: E731
    rp, col, w = dev(g.row_ptr, np.int64), dev(g.col, np.int32), dev(g.w, np.int32)
    d_src, out = dev(src, np.int32), torch.empty(n, dtype=torch.float64, device="cuda")
    status = torch.full((1,), 9, dtype=torch.int32, device="cuda")
    st = torch.cuda.Stream()
    st.wait_stream(torch.cuda.current_stream())  # the inputs are written on the current stream
    for _ in range(2):
        bc.bc_compute_noalloc(rp.data_ptr(), col.data_ptr(), w.data_ptr(), n, g.nnz, d_src.data_ptr(), len(src), 0.5,
                              out.data_ptr(), status.data_ptr(), st.cuda_stream)
        st.synchronize()
        assert int(status.item()) == bc.BC_OK
        assert_bc_close(out.cpu().numpy(), oracle.bc(g, src, 0.5))


def test_memory_fraction_that_only_holds_strict_slabs():
    """A sweep slab is a quarter larger than a strict one: a budget between the
    two runs the strict schedule on every entry point, as it did before."""
    torch = pytest.importorskip("torch")
    g = gen.ba_graph(3000, 4, 1, 100, seed=31)
    src = np.arange(0, g.n, 97, dtype=np.uint32)
    want = oracle.bc(g, src, 0.5)
    with bc.Graph(g) as G:
        sweep = G.info().slab_bytes
        bc.bc_set_config(algorithm=bc.BC_ALGO_STRICT)
        strict = G.info().slab_bytes
        assert strict < sweep
        free_b = torch.cuda.mem_get_info()[0]
        bc.bc_set_config(algorithm=bc.BC_ALGO_AUTO, mem_fraction=(strict + sweep) / 2 / free_b)
        assert_bc_close(G.compute(src, 0.5), want)
        assert G.stats().algorithm == bc.BC_ALGO_STRICT and G.stats().slots == 1
        ebc, _ = G.edge_compute(src, 0.5)
        assert_bc_close(ebc, oracle.edge_bc(g, src, 0.5))
        G.autotune(src)
        assert_bc_close(G.compute(src, 0.5), want)
        bc.bc_set_config(algorithm=bc.BC_ALGO_DELTA)
        with pytest.raises(bc.BCError) as ei:
            G.compute(src, 0.5)
        assert ei.value.code == bc.BC_ERR_NOMEM
