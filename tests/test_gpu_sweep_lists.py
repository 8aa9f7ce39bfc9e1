"""DAG lists and rows on both sides of the sweep kernel's tiers, where they survive to be walked.

A leaf is replaced by a count before sigma, so a list of leaves tests nothing
below it.  Here every listed successor has successors with two predecessors:
the lists reach sigma and the dependencies at their full length.  Same bar as the
other parity tests: BC zero exactly where the oracle's is, else 1e-9 relative."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import paper_1701_05975_gb300 as bc
from paper_1701_05975_gb300 import gen
from test_gpu_parity import assert_bc_close
from test_gpu_sweep import hubs, layers

pytestmark = pytest.mark.gpu
UNLIMITED = (1 << 64) - 1


@pytest.fixture(autouse=True)
def default_config():
    c0 = bc.bc_get_config()
    bc.bc_set_config(algorithm=bc.BC_ALGO_DELTA)
    yield
    bc.bc_set_config(c0)


def kept_star(spokes, seed):
    """A hub with `spokes` spokes of random length; child i hangs tied from spokes i and i + 1, all children
    at distance 1000 from the hub: the hub's list keeps every spoke, every spoke's list two children."""
    rng = np.random.default_rng(seed)
    w = rng.integers(1, 900, spokes)
    spoke, child = 1 + np.arange(spokes), 1 + spokes + np.arange(spokes)
    u = np.concatenate([np.zeros(spokes, np.int64), spoke, np.roll(spoke, -1)])
    v = np.concatenate([spoke, child, child])
    return gen.csr_from_undirected(1 + 2 * spokes, u, v, np.concatenate([w, 1000 - w, 1000 - np.roll(w, -1)]))


def check(g, src, team, flags=0, overflow=False):
    bc.bc_set_config(team_threads=team)
    want, wante = oracle.bc(g, src, 0.5, nthreads=8), oracle.edge_bc(g, src, 0.5)
    with bc.Graph(g, flags=flags) as G:
        for _ in range(2):  # the second run starts from what the first left in its slabs
            assert_bc_close(G.compute(src, 0.5), want)
            assert (G.stats().pair_overflows > 0) == overflow
        ebc, vbc = G.edge_compute(src, 0.5)
        assert_bc_close(ebc, wante)
        assert_bc_close(vbc, want)
        return G.stats(), G.info()


@pytest.mark.parametrize("team", [0, 32, 128, 1024])
@pytest.mark.parametrize("spokes", [4, 5, 20, 21, 68, 69, 700, 2048, 2049, 2300, 5000])
def test_lists_that_are_kept(spokes, team):
    """One thread up to 4 successors, eight lanes up to 68, a warp up to 2048, the whole team above; rows of 4 / 5
    and 20 / 21 entries as well, since the hub is among the sources."""
    g = kept_star(spokes, spokes)
    src = np.unique(np.concatenate([[0, 1, spokes, 1 + spokes], np.arange(0, g.n, max(1, g.n // 9))])).astype(np.uint32)
    check(g, src, team)


@pytest.mark.parametrize("entries", [4, 5, 20, 21, 128, 129])
@pytest.mark.parametrize("chords", [0, 3])
def test_rows_walked_from_their_hub(entries, chords):
    """A row of exactly `entries` entries in a graph whose every vertex is a source."""
    rng = np.random.default_rng(entries + chords)
    n = entries + 1 + 4
    u = np.concatenate([np.zeros(entries, np.int64), rng.integers(1, n, chords * n)])
    v = np.concatenate([1 + np.arange(entries), rng.integers(1, n, chords * n)])
    key = np.unique(np.minimum(u, v) * n + np.maximum(u, v), return_index=True)[1]
    key = key[u[key] != v[key]]
    g = gen.csr_from_undirected(n, u[key], v[key], rng.integers(1, 30, len(key)))
    assert int(np.diff(g.row_ptr)[0]) == entries
    for team in (0, 32, 256):
        check(g, np.arange(n, dtype=np.uint32), team)


@pytest.mark.parametrize("width,count", [(20, 12), (40, 60)])
def test_lists_that_overflow(width, count):
    g = layers(width, count)
    for team in (0, 32, 512):
        check(g, np.arange(0, g.n, max(1, g.n // 40), dtype=np.uint32), team, overflow=True)


@pytest.mark.parametrize("graph,bits,packed", [
    (lambda: hubs(3000, 15000, 100, 11), 16, True),
    (lambda: hubs(3000, 15000, 200000, 11, wmin=1000), 32, True),
    (lambda: hubs(3000, 24000, 3000000, 12, wmin=1000), 32, False),
], ids=["16-bit", "32-bit", "entries-do-not-pack"])
def test_landmark_tables_are_in_use(graph, bits, packed):
    g = graph()
    src = np.arange(0, g.n, 31, dtype=np.uint32)
    st, info = check(g, src, 0)
    assert st.bucket_width == UNLIMITED and info.relabeled and info.dist_bits == 32
    n, nnz = g.n, g.nnz
    rows = (n + 1) * 8 + nnz * (4 if packed else 8) + 4 * n + 8 * n + 8 * n + 4 * nnz
    assert info.device_bytes == rows + (12 if packed else 16) * nnz + ((n + 7) // 8 * 8) * 64 * bits // 8
