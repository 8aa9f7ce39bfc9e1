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
