"""Host-side rules of the sweep schedule (bc_slab.h), compiled for the CPU.

What bounds a kernel's indices is decided here, so it is checked without a
GPU: a wrong bound would be an access out of range there."""
from __future__ import annotations

import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1701_05975_gb300", "csrc")


def run_cpp(tmp_path, body, stdin=""):
    """Compile `body` (the main function's) against bc_slab.h and return its output's words."""
    cxx, nvcc = shutil.which("g++"), shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if cxx is None or not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    src, exe = tmp_path / "host.cpp", tmp_path / "host"
    src.write_text('#include <cstdint>\n#include <iostream>\n#include <vector>\n#include "bc_slab.h"\n'
                   "using namespace bcgpu;\nint main() {\n" + body + "\n}\n")
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, "-isystem", cuda, str(src), "-o", str(exe)], check=True)
    return subprocess.run([str(exe)], input=stdin, capture_output=True, text=True, check=True).stdout.split()


# rows as {vertex: neighbours}
CSRS = [
    (1, {}),
    (40, {}),
    (70, {0: [69]}),  # one direction only: the target has no row and the highest id
    (70, {3: [4], 4: [3]}),
    (100, {2: [64, 65], 64: [2]}),  # the targets' words lie past the last row's
    (100, {2: [1], 99: [0]}),
    (4097, {0: [32, 4095], 4000: [1]}),
]


def test_vertex_bits_cover_every_neighbour(tmp_path):
    text = [str(len(CSRS))]
    want = []
    for n, rows in CSRS:
        deg = np.zeros(n + 1, np.int64)
        for v, nb in rows.items():
            deg[v + 1] = len(nb)
        col = [u for v in sorted(rows) for u in rows[v]]
        text += [f"{n} {len(col)}", " ".join(map(str, np.cumsum(deg))), " ".join(map(str, col))]
        want.append(1 + max([-1] + [v for v in rows if rows[v]] + col))
    got = run_cpp(tmp_path, """
  int cases;
  for (std::cin >> cases; cases-- > 0;) {
    uint32_t n;
    uint64_t nnz;
    std::cin >> n >> nnz;
    std::vector<uint64_t> rp(n + 1ull);
    std::vector<uint32_t> col(nnz);
    for (auto& x : rp) std::cin >> x;
    for (auto& x : col) std::cin >> x;
    std::cout << active_vertices(n, rp.data(), col.data()) << "\\n";
  }""", "\n".join(text))
    assert [int(x) for x in got] == want


def test_teams_per_sm_by_registers_and_shared_memory(tmp_path):
    """32-bit words: 1024 threads; 64-bit ones 7/8 of that up to 256 a team; and what shared memory holds."""
    got = run_cpp(tmp_path, """
  for (uint32_t t : {128u, 256u, 512u, 1024u})
    std::cout << sweep_teams_per_sm(32, t, 0) << " " << sweep_teams_per_sm(64, t, 0) << " ";
  for (uint32_t n : {300u, 1024u, 1536u})
    std::cout << sweep_teams_per_sm(32, 256, make_layout(n, 32, SLAB_NONE).smem) << " "
              << sweep_teams_per_sm(32, 128, make_layout(n, 32, SLAB_NONE).smem) << " ";""")
    assert [int(x) for x in got] == [8, 7, 4, 3, 2, 2, 1, 1, 4, 8, 4, 4, 3, 3]


def test_sweep_counts_stay_in_32_bits(tmp_path):
    """A DAG of every entry with a list per vertex must not wrap the list counter."""
    sizes = [(1 << 20, 1 << 25), (1 << 31, 10), ((1 << 31) - 1, 0), (10**9, 2 * 10**9), (10**9, 23 * 10**8),
             (2, (1 << 32) - 65541), (2, (1 << 32) - 65540)]
    got = run_cpp(tmp_path, "".join(f'  std::cout << sweep_counts_fit({n}u, {m}ull) << " ";\n' for n, m in sizes))
    assert [x == "1" for x in got] == [n < 1 << 31 and m + 2 * n < (1 << 32) - (1 << 16) for n, m in sizes]
    assert got == ["1", "0", "0", "1", "0", "1", "0"]
