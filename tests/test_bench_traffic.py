"""The measured DRAM bytes of a committed profile describe one run only (CPU)."""
from __future__ import annotations

import re

import pytest

import bench


@pytest.mark.parametrize("workload", ["rmat20", "ba65k"])
def test_traffic_needs_the_captured_run(workload):
    text = open(f"{bench.ROOT}/profiles/bc_batched_{workload}.md").read()
    run = {k: re.search(rf"^captured_{k}:\s*(\S+)", text, re.M).group(1)
           for k in ("algorithm", "sources", "team_threads", "slots")}
    assert run["algorithm"] == "sweep"
    run = {k: v if k == "algorithm" else int(v) for k, v in run.items()}
    assert bench.load_traffic(workload, run) == bench.load_traffic(workload) > 0
    for other in (dict(algorithm="strict"), dict(sources=64), dict(team_threads=128), dict(slots=76)):
        assert bench.load_traffic(workload, {**run, **other}) is None


def test_digest_covers_what_sets_the_traffic():
    names = {p.rsplit("/", 1)[1] for p in bench.KERNEL_SRC}
    assert {"bc_sweep.cuh", "bc_team.cuh", "bc_land.cu", "bc_slab.h", "bc_common.h"} <= names
