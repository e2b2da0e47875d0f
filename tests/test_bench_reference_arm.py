"""The benchmark's reference arm (the oracle timed on the host cores) runs
without a GPU: check its JSON line against the benchmark contract."""
import json
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.slow
def test_reference_arm_prints_one_contract_line():
    r = subprocess.run([sys.executable, "bench.py", "--impl", "reference", "--steps", "1", "--warmup", "0"],
                       cwd=ROOT, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    lines = [l for l in r.stdout.splitlines() if l.strip()]
    assert len(lines) == 1
    d = json.loads(lines[0])
    assert d["impl"] == "reference" and d["unit"] == "images/s" and d["higher_is_better"] is True
    assert d["value"] > 0 and d["ms_per_step"] > 0 and d["steps"] == 1
    assert d["cpu_baseline"]["kind"] == "oracle" and d["cpu_baseline"]["cores"] >= 1
    assert d["cpu_baseline"]["value"] == d["value"]
    assert d["e2e"] == {"value": d["value"], "unit": "images/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}
    assert d["config"]["workload"].startswith("cfg4")


def test_reference_arm_other_ranks_exit_quietly():
    r = subprocess.run([sys.executable, "bench.py", "--impl", "reference", "--steps", "1", "--warmup", "0"],
                       cwd=ROOT, capture_output=True, text=True, timeout=600, env={**os.environ, "RANK": "1"})
    assert r.returncode == 0 and r.stdout.strip() == ""


def test_traffic_key_covers_what_decides_the_kernels():
    """The hash that keeps a committed DRAM capture with its sources: every convolution source, what it
    includes, and the planning (choice of kernel, tiles, chunks and stages) in hatq_api.cu."""
    import re

    import bench
    csrc = os.path.join(ROOT, "paper_2608_01653_gb300", "csrc")
    need, todo = set(), {f for f in os.listdir(csrc) if f.startswith("hatq_conv")} | {"hatq_api.cu"}
    while todo:
        f = todo.pop()
        need.add(f)
        if f != "hatq_api.cu":
            inc = re.findall(r'#include "(\w+\.\w+)"', open(os.path.join(csrc, f)).read())
            todo |= {i for i in inc if os.path.exists(os.path.join(csrc, i))} - need
    assert set(bench.CONV_SOURCES) == need
