"""Solve server under failing device allocations, on the CPU: the engine with a fake CUDA runtime (growth_harness.cu).

A step whose tables cannot grow returns ASCG_ERR_OOM. No launch may then get a table that is not there, the requests
that were not yet running are queued again, and later steps finish all of them.
"""
import os
import re
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.fixture(scope="module")
def lines(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("growth") / "growth")
    nvcc = "/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else "nvcc"
    subprocess.run([nvcc, "-std=c++17", "-w", "-gencode", "arch=compute_103a,code=sm_103a", "--expt-relaxed-constexpr",
                    "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_1701_03989_gb300", "csrc"),
                    os.path.join(HERE, "growth_harness.cu"), "-o", exe], check=True)
    return subprocess.run([exe], check=True, capture_output=True, text=True, timeout=120).stdout.splitlines()


def test_failed_growth_is_made_up_for(lines):
    rows = [dict(zip(m[0::2], map(int, m[1::2]))) for m in (re.split(r"\s+", l) for l in lines[:-1])]
    assert len(rows) > 5 and [r["hit"] for r in rows] == [1] * (len(rows) - 1) + [0]
    for r in rows:
        assert r["status"] == (2 if r["hit"] else 0)       # ASCG_ERR_OOM
        assert r["missing"] == 0                           # tables handed to a launch that are not there
        assert r["done"] == 4 and r["used"] == 0           # every request completed, every basis given back
        if r["hit"]:
            assert r["queued"] >= 1 and r["running"] + r["queued"] == 4
    assert lines[-1] == "leaked 0"
