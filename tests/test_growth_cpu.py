"""The lockstep engine on the CPU, with a fake CUDA runtime (growth_harness.cu): failing allocations, and what is launched.

A step whose tables cannot grow returns ASCG_ERR_OOM. No launch may then get a table that is not there, the requests
that were not yet running are queued again, and later steps finish all of them.
"""
import os
import re
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def _compile(tmp, name, *extra):
    exe = str(tmp.mktemp(name) / name)
    nvcc = "/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else "nvcc"
    subprocess.run([nvcc, "-std=c++17", "-w", "-gencode", "arch=compute_103a,code=sm_103a", "--expt-relaxed-constexpr",
                    "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_1701_03989_gb300", "csrc"),
                    os.path.join(HERE, name + "_harness.cu"), "-o", exe, *extra], check=True)
    return exe


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    exe = _compile(tmp_path_factory, "growth")
    return lambda what: subprocess.run([exe, what], check=True, capture_output=True, text=True, timeout=120).stdout.splitlines()


def _rows(lines):
    return [dict(zip(m[0::2], map(int, m[1::2]))) for m in (re.split(r"\s+", l) for l in lines)]


def test_failed_growth_is_made_up_for(run):
    lines = run("growth")
    rows = _rows(lines[:-1])
    assert len(rows) > 5 and [r["hit"] for r in rows] == [1] * (len(rows) - 1) + [0]
    for r in rows:
        assert r["status"] == (2 if r["hit"] else 0)       # ASCG_ERR_OOM
        assert r["missing"] == 0                           # tables handed to a launch that are not there
        assert r["done"] == 4 and r["used"] == 0           # every request completed, every basis given back
        if r["hit"]:
            assert r["queued"] >= 1 and r["running"] + r["queued"] == 4
    assert lines[-1] == "leaked 0"


def test_reported_launches_are_those_made(run):
    """Systems below the tensor-core line, with exponents recorded by the steps, with both chains in a thread (the exponents
    take a launch), and from 2^20 rows."""
    rows = _rows(run("count"))
    assert [r["n"] for r in rows] == [700, 3000, 250000, 1100000]
    for r in rows:
        assert r["reported"] == r["made"] > 0, r


def test_tuner_times_the_exponents_of_large_batches(run):
    """11 sizes, six Grams each; one exponent pass to prepare each size, and one with every Gram of the three sizes of at
    least 2^20 rows, in whose batches no system's steps record the exponents."""
    (r,) = _rows(run("tune"))
    assert r == {"sizes": 11, "grams": 66, "exponents": 11 + 3 * 6}


def test_server_memory_is_what_the_header_states(run):
    """A 1 GB budget, 16 systems at once: the basis matrix and the partials' first buffers as at creation, buffers at most
    twice what the systems have needed, tables, sums and records as the header gives them."""
    for r in _rows(run("memory")):
        w = 2 * r["s"] + 1
        pairs = w * (w + 1) // 2
        budget = 1 << 30
        first = (budget // (8 * w) // 1024 + 16) // 3 + 1          # partials per class at creation
        assert r["arena"] <= budget
        partials = 8 * pairs * max(2 * r["gitems"], 3 * first) + 8 * pairs * 2 * r["titems"]
        tables = 2 * 96 * r["units"] + 3 * (1024 * 16 + first * 16)
        sums = 2 * r["split"] * (16 * pairs + 4)
        assert r["peak"] <= r["arena"] + partials + tables + sums + 3 * 16 * 25000, r


def test_workspace_after_a_failed_growth(tmp_path_factory):
    """An operator's workspace whose k-th allocation failed: a later, smaller call finds every part, whether the workspace
    was new or already there. The kernels' launchers come from the library; none is called."""
    import __graft_entry__
    __graft_entry__.build()
    lib = os.path.join(ROOT, "paper_1701_03989_gb300")
    exe = _compile(tmp_path_factory, "workspace", "-L", lib, "-l:libascg.so", "-Xlinker", "-rpath," + lib)
    lines = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=120).stdout.splitlines()
    rows = _rows(lines[:-1])
    for grown in (0, 1):
        r = [q for q in rows if q["grown"] == grown]
        assert len(r) > 3 and [q["status"] for q in r] == [2] * (len(r) - 1) + [0]  # ASCG_ERR_OOM until nothing fails
    assert all(q["again"] == 0 and q["missing"] == 0 for q in rows)
    assert lines[-1] == "leaked 0"
