"""The rules that choose between kernels by size (csrc/dispatch.cuh): which side each size takes, where one was measured
faster by more than the runs of a side differ."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1701_03989_gb300", "csrc")


def _run(tmp_path, body):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text('#include <cstdio>\n#include "%s"\nusing namespace ascg;\nint main() {\n%s\n}\n'
                   % (os.path.join(CSRC, "dispatch.cuh"), body))
    subprocess.run(["g++", "-std=c++17", "-x", "c++", str(src), "-o", str(exe)], check=True)
    return subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()


# systems of a batch as (rows, entries of O per row), and which of them are summed by chain
BATCHES = [
    ([(131044, 4.0)], "1"), ([(262144, 4.0)], "0"), ([(1048576 - 1, 4.0)], "0"), ([(125000, 6.0)], "1"), ([(262144, 6.0)], "0"),
    ([(1000000, 6.0)], "0"), ([(131072, 8.0)], "1"), ([(750000, 8.0)], "0"), ([(400000, 12.0)], "1"), ([(600000, 12.0)], "0"),
    ([(1000000, 16.0)], "0"), ([(200000, 20.0)], "1"), ([(600000, 20.0)], "0"), ([(1000000, 48.0)], "1"), ([(400000, 96.0)], "1"),
    ([(32400, 4.0)] * 16, "0" * 16), ([(10000, 4.0)] * 30, "0" * 30), ([(10000, 4.0)] * 10, "1" * 10),
    ([(1000000, 4.0), (5000, 40.0)], "01"), ([(729000, 6.0), (3000, 100.0)], "01"), ([(512000, 6.0), (10000, 32.0)], "00"),
    ([(360000, 4.0), (100000, 60.0), (512000, 6.0)], "111"), ([(250000, 4.0), (50000, 128.0)], "11"),
    ([(1048576, 4.0)], "0"), ([(2000000, 48.0)], "0"), ([(2250000, 4.0), (20000, 120.0)], "00"),
]


@pytest.mark.parametrize("systems,want", BATCHES, ids=[str(k) for k in range(len(BATCHES))])
def test_items_by_chain(tmp_path, systems, want):
    body = "BatchRows b;\n"
    for n, l in systems:
        body += "b.rows += %d; b.mean_len += %r * %d; b.max_len = b.max_len > %r ? b.max_len : %r;\n" % (n, l, n, l, l)
    body += "b.mean_len /= (double)b.rows;\n" + "".join('std::printf("%%d ", (int)items_by_chain(b, %r));\n' % l for _, l in systems)
    assert "".join(_run(tmp_path, body)) == want


# classical CG: rows, entries a row, pipelined row sums?
CG_ROWS = [(20000, 13, 1), (20000, 81, 1), (50000, 49, 1), (20000, 5, 0), (70000, 13, 0), (70000, 49, 1), (80000, 21, 0), (90000, 33, 1),
           (100000, 13, 0), (100000, 49, 1), (110000, 13, 0), (110000, 21, 0), (110000, 61, 0), (116000, 61, 1), (130000, 21, 0),
           (130000, 81, 1), (150000, 13, 0), (150000, 33, 0), (150000, 49, 1), (160000, 13, 1), (160000, 81, 1), (175000, 49, 1),
           (190000, 33, 1), (190000, 61, 0), (200000, 49, 0), (200000, 201, 0), (230000, 33, 1), (262144, 21, 1), (262144, 33, 0),
           (262144, 201, 0), (300000, 21, 0), (600000, 81, 0)]


def test_cg_rows_pipelined(tmp_path):
    got = _run(tmp_path, "".join('std::printf("%%d ", (int)cg_rows_pipelined(%d, %d));\n' % (n, n * k) for n, k, _ in CG_ROWS))
    assert [int(v) for v in got] == [w for _, _, w in CG_ROWS]
