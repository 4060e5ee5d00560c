"""Room for a batch's rows after an allocation that was refused: what a buffer is said to hold is
what it holds, so the next call allocates again (or is refused) and never works on memory that
is gone.  Built for the host from the library's header; no GPU is involved."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(HERE, "grow_rows_host.cu")
HDR = os.path.join(os.path.dirname(HERE), "paper_2205_08941_gb300", "csrc", "cq_internal.cuh")
EXE = os.path.join(HERE, "_build", "grow_rows_host")


def run(limit, rows):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    if not os.path.exists(EXE) or any(os.path.getmtime(f) > os.path.getmtime(EXE) for f in (SRC, HDR)):
        os.makedirs(os.path.dirname(EXE), exist_ok=True)
        subprocess.run([nvcc, "-O1", "-std=c++17", SRC, "-o", EXE], check=True, capture_output=True)
    out = subprocess.run([EXE], input=" ".join(map(str, [limit, *rows])), text=True, capture_output=True,
                         check=True).stdout
    return [tuple(int(v) for v in line.split()) for line in out.splitlines()]


def test_a_refused_growth_leaves_no_room():
    got = run(100, [10, 5, 100, 101, 5, 100, 200, 200, 1])
    assert got == [(1, 10, 10), (1, 10, 10), (1, 100, 100), (0, 0, 0), (1, 5, 5), (1, 100, 100), (0, 0, 0),
                   (0, 0, 0), (1, 1, 1)]
    for ok, have, held in got:
        assert have == held and (ok or have == 0)
