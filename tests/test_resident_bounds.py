"""Bounds audit of the streaming sides, the wall masks and the resident tiles
(CPU): tests/c/resident_bounds.cc walks them over ragged and degenerate lattices
against its own in-lattice test (see the program's header)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_resident_index_arithmetic_stays_in_bounds(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    exe = str(tmp_path / "resident_bounds")
    r = subprocess.run([cxx, "-std=c++17", "-O2", "-Wall", "-Wextra", "-Werror",
                        "-I", os.path.join(ROOT, "paper_2502_00920_gb300", "csrc"),
                        os.path.join(ROOT, "tests", "c", "resident_bounds.cc"), "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    run = subprocess.run([exe], capture_output=True, text=True, timeout=600)
    assert run.returncode == 0 and run.stdout.startswith("ok "), run.stdout + run.stderr[-3000:]
