"""The server's edge tables (one row per lattice and iteration of a chunk):
their size is exact for every chunk length that a configuration may ask for,
and a chunk longer than the histories takes no more rows than these have."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2502_00920_gb300 import inputs as I

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = """
#include <stdio.h>
#include <stdlib.h>
#include "lbs_tiles.h"
int main(int argc, char **argv) {
  for (int i = 1; i + 1 < argc; i += 2)
    printf("%zu\\n", lbs::edge_tables_bytes((size_t)atoll(argv[i]), (int64_t)atoll(argv[i + 1])));
  printf("%d\\n", lbs::kEdgeStride);
}
"""


def test_table_bytes_are_exact_or_refused(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    src, exe = tmp_path / "t.cc", str(tmp_path / "t")
    src.write_text(PROGRAM)
    r = subprocess.run([cxx, "-std=c++17", "-Wall", "-Wextra", "-Werror", "-I",
                        os.path.join(ROOT, "paper_2502_00920_gb300", "csrc"), str(src), "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    cases = [(0, 64), (1, 0), (1, 64), (10, 64), (134, 1_000_000), (3, 1 << 27), (3, 1 << 30), (1000, 2 ** 31 - 1),
             (1 << 20, 1 << 40), (2, 2 ** 62)]
    out = subprocess.run([exe] + [str(v) for c in cases for v in c], capture_output=True, text=True, check=True)
    *got, stride = [int(x) for x in out.stdout.split()]
    most = (2 ** 64 - 1) // 2
    for (n, rows), b in zip(cases, got):
        assert b == min(n * rows * stride, most), (n, rows)


@pytest.mark.gpu
@pytest.mark.parametrize("chunk", [1 << 27, 1 << 30, 2 ** 31 - 1])
def test_chunks_longer_than_the_histories(chunk):
    """Three walled lattices whose whole histories are one chunk: the sizes of
    their tables do not fit 32 bits at this chunk's length."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2502_00920_gb300 import build
    build.build()
    from paper_2502_00920_gb300 import lbs as L
    trac = I.Edge("neumann", "linear_ramp", (0.01, 0.0), 0, 80)
    cases = [I.Case("a", 70, 40, n, model="svk", nu=0.2, edges=(I.CLAMPED, trac, I.FREE, I.FREE), precision="fp32")
             for n in (90, 40, 130)]
    with L.Server(precision="fp32", chunk=chunk) as srv:
        tickets = [srv.submit(c) for c in cases]
        srv.drain(60)
        results = [srv.result(t) for t in tickets]
    for c, (u, v, P, rc) in zip(cases, results):
        assert rc == L.OK
        with L.Simulation(c) as s:
            s.step(c.nsteps)
            s.sync()
            for a, b in zip((u, v, P), s.fields()):
                assert np.array_equal(a, b)
