"""Limits of the resident launches (small lattices: many iterations in one
cooperative launch): how long one may be, whatever the graph chunk."""
import numpy as np
import pytest

from paper_2502_00920_gb300 import inputs as I

pytestmark = pytest.mark.gpu

# (clamped walls stay bounded over thousands of iterations)
WALLS = (I.Edge("dirichlet", "half_sine", (0.001, -0.0004), 0, 50), I.CLAMPED, I.CLAMPED, I.CLAMPED)
MOST = 4096  # iterations of one launch at most


@pytest.fixture(scope="module")
def L():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2502_00920_gb300 import build
    build.build()
    from paper_2502_00920_gb300 import lbs
    return lbs


def same(a, b):
    return all(np.array_equal(x, y) for x, y in zip(a, b))


@pytest.mark.parametrize("nx,ny", [(16, 8), (33, 20), (70, 60)])  # one block, a cluster, a grid of them
def test_long_graph_chunks_go_out_in_bounded_launches(L, nx, ny):
    c = I.Case("r", nx, ny, 0, model="svk", nu=0.2, edges=WALLS, precision="fp32", dx=0.01, tau=0.6)
    steps = 2 * MOST + 8
    with L.Simulation(c, monitor_interval=0) as s:
        s.step(steps)
        s.sync()
        ref = s.fields()
        assert np.isfinite(ref[0]).all() and np.abs(ref[0]).max() > 0
    for chunk, monitor, launches in ((steps, 0, 3), (2 ** 31 - 2, 0, 3), (steps, 5, 3 + 2), (MOST + 2, 0, 5)):
        with L.Simulation(c, monitor_interval=monitor, graph_chunk=chunk) as s:
            before = s.launch_count
            s.step(steps)
            s.sync()
            assert s.iteration == steps
            assert s.launch_count - before == launches, (chunk, monitor)
            assert same(s.fields(), ref)
