"""Where resident launches begin and end: the largest lattice on each tile shape
and the next one up, by the number of launches (one for a run of iterations, at
least one an iteration otherwise), and the same bits as single launches on both
sides of the line."""
import numpy as np
import pytest

from paper_2502_00920_gb300 import inputs as I

pytestmark = pytest.mark.gpu

EDGES = (I.Edge("dirichlet", "half_sine", (0.01, -0.004), 0, 50), I.Edge("neumann", "sin2_ramp", (0.02, 0.01), 0, 60),
         I.FREE, I.CLAMPED)
# small and large tile, and the share of the SMs that large tiles may take, by wall reading
TILES = {"fp32": ((16, 8), (32, 14), {"own": 1, "linear": 2}), "fp16s": ((16, 8), (32, 14), {"own": 1, "linear": 2}),
         "fp64": ((8, 8), (16, 16), {"own": 2, "linear": 0})}


@pytest.fixture(scope="module")
def L():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2502_00920_gb300 import build
    build.build()
    from paper_2502_00920_gb300 import lbs
    return lbs


def run(L, c, **kw):
    u0, v0 = I.random_state(c.nx, c.ny, 3, amp_u=1e-4, amp_v=1e-3)
    with L.Simulation(c, u0=u0, v0=v0, monitor_interval=0, **kw) as s:
        before = s.launch_count
        s.step(40)
        launches = s.launch_count - before
        s.step(3)
        s.sync()
        return s.fields(), launches


@pytest.mark.parametrize("precision", list(TILES))
@pytest.mark.parametrize("extrap", ["own", "linear"])
def test_lines_of_the_resident_launches(L, precision, extrap):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    (sx, sy), (lx, ly), share = TILES[precision]
    large = sms // share[extrap] if share[extrap] else 0
    if sms % 8 or large % 4:
        pytest.skip("tiles cannot fill the SMs evenly as laid out here")
    rows = sms // 8
    cases = [(8 * sx, rows * sy, True), (8 * sx - 3, rows * sy - 2, True)]  # the last on small tiles
    if large:
        # past them, the last on large tiles, past those
        cases += [(8 * sx, rows * sy + 1, True), (4 * lx, large // 4 * ly, True), (4 * lx - 5, large // 4 * ly - 1, True),
                  (4 * lx, large // 4 * ly + 1, False), (4 * lx + 1, large // 4 * ly, False)]
    else:
        cases += [(8 * sx, rows * sy + 1, False), (8 * sx + 1, rows * sy, False)]
    for nx, ny, resident in cases:
        c = I.Case("r", nx, ny, 0, model="nh", nu=0.2, edges=EDGES, precision=precision, extrap=extrap, dx=0.01)
        got, launches = run(L, c)
        assert (launches == 1) if resident else launches >= 40, (nx, ny, launches)
        ref, single = run(L, c, graph_chunk=0)
        assert single >= 40
        for a, b in zip(got, ref):
            assert np.isfinite(b).all() and np.array_equal(a, b), (nx, ny)
