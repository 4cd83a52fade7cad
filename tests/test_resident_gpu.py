"""Resident launches (small lattices: many iterations in one cooperative
launch) against single launches of every iteration (graph chunk 0), which the
parity tests compare with the oracle: the same operations on every node, so
the same bits."""
import numpy as np
import pytest

from paper_2502_00920_gb300 import inputs as I

pytestmark = pytest.mark.gpu

MOVING = I.Edge("dirichlet", "half_sine", (0.01, -0.004), 0, 50)
TRACTION = I.Edge("neumann", "sin2_ramp", (0.02, 0.01), 0, 60)
WALLS = {
    "periodic": (I.PERIODIC,) * 4,
    "mixed": (MOVING, TRACTION, I.FREE, I.CLAMPED),
    "clamped": (MOVING, I.CLAMPED, I.Edge("dirichlet", "const", (0.003, 0.002)), MOVING),
    "traction": (TRACTION, I.FREE, I.Edge("neumann", "linear_ramp", (0.0, -0.02), 0, 50), I.FREE),
    "strip": (I.PERIODIC, I.PERIODIC, I.CLAMPED, TRACTION),
}


@pytest.fixture(scope="module")
def L():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2502_00920_gb300 import build
    build.build()
    from paper_2502_00920_gb300 import lbs
    return lbs


def fields(L, c, calls, **kw):
    u0, v0 = I.random_state(c.nx, c.ny, 3, amp_u=1e-3, amp_v=1e-2)
    with L.Simulation(c, u0=u0, v0=v0, **kw) as s:
        for n in calls:
            s.step(n)
        s.sync()
        assert s.iteration == sum(calls)
        return s.fields(), s.launch_count


# one node more and less than the tiles (8 x 8, 16 x 8, 16 x 16, 32 x 14), the
# smallest lattice, long strips, and the largest lattices on each tile
SIZES = [(3, 3), (4, 9), (8, 8), (9, 7), (17, 8), (33, 15), (3, 300), (301, 5), (96, 96), (128, 128), (131, 125),
         (256, 256), (303, 241)]


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16s"])
@pytest.mark.parametrize("walls", list(WALLS))
@pytest.mark.parametrize("nx,ny", SIZES)
def test_resident_launches_equal_single_ones_bitwise(L, nx, ny, walls, precision):
    for model, extrap in (("nh", "own"), ("svk", "linear")):
        if extrap == "linear" and walls == "periodic":
            continue
        c = I.Case("r", nx, ny, 0, model=model, nu=0.2, edges=WALLS[walls], precision=precision, extrap=extrap,
                   dx=1.0 / min(nx, ny), body=(0.001, -0.002))
        calls = [1, 37, 2]  # more than one batch of edge values, an odd count, a resumed run
        a, _ = fields(L, c, calls)
        b, _ = fields(L, c, calls, graph_chunk=0)
        for x, y in zip(a, b):
            assert np.isfinite(y).all() and np.array_equal(x, y)


def test_monitors_and_switches_keep_their_places(L):
    """Monitors split a resident run at the same iterations as graph chunks;
    a chosen variant and graph chunk 0 take the single launches; all mix."""
    c = I.Case("m", 60, 50, 0, model="svk", nu=0.2, edges=WALLS["mixed"], precision="fp32")
    ref, many = fields(L, c, [200], graph_chunk=0, monitor_interval=0)
    got, few = fields(L, c, [200], monitor_interval=0)
    assert few < many and all(np.array_equal(x, y) for x, y in zip(got, ref))
    with L.Simulation(c, *I.random_state(60, 50, 3, amp_u=1e-3, amp_v=1e-2), monitor_interval=30) as s:
        s.step(70)
        s.set_graph_chunk(0)
        s.step(13)
        s.set_graph_chunk(64)
        s.step(50)
        s.set_variant(1)
        s.step(67)
        s.sync()
        assert all(np.array_equal(x, y) for x, y in zip(s.fields(), ref))
    # a non-finite state is seen at the first chunk boundary past the interval
    u0 = np.zeros((50, 60, 2))
    u0[20, 20, 0] = np.nan
    with L.Simulation(c, u0=u0, monitor_interval=30) as s:
        s.step(200)
        with pytest.raises(L.LbsError) as e:
            s.sync()
        assert e.value.code == L.EUNSTABLE and s.unstable_iteration == 64
