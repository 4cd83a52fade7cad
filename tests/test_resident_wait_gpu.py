"""The barrier between the blocks of a resident launch gives up after a bounded
number of polls: every call that reads the state then reports it, and setting
the state anew makes the handle usable again."""
import time

import numpy as np
import pytest

from paper_2502_00920_gb300 import inputs as I

pytestmark = pytest.mark.gpu

EDGES = (I.CLAMPED, I.Edge("neumann", "sin2_ramp", (0.02, 0.01), 0, 60), I.FREE, I.CLAMPED)


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


# small and large tiles; which reading call meets the give-up first, which way
# the state is set anew (a wait takes the better part of a second)
@pytest.mark.parametrize("nx,ny,precision,first,again", [
    (70, 60, "fp32", 0, "load"), (160, 160, "fp32", 1, "initial"), (60, 50, "fp64", 2, "initial"),
    (128, 128, "fp64", 3, "load"), (70, 60, "fp16s", 4, "initial"), (160, 160, "fp16s", 5, "load"),
    (70, 60, "fp32", 6, "initial")])
def test_a_barrier_that_runs_out_is_reported_until_the_state_is_set_anew(L, nx, ny, precision, first, again):
    c = I.Case("w", nx, ny, 0, model="nh", nu=0.2, edges=EDGES, precision=precision, dx=0.01)
    u0, v0 = I.random_state(nx, ny, 3, amp_u=1e-4, amp_v=1e-3)
    with L.Simulation(c, u0=u0, v0=v0, monitor_interval=0) as s:
        s.step(6)
        state = s.save()
        s.step(5)
        ref = s.fields()
        assert np.isfinite(ref[0]).all()
        reads = [s.sync, s.fields, s.fields_static, s.save, lambda: s.probe([0]), s.monitor, lambda: s.grid_error(ref[0])]
        t = time.perf_counter()
        s.selftest_resident_wait()
        s.step(3)  # (not known yet: these do nothing)
        for f in reads[first:] + reads[:first] + [lambda: s.step(2)]:
            with pytest.raises(L.LbsError) as e:
                f()
            assert e.value.code == L.ETIMEOUT
        assert time.perf_counter() - t < 30.0
        if again == "load":
            s.load(state)
        else:
            s.set_initial(u0, v0)
            s.step(6)
        s.sync()
        assert s.iteration == 6
        s.step(5)
        assert same(s.fields(), ref)


def test_lattices_without_the_barrier_refuse_the_self_test(L):
    for nx, ny in ((16, 8), (40, 40), (512, 512)):  # one block, one cluster, single launches
        with L.Simulation(I.Case("w", nx, ny, 0, model="nh", nu=0.2, edges=EDGES, precision="fp32")) as s:
            with pytest.raises(L.LbsError) as e:
                s.selftest_resident_wait()
            assert e.value.code == L.EINVAL
            s.step(3)
            s.sync()
            assert s.iteration == 3
