"""The barrier between the blocks of a resident launch gives up after a bounded
number of polls: every call that reads the state then reports it, and setting
the state anew makes the handle usable again."""
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


# small and large tiles of each precision
@pytest.mark.parametrize("nx,ny,precision", [(70, 60, "fp32"), (160, 160, "fp32"), (60, 50, "fp64"), (128, 128, "fp64"),
                                             (70, 60, "fp16s"), (160, 160, "fp16s")])
def test_a_barrier_that_runs_out_is_reported_until_the_state_is_set_anew(L, nx, ny, precision):
    c = I.Case("w", nx, ny, 0, model="nh", nu=0.2, edges=EDGES, precision=precision, dx=0.01)
    u0, v0 = I.random_state(nx, ny, 3, amp_u=1e-4, amp_v=1e-3)
    with L.Simulation(c, u0=u0, v0=v0, monitor_interval=0) as s:
        s.step(6)
        state = s.save()
        s.step(5)
        ref = s.fields()
        assert np.isfinite(ref[0]).all()
        reads = [s.sync, s.fields, s.fields_static, s.save, lambda: s.probe([0]), s.monitor, lambda: s.grid_error(ref[0]),
                 lambda: s.step(2)]
        for again in (lambda: (s.set_initial(u0, v0), s.step(6)), lambda: s.load(state)):
            for first in range(len(reads) - 1):  # (whichever call meets it first; steps learn of it from the others)
                s.selftest_resident_wait(1000)
                s.step(3)  # (not known yet: these do nothing)
                for f in reads[first:] + reads[:first]:
                    with pytest.raises(L.LbsError) as e:
                        f()
                    assert e.value.code == L.ETIMEOUT
                again()
                s.sync()
                assert s.iteration == 6
                s.step(5)
                assert same(s.fields(), ref)


def test_lattices_without_the_barrier_refuse_the_self_test(L):
    for nx, ny in ((16, 8), (40, 40), (512, 512)):  # one block, one cluster, single launches
        with L.Simulation(I.Case("w", nx, ny, 0, model="nh", nu=0.2, edges=EDGES, precision="fp32")) as s:
            with pytest.raises(L.LbsError) as e:
                s.selftest_resident_wait(10)
            assert e.value.code == L.EINVAL
            s.step(3)
            s.sync()
            assert s.iteration == 3
            with pytest.raises(L.LbsError):
                s.selftest_resident_wait(0)
