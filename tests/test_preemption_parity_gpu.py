"""Preemption at odd iterations: a swapped-out lattice resumes from its own
state whatever the parity of the iteration at which it left (chunks of an odd
number of iterations)."""
import time

import numpy as np
import pytest

from paper_2502_00920_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2502_00920_gb300 import build
    build.build()
    from paper_2502_00920_gb300 import lbs
    return lbs


def test_swapped_out_lattices_resume_at_odd_iterations(L):
    clamped = (I.CLAMPED,) * 4
    long = I.Case("long", 700, 600, 30000, model="nh", nu=0.3, body=(0.0, -0.01), edges=clamped, precision="fp32")
    short = long.replace(name="short", nsteps=100, model="svk", nu=0.2, body=(0.01, 0.0))
    swaps = 0
    with L.Server(precision="fp32", hbm_budget=int(1.5 * L.footprint(long)), chunk=33, preempt_after_s=0.005) as srv:
        tl = srv.submit(long)
        shorts = []
        for _ in range(8):  # each swaps the long one out after some multiple of 33 iterations
            time.sleep(0.03)
            shorts.append(srv.submit(short))
            srv.wait(shorts[-1], 60)
        srv.drain(300)
        swaps = srv.poll(tl)["swaps"]
        got = [srv.result(t) for t in [tl] + shorts]
    assert swaps >= 6
    for case, r in zip([long] + [short] * 8, got):
        assert r[3] == L.OK
        with L.Simulation(case) as s:
            s.step(case.nsteps)
            s.sync()
            for a, b in zip(r[:3], s.fields()):
                assert np.isfinite(b).all() and np.array_equal(a, b), case.name
