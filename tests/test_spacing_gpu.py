"""The scheme has no length of its own: with u and dx times a power of two, and
nothing else that carries a length, every iteration computes the same numbers,
at spacings whose squares leave the range of a double too (there the neo-Hooke
law takes another, equivalent form: the results agree to rounding)."""
import numpy as np
import pytest

from paper_2502_00920_gb300 import inputs as I

pytestmark = pytest.mark.gpu

MOVING = I.Edge("dirichlet", "half_sine", (0.01, -0.004), 0, 50)
EDGES = {"periodic": (I.PERIODIC,) * 4, "walls": (MOVING, I.FREE, I.CLAMPED, I.Edge("neumann", "const", (0.002, 0.001)))}


@pytest.mark.parametrize("exponent", [-530, 530, -400])
@pytest.mark.parametrize("edges", list(EDGES))
@pytest.mark.parametrize("nx,ny", [(40, 30), (120, 100), (300, 200)])  # resident on both tiles, single launches
def test_double_precision_neo_hooke_scales_with_the_spacing(nx, ny, edges, exponent):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2502_00920_gb300 import build
    build.build()
    from paper_2502_00920_gb300 import lbs as L
    s = 2.0 ** exponent
    u0, v0 = I.random_state(nx, ny, 3, amp_u=1e-3, amp_v=1e-2)
    out = []
    for k in (1.0, s):
        c = I.Case("s", nx, ny, 0, model="nh", nu=0.2, edges=EDGES[edges], precision="fp64", dx=k / 64)
        with L.Simulation(c, u0=u0 * k, v0=v0) as sim:
            sim.step(20)
            sim.sync()
            out.append(sim.fields())
    (u, v, P), (us, vs, Ps) = out
    assert np.isfinite(u).all() and np.abs(u).max() > 0
    # (the bar that double-precision results hold against the oracle)
    for a, b in ((u, us / s), (v, vs), (P, Ps)):
        assert np.abs(a - b).max() <= 1e-12 * np.abs(a).max()
