"""The half-precision warp columns on the lattices that do not go whole through
them but are not walled all round: odd or narrow periodic ones, and those with
one periodic axis; their interiors march, their frame tiles wrap.  Every node's
operations are those of the tiles, so the bits are."""
import numpy as np
import pytest

from paper_2502_00920_gb300 import inputs as I

pytestmark = pytest.mark.gpu

PULL = I.Edge("neumann", "sin2_ramp", (0.02, 0.01), 0, 60)
EDGES = {"periodic": (I.PERIODIC,) * 4, "x": (I.PERIODIC, I.PERIODIC, I.CLAMPED, PULL),
         "y": (PULL, I.CLAMPED, I.PERIODIC, I.PERIODIC)}


@pytest.mark.parametrize("edges", list(EDGES))
@pytest.mark.parametrize("nx,ny", [(131, 77), (255, 64), (100, 130), (99, 60), (128, 50), (97, 201), (1021, 63)])
def test_half_periodic_and_odd_columns_equal_tiles_bitwise(nx, ny, edges):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2502_00920_gb300 import build
    build.build()
    from paper_2502_00920_gb300 import lbs as L
    column = next(v for v in range(len(L.tile_variants("fp16s")))
                  if L.tile_variant_name("fp16s", v) == "step_column_kernel")
    c = I.Case("c", nx, ny, 0, model="nh", nu=0.2, edges=EDGES[edges], precision="fp16s", dx=0.01)
    u0, v0 = I.random_state(nx, ny, 5, amp_u=1e-3, amp_v=1e-2)
    out = []
    for v in (0, column):
        with L.Simulation(c, u0=u0, v0=v0, variant=v, monitor_interval=0) as s:
            for n in (1, 2, 67):
                s.step(n)
            s.sync()
            out.append(s.fields())
    for a, b in zip(*out):
        assert np.isfinite(a).all() and np.array_equal(a, b)
