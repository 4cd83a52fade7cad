"""Warp columns (two lattice columns per lane, marching up the rows in
registers; two iterations per launch on periodic lattices) against the
global-memory tiles: every node's operations are the same, so the bits are."""
import numpy as np
import pytest

from paper_2502_00920_gb300 import inputs as I

pytestmark = pytest.mark.gpu

PERIODIC = (I.PERIODIC,) * 4
WALLS = (I.CLAMPED, I.Edge("neumann", "sin2_ramp", (0.02, 0.01), 0, 60), I.FREE,
         I.Edge("dirichlet", "const", (0.01, -0.004)))


@pytest.fixture(scope="module")
def L():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2502_00920_gb300 import build
    build.build()
    from paper_2502_00920_gb300 import lbs
    return lbs


def column(L, precision):
    return next(v for v in range(len(L.tile_variants(precision)))
                if L.tile_variant_name(precision, v) == "step_column_kernel")


def run(L, c, u0, v0, calls, **kw):
    with L.Simulation(c, u0=u0, v0=v0, monitor_interval=0, **kw) as s:
        for n in calls:
            s.step(n)
        s.sync()
        return s.fields()


def same(a, b):
    return all(np.array_equal(x, y, equal_nan=True) for x, y in zip(a, b))


# strips of 52 (two iterations) and 56 columns: widths at, before and past their
# multiples; the smallest lattice the columns take; segments that do not divide
SIZES = [(128, 64), (156, 65), (158, 71), (168, 64), (170, 333), (260, 100), (390, 177), (1040, 200)]


@pytest.mark.parametrize("precision", ["fp32", "fp16s"])
@pytest.mark.parametrize("nx,ny", SIZES)
def test_periodic_columns_equal_tiles_bitwise(L, nx, ny, precision):
    v = column(L, precision)
    for model in ("nh", "svk", "le"):
        c = I.Case("p", nx, ny, 0, model=model, nu=0.2, edges=PERIODIC, precision=precision, dx=0.01, body=(0.01, -0.02))
        u0, v0 = I.random_state(nx, ny, 3, amp_u=1e-3, amp_v=1e-2)
        # single, even and odd counts, a graph and what is left of it
        calls = [1, 2, 5, 67]
        ref = run(L, c, u0, v0, calls, variant=0)
        assert np.isfinite(ref[0]).all()
        assert same(run(L, c, u0, v0, calls, variant=v), ref)
        assert same(run(L, c, u0, v0, calls, variant=v, graph_chunk=0), ref)


# interior regions of one tile, one and several strips, odd sizes, padded rows
@pytest.mark.parametrize("nx,ny", [(40, 40), (70, 50), (100, 60), (131, 77), (500, 101), (1021, 130)])
def test_walled_half_precision_columns_equal_tiles_bitwise(L, nx, ny):
    for extrap in ("own", "linear"):
        c = I.Case("w", nx, ny, 0, model="nh", nu=0.2, edges=WALLS, precision="fp16s", extrap=extrap, dx=0.01)
        u0, v0 = I.random_state(nx, ny, 5, amp_u=1e-3, amp_v=1e-2)
        calls = [1, 30]
        ref = run(L, c, u0, v0, calls, variant=0)
        assert np.isfinite(ref[0]).all()
        assert same(run(L, c, u0, v0, calls, variant=column(L, "fp16s")), ref)


@pytest.mark.parametrize("precision", ["fp32", "fp16s"])
def test_strong_compression_and_non_finite_values(L, precision):
    """J < 1/2 (neo-Hooke in double precision) and a NaN take the same course."""
    nx, ny = 256, 128
    c = I.Case("j", nx, ny, 0, model="nh", nu=0.2, edges=PERIODIC, precision=precision, dx=1.0)
    x = 2 * np.pi * np.arange(nx) / nx
    u0 = np.zeros((ny, nx, 2))
    u0[:, :, 0] = -0.7 / (2 * np.pi / nx) * np.sin(x)[None, :]  # J down to 0.3
    ref = run(L, c, u0, None, [3], variant=0)
    assert np.isfinite(ref[0]).all()
    assert same(run(L, c, u0, None, [3], variant=column(L, precision)), ref)
    u0[60, 100, 0] = np.nan
    ref = run(L, c, u0, None, [5], variant=0)
    assert np.isnan(ref[0]).any() and not np.isnan(ref[0]).all()
    assert same(run(L, c, u0, None, [5], variant=column(L, precision)), ref)


def test_large_periodic_lattices_take_the_columns(L):
    """The default of a large periodic lattice; monitors keep their iterations
    (a call of two does not step over one that is due)."""
    c = I.roofline(1024, 0, nx=2048)
    u0, v0 = I.initial_fields(c)
    with L.Simulation(c, v0=v0, monitor_interval=3, graph_chunk=0) as s:
        assert L.tile_variant_name("fp32", s.variant) == "step_column_kernel"
        s.step(10)
        s.sync()
        a = s.fields()
    assert same(a, run(L, c, None, v0, [10], variant=0))
    bad = np.zeros((1024, 2048, 2))
    bad[5, 7, 1] = np.nan
    with L.Simulation(c, u0=bad, monitor_interval=3, graph_chunk=0) as s:
        s.step(4)
        with pytest.raises(L.LbsError):
            s.sync()
        assert s.unstable_iteration == 3
