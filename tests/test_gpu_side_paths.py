"""The two pulls of the boundary kernel: a warp with a column next to a side takes
the general one for all of its columns, which away from the side has to give the
values of the periodic one, on every run the same."""
import numpy as np
import pytest

from paper_2407_01651_gb300 import pf
from paper_2407_01651_gb300 import workload as wl
from tests.test_gpu_boundaries import F, P, S, W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(20, 33), (33, 20), (100, 41), (131, 40), (258, 24)])
@pytest.mark.parametrize("bc", [(W, W, P, P), (S, F, P, P), (P, P, W, F)])
@pytest.mark.parametrize("precision,thermal", [("fp32", 0), ("fp32", 1), ("fp64", 0), ("fp64", 1)])
def test_columns_away_from_a_side_step_as_periodic_ones(shape, bc, precision, thermal):
    """One step reaches two sites: beyond them a lattice with sides holds what the
    periodic one does.  The bound is that of the same sums in another order: the
    16-fold (W^2) Laplacian of values of order 1 rounded to a few ulp."""
    nx, ny = shape
    par = dict(wl.BASE_PARAMS, thermal=thermal, g=1e-5)
    x, y = np.meshgrid(np.arange(nx) / nx, np.arange(ny) / ny)
    wave = np.sin(2 * np.pi * x) * np.cos(2 * np.pi * y)
    phi, psi = 0.5 + 0.5 * np.tanh(3 * wave + 2), np.tanh(3 * np.cos(2 * np.pi * (x + y)))
    C, vx, vy = 0.9 + 0.05 * wave, 1e-3 * wave, -2e-3 * np.cos(2 * np.pi * y) * np.ones_like(x)
    out = []
    for sides in (bc, bc, None):
        sim = pf.Simulation([shape], par, precision)
        if sides:
            sim.set_boundaries(0, *sides)
        sim.set_fields(0, phi, psi, C, vx, vy, 1e-4 * wave)
        if thermal:
            sim.set_temperature(0, -0.5 + 0.1 * wave)
        sim.step(1)
        out.append(sim.get_state())
        sim.close()
    assert np.array_equal(out[0], out[1])
    bound = 16 * 8 * (2.3e-16 if precision == "fp64" else 1.2e-7)
    cut = (slice(None), slice(2, -2) if bc[2] else slice(None), slice(2, -2) if bc[0] else slice(None))
    for k, (a, b) in enumerate(zip(out[0][cut], out[2][cut])):
        assert np.abs(a - b).max() <= bound * max(1.0, np.abs(b).max()), k
