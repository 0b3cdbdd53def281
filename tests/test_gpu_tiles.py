"""Tiles of the y-march at the sizes where they can go wrong."""
import pytest

from paper_2407_01651_gb300 import pf
from paper_2407_01651_gb300 import workload as wl
from tests.test_gpu_boundaries import F, P, S, W, compare, pair

pytestmark = pytest.mark.gpu


def small(nx, ny):
    return wl.Layout(nx, ny, seeds=[(nx / 2, ny / 2, 0.4)], bubbles=[(nx / 4, ny / 4, min(nx, ny) / 8)])


@pytest.mark.parametrize("shape,bc,rows", [
    ((129, 40), (W, S, P, P), 0),     # a last strip of one column
    ((130, 40), (F, W, P, P), 0),
    ((70, 65), (P, P, W, F), 32),     # a last tile row of one row
    ((70, 66), (P, P, W, F), 32),
    ((129, 33), (S, S, W, F), 1),     # single rows: the second row's ring is the first
    ((70, 21), (S, W, F, W), 2),
])
def test_tiles_next_to_a_side(shape, bc, rows):
    """Tiles whose ring touches a side take the boundary kernel, whatever the
    tile height and however narrow the last tile is.  FP64 against the oracle
    with the bounds of test_gpu_boundaries."""
    lay = small(*shape)
    lay.bubbles = [(3.0, 4.0, 6.0), (shape[0] - 5.0, shape[1] - 4.0, 5.0)]
    o, sim = pair(lay, bc, "fp64", dict(lay.params, g=1e-5))
    if rows:
        sim.set_step_config(1, rows)
    for _ in range(4):
        o.step(1)
        sim.step(1)
        compare(o, sim, 1e-11, early=True)
