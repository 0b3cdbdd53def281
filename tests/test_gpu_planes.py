"""Planes per tile of the 3-D z-marches chosen by size: the state is that of
fixed lengths, bit for bit (a tile's warm-up planes are streamed by the same
arithmetic as its own)."""
import numpy as np
import pytest

from paper_2407_01651_gb300 import pf
from tests import test_gpu_3d as melt
from tests import test_gpu_3f as flow

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("shape", [(4, 4, 4), (37, 45, 51), (64, 64, 64), (96, 40, 130)])
def test_planes_by_size_give_the_state_of_fixed_lengths(shape, precision):
    centre = [0.5 * n for n in shape]
    R = 0.25 * min(shape)
    for params in (melt.P3, melt.T3):
        got = []
        for chunk in (None, 16, 3):
            sim = pf.Simulation3D(shape, dict(melt.wl.BASE_PARAMS, **params), precision)
            if chunk:
                sim.set_chunk(chunk)
            sim.init_seeds([tuple(centre)], R)
            sim.step(3)
            got.append(sim.get_state())
            sim.close()
        assert all(np.array_equal(g, got[0]) for g in got), "melt"
    planes = flow.flow_fields(shape, [tuple(centre)], R, [(1.0, 2.0, 1.5, R)])
    got = []
    for chunk in (None, 36, 3):
        sim = pf.Simulation3F(shape, dict(flow.wl.BASE_PARAMS, **flow.P3F), precision)
        if chunk:
            sim.set_chunk(chunk)
        sim.set_fields(*planes)
        sim.step(3)
        got.append(sim.get_state())
        sim.close()
    assert all(np.array_equal(g, got[0]) for g in got), "two-phase"
