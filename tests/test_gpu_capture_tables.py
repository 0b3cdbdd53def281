"""Caller's graphs of pf_step against calls that would move what they read."""
import numpy as np
import pytest

from paper_2407_01651_gb300 import pf
from paper_2407_01651_gb300 import workload as wl
from tests.test_gpu_boundaries import F, P, S, W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

DOMS = [(256, 200), (100, 36), (512, 300)]


def handle(bc=None):
    sim = pf.Simulation(DOMS, dict(wl.BASE_PARAMS, g=1e-5), "fp32")
    for d, (nx, ny) in enumerate(DOMS):
        if bc:
            sim.set_boundaries(d, *bc)
        sim.init_fields(d, [(nx / 2, ny / 2, 0.4)], 5.0, [(nx / 5, ny / 4, 6.0)])
    return sim


def capture(sim, stream, n):
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        sim.step(n)
    return g


def same(a, b):
    return all(np.array_equal(a.get_state(d), b.get_state(d)) for d in range(len(DOMS)))


def test_launch_mode_keeps_the_tiles_of_a_captured_step():
    """pf_set_launch chooses rows per tile by size again; a graph captured before
    holds the tables of the old rows, so a handle with one keeps them."""
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        sim, ref = handle(), handle()
        sim.step(1)
        ref.step(1)
        sim.sync()
        g = capture(sim, stream, 2)
        rows = sim.step_config()
        for mode in (1, 0, 1):
            sim.set_launch(mode)
            assert sim.step_config() == rows
            g.replay()
            sim.step(3)
            ref.step(5)
            assert same(sim, ref)
            sim.step(1)      # the graph starts from the buffer it was captured on
            ref.step(1)
        fresh = handle()     # without a graph the rows follow the launches
        fresh.set_launch(1)
        fresh.step(3)
        again = handle()
        again.step(3)
        assert same(fresh, again)
        del g
        for s in (sim, ref, fresh, again):
            s.close()


@pytest.mark.parametrize("bc", [None, (S, S, W, F), (P, P, W, W)])
def test_initialising_again_keeps_what_a_graph_reads(bc):
    """A domain initialised again behind the capture (another mean density): the
    graph steps the new state with the new buoyancy reference."""
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        sim, ref = handle(bc), handle(bc)
        sim.sync()
        g = capture(sim, stream, 2)
        for s in (sim, ref):
            s.init_fields(1, [(30.0, 18.0, 0.1)], 6.0, [(70.0, 18.0, 9.0)])
        g.replay()
        ref.step(2)
        assert same(sim, ref)
        f = ref.fields(0)
        for s in (sim, ref):
            s.set_fields(0, f["phi"][::-1], f["psi"], f["C"])
        g.replay()
        ref.step(2)
        assert same(sim, ref)
        del g
        sim.close()
        ref.close()
