"""pf_step captured into a caller's graph and replayed on states of pf_set_state
whose populations no collision made: every replay starts from the state that is
in the buffer when it runs."""
import numpy as np
import pytest

from paper_2407_01651_gb300 import pf
from paper_2407_01651_gb300 import workload as wl
from tests.test_gpu_boundaries import F, P, S, W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

FORMS = [("fp64", 0, None, (0, 0, 0)), ("fp32", 0, None, (0, 0, 0)), ("fp32", 1, None, (1, 0, 0)),
         ("fp16", 0, None, (0, 0, 0)), ("bf16", 0, None, (0, 1, 0)), ("fp64", 1, (S, S, W, F), (0, 0, 0)),
         ("fp32", 1, (P, P, W, F), (0, 0, 0)), ("fp32", 0, None, (0, 2, 0))]
DOMS = [(70, 52), (40, 36)]


def handle(precision, thermal, bc, launch):
    sim = pf.Simulation(DOMS, dict(wl.BASE_PARAMS, thermal=thermal, g=1e-5), precision)
    for d, (nx, ny) in enumerate(DOMS):
        if bc:
            sim.set_boundaries(d, *bc)
        sim.init_fields(d, [(nx / 2, ny / 2, 0.4)], 5.0, [(nx / 5, ny / 4, 5.0)])
    sim.set_launch(*launch)
    sim.step(2)
    return sim


def general(st, thermal, seed):
    """The state with every tied population moved on its own."""
    st, rng = st.copy(), np.random.default_rng(seed)
    for g in (slice(9, 18), slice(23, 28), slice(29, 34)) + ((slice(39, 44),) if thermal else ()):
        st[g] += 1e-3 * rng.standard_normal(st[g].shape)
    return st


def capture(sim, stream, n):
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        sim.step(n)
    return g


def states(sim):
    return [sim.get_state(d) for d in range(len(DOMS))]


@pytest.mark.parametrize("form", FORMS, ids=lambda f: "-".join(map(str, f)))
@pytest.mark.parametrize("first", ["capture", "state"])
def test_replays_from_a_state_set_by_hand(form, first):
    """A graph of two steps, the state set before or after it was captured, read
    back (what frees the planes of a used state) and set again between replays,
    against a handle that steps the same states without a graph."""
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        sim, ref = handle(*form), handle(*form)
        raws = [general(st, form[1], 5) for st in states(sim)]
        sim.sync()
        if first == "capture":
            g = capture(sim, stream, 2)
        for s in (sim, ref):
            s.set_state(1, raws[1])
        if first == "state":
            g = capture(sim, stream, 2)
        assert np.array_equal(sim.get_state(1), ref.get_state(1))
        for k in range(4):
            if k == 2:      # both domains now, and one of them back to an ordinary state
                for s in (sim, ref):
                    s.set_state(0, raws[0])
                    s.set_state(1, raws[1])
                    s.set_state(1, ordinary)
            g.replay()
            ref.step(2)
            a, b = states(sim), states(ref)
            assert all(np.array_equal(x, y) for x, y in zip(a, b)), k
            fa, fb = sim.fields(1), ref.fields(1)
            assert all(np.array_equal(fa[n], fb[n]) for n in fa), k
            ordinary = b[1]
        # a replay has used a state: steps outside the graph go on from there
        for s in (sim, ref):
            s.set_state(1, raws[1])
        g.replay()
        ref.step(2)
        for s in (sim, ref):
            s.step(3)
        assert all(np.array_equal(x, y) for x, y in zip(states(sim), states(ref)))
        del g
        sim.close()
        ref.close()


@pytest.mark.parametrize("form", FORMS[:4], ids=lambda f: "-".join(map(str, f)))
def test_graphs_of_one_step_in_turn(form):
    """Two graphs of one step, from either buffer to the other: a state stays what
    its buffer holds until a step overwrites that."""
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        sim, ref = handle(*form), handle(*form)
        raw = general(sim.get_state(0), form[1], 7)
        sim.sync()
        there, back = capture(sim, stream, 1), capture(sim, stream, 1)
        for s in (sim, ref):
            s.set_state(0, raw)
        there.replay()
        there.replay()          # from the same buffer again
        back.replay()
        ref.step(2)
        for _ in range(2):
            assert all(np.array_equal(x, y) for x, y in zip(states(sim), states(ref)))
            there.replay()
            back.replay()
            ref.step(2)
        del there, back
        sim.close()
        ref.close()


def test_thermal_calls_between_replays():
    """pf_reduce_thermal sees the state that a replay left behind."""
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        sim, ref = handle("fp64", 1, None, (0, 0, 0)), handle("fp64", 1, None, (0, 0, 0))
        g = capture(sim, stream, 2)
        raw = general(ref.get_state(0), 1, 9)
        for s in (sim, ref):
            s.set_state(0, raw)
        assert sim.reduce_thermal(0) == ref.reduce_thermal(0)
        g.replay()
        ref.step(2)
        assert sim.reduce_thermal(0) == ref.reduce_thermal(0)
        del g
        sim.close()
        ref.close()


def test_steps_behind_a_replay_do_not_wait():
    """pf_step on a state that a replay has used enqueues and returns, also while
    the host has not looked whether it is raw still."""
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        sim, ref = handle("fp32", 0, None, (0, 0, 0)), handle("fp32", 0, None, (0, 0, 0))
        raw = general(ref.get_state(1), 0, 11)
        sim.sync()
        g = capture(sim, stream, 30)
        for s in (sim, ref):
            s.set_state(1, raw)
        torch.cuda.synchronize()
        for _ in range(60):
            g.replay()
        done = torch.cuda.Event()
        done.record()
        sim.step(1)              # some 10 ms of replays are in front of it
        assert not done.query()
        ref.step(1801)
        assert all(np.array_equal(x, y) for x, y in zip(states(sim), states(ref)))
        del g
        sim.close()
        ref.close()
