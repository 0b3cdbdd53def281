"""Device memory of raw states (pf_set_state of populations that no collision
made): what they hold, and what an allocation that fails leaves behind."""
import numpy as np
import pytest

from paper_2407_01651_gb300 import pf
from paper_2407_01651_gb300 import workload as wl

pytestmark = pytest.mark.gpu


class Allocator:
    """PyTorch's allocator with a record of what is held and a switch to fail."""

    def __init__(self):
        import torch
        self.held, self.fail = {}, False
        dev = torch.cuda.current_device()

        def alloc(ctx, nbytes, stream):
            if self.fail:
                return None
            p = torch.cuda.caching_allocator_alloc(int(nbytes), dev, stream or 0)
            self.held[p] = int(nbytes)
            return p

        def free(ctx, ptr, stream):
            del self.held[ptr]
            torch.cuda.caching_allocator_delete(ptr)
        self.struct = pf.pf_allocator(None, pf._ALLOC_FN(alloc), pf._FREE_FN(free))

    def bytes(self):
        return sum(self.held.values())


@pytest.fixture
def allocator(monkeypatch):
    pytest.importorskip("torch")
    a = Allocator()
    monkeypatch.setattr(pf, "torch_allocator", lambda device=None: a.struct)
    return a


def general(sim, dom, seed):
    """The domain's state with the populations of the solute moved on their own."""
    st = sim.get_state(dom)
    st[29:34] += 1e-3 * np.random.default_rng(seed).standard_normal(st[29:34].shape)
    return st


def ensemble(doms, precision, thermal=0):
    sim = pf.Simulation(doms, dict(wl.BASE_PARAMS, thermal=thermal), precision,
                        use_torch_allocator=True)
    for d, (nx, ny) in enumerate(doms):
        sim.init_fields(d, [(nx / 2, ny / 2, 0.3)], 5.0, [])
    return sim


@pytest.mark.parametrize("precision,thermal,values", [
    ("fp32", 0, 19), ("fp32", 1, 25), ("fp64", 0, 19), ("fp16", 0, 19)])
def test_raw_states_hold_their_tied_planes_only(allocator, precision, thermal, values):
    """Every domain of an ensemble raw: 19 (25) values a site in the storage type,
    not a staging buffer each; they are released once a step has used them."""
    doms = [(64, 48)] * 6 + [(40, 36)]
    sim = ensemble(doms, precision, thermal)
    states = [general(sim, d, d) for d in range(len(doms))]   # staging is at its size now
    before = allocator.bytes()
    for d, st in enumerate(states):
        sim.set_state(d, st)
    elem = {"fp64": 8, "fp32": 4, "fp16": 2}[precision]
    assert allocator.bytes() - before == sum(values * elem * nx * ny for nx, ny in doms)
    sim.step(2)
    sim.get_state(0)
    assert allocator.bytes() == before
    sim.close()
    assert not allocator.held


@pytest.mark.parametrize("what", ["same domain", "other domain", "tied planes"])
def test_an_allocation_that_fails_leaves_the_state(allocator, what):
    """pf_set_state that runs out of memory: a raw state stays the raw state."""
    doms = [(32, 40), (64, 48)]
    sim = ensemble(doms, "fp64")
    st0 = general(sim, 0, 1)
    sim.set_state(0, st0)
    if what == "tied planes":
        new, dom = general(sim, 1, 2), 1   # the staging is large enough now
        want = sim.get_state(1)
        allocator.fail = True
    else:
        dom = 0 if what == "same domain" else 1
        new = np.random.default_rng(3).standard_normal((39, doms[dom][1], doms[dom][0]))
        allocator.fail = True
        with pytest.raises(pf.PFError) as e:
            sim.set_state(1, np.zeros((39, 48, 64)))   # the staging would have to grow
        assert e.value.code == pf.PF_ERR_OOM
        want = None
    with pytest.raises(pf.PFError) as e:
        sim.set_state(dom, new)
    assert e.value.code == pf.PF_ERR_OOM
    with pytest.raises(pf.PFError) as e:
        sim.set_fields(0, *[np.zeros((40, 32))] * 6) if what == "same domain" else sim.set_state(dom, new)
    assert e.value.code == pf.PF_ERR_OOM
    allocator.fail = False
    assert np.array_equal(sim.get_state(0), st0)
    if want is not None:
        assert np.array_equal(sim.get_state(1), want)
    sim.step(1)
    ref = ensemble(doms, "fp64")
    ref.set_state(0, st0)
    ref.step(1)
    for d in (0, 1):
        assert np.array_equal(sim.get_state(d), ref.get_state(d))


@pytest.mark.parametrize("wait", ["sync", "reduce", "reduce_thermal", "set_state"])
def test_every_wait_releases_used_planes(allocator, wait):
    """Planes that a step has used go at the next call that waits for the stream."""
    sim = ensemble([(64, 48)], "fp32", 1)
    ordinary, st = sim.get_state(0), general(sim, 0, 1)
    before = allocator.bytes()
    sim.set_state(0, st)
    sim.step(2)
    assert allocator.bytes() - before == 25 * 4 * 64 * 48
    sim.set_state(0, ordinary) if wait == "set_state" else getattr(sim, wait)()
    assert allocator.bytes() == before
