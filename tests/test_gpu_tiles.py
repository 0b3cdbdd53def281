"""Tiles chosen by size, tiles next to non-periodic sides, and the one-launch
FP64 reductions, at the sizes where they can go wrong."""
import numpy as np
import pytest

from paper_2407_01651_gb300 import pf
from paper_2407_01651_gb300 import workload as wl
from tests.test_gpu_boundaries import F, P, S, W, compare, pair

pytestmark = pytest.mark.gpu


def small(nx, ny):
    return wl.Layout(nx, ny, seeds=[(nx / 2, ny / 2, 0.4)], bubbles=[(nx / 4, ny / 4, min(nx, ny) / 8)])


@pytest.mark.parametrize("shape", [(4, 4), (64, 64), (129, 5), (300, 301), (512, 96)])
@pytest.mark.parametrize("precision,thermal", [("fp32", 0), ("fp32", 1), ("fp64", 0), ("fp16", 0)])
def test_rows_per_tile_do_not_change_the_bits(shape, precision, thermal):
    """The rows per tile follow the lattice's size; every choice gives the bits
    of 32-row tiles of the same traversal."""
    lay = small(*shape)
    par = dict(lay.params, thermal=thermal)
    res = []
    for fixed in (False, True):
        sim = pf.Simulation([shape], par, precision)
        if fixed:
            sim.set_step_config(sim.step_config()[0], 32)
        sim.init_fields(0, lay.seeds, lay.R_s, lay.bubbles)
        sim.step(5)
        res.append(sim.get_state())
        assert sim.step_config()[1] == 32 if fixed else 1 <= sim.step_config()[1] <= 48
    assert np.array_equal(res[0], res[1])


@pytest.mark.parametrize("shape", [(1024, 768), (1028, 800), (900, 900), (132, 6000)])
@pytest.mark.parametrize("thermal,bc", [(0, None), (1, None), (1, (S, S, W, F)), (0, (P, P, W, W))])
def test_staged_rows_give_the_bits_of_the_plain_march(shape, thermal, bc):
    """Large FP32 lattices stage their rows by bulk copies where the width allows
    it: the bits of the y-march set by hand, with the temperature lattice and
    beside tiles at a side."""
    lay = small(*shape)
    par = dict(lay.params, thermal=thermal, g=1e-5)
    res = []
    for plain in (False, True):
        sim = pf.Simulation([shape], par, "fp32")
        if bc:
            sim.set_boundaries(0, *bc)
        if plain:
            sim.set_step_config(1, sim.step_config()[1])
        sim.init_fields(0, lay.seeds, lay.R_s, lay.bubbles)
        sim.step(6)
        res.append(sim.get_state())
    assert np.array_equal(res[0], res[1])


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


@pytest.mark.parametrize("shape", [(4, 4), (16, 16), (33, 31), (700, 600)])
def test_reductions_equal_the_sums_of_the_fields(shape):
    """pf_reduce against numpy FP64 sums of the fields it reads; a sum of n
    terms in another order differs by at most n eps of the sum of magnitudes."""
    lay = small(*shape)
    sim = pf.Simulation([shape], lay.params, "fp64")
    sim.init_fields(0, lay.seeds, lay.R_s, lay.bubbles)
    sim.step(2)
    for _ in range(2):     # the block counter is back at zero after a call
        d, f = sim.reduce(0), sim.fields()
        x, y = np.arange(shape[0])[None, :], np.arange(shape[1])[:, None]
        gas = 1.0 - f["phi"]
        want = dict(sum_phi=f["phi"], sum_C=f["C"], sum_hpsi=0.5 * (1 + f["psi"]), gas=gas,
                    gas_x=x * gas, gas_y=y * gas)
        for k, v in want.items():
            assert abs(d[k] - v.sum()) <= v.size * 2.3e-16 * np.abs(v).sum() + 1e-300, k
        assert d["max_v"] == np.sqrt(f["vx"] ** 2 + f["vy"] ** 2).max() or np.isclose(
            d["max_v"], np.sqrt(f["vx"] ** 2 + f["vy"] ** 2).max(), rtol=1e-15)
        assert d["nonfinite"] == 0


@pytest.mark.parametrize("doms,bc", [
    ([(4, 4)], None), ([(128, 128)], None), ([(512, 300)], None), ([(1024, 800)], None),
    ([(64, 48), (33, 45)], None), ([(32, 40)], (S, S, W, F)), ([(200, 120)], (P, P, W, W)),
    ([(96, 200), (160, 64)], (W, W, W, F)), ([(700, 500)], (P, P, W, W)),
])
@pytest.mark.parametrize("precision,thermal", [("fp32", 0), ("fp32", 1), ("fp64", 0), ("fp16", 0)])
def test_steps_launched_behind_one_another(doms, bc, precision, thermal):
    """The steps of a call start while the one before ends: the bits of as many
    calls of one step, also when the call is captured into a caller's graph."""
    torch = pytest.importorskip("torch")
    if bc and precision == "fp16":
        pytest.skip("sides take FP32 or FP64 storage")
    lay = small(*doms[0])
    par = dict(lay.params, thermal=thermal, g=1e-5)
    res = []
    side = torch.cuda.Stream()
    for mode in ("call", "single", "captured"):
        with torch.cuda.stream(side):
            sim = pf.Simulation(doms, par, precision)
            for k, (nx, ny) in enumerate(doms):
                if bc:
                    sim.set_boundaries(k, *bc)
                l = small(nx, ny)
                sim.init_fields(k, l.seeds, l.R_s, l.bubbles)
            if mode == "single":
                for _ in range(31):
                    sim.step(1)
            elif mode == "call":
                sim.step(31)
            else:
                sim.step(1)      # what the first step allocates
                sim.sync()
                g = torch.cuda.CUDAGraph()
                with torch.cuda.graph(g, stream=side):
                    sim.step(30)
                g.replay()
            res.append([sim.get_state(k) for k in range(len(doms))])
            sim.close()
    for r in res[1:]:
        assert all(np.array_equal(a, b) for a, b in zip(res[0], r))
