"""Raw states of pf_set_state whose populations no collision made: the state is
stored as one population of each pair, and such a state has to survive until
its step all the same."""
import numpy as np
import pytest

import oracle
from paper_2407_01651_gb300 import pf
from paper_2407_01651_gb300 import workload as wl
from tests.test_gpu_boundaries import F, P, S, W

pytestmark = pytest.mark.gpu

FIELDS = ("phi", "psi", "C", "U", "p", "vx", "vy", "mu")
# groups of planes that a collision ties to each other
H, GPOST, SOL, E = slice(9, 18), slice(23, 28), slice(29, 34), slice(39, 44)


def layout(nx, ny):
    return wl.Layout(nx, ny, seeds=[(nx / 3, ny / 4, 0.4), (2 * nx / 3, ny / 2, 0.0)],
                     bubbles=[(nx / 4, 3 * ny / 4, min(nx, ny) / 8)])


def handle(shape, precision, thermal=0, bc=None, config=None):
    lay = layout(*shape)
    sim = pf.Simulation([shape], dict(lay.params, thermal=thermal, g=1e-5), precision)
    if bc:
        sim.set_boundaries(0, *bc)
    if config:
        sim.set_step_config(*config)
    sim.init_fields(0, lay.seeds, lay.R_s, lay.bubbles)
    return sim


def perturbed(sim, thermal, seed=3, size=1e-3):
    """A developed state with every tied population moved on its own."""
    sim.step(3)
    st = sim.get_state()
    rng = np.random.default_rng(seed)
    for g in (H, GPOST, SOL) + ((E,) if thermal else ()):
        st[g] += size * rng.standard_normal(st[g].shape)
    return st


def pull(st, i, q):
    """Population plane q + i of the D2Q9 direction i, streamed (periodic)."""
    c = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)][i]
    return np.roll(st[q + i], (c[1], c[0]), axis=(0, 1))


@pytest.mark.parametrize("shape", [(70, 52), (33, 9), (128, 64), (4, 4)])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_first_step_streams_every_population(shape, precision):
    """After one step phi and C are the sums of the streamed populations and
    psi that of the time-stretched ones, which a state projected onto pairs
    would miss by the size of the perturbation (1e-3)."""
    sim = handle(shape, precision)
    st = perturbed(sim, 0)
    sim.set_state(0, st)
    back = sim.get_state()
    eps = 2.3e-16 if precision == "fp64" else 1.2e-7
    assert np.abs(back - st).max() <= eps * np.abs(st).max()
    sim.step(1)
    f = sim.fields(0, ("phi", "psi", "C"))
    phi = sum(pull(st, i, 9) for i in range(9))
    C = sum(pull(st, i, 29) for i in range(5))
    roll = lambda a, i: pull(np.stack([a] * 9), i, 0)                       # noqa: E731
    psi = sum(st[18 + i] + roll(st[28], i) * (pull(st, i, 23) - st[18 + i]) for i in range(5))
    # sums of 9 terms of at most 1.3, each rounded to the storage type
    for got, want in ((f["phi"], phi), (f["C"], C), (f["psi"], psi)):
        assert np.abs(got - want).max() <= 32 * eps


@pytest.mark.parametrize("precision,thermal,bc,config", [
    ("fp64", 0, None, None), ("fp64", 1, None, None), ("fp64", 0, (S, S, W, F), None),
    ("fp64", 1, (F, W, P, P), None), ("fp32", 0, None, (0, 32, 8)), ("fp32", 0, None, (2, 16, 0)),
    ("fp32", 1, (S, S, W, F), None), ("fp16", 0, None, None), ("bf16", 0, None, (1, 8, 0)),
])
def test_general_and_paired_paths_agree_on_a_state_of_a_step(precision, thermal, bc, config):
    """A state that a step left behind, moved by less than the storage form
    resolves but more than the test of its pairs allows, takes the general
    path; it gives the fields of the paired path to rounding."""
    sim = handle((72, 52), precision, thermal, bc, config)
    sim.step(4)
    st = sim.get_state()
    res = []
    for general in (False, True):
        a = handle((72, 52), precision, thermal, bc, config)
        s = st.copy()
        if general:
            s[9, 3, 5] += 1e-5       # one rest population; taken out of its density's pair
            s[10, 3, 5] -= 1e-5
        a.set_state(0, s)
        a.step(3)
        res.append(a.fields(0, FIELDS))
    tol = {"fp64": 1e-4, "fp32": 1e-4, "fp16": 1e-3, "bf16": 2e-2}[precision]
    for k in ("phi", "psi", "C"):
        d = np.abs(res[0][k] - res[1][k])
        assert d.max() <= tol, k
        # beyond three steps of reach (two sites each) nothing moved but rounding
        far = np.ones_like(d, bool)
        far[:12, :14] = far[-6:, :14] = far[:12, -6:] = far[-6:, -6:] = False
        assert d[far].max() <= {"fp64": 1e-13, "fp32": 2e-6, "fp16": 1e-4, "bf16": 2e-3}[precision], k


def test_a_mixed_ensemble_and_every_launch_mode():
    """One domain from a raw state beside one without, through every launch mode
    and pf_get_state, pf_reduce_thermal and set_temperature around it."""
    lays = [wl.random_layout(48, 40, 1, 1, rng_seed=k, R_max=7) for k in (1, 2)]
    ref = None
    for mode in ((0, 0, 0), (1, 0, 0), (0, 1, 0), (0, 2, 0), (0, 0, 2)):
        sim = pf.Simulation([(48, 40), (48, 40)], lays[0].params, "fp64")
        for d, lay in enumerate(lays):
            sim.init_fields(d, lay.seeds, lay.R_s, lay.bubbles)
        sim.set_launch(*mode)
        sim.step(2)
        st = sim.get_state(1)
        st[9:18] += 1e-4 * np.random.default_rng(1).standard_normal(st[9:18].shape)
        sim.set_state(1, st)
        sim.step(5)
        out = np.stack([sim.get_state(d) for d in (0, 1)])
        assert np.isfinite(out).all()
        if ref is None:
            ref = out
        assert np.array_equal(out, ref), mode


def test_thermal_totals_and_temperature_of_a_raw_state():
    sim = handle((40, 36), "fp64", thermal=1)
    st = sim.get_state()
    st[E] += 1e-3 * np.random.default_rng(2).standard_normal(st[E].shape)
    sim.set_state(0, st)
    assert np.isclose(sim.reduce_thermal(0)["sum_e"], st[E].sum(), rtol=1e-12)
    sim.set_temperature(0, np.full((36, 40), -0.3))
    a = handle((40, 36), "fp64", thermal=1)
    a.set_temperature(0, np.full((36, 40), -0.3))
    for s in (sim, a):
        s.step(2)
    fa, fb = sim.fields(), a.fields()
    for k in ("phi", "psi", "C", "theta"):
        assert np.abs(fa[k] - fb[k]).max() <= 1e-12, k


def test_adjoint_from_a_raw_state():
    """J and its gradient from a raw state: central differences in FP64, and the
    same for every checkpoint interval."""
    sim = handle((48, 40), "fp64")
    st = perturbed(sim, 0, size=1e-4)
    lay = layout(48, 40)

    def run(par, K):
        s = pf.Simulation([(48, 40)], par, "fp64")
        s.init_fields(0, lay.seeds, lay.R_s, lay.bubbles)
        s.step(1)                      # not fresh: the state does not depend on Omega
        s.set_state(0, st)
        return s.adjoint_step(12, 1.0, 1.0, K)
    par = dict(lay.params, g=1e-5)
    J, g = run(par, 12)
    for K in (1, 5):
        J2, g2 = run(par, K)
        assert J2 == J and np.array_equal(g, g2)
    for i, n in enumerate(("eps_s", "Omega", "sigma")):
        h = 1e-5 * par[n]
        fd = (run(dict(par, **{n: par[n] + h}), 12)[0] - run(dict(par, **{n: par[n] - h}), 12)[0]) / (2 * h)
        # J is of order 1 and rounded to 1e-16; its third derivatives are of order 1e3 or less
        assert abs(g[i] - fd) <= 1e-15 / h + 1e3 * h * h + 1e-9 * abs(fd), (n, g[i], fd)


def test_paired_state_of_the_oracle():
    """The oracle's state (dense moment matrices) continues as the oracle does,
    whichever path its rounding takes."""
    lay = wl.random_layout(70, 52, 2, 2, rng_seed=21, R_max=10)
    o = oracle.Oracle(70, 52, lay.params)
    o.init_spec(lay.seeds, lay.R_s, lay.bubbles)
    o.step(30)
    sim = pf.Simulation([(70, 52)], lay.params, "fp64")
    sim.init_fields(0, lay.seeds, lay.R_s, lay.bubbles)
    sim.set_state(0, o.state())
    o.step(3)
    sim.step(3)
    fo, fg = o.fields(), sim.fields()
    for k in ("phi", "psi", "C", "vx", "vy"):
        assert np.abs(fo[k] - fg[k]).max() <= 1e-11 * np.abs(fo[k]).max(), k
