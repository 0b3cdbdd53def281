"""pf_adjoint_step that fails behind its forward sweep, from a state of
pf_set_state whose populations no collision made."""
import numpy as np
import pytest

from paper_2407_01651_gb300 import pf
from paper_2407_01651_gb300 import workload as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("n,every", [(4, 4), (5, 5), (5, 2), (6, 2), (2, 1), (1, 1)])
def test_failed_objective_leaves_the_state_after_the_steps(precision, n, every):
    """Without gas the centroid objective is refused after the forward sweep: the
    handle holds the state n steps on, as if it had stepped."""
    shape = (48, 40)
    par = dict(wl.BASE_PARAMS, g=1e-5)
    sims = []
    for _ in range(2):
        sim = pf.Simulation([shape], par, precision)
        sim.init_fields(0, [(20.0, 18.0, 0.3)], 6.0, [])
        # phi above 1 everywhere: no gas, at the start and after the steps
        f = sim.fields()
        sim.set_fields(0, np.full_like(f["phi"], 1.001), f["psi"], f["C"])
        st = sim.get_state()
        st[29:34] += 1e-4 * np.random.default_rng(1).standard_normal(st[29:34].shape)
        sim.set_state(0, st)
        sims.append(sim)
    a, b = sims
    with pytest.raises(pf.PFError) as e:
        a.adjoint_step(n, 1.0, 1.0, every)
    assert e.value.code == pf.PF_ERR_BAD_ARG and "gas" in str(e.value)
    b.step(n)
    assert np.array_equal(a.get_state(), b.get_state())
    a.step(1)
    b.step(1)
    assert np.array_equal(a.get_state(), b.get_state())
    a.set_state(0, st)      # and a raw state again
    b.set_state(0, st)
    a.step(3)
    b.step(3)
    assert np.array_equal(a.get_state(), b.get_state())
