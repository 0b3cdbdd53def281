"""pf_get_step_config handed back to pf_set_step_config: the same kernels run."""
import pytest

from paper_2407_01651_gb300 import pf
from paper_2407_01651_gb300 import workload as wl
from tests.test_gpu_boundaries import F, S, W

pytestmark = pytest.mark.gpu


def handle(shape, precision, thermal, bc):
    sim = pf.Simulation([shape], dict(wl.BASE_PARAMS, thermal=thermal), precision)
    if bc:
        sim.set_boundaries(0, *bc)
    sim.init_fields(0, [(shape[0] / 2, shape[1] / 2, 0.4)], 5.0, [])
    return sim


def stages(sim):
    """Whether the steps stage their rows: with the copies dropped their waits give
    up after a second each and the call that waits says so."""
    sim.test_drop_staged_copies(True)
    try:
        sim.step(1)
        sim.sync()
        return False
    except pf.PFError as e:
        assert e.code == pf.PF_ERR_TIMEOUT
        return True
    finally:
        sim.test_drop_staged_copies(False)
        sim.init_fields(0, [(9.0, 9.0, 0.4)], 5.0, [])


@pytest.mark.parametrize("shape,precision,thermal,bc,staged", [
    ((1024, 768), "fp32", 1, None, True), ((1024, 768), "fp32", 1, (S, S, W, F), True),
    ((1022, 772), "fp32", 1, None, False), ((256, 96), "fp32", 1, None, False),
    ((256, 96), "fp64", 0, None, False),
])
def test_the_reported_configuration_keeps_the_kernels(shape, precision, thermal, bc, staged):
    sim = handle(shape, precision, thermal, bc)
    cfg = sim.step_config()
    assert cfg[0] == (2 if staged else 1)
    for _ in range(2):
        sim.set_step_config(*cfg)
        assert sim.step_config() == cfg
    assert stages(sim) == staged
    sim.set_step_config(1, cfg[1] + 1)        # a march set by hand is the plain one
    assert sim.step_config() == (1, cfg[1] + 1, 0)
    assert not stages(sim)
    if thermal or bc:                         # and the staged one is still not for setting
        with pytest.raises(pf.PFError) as e:
            sim.set_step_config(2, 16)
        assert e.value.code == pf.PF_ERR_BAD_ARG


def test_a_small_16_bit_march_stays_unstaged():
    """128^2 FP16 steps in 4.8 us unstaged and 12 us staged: the reported pair keeps
    the first (half way between them is the bound)."""
    torch = pytest.importorskip("torch")

    def us(sim):
        best = 1e9
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            sim.step(200)
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b) * 5)
        return best
    sim = handle((128, 128), "fp16", 0, None)
    by_size = us(sim)
    sim.set_step_config(*sim.step_config())
    assert us(sim) < 1.6 * by_size
