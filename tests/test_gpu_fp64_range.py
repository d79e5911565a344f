"""FP64 quotients over the whole range of magnitudes: the step's reciprocal-based divisions fall
back to the general division outside 2^+-450, and both sides of that limit are the oracle's bits."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2604_13407_gb300 import lbm
from tests import gpu_cases as GC
from tests.setups import cs_params, vdw_params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("params", [cs_params, lambda **k: vdw_params(1.895, 0.54, **k)], ids=["cs", "vdw"])
@pytest.mark.parametrize("scheme", [0, 1])
@pytest.mark.parametrize("log2", [0, -100, -440, -449, -452, -455, -500])
def test_fp64_step_is_the_oracles_at_any_magnitude(params, scheme, log2):
    """One step from populations of size 2^log2 (positive, irregular; one row at rest, so that exact
    zeros are divided too) equals the oracle bit for bit."""
    op = params(nx=33, ny=11, periodic_x=True, periodic_y=False, scheme=scheme, tau_l=0.9, tau_g=0.9)
    rng = np.random.default_rng(5)
    w = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)[:, None, None]
    A = 0.2 * w * (1.0 + 0.1 * rng.standard_normal((9, 11, 33)))
    A[:, 5:9] = 0.2 * w
    A = np.ldexp(A, log2)
    ref = O.OracleSim(op)
    ref.set_state(A)
    ref.step(1)
    want = ref.get_state()
    assert np.all(np.isfinite(want))
    gp = GC.gpu_params(op, lbm.F64)
    gp.rho_max = 0.3  # psi is real up to there in both equations of state
    sim = lbm.Simulation(gp)
    sim.set_state(A)
    sim.step(1)
    assert np.array_equal(sim.get_state(), want)
    sim.close()


@pytest.mark.parametrize("params", [cs_params, lambda **k: vdw_params(1.895, 0.54, **k)], ids=["cs", "vdw"])
@pytest.mark.parametrize("signs", [1.0, -1.0, 0.0])
def test_signs_of_zero_are_the_oracles(params, signs):
    """Populations at rest of +0, -0 or either sign beside the rest population (the sum of the forces and momenta is then
    an exact zero): the bits of the moments and of the state after one step, signs of zero included."""
    op = params(nx=33, ny=11, periodic_x=True, periodic_y=False, scheme=1, tau_l=0.9, tau_g=0.9)
    A = np.zeros((9, 11, 33))
    A[1:] *= signs if signs else np.where(np.random.default_rng(3).random((8, 11, 33)) < 0.5, -1.0, 1.0)
    A[0] = 0.2
    ref = O.OracleSim(op)
    ref.set_state(A)
    gp = GC.gpu_params(op, lbm.F64)
    gp.rho_max = 0.3
    sim = lbm.Simulation(gp)
    sim.set_state(A)
    bits = lambda a: np.ascontiguousarray(a).view(np.int64)  # noqa: E731
    for g, w in zip(sim.moments(), ref.moments()):
        assert np.array_equal(bits(g), bits(w))
    sim.step(1)
    ref.step(1)
    assert np.array_equal(bits(sim.get_state()), bits(ref.get_state()))
    sim.close()
