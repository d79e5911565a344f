"""16-bit storage on lattices where LBM_KERNEL_FUSED is granted: LBM_KERNEL_AUTO leaves the states that
LBM_KERNEL_FUSED leaves, bit for bit, whether its size gets the staged kernel or the tile kernel.  (A stored
deviation is rounded to the storage type, so a last-bit difference of the FP32 arithmetic before it would show
as a whole ulp of that type.)"""
import numpy as np
import pytest

from paper_2604_13407_gb300 import inputs as I
from paper_2604_13407_gb300 import lbm
from tests import gpu_cases as GC
from tests.setups import cs_case, cs_params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [lbm.F16DEV, lbm.BF16DEV])
@pytest.mark.parametrize("kw", [dict(per_node_ref=1), dict(per_node_ref=1, storage_rounding=0), dict(per_node_ref=0)],
                         ids=["node_ref", "nearest", "one_ref"])
@pytest.mark.parametrize("scheme", [0, 1])
@pytest.mark.parametrize("force_mode,tau_g", [(0, 1.0), (0, 0.7), (1, 1.0), (1, 0.7), (2, 1.0)])
@pytest.mark.parametrize("nx,ny", [(512, 512), (520, 517)])
def test_auto_is_the_fused_step(nx, ny, force_mode, tau_g, scheme, kw, prec):
    """Whole and ragged tiles; every force law, one and two relaxation times, both schemes: the options that
    either kernel fixes at compile time."""
    T, rg, rl = cs_case()
    op = cs_params(nx=nx, ny=ny, periodic_x=True, periodic_y=True, scheme=scheme, force_mode=force_mode, Fx=1e-6, Fy=-2e-6,
                   tau_l=1.0, tau_g=tau_g)
    u = I.uniform(7, 2 * nx * ny, -0.02, 0.02).reshape(2, ny, nx)
    field = I.uniform(13, 2 * nx * ny, -1e-5, 1e-5).reshape(2, ny, nx)
    rho = I.droplet(nx, ny, rl, rg, 90, 0.47 * nx, 0.55 * ny, periodic_x=True, periodic_y=True)
    state = {}
    for kernel in (lbm.KERNEL_AUTO, lbm.KERNEL_FUSED):
        sim = lbm.Simulation(GC.gpu_params(op, prec, kernel, **kw))
        if force_mode == 2:
            sim.set_geometry(None, None, None, field)
        assert sim.kernel_in_use == lbm.KERNEL_FUSED
        sim.init_fields(rho, u[0], u[1])
        sim.step(3)
        state[kernel] = sim.get_state()
        sim.close()
    assert np.all(np.isfinite(state[lbm.KERNEL_AUTO]))
    assert np.array_equal(state[lbm.KERNEL_AUTO], state[lbm.KERNEL_FUSED])
