"""FP32 arithmetic: LBM_KERNEL_AUTO leaves the states of the kernel that lbm_kernel_in_use names, bit for bit.  Where that
is LBM_KERNEL_FUSED, whether the size gets the staged kernel or the tile kernel; where it is LBM_KERNEL_TWO_PASS, with
interpolated and moving walls too.  (A 16-bit deviation is rounded to the storage type, so a last-bit difference of
the FP32 arithmetic before it would show as a whole ulp of that type.)"""
import numpy as np
import pytest

from paper_2604_13407_gb300 import inputs as I
from paper_2604_13407_gb300 import lbm
from tests import gpu_cases as GC
from tests.setups import cs_case, cs_params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,kw", [(p, kw) for p in (lbm.F16DEV, lbm.BF16DEV)
                                     for kw in (dict(per_node_ref=1), dict(per_node_ref=1, storage_rounding=0), dict(per_node_ref=0))] +
                         [(lbm.F32, {})])
@pytest.mark.parametrize("scheme", [0, 1])
@pytest.mark.parametrize("force_mode,tau_g", [(0, 1.0), (0, 0.7), (1, 1.0), (1, 0.7), (2, 1.0)])
@pytest.mark.parametrize("nx,ny", [(512, 512), (520, 517)])
def test_auto_is_the_fused_step(nx, ny, force_mode, tau_g, scheme, prec, kw):
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


@pytest.mark.parametrize("prec,kw", [(lbm.F32, {}), (lbm.F16DEV, dict(per_node_ref=1)), (lbm.BF16DEV, dict(per_node_ref=1)),
                                     (lbm.F16DEV, dict(per_node_ref=0, storage_rounding=0))])
@pytest.mark.parametrize("walls", ["interpolated", "moving", "both"])
@pytest.mark.parametrize("px,py", [(True, True), (False, False)])
def test_link_walls_are_the_two_pass_steps(px, py, walls, prec, kw):
    """An annulus (fractions of both halves, some of exactly 1/2) and scattered solid nodes with random fractions and
    velocities, some links with no second node."""
    T, rg, rl = cs_case()
    for nx, ny, scattered in ((101, 101, False), (67, 37, True)):
        if scattered:
            r = I.uniform(11, nx * ny).reshape(ny, nx)
            solid = (r < 0.15).astype(np.uint8)
            wall_u = 0.01 * np.stack([np.cos(9 * r), np.sin(9 * r)]) * (solid == 1)
            q = I.uniform(19, 8 * nx * ny, 0.05, 1.0).reshape(8, ny, nx)
            q[:, ::3] = 0.5
        else:
            solid, wall_u, q = I.annulus(nx, ny, 13.3, 46.6, u_wall_out=0.01)
        geometry = (solid, None if walls == "interpolated" else wall_u, None if walls == "moving" else q, None)
        op = cs_params(nx=nx, ny=ny, periodic_x=px, periodic_y=py, scheme=1, Fx=1e-6, tau_l=1.0, tau_g=0.8)
        u = I.uniform(7, 2 * nx * ny, -0.02, 0.02).reshape(2, ny, nx)
        state = {}
        for kernel in (lbm.KERNEL_AUTO, lbm.KERNEL_TWO_PASS):
            sim = lbm.Simulation(GC.gpu_params(op, prec, kernel, **kw))
            sim.set_geometry(*geometry)
            assert sim.kernel_in_use == lbm.KERNEL_TWO_PASS
            sim.init_fields(I.spinodal(nx, ny, 0.18, 0.3, 3), u[0], u[1])
            sim.step(5)
            state[kernel] = sim.get_state()[:, solid == 0]
            sim.close()
        assert np.all(np.isfinite(state[lbm.KERNEL_AUTO]))
        assert np.array_equal(state[lbm.KERNEL_AUTO], state[lbm.KERNEL_TWO_PASS]), (nx, ny)
