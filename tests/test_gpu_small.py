"""Many steps of a small lattice in one launch (LBM_KERNEL_AUTO) against one launch per step and the
two-pass kernels, bit for bit: strips of one row, fewer rows than CTAs, uneven strips, the largest
lattices taken and the first ones not, one-node lattices, odd and even step counts."""
import numpy as np
import pytest

from paper_2604_13407_gb300 import inputs as I
from paper_2604_13407_gb300 import lbm
from tests import gpu_cases as GC
from tests.setups import cs_case, cs_params

pytestmark = pytest.mark.gpu

SIZES = [(1, 1), (3, 2), (1, 40), (33, 5), (37, 23), (4, 181), (700, 1), (1024, 15), (61, 33), (128, 128), (129, 127), (300, 17)]
PRECS = {"f64": (lbm.F64, {}), "f32": (lbm.F32, {}), "f16": (lbm.F16DEV, {"per_node_ref": 1}),
         "f16_nearest": (lbm.F16DEV, {"per_node_ref": 0, "storage_rounding": 0}), "bf16": (lbm.BF16DEV, {"per_node_ref": 1})}


def _run(op, prec, kernel, steps, geometry=None, wall_rho=None):
    pid, kw = PRECS[prec]
    nx, ny = op.nx, op.ny
    sim = lbm.Simulation(GC.gpu_params(op, pid, kernel, **kw))
    if geometry is not None:
        sim.set_geometry(*geometry)
    if wall_rho is not None:
        sim.set_wall_density(wall_rho)
    u = I.uniform(7, 2 * nx * ny, -0.02, 0.02).reshape(2, ny, nx)
    sim.init_fields(I.spinodal(nx, ny, 0.18, 0.3, 3), u[0], u[1])
    for n in steps:
        sim.step(n)
    A = sim.get_state()
    assert sim.step_count == sum(steps)
    sim.close()
    return A


@pytest.mark.parametrize("prec", sorted(PRECS))
@pytest.mark.parametrize("nx,ny", SIZES)
def test_one_launch_is_step_by_step(nx, ny, prec):
    for k, (px, py) in enumerate(((True, True), (True, False), (False, True), (False, False))):
        op = cs_params(nx=nx, ny=ny, periodic_x=px, periodic_y=py, scheme=k % 2, force_mode=k // 2, Fx=1e-5, Fy=-2e-5,
                       tau_l=1.0, tau_g=0.8 if k % 3 else 1.0)
        a = _run(op, prec, lbm.KERNEL_AUTO, [7, 6])
        assert np.all(np.isfinite(a))
        assert np.array_equal(a, _run(op, prec, lbm.KERNEL_AUTO, [1] * 13)), (px, py)
        assert np.array_equal(a, _run(op, prec, lbm.KERNEL_TWO_PASS, [13])), (px, py)


@pytest.mark.parametrize("prec", ["f32", "f16", "f16_nearest", "bf16"])
@pytest.mark.parametrize("nx,ny", [(32, 64), (43, 48), (128, 64), (171, 48)])
def test_edges_of_one_and_two_nodes_a_thread(nx, ny, prec):
    """Strips of 128, 129, 512 and 513 nodes: the last of the small blocks, the first of the large ones, the
    last with one node a thread and the first (odd) with two."""
    for px, force_mode in ((True, 0), (False, 1)):
        op = cs_params(nx=nx, ny=ny, periodic_x=px, periodic_y=True, scheme=1, force_mode=force_mode, Fx=1e-5, Fy=-2e-5, tau_l=1.0, tau_g=0.8)
        a = _run(op, prec, lbm.KERNEL_AUTO, [5, 4])
        assert np.all(np.isfinite(a)) and np.array_equal(a, _run(op, prec, lbm.KERNEL_TWO_PASS, [9])), (px, force_mode)


@pytest.mark.parametrize("prec", sorted(PRECS))
@pytest.mark.parametrize("nx,ny", [(9, 9), (67, 37), (40, 18)])
def test_solid_nodes_force_field_and_wall_densities(nx, ny, prec):
    T, rg, rl = cs_case()
    r = I.uniform(11, nx * ny).reshape(ny, nx)
    solid = (r < 0.15).astype(np.uint8)
    solid[1:4, 1:4] = 1
    solid[2, 2] = 0
    field = I.uniform(13, 2 * nx * ny, -1e-5, 1e-5).reshape(2, ny, nx)
    wall_rho = I.uniform(17, nx * ny, rg, rl).reshape(ny, nx)
    for px, py in ((True, True), (False, True), (False, False)):
        op = cs_params(nx=nx, ny=ny, periodic_x=px, periodic_y=py, scheme=1, force_mode=2, tau_l=1.0, tau_g=1.0)
        g = (solid, None, None, field)
        a = _run(op, prec, lbm.KERNEL_AUTO, [5], g, wall_rho)
        assert np.all(np.isfinite(a[:, solid == 0]))
        assert np.array_equal(a, _run(op, prec, lbm.KERNEL_AUTO, [1] * 5, g, wall_rho)), (px, py)
        assert np.array_equal(a, _run(op, prec, lbm.KERNEL_TWO_PASS, [5], g, wall_rho)), (px, py)


def test_more_steps_than_a_launch_takes():
    op = cs_params(nx=12, ny=9, periodic_x=True, periodic_y=False, Fx=1e-6)
    for prec in ("f32", "f16"):
        assert np.array_equal(_run(op, prec, lbm.KERNEL_AUTO, [4099]), _run(op, prec, lbm.KERNEL_TWO_PASS, [4099]))
