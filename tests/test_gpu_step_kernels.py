"""The kernels that the automatic choice takes on the GPU: where the many-step kernel of small lattices runs and where it
does not, and the tile kernel, one step a call so that it takes every one of them, against the two-pass kernels at the
sizes where a tile can go wrong."""
import numpy as np
import pytest

from paper_2604_13407_gb300 import inputs as I
from paper_2604_13407_gb300 import lbm
from tests import gpu_cases as GC
from tests.setups import cs_case, cs_params
from tests.test_gpu_tile import PRECS, SIZES

pytestmark = pytest.mark.gpu


def _one_by_one(op, prec, kernel, steps, geometry=None, wall_rho=None):
    pid, kw = PRECS[prec]
    nx, ny = op.nx, op.ny
    sim = lbm.Simulation(GC.gpu_params(op, pid, kernel, **kw))
    if geometry is not None:
        sim.set_geometry(*geometry)
    if wall_rho is not None:
        sim.set_wall_density(wall_rho)
    assert sim.step_launches(1) == ((1, "tile") if kernel == lbm.KERNEL_AUTO else (2, "two_pass"))
    u = I.uniform(7, 2 * nx * ny, -0.02, 0.02).reshape(2, ny, nx)
    sim.init_fields(I.spinodal(nx, ny, 0.18, 0.3, 3), u[0], u[1])
    for _ in range(steps):
        sim.step(1)
    A = sim.get_state()
    sim.close()
    return A


@pytest.mark.parametrize("prec", sorted(PRECS))
@pytest.mark.parametrize("nx,ny", SIZES)
def test_tile_step_is_the_two_pass_step(nx, ny, prec):
    """Bit for bit, with every combination of periodic directions, both schemes, constant and buoyant force, one and
    two relaxation times in turn."""
    for k, (px, py) in enumerate(((True, True), (True, False), (False, True), (False, False))):
        op = cs_params(nx=nx, ny=ny, periodic_x=px, periodic_y=py, scheme=k % 2, force_mode=k // 2, Fx=1e-5, Fy=-2e-5,
                       tau_l=1.0, tau_g=0.8 if k % 3 else 1.0)
        a, b = (_one_by_one(op, prec, kern, 7) for kern in (lbm.KERNEL_TWO_PASS, lbm.KERNEL_AUTO))
        assert np.all(np.isfinite(a)) and np.array_equal(a, b), (px, py)


@pytest.mark.parametrize("prec", sorted(PRECS))
@pytest.mark.parametrize("nx,ny", [(9, 9), (33, 16), (67, 37), (131, 40)])
def test_tile_step_with_solid_nodes(nx, ny, prec):
    """Half-way links on scattered solid nodes (a node walled in on all sides among them), a force field and wall
    densities: bit for bit."""
    T, rg, rl = cs_case()
    r = I.uniform(11, nx * ny).reshape(ny, nx)
    solid = (r < 0.15).astype(np.uint8)
    solid[1:4, 1:4] = 1
    solid[2, 2] = 0
    field = I.uniform(13, 2 * nx * ny, -1e-5, 1e-5).reshape(2, ny, nx)
    wall_rho = I.uniform(17, nx * ny, rg, rl).reshape(ny, nx)
    for px, py in ((True, True), (False, True), (False, False)):
        op = cs_params(nx=nx, ny=ny, periodic_x=px, periodic_y=py, scheme=1, force_mode=2, tau_l=1.0, tau_g=1.0)
        a, b = (_one_by_one(op, prec, kern, 4, (solid, None, None, field), wall_rho)[:, solid == 0]
                for kern in (lbm.KERNEL_TWO_PASS, lbm.KERNEL_AUTO))
        assert np.all(np.isfinite(a)) and np.array_equal(a, b), (px, py)


@pytest.mark.parametrize("nx,ny,fp32,fp64", [
    # strips of at most 1024 nodes (FP64: 128) over at most 16 CTAs, at most 16384 (2048) nodes
    (1, 1, True, True), (3, 2, True, True), (1, 40, True, True), (33, 5, True, True), (37, 23, True, True), (4, 181, True, True),
    (4, 512, True, True), (128, 16, True, True), (129, 16, True, False), (4, 513, True, False), (61, 33, True, False),
    (700, 1, True, False), (1024, 16, True, False), (1024, 15, False, False), (128, 128, True, False), (129, 127, False, False),
    (128, 129, False, False), (300, 17, True, False)])
def test_where_the_small_lattice_kernel_runs(nx, ny, fp32, fp64):
    for prec, want in ((lbm.F32, fp32), (lbm.F16DEV, fp32), (lbm.BF16DEV, fp32), (lbm.F64, fp64)):
        sim = lbm.Simulation(lbm.default_params(nx=nx, ny=ny, precision=prec, per_node_ref=1))
        assert sim.step_launches(7) == ((1, "small") if want else (7, "tile")), prec
        assert sim.step_launches(3) == (3, "tile")
        sim.set_geometry(None, None, np.full((8, ny, nx), 0.5))
        assert sim.step_launches(7) == (7, "tile")
        sim.close()
