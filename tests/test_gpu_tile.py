"""The one-pass step on tiles (LBM_KERNEL_AUTO below the staged kernel's sizes) against the two-pass
kernels, at the sizes where a tile can go wrong: lattices narrower and shorter than a tile, one node
more and less than a whole number of tiles, rings that wrap onto the tile itself, one-node lattices."""
import numpy as np
import pytest

from paper_2604_13407_gb300 import inputs as I
from paper_2604_13407_gb300 import lbm
from tests import gpu_cases as GC
from tests.setups import cs_case, cs_params

pytestmark = pytest.mark.gpu

SIZES = [(1, 1), (1, 5), (2, 3), (5, 1), (31, 8), (32, 9), (33, 16), (34, 17), (36, 21), (66, 20), (97, 35), (130, 41), (4, 130), (300, 7)]
PRECS = {"f64": (lbm.F64, {}), "f32": (lbm.F32, {}), "f16": (lbm.F16DEV, {"per_node_ref": 1}),
         "f16_nearest": (lbm.F16DEV, {"per_node_ref": 0, "storage_rounding": 0}), "bf16": (lbm.BF16DEV, {"per_node_ref": 1})}


def _state(case_params, nx, ny, prec, kw, kernel, geometry=(None, None, None, None), wall_rho=None, steps=7):
    T, rg, rl = cs_case()
    sim = lbm.Simulation(GC.gpu_params(case_params, prec, kernel, **kw))
    if any(g is not None for g in geometry):
        sim.set_geometry(*geometry)
    if wall_rho is not None:
        sim.set_wall_density(wall_rho)
    u = I.uniform(7, 2 * nx * ny, -0.02, 0.02).reshape(2, ny, nx)
    sim.init_fields(I.spinodal(nx, ny, 0.18, 0.3, 3), u[0], u[1])
    sim.step(steps)
    A = sim.get_state()
    sim.close()
    return A


@pytest.mark.parametrize("prec", sorted(PRECS))
@pytest.mark.parametrize("nx,ny", SIZES)
def test_tile_step_is_the_two_pass_step(nx, ny, prec):
    """Bit for bit, with every combination of periodic directions, both schemes, constant and
    buoyant force, one and two relaxation times in turn."""
    pid, kw = PRECS[prec]
    for k, (px, py) in enumerate(((True, True), (True, False), (False, True), (False, False))):
        op = cs_params(nx=nx, ny=ny, periodic_x=px, periodic_y=py, scheme=k % 2, force_mode=k // 2, Fx=1e-5, Fy=-2e-5,
                       tau_l=1.0, tau_g=0.8 if k % 3 else 1.0)
        a, b = (_state(op, nx, ny, pid, kw, kern) for kern in (lbm.KERNEL_TWO_PASS, lbm.KERNEL_AUTO))
        assert np.all(np.isfinite(a)) and np.array_equal(a, b), (px, py)


@pytest.mark.parametrize("prec", sorted(PRECS))
@pytest.mark.parametrize("nx,ny", [(9, 9), (33, 16), (67, 37), (131, 40)])
def test_tile_step_with_solid_nodes(nx, ny, prec):
    """Half-way links on scattered solid nodes (a node walled in on all sides among them), a force
    field and wall densities: bit for bit.  Interpolated and moving walls: FP64 bit for bit; FP32
    arithmetic to rounding, since the tile kernel's link coefficients are rounded once from FP64 where
    the two-pass kernels form them from rounded factors: a few ulps (2^-23) of a population per step."""
    pid, kw = PRECS[prec]
    T, rg, rl = cs_case()
    r = I.uniform(11, nx * ny).reshape(ny, nx)
    solid = (r < 0.15).astype(np.uint8)
    solid[1:4, 1:4] = 1
    solid[2, 2] = 0
    field = I.uniform(13, 2 * nx * ny, -1e-5, 1e-5).reshape(2, ny, nx)
    wall_rho = I.uniform(17, nx * ny, rg, rl).reshape(ny, nx)
    wall_u = 0.01 * np.stack([np.cos(9 * r), np.sin(9 * r)]) * (solid == 1)
    q = I.uniform(19, 8 * nx * ny, 0.05, 1.0).reshape(8, ny, nx)
    q[:, ::3] = 0.5
    fluid = solid == 0
    for px, py in ((True, True), (False, True), (False, False)):
        op = cs_params(nx=nx, ny=ny, periodic_x=px, periodic_y=py, scheme=1, force_mode=2, tau_l=1.0, tau_g=1.0)
        for geometry, exact in (((solid, None, None, field), True), ((solid, wall_u, q, field), pid == lbm.F64),
                                ((None, None, q, field), pid == lbm.F64)):
            rho = wall_rho if geometry[0] is not None else None
            a, b = (_state(op, nx, ny, pid, kw, kern, geometry, rho, steps=4) for kern in (lbm.KERNEL_TWO_PASS, lbm.KERNEL_AUTO))
            if geometry[0] is not None:
                a, b = a[:, fluid], b[:, fluid]
            assert np.all(np.isfinite(a))
            if exact:
                assert np.array_equal(a, b), (px, py)
            else:
                # 16-bit storage: a last-bit difference before rounding can move a stored deviation by one ulp of its type
                ulp = 2.0 ** -23 if pid == lbm.F32 else 2.0 ** -10 if pid == lbm.F16DEV else 2.0 ** -7
                assert np.abs(a - b).max() <= 4 * 8 * ulp * np.abs(a).max(), (px, py)


@pytest.mark.parametrize("prec", ["f32", "f16", "f16_nearest", "bf16"])
@pytest.mark.parametrize("force_mode", [0, 1, 2])
@pytest.mark.parametrize("tau_g", [1.0, 0.7])
def test_every_compiled_combination_of_options(prec, force_mode, tau_g):
    """Force law, relaxation and reference plane are fixed at compile time in the tile kernel: bit for bit
    the two-pass step in each, with and without solid nodes (three steps: none in the kernel of small
    lattices), on a lattice with tiles at the edges and inside."""
    pid, kw = PRECS[prec]
    nx, ny = 131, 41
    solid = (I.uniform(11, nx * ny).reshape(ny, nx) < 0.1).astype(np.uint8)
    field = I.uniform(13, 2 * nx * ny, -1e-5, 1e-5).reshape(2, ny, nx) if force_mode == 2 else None
    op = cs_params(nx=nx, ny=ny, periodic_x=True, periodic_y=False, scheme=1, force_mode=force_mode, Fx=1e-5, Fy=-2e-5, tau_l=1.0, tau_g=tau_g)
    for mask in (None, solid):
        a, b = (_state(op, nx, ny, pid, kw, kern, (mask, None, None, field), steps=3) for kern in (lbm.KERNEL_TWO_PASS, lbm.KERNEL_AUTO))
        if mask is not None:
            a, b = a[:, mask == 0], b[:, mask == 0]
        assert np.all(np.isfinite(a)) and np.array_equal(a, b)


@pytest.mark.parametrize("masked", [False, True])
@pytest.mark.parametrize("prec", ["f64", "f32", "f16", "bf16"])
@pytest.mark.parametrize("nx,ny", [(1, 5), (33, 17), (70, 37), (131, 40)])
def test_readings_of_a_state(nx, ny, prec, masked):
    """Moments and diagnostics of a stored state against the oracle's of the same (decoded) state: FP64 to
    1e-12 of the mass (sums in another order) and bit for bit per node; FP32 arithmetic per node to
    1e-6, some ten roundings (2^-24) of terms no larger than the density, and its sums to 1e-6 of the
    mass."""
    from oracle import oracle as O
    pid, kw = PRECS[prec]
    T, rg, rl = cs_case()
    solid = (I.uniform(11, nx * ny).reshape(ny, nx) < 0.12).astype(np.uint8) if masked else None
    for px, py in ((True, True), (True, False), (False, False)):
        op = cs_params(nx=nx, ny=ny, periodic_x=px, periodic_y=py, scheme=1, force_mode=1, Fx=1e-5, Fy=-2e-5)
        sim = lbm.Simulation(GC.gpu_params(op, pid, **kw))
        if masked:
            sim.set_geometry(solid)
        u = I.uniform(7, 2 * nx * ny, -0.02, 0.02).reshape(2, ny, nx)
        sim.init_fields(I.spinodal(nx, ny, 0.18, 0.3, 3), u[0], u[1])
        sim.step(3)
        ref = O.OracleSim(op, solid=solid)
        ref.set_state(sim.get_state())
        got, want = sim.moments(), ref.moments()
        a, b = sim.diagnostics(), ref.diagnostics()
        sim.close()
        for g, w in zip(got, want):
            assert np.array_equal(g, w) if prec == "f64" else np.abs(g - w).max() <= 1e-6
        mass = b[0]
        tol = 1e-12 if prec == "f64" else 1e-6
        assert np.abs(a[:9] - b[:9]).max() <= tol * mass, (a, b)
        assert abs(a[9] - b[9]) <= (1e-15 if prec == "f64" else 1e-6)
