"""The transposed step from 2^19 nodes on (an instantiation of its own: short tiles, five blocks an SM): against FP64
autograd through the FP64 reference step, and against the smaller lattices' instantiation."""
import numpy as np
import pytest

from oracle import adjoint_ref as AR
from paper_2604_13407_gb300 import inputs as I
from paper_2604_13407_gb300 import lbm
from tests import gpu_cases as GC
from tests.setups import cs_case, cs_params

pytestmark = pytest.mark.gpu

PRECS = {"f32": lbm.F32, "f16": lbm.F16DEV, "bf16": lbm.BF16DEV}


def _sim(nx, ny, prec, px, py, solid=None, copies=1, rho=None, **kw):
    """A droplet in a drifting gas; `copies` by `copies` of it on a lattice that much larger."""
    T, rg, rl = cs_case()
    op = cs_params(nx=nx * copies, ny=ny * copies, periodic_x=px, periodic_y=py, scheme=1, force_mode=1, Fx=1e-6, Fy=-2e-6, tau_l=1.0, tau_g=1.0)
    s = lbm.Simulation(GC.gpu_params(op, prec, **dict(dict(per_node_ref=1), **kw)))
    if solid is not None:
        s.set_geometry(np.tile(solid, (copies, copies)))
    rho = I.droplet(nx, ny, rl, rg, 0.25 * min(nx, ny), 0.47 * nx, 0.55 * ny, periodic_x=px, periodic_y=py) if rho is None else rho
    u = I.uniform(7, 2 * nx * ny, 0.01, 0.03).reshape(2, ny, nx)
    again = lambda a: np.tile(a, (copies, copies))  # noqa: E731
    s.init_fields(again(rho), again(u[0]), again(u[1]))
    return s, op


@pytest.mark.parametrize("masked", [False, True])
@pytest.mark.parametrize("prec", sorted(PRECS))
@pytest.mark.parametrize("nx,ny,px,py", [(1024, 512, True, False), (725, 727, False, True)])
def test_matches_the_reference_adjoint(nx, ny, px, py, prec, masked):
    """Whole and ragged tiles, walls at the edges and at scattered solid nodes.  FP32 over two steps, so that a
    transposed step takes what the one after it left; 16-bit storage over one, whose result depends on the stored
    state alone, and with the solid nodes, whose gas-like walls inside the liquid leave the equation of state's
    range in the second step (in 64 bits too).  Tolerances as in test_gpu_adjoint.py for FP32 arithmetic: 1e-5 of the largest magnitude
    (the wall force's gradient cancels between opposite walls and is left to lambda_0)."""
    solid = (I.uniform(5, nx * ny).reshape(ny, nx) < 0.1).astype(np.uint8) if masked else None
    fluid = np.ones((ny, nx), bool) if solid is None else solid == 0
    n = 2 if prec == "f32" and not masked else 1
    s, op = _sim(nx, ny, PRECS[prec], px, py, solid)
    A0 = s.get_state()
    snap = s.save_state()
    for obj, oid in (("wall_force_y", lbm.OBJ_WALL_FORCE_Y), ("mean_jx", lbm.OBJ_MEAN_JX)):
        J, g, lam = AR.objective_and_grad(op, A0, n, obj, solid)
        s.load_state(snap)
        J2, g2, lam2 = s.adjoint(n, 2, oid, want_lambda0=True)
        k = [0, 1, 3]
        if obj == "mean_jx":
            assert np.abs(g[k] - g2[k]).max() <= 1e-5 * np.abs(g[k]).max(), (g, g2)
        assert np.abs(lam - lam2)[:, fluid].max() <= 1e-5 * np.abs(lam).max(), obj
    s.close()


@pytest.mark.parametrize("banded", [False, True])
@pytest.mark.parametrize("prec", sorted(PRECS))
def test_four_copies_of_a_small_lattice(prec, banded):
    """512^2 periodic nodes and four copies of them on 1024^2 (each side of the threshold), without walls and between
    solid bands, rounded to nearest so that every copy takes the same trajectory: the mean objective's lambda_0 is a
    quarter of the small lattice's in each copy and its gradient the same, to the FP32 arithmetic of seven steps (1e-5,
    as above)."""
    T, rg, rl = cs_case()
    n = 512
    solid, rho = (I.oblique_band_walls(n), I.oblique_slab(n, rl, rg, n // 2)) if banded else (None, None)
    got = {}
    for copies in (1, 2):
        s, _ = _sim(n, n, PRECS[prec], True, True, solid, copies, rho, storage_rounding=0)
        got[copies] = s.adjoint(7, 3, lbm.OBJ_MEAN_JX, want_lambda0=True)
        s.close()
    (J1, g1, l1), (J2, g2, l2) = got[1], got[2]
    k = [0, 1, 3]
    assert abs(J1 - J2) <= 1e-5 * abs(J1)
    assert np.abs(g1[k] - g2[k]).max() <= 1e-5 * np.abs(g1[k]).max(), (g1, g2)
    assert np.abs(4 * l2 - np.tile(l1, (1, 2, 2))).max() <= 1e-5 * np.abs(l1).max()
