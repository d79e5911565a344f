"""The transposed step on tiles: lattices with tiles that touch no edge, ragged ones, solid nodes; odd and
even step counts (which of the context's buffers the forward sweep ends in) and checkpoint intervals."""
import numpy as np
import pytest

from oracle import adjoint_ref as AR
from paper_2604_13407_gb300 import inputs as I
from paper_2604_13407_gb300 import lbm
from tests import gpu_cases as GC
from tests.setups import cs_case, cs_params

pytestmark = pytest.mark.gpu

PRECS = {"f64": lbm.F64, "f32": lbm.F32, "f16": lbm.F16DEV}


def _sim(nx, ny, prec, px, py, solid, kernel=lbm.KERNEL_AUTO, tau_g=0.8):
    T, rg, rl = cs_case()
    op = cs_params(nx=nx, ny=ny, periodic_x=px, periodic_y=py, scheme=1, force_mode=1, Fx=1e-6, Fy=-2e-6, tau_l=1.0, tau_g=tau_g)
    s = lbm.Simulation(GC.gpu_params(op, prec, kernel, per_node_ref=1))
    if solid is not None:
        s.set_geometry(solid)
    u = 0.02 * np.stack([np.ones((ny, nx)), np.ones((ny, nx))])
    s.init_fields(I.droplet(nx, ny, rl, rg, 0.25 * min(nx, ny), 0.47 * nx, 0.55 * ny, periodic_x=px, periodic_y=py), u[0], u[1])
    return s, op


@pytest.mark.parametrize("masked", [False, True])
@pytest.mark.parametrize("walls", [(False, True), (True, False), (True, True)])
@pytest.mark.parametrize("nx,ny", [(3, 2), (33, 17), (70, 37), (101, 52)])
def test_matches_the_reference_adjoint(nx, ny, walls, masked):
    """Against FP64 autograd through the FP64 reference step, with the tolerances of test_gpu_adjoint.py:
    FP64 over three steps to 1e-9; FP32 arithmetic over one step from the stored state (which lambda_0 and
    the gradient then depend on alone) to 1e-5.  One relaxation time: with two, the derivative of nu(rho)
    jumps at rho_g, where the last bit of the gas density would decide."""
    solid = (I.uniform(5, nx * ny).reshape(ny, nx) < 0.1).astype(np.uint8) if masked else None
    fluid = np.ones((ny, nx), bool) if solid is None else solid == 0
    for prec in sorted(PRECS):
        n, tol = (3, 1e-9) if prec == "f64" else (1, 1e-5)
        for obj, oid in (("wall_force_y", lbm.OBJ_WALL_FORCE_Y), ("mean_jx", lbm.OBJ_MEAN_JX)):
            s, op = _sim(nx, ny, PRECS[prec], *walls, solid, tau_g=1.0)
            A0 = s.get_state()
            J, g, lam = AR.objective_and_grad(op, A0, n, obj, solid)
            J2, g2, lam2 = s.adjoint(n, 2, oid, want_lambda0=True)
            s.close()
            k = [0, 1, 3]
            if prec == "f64":
                assert abs(J - J2) <= 1e-11 * abs(J) + 1e-15
            if prec == "f64" or obj == "mean_jx":  # (the wall force's gradient cancels between opposite walls)
                assert np.abs(g[k] - g2[k]).max() <= tol * np.abs(g[k]).max() + 1e-15, (prec, obj, g, g2)
            assert np.abs(lam - lam2)[:, fluid].max() <= tol * np.abs(lam).max() + 1e-15, (prec, obj)


@pytest.mark.parametrize("prec", sorted(PRECS))
@pytest.mark.parametrize("kernel", [lbm.KERNEL_AUTO, lbm.KERNEL_TWO_PASS])
@pytest.mark.parametrize("n", [1, 6, 7])
def test_state_and_checkpoints(prec, kernel, n):
    """Any checkpoint interval gives the same lambda_0 bit for bit and the same sums to rounding; the state
    afterwards, solid nodes included, and what follows it are what n steps give."""
    solid = (I.uniform(5, 70 * 37).reshape(37, 70) < 0.05).astype(np.uint8)
    want = None
    for K in (1, 2, 3, n, 50):
        a, b = (_sim(70, 37, PRECS[prec], True, False, solid, kernel)[0] for _ in range(2))
        J, g, lam = a.adjoint(n, K, lbm.OBJ_MEAN_JX, want_lambda0=True)
        b.step(n)
        assert a.step_count == n and np.array_equal(a.get_state(), b.get_state())
        a.step(3), b.step(3)
        assert np.array_equal(a.get_state(), b.get_state())
        if want is None:
            want = (J, g, lam)
        assert np.array_equal(lam, want[2])
        assert abs(J - want[0]) <= 1e-12 * abs(want[0]) and np.abs(g - want[1]).max() <= 1e-12 * np.abs(want[1]).max()
        a.close(), b.close()
