"""Which kernel steps a context, on a fake device: both sides of every threshold of the automatic choice, and
lbm_step_launches against what lbm_step then launches."""
import ctypes

import numpy as np
import pytest

from paper_2604_13407_gb300 import lbm
from tests import fake


@pytest.fixture(scope="module")
def fakelib(tmp_path_factory):
    saved, lbm._lib = lbm._lib, None
    try:
        yield fake.load(tmp_path_factory.mktemp("fake"))
    finally:
        lbm._lib = saved


ANY = np.zeros(8)


def _sim(fakelib, nx, ny, prec, kernel=lbm.KERNEL_AUTO, small=0, geom=None, **kw):
    fakelib.fake_reset(small)
    sim = lbm.Simulation(lbm.default_params(**dict(dict(nx=nx, ny=ny, periodic_x=1, periodic_y=1, precision=prec, kernel=kernel,
                                                        per_node_ref=1), **kw)))
    solid = np.zeros((ny, nx), np.uint8)
    solid[:, :2] = 1
    if geom == "solid":
        sim.set_geometry(solid)
    elif geom == "q":
        sim.set_geometry(solid, None, np.full((8, ny, nx), 0.5))
    assert fakelib.lbm_init_fields(sim._h, ANY.ctypes.data, None, None, 1) == 0  # (the fake kernels read no field)
    return sim


def _check(fakelib, sim, nsteps, kernel, ran):
    n, k = sim.step_launches(nsteps)
    before = fakelib.fake_launches()
    sim.step(nsteps)
    assert (k, fakelib.fake_last_step().decode(), n) == (kernel, ran, fakelib.fake_launches() - before)
    fake.sound(fakelib)


F16, F32, F64 = lbm.F16DEV, lbm.F32, lbm.F64


@pytest.mark.parametrize("nx,ny,prec,kw,kernel,ran,in_use", [
    # periodic: staged rows from 2^25 nodes in FP32, from 3 2^20 in 16 bits, never in FP64
    (4096, 8192, F32, {}, "staged", "staged", 2),
    (4096, 8191, F32, {}, "tile", "tile packed", 2),
    (512, 512, F32, {}, "tile", "tile packed", 2),
    (512, 511, F32, {}, "tile", "tile", 1),
    (1024, 3072, F16, {}, "staged", "staged", 2),
    (1024, 3071, F16, {}, "tile", "tile packed", 2),
    (1024, 3071, lbm.BF16DEV, {}, "tile", "tile packed", 2),
    (4096, 8192, F64, {}, "tile", "tile", 2),
    # a width that no staged row can have
    (4098, 8192, F32, {}, "tile", "tile", 1),
    (1028, 3072, F16, {}, "tile", "tile", 1),
    # walls: tiles at every size, rounded as the staged kernel where the step is that of LBM_KERNEL_FUSED
    (4096, 8192, F32, dict(periodic_x=0), "tile", "tile packed", 2),
    (256, 2048, F32, dict(periodic_x=0), "tile", "tile", 1),
    (512, 512, F16, dict(periodic_y=0), "tile", "tile packed", 2),
    (512, 511, F16, dict(periodic_y=0), "tile", "tile", 1),
    (256, 2048, F16, dict(periodic_x=0), "tile", "tile", 1),
    (512, 512, F16, dict(geom="solid"), "tile", "tile packed", 2),
    (512, 511, F16, dict(geom="solid"), "tile", "tile", 1),
    (512, 512, F32, dict(geom="solid"), "tile", "tile", 1),
    (1024, 512, F32, dict(geom="solid"), "tile", "tile packed", 2),
    (512, 512, F64, dict(geom="solid"), "tile", "tile", 1),
    (1024, 1024, F16, dict(geom="q"), "tile", "tile", 1),
    # on request
    (256, 64, F32, dict(kernel=lbm.KERNEL_FUSED), "staged", "staged", 2),
    (256, 64, F32, dict(kernel=lbm.KERNEL_FUSED, periodic_x=0), "tile", "tile packed", 2),
    (256, 64, F16, dict(kernel=lbm.KERNEL_FUSED, geom="solid"), "tile", "tile packed", 2),
    (255, 64, F32, dict(kernel=lbm.KERNEL_FUSED), "two_pass", "two_pass", 1),
    (256, 64, F64, dict(kernel=lbm.KERNEL_FUSED, geom="solid"), "two_pass", "two_pass", 1),
    (4096, 8192, F32, dict(kernel=lbm.KERNEL_TWO_PASS), "two_pass", "two_pass", 1),
    (64, 64, F32, dict(kernel=lbm.KERNEL_TWO_PASS, small=16), "two_pass", "two_pass", 1),
    (256, 64, F32, dict(kernel=lbm.KERNEL_FUSED, small=16), "staged", "staged", 2)])
def test_the_kernel_that_steps(fakelib, nx, ny, prec, kw, kernel, ran, in_use):
    sim = _sim(fakelib, nx, ny, prec, **kw)
    assert sim.kernel_in_use == in_use
    for n in (1, 3, 4, 9):
        _check(fakelib, sim, n, kernel, ran)
    sim.close()


@pytest.mark.parametrize("prec", [F64, F32, F16])
def test_small_lattices(fakelib, prec):
    """Calls of four steps and more in launches of at most 4096; a rest of fewer one by one; with diagnostics every
    D steps up to each of them."""
    sim = _sim(fakelib, 64, 64, prec, small=16)
    for n, ran in ((1, "tile"), (3, "tile"), (4, "small"), (4096, "small"), (4099, "tile"), (4100, "small"), (8192 + 7, "small")):
        _check(fakelib, sim, n, "tile" if n < 4 else "small", ran)
    assert sim.step_launches(0)[0] == 0
    sim.close()
    sim = _sim(fakelib, 64, 64, prec, small=16, diag_every=5)
    for n in (1, 2, 3, 14, 23):
        m, k = sim.step_launches(n)
        before, steps = fakelib.fake_launches(), sim.step_count
        sim.step(n)
        stops = sim.step_count // 5 - steps // 5
        assert m == fakelib.fake_launches() - before - stops, n  # (one reading each)
    fake.sound(fakelib)
    sim.close()
    sim = _sim(fakelib, 64, 64, prec, small=16, geom="q")  # link fractions: not in the small-lattice kernel
    _check(fakelib, sim, 9, "tile", "tile")
    sim.close()


def test_the_small_lattice_kernel_is_asked_for_when_a_call_can_use_it(fakelib):
    """Creating a context, geometry and single steps load nothing for it."""
    sim = _sim(fakelib, 64, 64, F32, small=16, geom="solid")
    for n in (1, 2, 3):
        sim.step(n)
    assert fakelib.fake_small_asked() == 0
    sim.step(4)
    assert fakelib.fake_small_asked() == 1 and fakelib.fake_last_step() == b"small"
    sim.close()
    sim = _sim(fakelib, 64, 64, F32, small=16, kernel=lbm.KERNEL_TWO_PASS)
    sim.step(9)
    assert fakelib.fake_small_asked() == 0
    sim.close()
