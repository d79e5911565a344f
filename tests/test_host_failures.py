"""What the host side of the library does when an allocation fails, on a fake device: a call that fails leaves
a context that later calls may use, with nothing freed that a launch still names."""
import numpy as np
import pytest

from paper_2604_13407_gb300 import lbm
from tests import fake

ENOMEM = 2


@pytest.fixture(scope="module")
def fakelib(tmp_path_factory):
    saved, lbm._lib = lbm._lib, None
    try:
        yield fake.load(tmp_path_factory.mktemp("fake"))
    finally:
        lbm._lib = saved


def _arrays(nx, ny):
    solid = np.zeros((ny, nx), np.uint8)
    solid[:, :2] = 1
    wall_u = 0.01 * np.ones((2, ny, nx)) * solid
    return solid, wall_u, np.full((8, ny, nx), 0.4), np.full((2, ny, nx), 1e-6)


@pytest.mark.parametrize("prec", [lbm.F64, lbm.F32, lbm.F16DEV])
@pytest.mark.parametrize("before", [False, True])
def test_set_geometry_that_runs_out_of_memory(fakelib, prec, before):
    """Fails at its first, second, ... allocation, on a context with and without a geometry; then the steps,
    the readings and calls that refresh the kernels' parameters."""
    nx, ny = 40, 24
    geometry = _arrays(nx, ny)
    k = failed = 0
    while failed == k:
        fakelib.fake_reset(0)
        sim = lbm.Simulation(lbm.default_params(nx=nx, ny=ny, periodic_x=1, periodic_y=1, precision=prec, force_mode=2))
        sim.init_fields(np.full((ny, nx), 0.2))
        if before:
            sim.set_geometry(*geometry)
        fake.limit(fakelib, mallocs=k)
        try:
            sim.set_geometry(*geometry)
        except lbm.LbmError as e:
            assert e.status == ENOMEM
            failed += 1
        fake.limit(fakelib)
        sim.step(2)
        sim.set_param(lbm.PARAM_T, sim.params.T)
        sim.step(1)
        sim.moments()
        sim.set_wall_density(np.full((ny, nx), 0.1))
        sim.step(1)
        fake.sound(fakelib)
        sim.set_geometry(*geometry)  # and the same call with memory to be had succeeds
        sim.step(1)
        sim.close()
        fake.sound(fakelib)
        assert fakelib.fake_bytes() == 0
        k += 1
    assert k >= 5


@pytest.mark.parametrize("prec", [lbm.F64, lbm.F32, lbm.F16DEV])
@pytest.mark.parametrize("before", [False, True])
def test_set_wall_density_that_runs_out_of_memory(fakelib, prec, before):
    nx, ny = 40, 24
    solid = _arrays(nx, ny)[0]
    k = failed = 0
    while failed == k:
        fakelib.fake_reset(0)
        sim = lbm.Simulation(lbm.default_params(nx=nx, ny=ny, periodic_x=1, periodic_y=1, precision=prec))
        sim.set_geometry(solid)
        sim.init_fields(np.full((ny, nx), 0.2))
        if before:
            sim.set_wall_density(np.full((ny, nx), 0.1))
        fake.limit(fakelib, mallocs=k)
        try:
            sim.set_wall_density(np.full((ny, nx), 0.05))
        except lbm.LbmError as e:
            assert e.status == ENOMEM
            failed += 1
        fake.limit(fakelib)
        sim.step(2)
        sim.set_param(lbm.PARAM_FX, 1e-7)
        sim.step(1)
        sim.set_geometry(solid)
        sim.step(1)
        sim.close()
        fake.sound(fakelib)
        k += 1
    assert k >= (2 if prec == lbm.F64 else 3)


def test_a_reset_device_is_asked_again(fakelib):
    """What a kernel was allowed (shared memory, cluster size) is gone after a reset of the device: it is set
    again for the new context, and only once for each."""
    fakelib.fake_reset(0)
    for _ in range(3):
        assert fakelib.fake_cluster_fits(16) == 1
    assert fakelib.fake_attributes() == 2
    fakelib.fake_device_reset()
    for _ in range(3):
        assert fakelib.fake_cluster_fits(16) == 1
    assert fakelib.fake_attributes() == 4


@pytest.mark.parametrize("prec", [lbm.F64, lbm.F32, lbm.F16DEV])
@pytest.mark.parametrize("nx,ny", [(1, 1), (1, 3000), (40, 24), (700, 1)])
def test_diagnostics_allocate_nothing(fakelib, prec, nx, ny):
    fakelib.fake_reset(0)
    sim = lbm.Simulation(lbm.default_params(nx=nx, ny=ny, precision=prec, diag_every=2))
    sim.init_fields(np.full((ny, nx), 0.2))
    fake.limit(fakelib, mallocs=0)
    sim.diagnostics()
    sim.step(5)
    sim.close()
    fake.sound(fakelib)
