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
    assert k == 2  # (one allocation)


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
    assert k == 2


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


def _two_pass_adjoint_bytes(nx, ny, prec, n, K):
    """What an adjoint call took while its transposed step ran in two passes: every checkpoint, two sets of
    segment states (one state at least) and psi fields, 24 planes, and a row of 64 bytes for each 128 nodes of a lattice row."""
    elem, real = {lbm.F64: (8, 8), lbm.F32: (4, 4), lbm.F16DEV: (2, 4)}[prec]
    per_line = 128 // elem
    plane = (nx + per_line - 1) // per_line * per_line * ny
    up = lambda b: (b + 255) // 256 * 256  # noqa: E731
    state = 9 * plane * elem if prec != lbm.F16DEV else up(9 * plane * elem) + 4 * plane
    K = min(K, n)
    parts = up((nx + 127) // 128 * ny * 64)
    return ((n + K - 1) // K * up(state) + 2 * max(K - 1, 1) * up(state) + 2 * K * up(nx * ny * real) +
            2 * up(9 * plane * real) + up(2 * plane * real) + 4 * up(plane * real) + parts + 512)


@pytest.mark.parametrize("tight", [False, True])
@pytest.mark.parametrize("prec", [lbm.F64, lbm.F32, lbm.F16DEV])
@pytest.mark.parametrize("kernel", [lbm.KERNEL_AUTO, lbm.KERNEL_TWO_PASS])
def test_adjoint_in_the_memory_it_used_to_take(fakelib, prec, kernel, tight):
    """Every number of steps and checkpoint interval, with all the memory there is and with what the two-pass
    transposed step took: each kernel reads the state, psi field and planes of its step, whichever buffers hold them."""
    nx, ny = 33, 18
    for n in range(1, 10):
        for K in range(1, n + 2):
            fakelib.fake_reset(0)
            sim = lbm.Simulation(lbm.default_params(nx=nx, ny=ny, precision=prec, kernel=kernel, per_node_ref=1))
            sim.init_fields(np.full((ny, nx), 0.2))
            if tight:
                fake.limit(fakelib, nbytes=_two_pass_adjoint_bytes(nx, ny, prec, n, K))
            for call in range(2):  # (the second keeps the first one's memory)
                J, g, _ = sim.adjoint(n, K, lbm.OBJ_MEAN_JX)
                assert J == 1.0 and sim.step_count == n  # (the fake objective is the number of the state)
                fake.sound(fakelib)
                fake.limit(fakelib, mallocs=0)
                sim.init_fields(np.full((ny, nx), 0.2))
            fake.limit(fakelib)
            sim.init_fields(np.full((ny, nx), 0.2))
            sim.adjoint(n, K, lbm.OBJ_MEAN_JX, want_lambda0=True)
            sim.step(1)
            fake.sound(fakelib)
            sim.close()
