"""Forms of the D3Q19 step: which one the sides choose, each against the FP64 oracle on
shapes at the edges of its tiles (small ones are windowed only when asked), and a change of
form in the middle of a run (the graphs of the other form are dropped).  Tolerances as in
test_gpu_d3_tiles (FP32 2e-5 of the largest population over 20 steps), over 201 steps 2e-4."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def o3():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle import d3q19
    from paper_1809_02390_gb300 import build

    build.build()
    d3q19.build()
    return d3q19


def _rho(p, shape):
    nz, ny, nx = shape
    rng = np.random.default_rng(nx + 7 * ny)
    z, y, x = np.mgrid[0:nz, 0:ny, 0:nx].astype(float)
    wave = np.cos(2 * np.pi * (x / nx + y / ny)) + np.cos(2 * np.pi * (y / ny - z / nz) + 0.7)
    rho0 = 0.5 * (p.rho_g + p.rho_l) + 0.4 * (p.rho_l - p.rho_g) * np.tanh(wave)
    return rho0 * (1 + 0.01 * rng.uniform(-1, 1, shape))


def _error(o3, p, lat, rho0, steps):
    ore = [tuple(int(v) for v in c) for c in o3.velocities().T]
    perm = [ore.index(tuple(e)) for e in lat.velocities]
    ref = o3.step(p, o3.init_eq(p, rho0), steps)[perm]
    return np.abs(lat.populations().cpu().numpy() - ref).max() / np.abs(ref).max()


# Windows: one tensor-copy tile, several, ragged ones, the smallest, one and many planes.
@pytest.mark.parametrize("shape", [(5, 18, 72), (7, 34, 104), (4, 21, 100), (3, 26, 68), (2, 8, 40), (6, 12, 80),
                                   (1, 24, 96), (70, 9, 44), (33, 40, 64)])
def test_windows_match_the_oracle(o3, shape):
    from oracle import params as op
    from paper_1809_02390_gb300 import Lattice3, capi

    p = op.from_physical_3d(Tr=0.85, K_int=1.2)
    rho0 = _rho(p, shape)
    lat = Lattice3(rho0, precision="fp32", Tr=0.85, K_int=1.2)
    capi.lb_d3_set_form(lat.h, capi.LB_D3_WINDOWS)
    assert capi.lb_d3_form(lat.h) == capi.LB_D3_WINDOWS
    lat.step(20)
    assert _error(o3, p, lat, rho0, 20) <= 2e-5
    capi.check_d3(capi.lib().lb_d3_status(lat.h), lat.h)


def test_change_of_form_in_a_run(o3):
    from oracle import params as op
    from paper_1809_02390_gb300 import Lattice3, capi

    p = op.from_physical_3d(Tr=0.85, K_int=1.2)
    rho0 = _rho(p, (12, 20, 48))
    a, b = (Lattice3(rho0, precision="fp32", Tr=0.85, K_int=1.2) for _ in range(2))
    for form, n in ((capi.LB_D3_WINDOWS, 70), (capi.LB_D3_PULLS, 66), (capi.LB_D3_WINDOWS, 65)):
        for lat in (a, b):
            capi.lb_d3_set_form(lat.h, form)
            assert capi.lb_d3_form(lat.h) == form
        a.step(n)  # a replayed graph of 64 steps and single launches
        for _ in range(n):
            b.step(1)
    assert torch.equal(a.state(), b.state())
    assert _error(o3, p, a, rho0, 201) <= 2e-4


# (nz, ny, nx): small or ragged lattices by pulls, ones whose tiles are full by windows.
@pytest.mark.parametrize("shape,windows", [((40, 40, 40), False), ((32, 32, 48), False), ((101, 72, 40), False),
                                           ((104, 104, 104), False), ((40, 40, 75), False), ((40, 64, 36), False),
                                           ((64, 64, 64), True), ((96, 96, 96), True), ((48, 35, 196), True)])
def test_the_rule(o3, shape, windows):
    from paper_1809_02390_gb300 import LBError, Lattice3, capi

    lat = Lattice3(np.full(shape, 1.0), precision="fp32", Tr=0.85)
    assert capi.lb_d3_form(lat.h) == (capi.LB_D3_WINDOWS if windows else capi.LB_D3_PULLS)
    capi.lb_d3_set_form(lat.h, capi.LB_D3_PULLS)
    if shape[2] % 4 or shape[2] < 40:
        with pytest.raises(LBError):
            capi.lb_d3_set_form(lat.h, capi.LB_D3_WINDOWS)
    else:
        capi.lb_d3_set_form(lat.h, capi.LB_D3_WINDOWS)
    capi.lb_d3_set_form(lat.h, capi.LB_D3_AUTO)
    assert capi.lb_d3_form(lat.h) == (capi.LB_D3_WINDOWS if windows else capi.LB_D3_PULLS)
    with pytest.raises(LBError):
        capi.lb_d3_set_form(lat.h, 2)
    f = Lattice3(np.full((8, 8, 8), 1.0), precision="fp64", Tr=0.85)
    assert capi.lb_d3_form(f.h) == capi.LB_D3_WINDOWS
    with pytest.raises(LBError):
        capi.lb_d3_set_form(f.h, capi.LB_D3_PULLS)
