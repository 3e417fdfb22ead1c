"""D3Q19 step: how a tile's windows arrive and how a lattice is cut.  Shapes at the edges
of the tiles against the FP64 oracle: tiles with tensor copies beside tiles that wrap,
ragged last tiles, rows that are no multiple of 16 bytes, lattices below one tile, and
z-chunks with a remainder.  Tolerances as in test_gpu_d3q19 (FP64 1e-12 of the largest
population, FP32 2e-5: about 700 operations of relative error 6e-8 a node, 20 steps)."""
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


# (nz, ny, nx).  FP32: 72 x 18 holds one tensor-copy tile, 104 x 34 several; 100 x 21 and 68 x 26
# are ragged; 40 x 8 is the smallest with windows; 36, 75 and 12 rows take the pulled form.
FP32 = [(5, 18, 72), (7, 34, 104), (4, 21, 100), (3, 26, 68), (2, 8, 40), (5, 17, 36), (4, 19, 75), (6, 12, 80),
        (1, 24, 96), (70, 9, 44)]
# FP64: tiles chosen by size (24 x 10, 8 x 12, 12 x 10 nodes), odd rows, one chunk and several.
FP64 = [(5, 40, 48), (24, 24, 24), (9, 33, 41), (3, 7, 130), (2, 50, 8), (71, 10, 12)]


@pytest.mark.parametrize("precision,shape", [("fp32", s) for s in FP32] + [("fp64", s) for s in FP64])
def test_steps_match_the_oracle(o3, precision, shape):
    from oracle import params as op
    from paper_1809_02390_gb300 import Lattice3, capi

    p = op.from_physical_3d(Tr=0.85, K_int=1.2)
    nz, ny, nx = shape
    rng = np.random.default_rng(nx + 7 * ny)
    z, y, x = np.mgrid[0:nz, 0:ny, 0:nx].astype(float)
    wave = np.cos(2 * np.pi * (x / nx + y / ny)) + np.cos(2 * np.pi * (y / ny - z / nz) + 0.7)
    rho0 = 0.5 * (p.rho_g + p.rho_l) + 0.4 * (p.rho_l - p.rho_g) * np.tanh(wave)
    rho0 *= 1 + 0.01 * rng.uniform(-1, 1, shape)
    lat = Lattice3(rho0, precision=precision, Tr=0.85, K_int=1.2)
    ore = [tuple(int(v) for v in c) for c in o3.velocities().T]
    perm = [ore.index(tuple(e)) for e in lat.velocities]
    lat.step(20)
    ref = o3.step(p, o3.init_eq(p, rho0), 20)[perm]
    got = lat.populations().cpu().numpy()
    assert np.abs(got - ref).max() <= (1e-12 if precision == "fp64" else 2e-5) * np.abs(ref).max()
    capi.check_d3(capi.lib().lb_d3_status(lat.h), lat.h)


def test_mass_stays_in_fp32():
    """400 steps: the rounding of the collision's constants does not add up to a drift
    (a rest population from the other moments lost 3e-8 of it a step)."""
    from paper_1809_02390_gb300 import Lattice3

    rng = np.random.default_rng(1)
    lat = Lattice3(3.8 * (1 + 0.01 * rng.uniform(-1, 1, (24, 40, 72))), precision="fp32", Tr=0.8, K_int=1.5)
    m0 = lat.reduce()["mass"]
    lat.step(400)
    assert abs(lat.reduce()["mass"] / m0 - 1) <= 2e-6
