"""Adjoint steps with 8-row tiles (one or two nodes a thread, by the number of tiles)
against those with 16-row tiles, which a scratch without room for the partial sums of the
smaller tiles selects."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("nx,ny", [(9, 7), (33, 17), (32, 16), (45, 24), (256, 256), (301, 299), (608, 128), (609, 128)])
@pytest.mark.parametrize("k", [1, 4])
def test_tile_heights_agree(nx, ny, k):
    """The formulas and their order are the same, so only the contraction of products and
    the order of the parameters' sums can differ: a few units of 6e-8 a step, bounded by
    1e-5 of the largest entry as for the steps of lb_adjoint_step."""
    from paper_1809_02390_gb300 import Lattice, build, capi

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    rng = np.random.default_rng(nx + k)
    lat = Lattice(3.8 * (1 + 0.02 * rng.uniform(-1, 1, (ny, nx))), precision="fp32", Tr=0.8)
    states = []
    for _ in range(k):
        lat.step(1)
        states.append(lat.state().clone())
    lam0 = torch.from_numpy(rng.standard_normal((9, ny, nx))).to("cuda", torch.float32)
    full = capi.lb_adjoint_steps_scratch_bytes(lat.p)
    former = 2 * ((11 * nx * ny * 4 + 255) // 256 * 256) + -(-nx // 32) * -(-ny // 16) * 24
    assert former <= full
    out = []
    for size in (full, former):
        scr = torch.empty(size, dtype=torch.uint8, device="cuda")
        lam, th = lam0.clone(), torch.zeros(3, dtype=torch.float64, device="cuda")
        capi.lb_adjoint_steps(lat.h, [s.data_ptr() for s in states], lam.data_ptr(), th.data_ptr(), scr.data_ptr(), size)
        out.append((lam, th))
    with pytest.raises(capi.LBError):
        capi.lb_adjoint_steps(lat.h, [states[0].data_ptr()], lam0.data_ptr(), None, scr.data_ptr(), former - 1)
    (a, ta), (b, tb) = out
    assert bool(torch.isfinite(b).all()) and float((a - b).abs().max()) <= 1e-5 * float(b.abs().max())
    assert float((ta - tb).abs().max()) <= 1e-5 * float(tb.abs().max())
    lat.close()
