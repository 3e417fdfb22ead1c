"""Which kernel a step call takes (lb_step_form), and that every form gives the same bits."""
import pytest

from paper_1809_02390_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1809_02390_gb300 import build

    build.build()


def _lat(nx, ny, **kw):
    from paper_1809_02390_gb300 import Lattice, derive

    d = derive(nx, ny, Tr=0.85)
    rho = inputs.droplet(nx, ny, min(nx, ny) / 4, 5, d["rho_g"], d["rho_l"], center=(0.37 * nx, 0.58 * ny))
    rho = rho * (1 + 0.01 * (2 * inputs.uniform(7, nx * ny).reshape(ny, nx) - 1))
    return Lattice(rho, Tr=0.85, **kw)


def _forms(lat):
    from paper_1809_02390_gb300 import capi

    return tuple(capi.lb_step_form(lat.h, n) for n in (1, 3, 4, 11, 12, 300))


def test_asked_dispatch_is_taken():
    """A small lattice steps by plain loads or resident unless a tensor-copy form is asked
    for, which then serves calls of every length; all with the same bits."""
    from paper_1809_02390_gb300 import capi

    P, W, T, R = (capi.LB_STEP_PLAIN, capi.LB_STEP_TENSOR_WALK, capi.LB_STEP_TENSOR_TICKETS, capi.LB_STEP_RESIDENT)
    for precision in ("fp32", "fp16s"):
        a, b, c = (_lat(512, 300, precision=precision) for _ in range(3))
        assert _forms(a) == (P, P, P, P, R, R)
        capi.lb_set_tile_dispatch(b.h, True)
        assert _forms(b) == (T,) * 6 and capi.lb_tile_dispatch(b.h) == 1
        capi.lb_set_tile_dispatch(c.h, False)
        assert _forms(c) == (W,) * 6 and capi.lb_tile_dispatch(c.h) == 0
        rec = [torch.zeros((2, *a.f_a.shape), dtype=a.dtype, device="cuda") for _ in range(3)]
        for lat, r in zip((a, b, c), rec):
            for n in (1, 12, 70):
                lat.step(n)
            capi.lb_step_record(lat.h, 13, 6, r.data_ptr())
            capi.lb_status(lat.h)
        assert torch.equal(a.buffer(), b.buffer()) and torch.equal(a.buffer(), c.buffer())
        assert torch.equal(rec[0], rec[1]) and torch.equal(rec[0], rec[2])


def test_dispatch_of_lattices_without_tensor_copies_changes_nothing():
    from paper_1809_02390_gb300 import LBError, capi

    P, R = capi.LB_STEP_PLAIN, capi.LB_STEP_RESIDENT
    for kw, want in ((dict(precision="fp32"), (P, P, P, P, R, R)), (dict(precision="fp64"), (P, P, R, R, R, R)),
                     (dict(precision="fp32", variant="two_pass"), (capi.LB_STEP_TWO_PASS,) * 6)):
        lat = _lat(75, 61, **kw)
        assert _forms(lat) == want
        with pytest.raises(LBError):
            capi.lb_set_tile_dispatch(lat.h, True)
        capi.lb_set_tile_dispatch(lat.h, False)
        assert _forms(lat) == want
    with pytest.raises(LBError):
        capi.lb_step_form(lat.h, 0)
