"""lb_step_record: the recorded states are those that lb_step and lb_get_state in turn
give, bit for bit, on every path (resident, step into the record, step and copy)."""
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
    rho = inputs.droplet(nx, ny, min(nx, ny) / 4, 5, d["rho_g"], d["rho_l"], center=(0.4 * nx, 0.6 * ny))
    return Lattice(rho, Tr=0.85, **kw)


@pytest.mark.parametrize("nx,ny,kw", [(96, 80, dict(precision="fp32")), (70, 33, dict(precision="fp64")),
                                      (96, 80, dict(precision="fp16s", layout="rows")),
                                      (1000, 700, dict(precision="fp32")), (1001, 700, dict(precision="fp32")),
                                      (1000, 704, dict(precision="fp16s", layout="rows")),
                                      (96, 80, dict(precision="fp32", variant="two_pass"))])
@pytest.mark.parametrize("steps,every", [(1, 1), (6, 1), (7, 1), (13, 5), (12, 4), (3, 5), (0, 1)])
def test_record_equals_single_steps(nx, ny, kw, steps, every):
    from paper_1809_02390_gb300 import capi

    a, b = _lat(nx, ny, **kw), _lat(nx, ny, **kw)
    rec = torch.zeros((max(1, steps // every), *a.f_a.shape), dtype=a.dtype, device="cuda")
    capi.lb_step_record(a.h, steps, every, rec.data_ptr())
    for j in range(steps):
        b.step(1)
        if (j + 1) % every == 0:
            assert torch.equal(rec[j // every], b.buffer()), j
    assert torch.equal(a.buffer(), b.buffer()) and a.steps_done == b.steps_done == steps
    a.step(3)
    for _ in range(3):
        b.step(1)
    assert torch.equal(a.buffer(), b.buffer())


def test_invalid_records_are_refused():
    from paper_1809_02390_gb300 import capi

    lat = _lat(64, 48)
    rec = torch.empty_like(lat.f_a)
    for n, e, p in ((-1, 1, rec.data_ptr()), (4, 0, rec.data_ptr()), (4, 2, 0)):
        with pytest.raises(capi.LBError):
            capi.lb_step_record(lat.h, n, e, p)
    assert lat.steps_done == 0
