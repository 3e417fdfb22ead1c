"""lb_step_record into records that start at any element's address: the states of single
steps, bit for bit."""
import pytest

from paper_1809_02390_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


# FP16 even and odd widths without tensor copies, with them, resident calls (14 steps); FP32, FP64.
@pytest.mark.parametrize("nx,ny,kw", [(100, 80, dict(precision="fp16s")), (101, 80, dict(precision="fp16s", layout="rows")),
                                      (128, 96, dict(precision="fp16s")), (128, 96, dict(precision="fp32")),
                                      (70, 33, dict(precision="fp64"))])
@pytest.mark.parametrize("steps", [3, 14])
@pytest.mark.parametrize("offset", [0, 1, 2, 3, 8])  # elements
def test_records_at_any_element(nx, ny, kw, steps, offset):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1809_02390_gb300 import Lattice, capi, derive

    d = derive(nx, ny, Tr=0.85)
    rho = inputs.droplet(nx, ny, min(nx, ny) / 4, 5, d["rho_g"], d["rho_l"], center=(0.4 * nx, 0.6 * ny))
    a, b = (Lattice(rho, Tr=0.85, **kw) for _ in range(2))
    n = a.f_a.numel()
    buf = torch.zeros(steps * n + 16, dtype=a.dtype, device="cuda")
    rec = buf[offset:offset + steps * n]
    assert rec.data_ptr() % 16 == offset * buf.element_size() % 16
    capi.lb_step_record(a.h, steps, 1, rec.data_ptr())
    for j in range(steps):
        b.step(1)
        assert torch.equal(rec[j * n:(j + 1) * n].view(b.f_a.shape), b.buffer()), j
    assert torch.equal(a.buffer(), b.buffer())
    assert not buf[:offset].any() and not buf[offset + steps * n:].any()
