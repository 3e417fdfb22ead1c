"""Resident runs of more steps than one launch takes: the bits of single steps, with
recorded states on both sides of the seam."""
import pytest

from paper_1809_02390_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("nx,ny,kw,steps,every", [(410, 400, dict(precision="fp64"), 150, 7),
                                                  (333, 250, dict(precision="fp64"), 301, 60),
                                                  (583, 580, dict(precision="fp32"), 1230, 611),
                                                  (130, 75, dict(precision="fp16s"), 2601, 1300)])
def test_bits_across_launches(nx, ny, kw, steps, every):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1809_02390_gb300 import Lattice, capi, derive

    d = derive(nx, ny, Tr=0.85)
    rho = inputs.droplet(nx, ny, min(nx, ny) / 4, 5, d["rho_g"], d["rho_l"], center=(0.37 * nx, 0.58 * ny))
    a, b, c = (Lattice(rho, Tr=0.85, **kw) for _ in range(3))
    assert capi.lb_step_form(a.h, steps) == capi.LB_STEP_RESIDENT
    a.step(steps)
    rec = torch.zeros((steps // every, *c.f_a.shape), dtype=c.dtype, device="cuda")
    capi.lb_step_record(c.h, steps, every, rec.data_ptr())
    for j in range(steps):
        b.step(1)
        if (j + 1) % every == 0:
            assert torch.equal(rec[j // every], b.buffer()), j
    assert torch.equal(a.buffer(), b.buffer()) and torch.equal(c.buffer(), b.buffer())
    assert a.steps_done == b.steps_done == c.steps_done == steps
    capi.lb_status(a.h)
    capi.lb_status(c.h)
