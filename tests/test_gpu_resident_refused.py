"""A resident launch that the device refuses: the call goes on by single launches and gives
the same bits and records, whichever launch it was.  (The refusal is made on the host.)"""
import pytest

from paper_1809_02390_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("launches", [0, 1, 2])
@pytest.mark.parametrize("every", [0, 1, 7, 100, 150])  # 0: no record
def test_steps_go_on(launches, every):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1809_02390_gb300 import LBError, Lattice, capi, derive

    nx, ny, steps = 410, 330, 245  # some 80 steps a launch
    d = derive(nx, ny, Tr=0.85)
    rho = inputs.droplet(nx, ny, 80, 5, d["rho_g"], d["rho_l"], center=(0.37 * nx, 0.58 * ny))
    a, b = (Lattice(rho, Tr=0.85, precision="fp64") for _ in range(2))
    assert capi.lb_step_form(a.h, steps) == capi.LB_STEP_RESIDENT
    capi.lb_resident_selftest(a.h, launches)
    if every:
        rec = torch.zeros((steps // every, *a.f_a.shape), dtype=a.dtype, device="cuda")
        capi.lb_step_record(a.h, steps, every, rec.data_ptr())
    else:
        a.step(steps)
    assert capi.lb_step_form(a.h, steps) == capi.LB_STEP_PLAIN
    for j in range(steps):
        b.step(1)
        if every and (j + 1) % every == 0:
            assert torch.equal(rec[j // every], b.buffer()), j
    assert torch.equal(a.buffer(), b.buffer()) and a.steps_done == b.steps_done == steps
    with pytest.raises(LBError):
        capi.lb_resident_selftest(a.h, 0)
    capi.lb_status(a.h)
