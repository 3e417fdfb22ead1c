"""Resident runs and several streams: while lattices on more streams make long calls than runs
of one fit the GPU side by side, calls take single launches again; lb_set_resident decides
otherwise.  Lattices that make none do not count.  The bits are the same."""
import pytest

from paper_1809_02390_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _lats(streams, nx=200, ny=160, **kw):
    from paper_1809_02390_gb300 import Lattice, derive

    d = derive(nx, ny, Tr=0.85)
    rho = inputs.droplet(nx, ny, 40, 5, d["rho_g"], d["rho_l"], center=(0.37 * nx, 0.58 * ny))
    return [Lattice(rho * (1 + 0.01 * k), Tr=0.85, stream=s, **kw) for k, s in enumerate(streams)]


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_many_streams_leave_resident_runs(precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import gc

    from paper_1809_02390_gb300 import LBError, capi

    gc.collect()  # lattices of earlier tests count while they live
    R = capi.LB_STEP_RESIDENT
    one = torch.cuda.Stream()
    lats = _lats([one], precision=precision)
    assert capi.lb_step_form(lats[0].h, 40) == R
    lats += _lats([one] * 12, precision=precision)  # many lattices, one stream
    for lat in lats:
        lat.step(40)
    assert all(capi.lb_step_form(lat.h, 40) == R for lat in lats)
    others = [_lats([torch.cuda.Stream()], precision=precision)[0] for _ in range(12)]
    for lat in others:
        lat.step(3)  # too short for a resident run
    assert all(capi.lb_step_form(lat.h, 40) == R for lat in lats)
    for lat in others:
        lat.step(37)
    assert all(capi.lb_step_form(lat.h, 40) == capi.LB_STEP_PLAIN for lat in lats + others)
    capi.lb_set_resident(others[3].h, 1)
    assert capi.lb_step_form(others[3].h, 40) == R
    ref = _lats([one], precision=precision)[0]
    torch.cuda.synchronize()
    for _ in range(3):
        for lat in others:
            lat.step(40)
    for _ in range(160):
        ref.step(1)
    torch.cuda.synchronize()
    for lat in others:
        assert torch.equal(lat.buffer(), ref.buffer())
    for lat in others:
        lat.close()
    assert all(capi.lb_step_form(lat.h, 40) == R for lat in lats)
    capi.lb_set_resident(lats[0].h, 0)
    assert capi.lb_step_form(lats[0].h, 40) == capi.LB_STEP_PLAIN
    capi.lb_set_resident(lats[0].h, -1)
    assert capi.lb_step_form(lats[0].h, 40) == R
    for mode in (-2, 2):
        with pytest.raises(LBError):
            capi.lb_set_resident(lats[0].h, mode)
    big = _lats([one], 1000, 700, precision=precision)[0]
    with pytest.raises(LBError):
        capi.lb_set_resident(big.h, 1)
    for lat in (*lats, ref, big):
        lat.close()
