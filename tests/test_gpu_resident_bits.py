"""Resident runs against single steps, bit for bit, with the form asserted: step counts at the
least that runs resident and above it, written in place (even) and into the other buffer
(odd); the largest lattices that fit and ones just above; a NaN through the exchange."""
import pytest

from paper_1809_02390_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _lat(nx, ny, **kw):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1809_02390_gb300 import Lattice, capi, derive

    d = derive(nx, ny, Tr=0.85)
    r = inputs.droplet(nx, ny, max(1.5, min(nx, ny) / 4), 5, d["rho_g"], d["rho_l"], center=(0.37 * nx, 0.58 * ny))
    lat = Lattice(r * (1 + 0.01 * (2 * inputs.uniform(3, nx * ny).reshape(ny, nx) - 1)), Tr=0.85, **kw)
    try:
        capi.lb_set_resident(lat.h, 1)  # whatever other lattices live
    except capi.LBError:
        pass
    return lat


# One tile, strips, tiles that are all edge, uneven tiles, one and several slots a thread, and
# the largest by precision: 410^2 in FP64, 340,000 nodes else.
SHAPES = [(3, 3), (5, 7), (1024, 4), (4, 300), (100, 31), (97, 203), (301, 299)]
LARGEST = {"fp64": [(410, 410), (409, 401)], "fp32": [(583, 583), (2000, 170)], "fp16s": [(583, 583), (60000, 5)]}
ABOVE = {"fp64": [(411, 411)], "fp32": [(584, 583), (60000, 5)], "fp16s": [(584, 583)]}
CASES = [(p, layout, s) for p, layout in (("fp32", "planes"), ("fp32", "rows"), ("fp16s", "rows"), ("fp64", "planes"))
         for s in SHAPES + LARGEST[p]]


@pytest.mark.parametrize("precision,layout,shape", CASES)
def test_bits_of_single_steps(precision, layout, shape):
    from paper_1809_02390_gb300 import capi

    a, b = (_lat(*shape, precision=precision, layout=layout) for _ in range(2))
    least = 4 if precision == "fp64" else 12
    assert capi.lb_step_form(a.h, least - 1) != capi.LB_STEP_RESIDENT
    total = 0
    for n in (least, least + 1, 24, least, 33):
        assert capi.lb_step_form(a.h, n) == capi.LB_STEP_RESIDENT
        a.step(n)
        total += n
        for _ in range(n):
            b.step(1)
        assert (a.buffer() is a.f_a) == (b.buffer() is b.f_a)
        assert torch.equal(a.buffer(), b.buffer()), n
    assert a.steps_done == b.steps_done == total
    capi.lb_status(a.h)


@pytest.mark.parametrize("precision", sorted(ABOVE))
def test_lattices_above_the_bounds_do_not(precision):
    from paper_1809_02390_gb300 import LBError, capi

    for shape in ABOVE[precision]:
        lat = _lat(*shape, precision=precision)
        assert capi.lb_step_form(lat.h, 100) == capi.LB_STEP_PLAIN
        with pytest.raises(LBError):
            capi.lb_set_resident(lat.h, 1)
        lat.close()


@pytest.mark.parametrize("precision", ["fp32", "fp64", "fp16s"])
def test_nan_crosses_the_exchange(precision):
    from paper_1809_02390_gb300 import LBError, capi

    a, b = (_lat(200, 120, precision=precision) for _ in range(2))
    for lat in (a, b):
        lat.buffer()[4, 60, 100] = float("nan")
    assert capi.lb_step_form(a.h, 21) == capi.LB_STEP_RESIDENT  # tiles of some 14 x 15 nodes: 21 steps cross two
    a.step(21)
    for _ in range(21):
        b.step(1)
    nan = torch.isnan(a.buffer())
    assert torch.equal(nan, torch.isnan(b.buffer())) and int(nan.any(0).sum()) > 40 * 40
    assert torch.equal(a.buffer()[~nan], b.buffer()[~nan])
    with pytest.raises(LBError):
        capi.lb_reduce(a.h)
