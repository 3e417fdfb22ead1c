"""Resident runs (many steps per launch, lattice in shared memory): lb_step takes them
for calls of at least four steps on lattices that fit.  The arithmetic per node is
that of the per-step kernels, so every comparison is bit for bit with the same number
of single-step calls (which are never resident)."""
import numpy as np
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


def _rho(nx, ny, seed=3):
    from paper_1809_02390_gb300 import derive

    d = derive(max(nx, 3), max(ny, 3), Tr=0.85)
    r = inputs.droplet(nx, ny, max(1.5, min(nx, ny) / 4), 5, d["rho_g"], d["rho_l"], center=(0.37 * nx, 0.58 * ny))
    return r * (1 + 0.01 * (2 * inputs.uniform(seed, nx * ny).reshape(ny, nx) - 1))


def _lat(rho, **kw):
    from paper_1809_02390_gb300 import Lattice

    return Lattice(rho, Tr=0.85, **kw)


# One tile (3 x 3, 5 x 7); strips of one tile row or column; tiles that are all edge (100 x 31);
# uneven tiles (97 x 203, 301 x 299); one and several slots per thread; the largest that fit.
SHAPES = [(3, 3), (5, 7), (1024, 4), (4, 300), (100, 31), (97, 203), (301, 299), (440, 460), (613, 590)]


@pytest.mark.parametrize("nx,ny", SHAPES)
@pytest.mark.parametrize("precision,layout", [("fp32", "planes"), ("fp32", "rows"), ("fp16s", "rows"), ("fp64", "planes")])
def test_bits_of_single_steps(nx, ny, precision, layout):
    from paper_1809_02390_gb300 import capi

    rho = _rho(nx, ny)
    a, b = (_lat(rho, precision=precision, layout=layout) for _ in range(2))
    for n in (4, 7, 21):  # even: written in place; odd: into the other buffer
        a.step(n)
        for _ in range(n):
            b.step(1)
        assert (a.buffer() is a.f_a) == (b.buffer() is b.f_a)
        assert torch.equal(a.buffer(), b.buffer()), n
    assert a.steps_done == b.steps_done == 32
    capi.lb_status(a.h)


def test_long_call_and_cs():
    """More steps than one launch takes, Carnahan-Starling, nearest rounding."""
    from paper_1809_02390_gb300 import capi

    rho = _rho(70, 52) * 0.05
    for kw in (dict(precision="fp32", eos="cs", eos_a=1.0, eos_b=4.0), dict(precision="fp16s", rounding=1)):
        r = rho if "eos" in kw else _rho(70, 52)
        a, b = _lat(r, **kw), _lat(r, **kw)
        a.step(4097)
        for _ in range(4097):
            b.step(1)
        assert torch.equal(a.buffer(), b.buffer())
        capi.lb_status(a.h)


def test_two_lattices_on_two_streams():
    rho = _rho(256, 256)
    s = [torch.cuda.Stream() for _ in range(2)]
    lats = [_lat(rho * (1 + 0.01 * k), stream=s[k]) for k in range(2)]
    ref = [_lat(rho * (1 + 0.01 * k)) for k in range(2)]
    torch.cuda.synchronize()
    for _ in range(10):
        for lat in lats:
            lat.step(50)
    for lat in ref:
        for _ in range(10):
            lat.step(50)
    torch.cuda.synchronize()
    for a, b in zip(lats, ref):
        assert torch.equal(a.buffer(), b.buffer())


def test_scratch_of_the_former_size_still_works():
    """A scratch buffer without room for the exchange words is accepted; the steps are
    then launched one by one."""
    from paper_1809_02390_gb300 import capi

    rho = torch.from_numpy(_rho(128, 96)).cuda()
    p = capi.make_params(128, 96, Tr=0.85, rho_ref=1.0)
    base = (128 * 96 * 4 + 255) // 256 * 256 + 65536 + 256 + 256
    assert capi.lb_scratch_bytes(p) > base
    f = [torch.empty((9, 96, 128), dtype=torch.float32, device="cuda") for _ in range(2)]
    scratch = torch.empty(base, dtype=torch.uint8, device="cuda")
    h = capi.lb_init(p, f[0].data_ptr(), f[1].data_ptr(), scratch.data_ptr(), base, rho.data_ptr(), True,
                     torch.cuda.current_stream().cuda_stream)
    capi.lb_step(h, 40)
    ref = _lat(rho, rho_ref=1.0)
    ref.step(40)
    torch.cuda.synchronize()
    assert torch.equal(f[0], ref.buffer())
    capi.lb_free(h)


def test_non_finite_state_stays_reported():
    """A planted NaN spreads through the exchange like through single steps."""
    from paper_1809_02390_gb300 import LBError, capi

    a, b = _lat(_rho(200, 120)), _lat(_rho(200, 120))
    for lat in (a, b):
        lat.buffer()[4, 60, 100] = float("nan")
    a.step(9)
    for _ in range(9):
        b.step(1)
    assert torch.equal(torch.isnan(a.buffer()), torch.isnan(b.buffer())) and bool(torch.isnan(a.buffer()).any())
    with pytest.raises(LBError):
        capi.lb_reduce(a.h)
