"""Each form of the step held to what it should give, with the form asserted: tickets and
tensor copies against the oracle, graph replay of the plain step (whose launches overlap
there too) against single launches across buffer flips and new states, both layouts.  Small
lattices are kept from running resident by lb_set_resident or by the dispatch they ask for."""
import pytest

from gpu_util import lattice, oracle_params, rel_inf
from paper_1809_02390_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1809_02390_gb300 import build

    build.build()


def _droplet(nx, ny):
    p = oracle_params(Tr=0.85, K_int=1.0)
    return p, inputs.droplet(nx, ny, min(nx, ny) / 4, 5, p.rho_g, p.rho_l, center=(0.41 * nx, 0.53 * ny))


# Tolerances: those of the tensor-copy tests in test_gpu_parity (300 FP32 and 500 FP16 steps).
@pytest.mark.parametrize("precision,layout,nx,ny,steps,tol", [("fp32", "rows", 208, 83, 300, 2e-5),
                                                              ("fp32", "planes", 160, 96, 300, 2e-5),
                                                              ("fp16s", "planes", 160, 96, 500, 8e-3)])
@pytest.mark.parametrize("tickets", [True, False])
def test_tensor_copies_match_the_oracle(orc, precision, layout, nx, ny, steps, tol, tickets):
    from paper_1809_02390_gb300 import capi

    p, rho0 = _droplet(nx, ny)
    lat = lattice(rho0, precision, layout=layout, Tr=0.85, K_int=1.0)
    form = capi.LB_STEP_TENSOR_TICKETS if tickets else capi.LB_STEP_TENSOR_WALK
    capi.lb_set_tile_dispatch(lat.h, tickets)
    assert capi.lb_step_form(lat.h, 1) == capi.lb_step_form(lat.h, steps) == form
    assert capi.lb_wait_selftest(lat.h, 2000) == capi.LB_ETIMEOUT  # a wait that gave up leaves the form usable
    capi.lb_status(lat.h)
    lat.step(steps)
    capi.lb_status(lat.h)
    ref = orc.macro(p, orc.step(p, orc.init_feq(p, rho0), steps))[0]
    assert rel_inf(lat.moments(velocity=False).double().cpu().numpy(), ref) <= tol


# Above the largest resident lattice, and small ones with resident runs forbidden.
GRAPHS = [("fp32", "planes", 1003, 517), ("fp16s", "rows", 1000, 512), ("fp16s", "planes", 701, 600),
          ("fp64", "planes", 512, 500), ("fp32", "rows", 70, 45), ("fp16s", "rows", 160, 96), ("fp16s", "planes", 75, 61),
          ("fp64", "rows", 64, 64)]


@pytest.mark.parametrize("precision,layout,nx,ny", GRAPHS)
def test_graphs_of_the_plain_step(precision, layout, nx, ny):
    from paper_1809_02390_gb300 import capi

    _, rho0 = _droplet(nx, ny)
    a, b = (lattice(rho0, precision, layout=layout, Tr=0.85, K_int=1.0) for _ in range(2))
    if nx * ny < 20000:
        for lat in (a, b):
            capi.lb_set_resident(lat.h, 0)
    assert capi.lb_step_form(a.h, 1) == capi.lb_step_form(a.h, 200) == capi.LB_STEP_PLAIN

    def same_run(n):
        a.step(n)
        for _ in range(n):
            b.step(1)
        torch.cuda.synchronize()
        assert (a.buffer() is a.f_a) == (b.buffer() is b.f_a)
        assert torch.equal(a.buffer(), b.buffer()), n

    same_run(2 * 64 + 7)  # two replays, and single launches that flip the buffer
    for lat in (a, b):
        capi.lb_stream_copy(lat.h)
    same_run(64 + 5)
    other = a.buffer().clone()
    same_run(64)
    for lat in (a, b):
        capi.lb_set_state(lat.h, other.data_ptr())
    same_run(128)
    assert a.steps_done == b.steps_done


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16s"])
def test_layouts_of_the_plain_step_agree(precision):
    """Rows and planes, replayed and resident: one set of bits."""
    from paper_1809_02390_gb300 import capi

    _, rho0 = _droplet(75, 60)
    states = []
    for layout in ("planes", "rows"):
        for mode in (0, 1):
            lat = lattice(rho0, precision, layout=layout, Tr=0.85, K_int=1.0)
            capi.lb_set_resident(lat.h, mode)
            assert capi.lb_step_form(lat.h, 80) == (capi.LB_STEP_RESIDENT if mode else capi.LB_STEP_PLAIN)
            lat.step(80)
            states.append(lat.state().clone())
    assert all(torch.equal(s, states[0]) for s in states[1:])
