"""Plain fused step of lattices with more rows of tiles than a grid has in y (65,535 of
eight rows).  A lattice that repeats a 3 x 3 one stays its repetition, bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("ny", [524_280, 524_289, 1_048_560])
def test_tall_lattice_repeats_a_small_one(precision, ny):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1809_02390_gb300 import Lattice, capi

    rho = 2.0 + 0.05 * np.random.default_rng(5).uniform(-1, 1, (3, 3))
    kw = dict(precision=precision, Tr=0.85, rho_ref=2.0)
    small, tall = Lattice(rho, **kw), Lattice(np.tile(rho, (ny // 3, 1)), **kw)
    assert capi.lb_step_form(tall.h, 3) == capi.LB_STEP_PLAIN
    for n in (1, 3, 66):  # single launches, and a graph
        tall.step(n)
        for _ in range(n):
            small.step(1)
        assert torch.equal(tall.state(), small.state().repeat(1, ny // 3, 1)), n
