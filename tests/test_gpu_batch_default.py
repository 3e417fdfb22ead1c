"""The launch form a batch starts with (chosen by the size of its pool) gives each
lattice the single-lattice trajectory, on both sides of the rule."""
import pytest

from paper_1809_02390_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("sizes,tickets", [([(64, 64), (33, 45)], False), ([(1200, 1100), (40, 17)], False),
                                           ([(1300, 1200), (33, 45), (64, 64)], True)])
def test_the_default_form_equals_single_lattices(sizes, tickets):
    from paper_1809_02390_gb300 import Batch, Lattice, build, derive

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    rhos = []
    for k, (nx, ny) in enumerate(sizes):
        d = derive(nx, ny, Tr=0.8)
        rhos.append(inputs.spinodal(nx, ny, 0.5 * (d["rho_g"] + d["rho_l"]), 0.01, k))
    b = Batch(rhos, [dict(Tr=0.8) for _ in rhos])
    assert b.config()["tensor_copies"] == tickets
    b.run(5)
    b.status()
    for i, r in enumerate(rhos):
        lat = Lattice(r, precision="fp32", Tr=0.8)
        lat.step(5)
        assert torch.equal(b.state(i), lat.state()), i
        lat.close()
    b.close()
