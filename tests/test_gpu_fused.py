"""The plain fused step (8-row tiles) against other kernels of the same arithmetic: the
same bits at the edges of its tiles and on both sides of the rule that prefers it on
small lattices."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1809_02390_gb300 import build

    build.build()


def _rho(nx, ny):
    return 3.8 * (1 + 0.02 * np.random.default_rng(nx + ny).uniform(-1, 1, (ny, nx)))


@pytest.mark.parametrize("nx,ny", [(9, 7), (31, 7), (32, 8), (33, 9), (65, 15), (64, 17), (97, 23), (301, 250)])
def test_equals_the_batch_step(nx, ny):
    """The batch's persistent form steps 16-row tiles with the same tile code."""
    from paper_1809_02390_gb300 import Batch, Lattice

    lat = Lattice(_rho(nx, ny), precision="fp32", Tr=0.8)
    b = Batch([_rho(nx, ny)], [dict(Tr=0.8)])
    b.set_config(0, 1)
    for _ in range(5):
        lat.step(1)  # (a call of one step never runs resident)
    b.run(5)
    assert torch.equal(lat.state(), b.state(0))
    b.close()
    lat.close()


@pytest.mark.parametrize("precision,nx,ny", [("fp32", 104, 50), ("fp32", 512, 300), ("fp32", 1024, 1000),
                                             ("fp32", 1500, 1200), ("fp16s", 208, 100), ("fp16s", 1600, 1000)])
@pytest.mark.parametrize("layout", ["planes", "rows"])
def test_equals_the_tensor_copy_step(precision, nx, ny, layout):
    from paper_1809_02390_gb300 import Lattice, capi

    a, b = (Lattice(_rho(nx, ny), precision=precision, layout=layout, Tr=0.8) for _ in range(2))
    assert capi.lb_uses_tma(a.h)
    capi.lb_set_tile_dispatch(b.h, True)
    for n in (1, 2, 3, 1):
        a.step(n)
        b.step(n)
    assert torch.equal(a.buffer(), b.buffer())
    capi.lb_status(b.h)
    a.close()
    b.close()


@pytest.mark.parametrize("layout", ["planes", "rows"])
def test_half_tiles_of_a_batch(layout):
    """One block per tile in the 80-register form takes 8-row halves of the 16-row tiles:
    lattices whose last tile is a half, part of one or whole."""
    from paper_1809_02390_gb300 import Batch, Lattice

    sizes = [(33, 8), (40, 9), (64, 16), (31, 17), (65, 24), (130, 31)]
    b = Batch([_rho(*s) for s in sizes], [dict(Tr=0.8, layout=layout) for _ in sizes])
    b.set_config(1, 0)
    b.run(64 + 3)
    for i, s in enumerate(sizes):
        lat = Lattice(_rho(*s), precision="fp32", Tr=0.8)
        lat.step(64 + 3)
        assert torch.equal(b.state(i), lat.state()), s
        lat.close()
    b.close()


@pytest.mark.parametrize("nx,ny,n,tickets", [(130, 100, 120, False), (900, 800, 3, True)])
def test_default_form_of_a_large_pool(nx, ny, n, tickets):
    """Above 100 MB: tickets only if most tiles lie inside their lattices."""
    from paper_1809_02390_gb300 import Batch, Lattice

    b = Batch([_rho(nx, ny)] * n, [dict(Tr=0.8) for _ in range(n)])
    assert b.config()["tensor_copies"] == tickets
    b.run(3)
    lat = Lattice(_rho(nx, ny), precision="fp32", Tr=0.8)
    lat.step(3)
    for i in (0, n // 2, n - 1):
        assert torch.equal(b.state(i), lat.state())
    b.close()
    lat.close()
