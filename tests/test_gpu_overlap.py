"""Steps whose launches overlap the end of their predecessor: a run of single steps,
with other work on the buffers between some of them, gives the bits of the run that a
caller captures (whose launches are ordinary ones)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _lattice(kind, precision, shape):
    from paper_1809_02390_gb300 import Lattice, Lattice3

    rng = np.random.default_rng(5)
    rho = 3.8 * (1 + 0.01 * rng.uniform(-1, 1, shape))
    kw = dict(Tr=0.8, K_int=1.2)
    return Lattice(rho, precision=precision, **kw) if kind == 2 else Lattice3(rho, precision=precision, **kw)


@pytest.mark.parametrize("kind,precision,shape", [
    (2, "fp64", (33, 40)), (2, "fp32", (517, 1003)), (2, "fp32", (9, 7)), (2, "fp32", (1024, 1024)),
    (2, "fp16s", (1000, 1200)), (3, "fp32", (24, 40, 72)), (3, "fp32", (12, 31, 33)), (3, "fp64", (12, 31, 33))])
def test_overlapping_launches_equal_ordinary_ones(kind, precision, shape):
    from paper_1809_02390_gb300 import build

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    states = []
    for captured in (False, True):
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            lat = _lattice(kind, precision, shape)
            for _ in range(4):
                if captured:
                    s.synchronize()
                    g = torch.cuda.CUDAGraph()
                    with torch.cuda.graph(g, stream=s):
                        for _ in range(6):
                            lat.step(1)
                    g.replay()
                else:
                    for _ in range(6):
                        lat.step(1)
                # Other work that reads and rewrites the buffer, right behind the last step.
                f = lat.state()
                f.copy_(f.flip(-1).clone())
            states.append(lat.state().clone())
            s.synchronize()
            lat.close()
    assert torch.equal(*states)
