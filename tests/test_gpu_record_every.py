"""Distances between recorded states beyond the run, and checkpoint distances that mean
"none": accepted whatever their size, as a plain run."""
import pytest

from paper_1809_02390_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("every", [6, 2 ** 31 - 1, 2 ** 31, 2 ** 40, 2 ** 62])
@pytest.mark.parametrize("steps", [5, 30])
def test_distances_beyond_the_run(every, steps):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1809_02390_gb300 import Lattice, capi

    a, b = (Lattice(inputs.droplet(96, 64, 20, 5, 1.0, 6.0), Tr=0.85) for _ in range(2))
    rec = torch.zeros((max(1, steps // every), *a.f_a.shape), device="cuda")
    capi.lb_step_record(a.h, steps, every, rec.data_ptr() if steps >= every else 0)
    b.step(steps)
    assert torch.equal(a.buffer(), b.buffer()) and a.steps_done == steps


@pytest.mark.parametrize("every", [40, 40.0, 2 ** 31, 10 ** 15])
def test_rollout_without_checkpoints(every):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1809_02390_gb300 import adjoint

    spec = adjoint.RolloutSpec(48, 32, precision="fp64", Tr_ref=0.85)
    theta = [0.85, spec.G2_ref, 1.0]
    f0 = adjoint.initial_state(spec, inputs.droplet(48, 32, 10, 5, spec.rho_g, spec.rho_l), theta)
    grads = []
    for e in (every, None):
        t = torch.tensor(theta, dtype=torch.float64, requires_grad=True)
        out = adjoint.rollout(t, f0, spec, 30, e)
        (out ** 2).sum().backward()
        grads.append((out.detach(), t.grad))
    assert torch.equal(grads[0][0], grads[1][0])
    assert torch.allclose(grads[0][1], grads[1][1], rtol=1e-9)
