"""Resident runs take nothing from what their scratch buffer held before: handles that share
one in turn (which lb_init allows to all but concurrent ones), and exchange words planted
with every number a run's steps carry, give the bits of handles with a buffer of their own."""
import numpy as np
import pytest

from paper_1809_02390_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

PRECISION = {"fp64": (0, torch.float64, 8), "fp32": (1, torch.float32, 4), "fp16s": (2, torch.float16, 4)}


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1809_02390_gb300 import build

    build.build()


class Handle:
    def __init__(self, nx, ny, precision, scratch=None, seed=3):
        from paper_1809_02390_gb300 import capi

        code, dtype, self.real_bytes = PRECISION[precision]
        p = capi.make_params(nx, ny, precision=code, Tr=0.85, rho_ref=0.0 if precision == "fp64" else 3.0)
        assert p.precision == code
        rho = inputs.droplet(nx, ny, min(nx, ny) / 4, 5, 1.0, 6.0, center=(0.37 * nx, 0.58 * ny))
        rho = torch.from_numpy(rho * (1 + 0.01 * (2 * inputs.uniform(seed, nx * ny).reshape(ny, nx) - 1))).cuda()
        self.size = capi.lb_scratch_bytes(p)
        # One density plane, the reduction workspace, the tile tickets; then the exchange words.
        self.mail = (nx * ny * self.real_bytes + 255) // 256 * 256 + 65536 + 256 + 256
        self.scratch = torch.zeros(self.size, dtype=torch.uint8, device="cuda") if scratch is None else scratch
        self.f = [torch.empty((9, ny, nx), dtype=dtype, device="cuda") for _ in range(2)]
        self.h = capi.lb_init(p, self.f[0].data_ptr(), self.f[1].data_ptr(), self.scratch.data_ptr(), self.size,
                              rho.data_ptr(), True, torch.cuda.current_stream().cuda_stream)

    def step(self, n):
        from paper_1809_02390_gb300 import capi

        capi.lb_step(self.h, n)

    def state(self):
        from paper_1809_02390_gb300 import capi

        capi.lb_status(self.h)
        return self.f[0] if capi.lb_state(self.h) == self.f[0].data_ptr() else self.f[1]

    def close(self):
        from paper_1809_02390_gb300 import capi

        capi.lb_free(self.h)


# Calls on two handles in turn whose step counts make the words that one leaves carry the
# numbers that the other waits for.
TURNS = {"fp64": [(0, 4), (1, 4), (0, 5), (1, 4), (0, 4), (1, 7)],
         "fp32": [(1, 20), (0, 12), (0, 12), (1, 12), (0, 13), (1, 14)],
         "fp16s": [(1, 20), (0, 12), (0, 12), (1, 12), (0, 13), (1, 14)]}


@pytest.mark.parametrize("precision", sorted(TURNS))
@pytest.mark.parametrize("sizes", [((64, 48), (64, 48)), ((200, 120), (200, 120)), ((128, 96), (150, 101))])
def test_two_handles_share_a_scratch_buffer_in_turn(precision, sizes):
    own = [Handle(*s, precision, seed=3 + k) for k, s in enumerate(sizes)]
    both = torch.zeros(max(h.size for h in own), dtype=torch.uint8, device="cuda")
    shared = [Handle(*s, precision, scratch=both, seed=3 + k) for k, s in enumerate(sizes)]
    for _ in range(20):
        for k, n in TURNS[precision]:
            own[k].step(n)
            shared[k].step(n)
    for a, b in zip(own, shared):
        assert torch.equal(a.state(), b.state())
        a.close()
        b.close()


@pytest.mark.parametrize("precision", sorted(TURNS))
def test_planted_words_are_not_read(precision):
    a, b = (Handle(64, 48, precision) for _ in range(2))
    assert b.size > b.mail  # the exchange words are there
    n = 12
    for number in range(0, 3 * n):
        b.scratch[b.mail:].view(torch.int32).fill_(number)
        a.step(n)
        b.step(n)
        assert torch.equal(a.state(), b.state()), number
    a.close()
    b.close()
