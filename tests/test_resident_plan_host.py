"""The cut of a lattice for resident runs, on the host: bounds on tiles, shared memory,
exchange words and the steps of one launch."""
import ctypes

import pytest


class Plan(ctypes.Structure):
    _fields_ = [(k, ctypes.c_int) for k in ("gx", "gy", "wmax", "hmax", "pitch", "threads")] + [
        ("smem", ctypes.c_uint), ("words", ctypes.c_size_t), ("steps", ctypes.c_int)]


@pytest.fixture(scope="module")
def plan():
    from paper_1809_02390_gb300 import build as b

    b.build()
    from paper_1809_02390_gb300 import capi

    f = ctypes.CDLL(capi.lib()._name)["_ZN3lbm8res_planEiiiPNS_7ResPlanE"]  # lbm::res_plan
    f.restype = ctypes.c_bool

    def call(nx, ny, precision):
        p = Plan()
        return p if f(nx, ny, precision, ctypes.byref(p)) else None

    return call


@pytest.mark.parametrize("precision", [0, 1, 2])
def test_cuts_stay_within_their_bounds(plan, precision):
    sides = [3, 5, 17, 64, 100, 203, 256, 301, 409, 410, 512, 583]
    seen = 0
    for nx in sides + [1024, 5000]:
        for ny in sides + [1024, 5000]:
            p = plan(nx, ny, precision)
            if p is None:
                continue
            seen += 1
            assert p.gx * p.gy <= 152 and p.gx * p.wmax >= nx and p.gy * p.hmax >= ny
            assert (p.gx == 1 or nx // p.gx >= 4) and (p.gy == 1 or ny // p.gy >= 4)
            assert p.smem <= 226 * 1024 and p.pitch >= p.wmax + 4 and p.threads % 32 == 0
            assert p.words == p.gx * p.gy * 6 * (p.wmax + p.hmax) * (2 if precision == 0 else 1)
    assert seen > 100


def test_a_launch_is_bounded_by_time(plan):
    """About 5 ms a launch at 2 GHz: a warp of FP64 nodes takes 64 cycles of a scheduler an
    instruction and some 235 instructions a step (15,000 cycles per round of four warps)."""
    for n in (48, 64, 200, 300, 410):
        p = plan(n, n, 0)
        rounds = -(-(-(-p.wmax * p.hmax // 32)) // 4)
        assert p.steps % 2 == 0 and 16 <= p.steps <= 4096
        assert p.steps * rounds * 15000 <= 1.0e7 * 1.01
    for n in (3, 64, 256, 512, 583):
        p = plan(n, n, 1)
        assert p.steps % 2 == 0 and 1000 <= p.steps <= 4096
