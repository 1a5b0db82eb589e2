"""When the local CG runs on chip (resident_plan, a host function): never in more waves of
clusters than were measured to pay, for every cluster size the rule can pick.  The limits
are the measured break-even points between on-chip and streaming builds."""
import ctypes

import pytest

SMS = 152


class _Plan(ctypes.Structure):
    _fields_ = [("S", ctypes.c_int), ("smem", ctypes.c_size_t)]


@pytest.fixture(scope="module")
def plan():
    from paper_2404_06260_gb300 import _build
    lib = ctypes.CDLL(_build.build())
    fn = {}
    for t, c in ((8, "d"), (4, "f")):
        fn[t] = getattr(lib, "_ZN3mor13resident_planI%sEENS_12ResidentPlanEiiiii" % c)
        fn[t].restype = _Plan
    return lambda t, *a: fn[t](*a)


# (bytes of the working precision, CTAs per subdomain): waves up to which on-chip builds were
# measured faster, and from which on slower
BREAK_EVEN = {(8, 1): (11.4, 13.3), (8, 2): (13.5, 22), (8, 4): (6.7, 13.5), (8, 8): (5.7, 11.4),
              (4, 1): (13.5, 18.0), (4, 2): (23, 37.1), (4, 4): (11.9, 22.1), (4, 8): (5.7, 11.4)}


@pytest.mark.parametrize("size", [8, 4])
def test_waves_stay_below_the_break_even(plan, size):
    seen = {}
    for rows in (150, 398, 724, 1100, 1331, 2200, 3375, 4600):
        for n_sd in (1, 2, 8, 27, 64, 125, 216, 343, 512, 1000, 4000):
            for kp in (4, 8, 16, 32, 52, 80):
                p = plan(size, n_sd, rows, 15, 40, kp)
                if p.S == 0:
                    continue
                assert p.S in (1, 2, 4, 8) and 0 < p.smem <= 227 * 1024
                waves = p.S * n_sd * (kp * size // 16) / SMS
                seen[p.S] = max(seen.get(p.S, 0), waves)
    assert set(seen) == {1, 2, 4, 8}
    for S, waves in seen.items():
        assert waves < BREAK_EVEN[size, S][1], (S, waves)


@pytest.mark.parametrize("size", [8, 4])
def test_few_waves_run_on_chip(plan, size):
    for n_sd, kp in ((1, 4), (8, 16), (27, 16), (64, 8)):
        assert plan(size, n_sd, 398, 15, 12, kp).S >= 1
