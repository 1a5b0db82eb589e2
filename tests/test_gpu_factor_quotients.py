"""The quotients of the dense triangular solves of step 2 (a rounded reciprocal and one
correction step) against true ones: systems of order one, x = b / d, over the range of binary64.

The correction leaves at most one unit in the last place; numpy's quotient is correctly
rounded, so they differ by at most one spacing.  Where the reciprocal or the remainder
leaves the normal numbers, and for infinities and NaN, the solve divides: bit for bit.
"""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
TRSV = "_ZN3mor16launch_trsv_colsEiiiPKdPKlPKiS5_S5_PdS3_iS5_iP11CUstream_st"


def _solve(b, d):
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2404_06260_gb300 import _build
    lib, n = ctypes.CDLL(_build.build()), len(b)
    x, T = (torch.as_tensor(np.array(v), device="cuda") for v in (b, d))
    idx = torch.arange(n, dtype=torch.int64, device="cuda")
    one = torch.ones(n, dtype=torch.int32, device="cuda")
    zero = torch.zeros(n, dtype=torch.int32, device="cuda")
    p = [ctypes.c_void_p(t.data_ptr()) for t in (T, idx, one, one, zero, x, idx)]
    getattr(lib, TRSV)(n, 1, 1, *p, 1, ctypes.c_void_p(one.data_ptr()), 1, None)
    torch.cuda.synchronize()
    return x.cpu().numpy()


def _draw(rng, n, lo, hi):
    return np.ldexp(rng.uniform(1.0, 2.0, n) * rng.choice([-1.0, 1.0], n),
                    rng.integers(lo, hi + 1, n))


@pytest.mark.parametrize("lo,hi", [(-8, 8), (-500, 500), (-1021, 1021)])
def test_within_one_unit_in_the_last_place(lo, hi):
    rng = np.random.default_rng(hi)
    b, d = _draw(rng, 200000, lo, hi), _draw(rng, 200000, lo, hi)
    b[:100] = 0.0
    d[100:200] = b[100:200]
    with np.errstate(over="ignore", under="ignore"):
        want = b / d
    got = _solve(b, d)
    fin = np.isfinite(want)
    assert np.array_equal(got[~fin], want[~fin])
    assert np.all(np.abs(got[fin] - want[fin]) <= np.spacing(np.abs(want[fin])))


def test_divides_outside_the_range_of_the_correction():
    rng = np.random.default_rng(3)
    tiny = np.ldexp(rng.uniform(0.001, 0.9, 1000), -1022)        # subnormal pivots
    d = np.concatenate([tiny, _draw(rng, 1000, 1022, 1023), _draw(rng, 1000, -1000, -960),
                        np.full(3, 2.0), [np.inf, np.nan, 0.0]])
    b = np.concatenate([_draw(rng, 1000, -1000, -900), _draw(rng, 1000, 0, 1000),
                        _draw(rng, 1000, -1020, -960), [np.inf, -np.inf, np.nan], [1.0, 1.0, 1.0]])
    with np.errstate(all="ignore"):
        want = b / d
    got = _solve(b, d)
    assert np.array_equal(got, want, equal_nan=True)
