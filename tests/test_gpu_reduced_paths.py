"""The allocation-free reduced solve's choice of launch: it does not know the neighbour lists,
which are on the device, so it tries one cluster by a guess of nine neighbours per block row;
a matrix that has more and does not fit there takes a second launch, on every SM, and every
one that fits (or is large by the guess) a single one.  Solutions as in
test_gpu_reduced_solve: condition number at most 19, residual 1e-13, 1e-11.
"""
import ctypes

import numpy as np
import pytest

from test_gpu_reduced_solve import _system, mor  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,kq,nbrs,launches", [
    (27, 12, 6, 1), (64, 12, 4, 1), (64, 12, 10, 2), (70, 12, 12, 2), (40, 36, 7, 1),
    (90, 12, 10, 1)])
def test_launches_and_solution(mor, n, kq, nbrs, launches):  # noqa: F811
    import torch
    K, blocks, ptr, flat, b = _system(n, kq, nbrs, n + kq)
    d = [torch.as_tensor(np.ascontiguousarray(a), device="cuda")
         for a in (ptr, flat[:, 0], flat[:, 1], blocks, b)]
    x = torch.full((n * kq,), float("nan"), dtype=torch.float64, device="cuda")
    info, ref = mor.SolveInfo(), np.linalg.solve(K, b)
    for _ in range(2):
        n0 = mor.kernel_launches()
        rc = mor._lib.mor_solve_reduced_noalloc(
            n, kq, *[ctypes.c_void_p(t.data_ptr()) for t in d], 1e-13, 500, None,
            ctypes.c_void_p(x.data_ptr()), ctypes.byref(info))
        assert rc == 0 and info.converged == 1
        assert mor.kernel_launches() - n0 == launches
        assert np.linalg.norm(x.cpu().numpy() - ref) <= 1e-11 * np.linalg.norm(ref)
        assert abs(info.energy - b @ ref) <= 1e-11 * abs(b @ ref)
