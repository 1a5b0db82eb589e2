"""The reduced CG (mor_solve_reduced_noalloc) on caller-made block systems against a dense
solve: the edges of its work split.

Units of four rows (kq below, at and between multiples of four), one subdomain without
neighbours, fewer units than CTAs, the cluster launch and the launch on every SM, and
block rows with more neighbour columns than are staged at a time.  K = I + O with
||O||_2 <= 0.9, so K's condition number is at most 19; the CG stops at a relative
residual of 1e-13 and x is then within 19e-13 (plus rounding) of the solution: 1e-11.
"""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mor():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2404_06260_gb300 import _build
    _build.build()
    from paper_2404_06260_gb300 import mor as m
    return m


def _system(n, kq, nbrs, seed):
    """Dense K and its block-sparse form: block row i coupled to the nbrs next ones on
    either side of a ring."""
    rng = np.random.default_rng(seed)
    pairs = sorted({(min(i, (i + d) % n), max(i, (i + d) % n)) for i in range(n)
                    for d in range(1, nbrs + 1) if (i + d) % n != i})
    K, blocks, rows = np.zeros((n * kq, n * kq)), [], [[] for _ in range(n)]
    for i, j in pairs:
        B = rng.standard_normal((kq, kq))
        rows[i].append((j, len(blocks)))
        rows[j].append((i, len(blocks) + 1))
        blocks += [B, B.T]
        K[i * kq:(i + 1) * kq, j * kq:(j + 1) * kq] = B
        K[j * kq:(j + 1) * kq, i * kq:(i + 1) * kq] = B.T
    s = 0.9 / max(np.linalg.norm(K, 2), 1e-300) if pairs else 0.0
    K = s * K + np.eye(n * kq)
    blocks = np.ascontiguousarray(np.stack(blocks) * s) if blocks else np.zeros((1, kq, kq))
    ptr = np.cumsum([0] + [len(r) for r in rows]).astype(np.int32)
    flat = [e for r in rows for e in sorted(r)] or [(0, 0)]
    return K, blocks, ptr, np.array(flat, np.int32), rng.standard_normal(n * kq)


@pytest.mark.parametrize("n,kq,nbrs", [
    (1, 5, 0), (1, 1, 0), (2, 1, 1), (3, 4, 1), (5, 7, 2), (9, 12, 4), (27, 12, 6),
    (12, 33, 5), (40, 36, 7), (10, 128, 5), (30, 110, 14), (330, 3, 3)])
def test_reduced_solve_matches_dense(mor, n, kq, nbrs):
    import torch
    K, blocks, ptr, flat, b = _system(n, kq, nbrs, n * 1000 + kq)
    d = [torch.as_tensor(np.ascontiguousarray(a), device="cuda")
         for a in (ptr, flat[:, 0], flat[:, 1], blocks, b)]
    x = torch.full((n * kq,), float("nan"), dtype=torch.float64, device="cuda")
    P = [ctypes.c_void_p(t.data_ptr()) for t in d]
    info = mor.SolveInfo()
    st = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)

    def solve(max_iter):
        return mor._lib.mor_solve_reduced_noalloc(n, kq, *P, 1e-13, max_iter, st,
                                                  ctypes.c_void_p(x.data_ptr()),
                                                  ctypes.byref(info))

    ref = np.linalg.solve(K, b)
    for _ in range(2):   # the second call finds the first one's work space
        assert solve(500) == 0 and info.converged == 1
        assert np.linalg.norm(x.cpu().numpy() - ref) <= 1e-11 * np.linalg.norm(ref)
        assert abs(info.energy - b @ ref) <= 1e-11 * abs(b @ ref)
    if nbrs > 1:
        assert solve(2) == -4 and info.iterations == 2 and info.converged == 0
        assert np.isfinite(x.cpu().numpy()).all()
