"""The eigensolver of step 2 (mor_debug_sym_eig) against LAPACK, at the orders where its
kernels change (8 E rows per column, one CTA / a cluster, factor in shared / global memory).

G = X^T X with singular values of X from 1 down to 1e-6 in random directions.  LAPACK's and
the solver's eigenvalues both carry the backward error of a binary64 factorisation, at most
about n 2^-53 ||G||: 4 n 2^-53 covers the two.  The residual ||G V - V diag(ev)|| has the
same bound; V is orthonormal to the rotation threshold, sqrt(n) 2^-53 per pair, so
||V^T V - I||_F <= n^(3/2) 2^-53, times 4 for the normalisation and the sweeps.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


@pytest.fixture(scope="module")
def mor():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2404_06260_gb300 import _build
    _build.build()
    from paper_2404_06260_gb300 import mor as m
    return m


def _gram(n, rng, smallest=1e-6):
    Q = np.linalg.qr(rng.standard_normal((n, n)))[0]
    s = np.logspace(0, np.log10(smallest), n) if n > 1 else np.ones(1)
    X = (rng.permutation(s)[:, None] * Q)
    return X.T @ X


def _solve(mor, G):
    import torch
    ev, V = mor.sym_eig(torch.as_tensor(np.ascontiguousarray(G), device="cuda"))
    return ev.cpu().numpy(), V.cpu().numpy()


@pytest.mark.parametrize("n,batch", [
    (1, 3), (2, 2), (7, 1), (16, 5), (17, 2), (43, 4), (64, 2), (80, 3), (97, 2), (128, 2),
    (129, 3), (200, 40), (425, 2), (513, 1), (1024, 1)])
def test_against_lapack(mor, n, batch):
    rng = np.random.default_rng(n)
    G = np.stack([_gram(n, rng) * 10.0 ** (3 * b - 3) for b in range(batch)])
    ev, V = _solve(mor, G)
    for g, e, v in zip(G, ev, V):
        top = np.linalg.norm(g, 2)
        ref = np.linalg.eigvalsh(0.5 * (g + g.T))[::-1]
        assert np.all(np.diff(e) <= 0)
        assert np.abs(e - ref).max() <= 4 * n * U * top
        assert np.linalg.norm(g @ v - v * e, 2) <= 4 * n * U * top
        assert np.linalg.norm(v.T @ v - np.eye(n)) <= 4 * n ** 1.5 * U


@pytest.mark.parametrize("n", [12, 60, 200])
def test_graded_null_and_nonfinite(mor, n):
    """Graded columns keep relative accuracy, null columns and a rank deficiency complete
    the basis with eigenvalue 0, and a NaN comes back as NaN."""
    rng = np.random.default_rng(n)
    d = np.logspace(0, -9, n)
    C = np.eye(n) + 0.1 / n * rng.standard_normal((n, n))
    C = 0.5 * (C + C.T)          # well conditioned: D C D has relatively accurate eigenvalues
    G = d[:, None] * C * d
    ref = np.sort(np.linalg.svd(np.linalg.cholesky(C).T * d, compute_uv=False) ** 2)[::-1]
    low = np.zeros((n, n))       # rank 5, and two null columns
    X = rng.standard_normal((5, n))
    X[:, [1, n - 2]] = 0.0
    low[:] = X.T @ X
    ev, V = _solve(mor, np.stack([G, low]))
    # scaled condition number < 2: Cholesky and Jacobi are relatively accurate to about
    # n 2^-53; the reference SVD to n 2^-53 of each row-graded singular value
    top = ref > 2.0 ** -60 * ref[0]
    assert np.abs(ev[0][top] / ref[top] - 1).max() <= 16 * n * U
    s = np.linalg.svd(X, compute_uv=False) ** 2
    assert np.abs(ev[1][:5] - s).max() <= 4 * n * U * s[0]
    assert np.all(ev[1][5:] <= 4 * n * U * s[0])
    assert np.linalg.norm(V[1].T @ V[1] - np.eye(n)) <= 4 * n ** 1.5 * U
    low[0, 3] = low[3, 0] = np.nan
    assert np.isnan(_solve(mor, low[None])[0]).all()
