"""The eigensolver of step 2 on matrices whose columns differ by many orders of magnitude,
with and without a rank deficiency: eigenvalues keep their relative accuracy however small
they are, and the eigenvectors stay orthonormal.

Eigenvalues: G = D C D with C within 0.3 of I in norm, so Cholesky and one-sided Jacobi are
relatively accurate to about n 2^-53 (Demmel & Veselic), and so are the singular values of
chol(C)^T D by LAPACK only where the rows are ordered by size; the reference is therefore a
one-sided Jacobi in long double on the same factor, exact here.  16 n 2^-53 for the two.
Orthogonality: every pair ends at sqrt(n) 2^-53, so ||V^T V - I||_F <= n^(3/2) 2^-53, times 4
for the normalisation and the sweeps.  Residual: 4 n 2^-53 ||G||.
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


def _solve(mor, G):
    import torch
    ev, V = mor.sym_eig(torch.as_tensor(np.ascontiguousarray(G), device="cuda"))
    return ev.cpu().numpy(), V.cpu().numpy()


def _eigenvalues(C, d):
    """Eigenvalues of D C D, descending, by Cholesky and one-sided Jacobi in long double."""
    n = len(d)
    L = np.zeros((n, n), np.longdouble)
    A = C.astype(np.longdouble)
    for j in range(n):
        L[j:, j] = A[j:, j] / np.sqrt(A[j, j])
        A[j + 1:, j + 1:] -= np.outer(L[j + 1:, j], L[j + 1:, j])
    order = np.argsort(-d, kind="stable")  # large rows first: few sweeps
    W = (L * d.astype(np.longdouble)[:, None])[order].T.copy().T  # rows to be made orthogonal
    m = n + n % 2
    W = np.vstack([W, np.zeros((m - n, n), np.longdouble)])
    idx = np.arange(m)
    for _ in range(30):
        worst = 0.0
        for _ in range(m - 1):
            p, q = idx[:m // 2], idx[m // 2:][::-1]
            a, b = W[p], W[q]
            pq, pp, qq = (a * b).sum(1), (a * a).sum(1), (b * b).sum(1)
            prod = pp * qq
            cos = np.where(prod > 0, np.abs(pq) / np.sqrt(np.where(prod > 0, prod, 1)), 0)
            worst = max(worst, float(cos.max()))
            rot = cos > 2.0 ** -58
            tau = np.where(rot, (qq - pp) / np.where(rot, 2 * pq, 1), 0)
            t = np.where(rot, np.where(tau >= 0, 1, -1) / (np.abs(tau) + np.sqrt(1 + tau * tau)), 0)
            c = 1 / np.sqrt(1 + t * t)
            W[p], W[q] = (c[:, None] * a - (c * t)[:, None] * b, (c * t)[:, None] * a + c[:, None] * b)
            idx = np.concatenate([idx[:1], idx[-1:], idx[1:-1]])
        if worst <= 2.0 ** -58:
            break
    return np.sort((W * W).sum(1))[::-1][:n]


def _check(G, e, v):
    n = len(G)
    top = np.linalg.norm(G, 2)
    assert np.all(np.diff(e) <= 0) and e[-1] >= 0
    assert np.linalg.norm(v.T @ v - np.eye(n)) <= 4 * n ** 1.5 * U
    assert np.linalg.norm(G @ v - v * e, 2) <= 4 * n * U * top


# orders of the one-CTA kernel and of the clusters
@pytest.mark.parametrize("n", [12, 47, 60, 129])
@pytest.mark.parametrize("decades", [12, 20, 60])
def test_small_eigenvalues_keep_their_relative_accuracy(mor, n, decades):
    rng = np.random.default_rng(n + decades)
    C = rng.standard_normal((n, n))
    C = np.eye(n) + 0.15 * (C + C.T) / np.linalg.norm(C + C.T, 2)
    d = rng.permutation(np.logspace(0, -decades, n))
    d = 2.0 ** np.round(np.log2(d))     # D C D is then exact
    G = d[:, None] * C * d
    ref = _eigenvalues(C, d)
    ev, V = _solve(mor, G[None])
    assert np.abs(ev[0] / ref - 1).max() <= 16 * n * U
    _check(G, ev[0], V[0])


@pytest.mark.parametrize("n,rank", [(12, 5), (47, 9), (60, 20), (129, 43), (261, 60)])
@pytest.mark.parametrize("last", [30, 80])
def test_graded_and_rank_deficient(mor, n, rank, last):
    rng = np.random.default_rng(n * rank + last)
    few, smooth = np.ones(n), 2.0 ** np.round(np.linspace(0, -last, n))
    few[-max(5, n // 4):] = 2.0 ** -last
    null = smooth.copy()
    null[[1, n - 2]] = 0.0
    for d in (few, smooth, null):
        X = rng.standard_normal((rank, n)) * d
        G = X.T @ X
        ev, V = _solve(mor, G[None])
        _check(G, ev[0], V[0])
        s = np.linalg.svd(X, compute_uv=False) ** 2
        assert np.abs(ev[0][:rank] - s).max() <= 4 * n * U * s[0]
