"""The interface couplings a_uv, the blocks K~_ij = sum a_uv Q[u]^T Q[v] of the reduced
matrix and the energy norm against a plain binary64 assembly.

Every quantity is a sum of products in binary64, in another order than here: its error is at
most (number of terms) x 2^-53 x the sum of the absolute products.  An element coupling is
about 30 rounded operations, an entry has at most 24 elements and a block sum at most 32
terms per pass; 400 x 2^-53 covers them.  Shapes: one pair and many, 4 to 128 basis columns
(one slice of a block per pair to several, odd remainders), pairs with fewer entries than a
pass and with several passes, and a cylinder mesh of 24 elements around its axis edges (the
element lists of an entry hold 16).
"""
import numpy as np
import pytest

import synth

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


def _cube(n, parts):
    m = synth.kuhn_cube(n)
    return m.xyz, m.tets, m.dirichlet, synth.box_owner(n, parts)


def _cylinder(around, rings, layers, parts):
    """Prisms over a fan of triangles, cut into tetrahedra by ascending node number."""
    per = 1 + around * rings
    ang = 2 * np.pi * np.arange(around) / around
    disc = [(0.0, 0.0)] + [(r * np.cos(t), r * np.sin(t))
                           for r in range(1, rings + 1) for t in ang]
    tri = []
    for t in range(around):
        s = (t + 1) % around
        tri.append((0, 1 + t, 1 + s))
        for r in range(rings - 1):
            a, b = 1 + r * around, 1 + (r + 1) * around
            tri += [(a + t, b + t, b + s), (a + t, a + s, b + s)]
    xyz = np.array([(x, y, 0.7 * z) for z in range(layers) for x, y in disc])
    tets = []
    for z in range(layers - 1):
        for t in tri:
            i, j, k = sorted(t)
            lo, hi = z * per, (z + 1) * per
            tets += [(lo + i, lo + j, lo + k, hi + k), (lo + i, lo + j, hi + j, hi + k),
                     (lo + i, hi + i, hi + j, hi + k)]
    tets = np.array(tets, dtype=np.int32)
    e = xyz[tets[:, 1:]] - xyz[tets[:, :1]]
    flip = np.linalg.det(e) < 0
    tets[flip, 2:] = tets[flip, 3:1:-1]
    layer = np.arange(layers * per) // per
    dirichlet = np.isin(np.arange(layers * per) % per, range(per - around, per)).astype(np.uint8)
    return xyz, tets, dirichlet, (layer * parts // layers).astype(np.int32)


def _couplings(xyz, tets, kappa):
    """A and the sums of the absolute products it is made of (every product of the
    cofactors and of their dots taken absolutely)."""
    e = xyz[tets[:, 1:]] - xyz[tets[:, :1]]

    def cross(p, q, s):
        return np.stack([p[:, (i + 1) % 3] * q[:, (i + 2) % 3]
                         + s * p[:, (i + 2) % 3] * q[:, (i + 1) % 3] for i in range(3)], 1)

    def element(x, s):
        c = np.stack([cross(x[:, 1], x[:, 2], s), cross(x[:, 2], x[:, 0], s),
                      cross(x[:, 0], x[:, 1], s)], 1)
        g = np.concatenate([s * c.sum(1, keepdims=True), c], 1) / det[:, None, None]
        return np.einsum("tai,tbi->tab", g, g) * (kappa * det / 6)[:, None, None]

    det = np.einsum("ti,ti->t", e[:, 0], cross(e[:, 1], e[:, 2], -1))
    k, kabs = element(e, -1), element(np.abs(e), 1)
    n = len(xyz)
    A, Aabs = np.zeros((n, n)), np.zeros((n, n))
    for a in range(4):
        for b in range(4):
            np.add.at(A, (tets[:, a], tets[:, b]), k[:, a, b])
            np.add.at(Aabs, (tets[:, a], tets[:, b]), kabs[:, a, b])
    return A, Aabs


@pytest.mark.parametrize("mesh,rank,over", [
    (_cube(8, 2), 2, 1), (_cube(11, 3), 7, 2), (_cube(11, 2), 30, 5), (_cube(14, 2), 122, 5),
    (_cylinder(24, 3, 12, 2), 9, 3), (_cylinder(24, 3, 12, 3), 19, 3)])
def test_blocks_and_energy(mor, mesh, rank, over):
    import torch
    xyz, tets, dirichlet, owner = mesh
    rng = np.random.default_rng(5)
    kappa = np.exp(rng.standard_normal(len(tets)))
    sd = mor.Subdomains(mor.Mesh(xyz, tets, kappa, dirichlet), owner, 2)
    b = mor.Bases(sd, mor.basis_opts(rank=rank, oversample=over, seed=3, cg_rtol=1e-8))
    kq = b.kq
    assert kq >= rank
    K = mor.Reduced(sd, b).dense()
    A, Aabs = _couplings(xyz, tets, kappa)
    rows = [np.flatnonzero((owner == i) & (dirichlet == 0)) for i in range(sd.n_sub)]
    Q = [b.Q(i) for i in range(sd.n_sub)]
    pairs = 0
    for i in range(sd.n_sub):
        for j in range(sd.n_sub):
            if i == j:
                continue
            ij = np.ix_(rows[i], rows[j])
            pairs += np.abs(A[ij]).max() > 0
            got = K[i * kq:(i + 1) * kq, j * kq:(j + 1) * kq]
            bound = 400 * U * (np.abs(Q[i]).T @ Aabs[ij] @ np.abs(Q[j]))
            assert np.all(np.abs(got - Q[i].T @ A[ij] @ Q[j]) <= bound), (i, j)
    assert pairs > 0
    u1, u2 = rng.standard_normal((2, len(xyz)))
    dev = lambda x: torch.from_numpy(x).cuda()
    for got, d in ((mor.energy_norm(sd, dev(u1)), u1), (mor.energy_norm(sd, dev(u1), dev(u2)),
                                                        u1 - u2)):
        want = np.sqrt(d @ A @ d)
        assert abs(got - want) <= 400 * U * (np.abs(d) @ Aabs @ np.abs(d)) / want
