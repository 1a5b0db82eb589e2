"""Batched dense Cholesky (mor_explicit.cu: 64-column panels, 32-row panel blocks) and the
triangular solves of the explicit SVD (two vectors per warp) at orders around their tiles,
against the oracle's LAPACK factors.

A Cholesky factor computed in binary64 is exact for a matrix perturbed by at most
(n + 1) 2^-53 of |L||L^T|, which moves it by that times the condition number: 4 n 2^-53
cond(H^+) bounds the difference of two such factors relative to their norm.  The explicit
singular values keep the 1e-10 sigma_1 of the 16^3 comparison (smaller systems here).
Orders: below one panel, one panel exactly and one row more, several panels with ragged
ends, subdomains of different orders, odd and even numbers of vectors.
"""
import numpy as np
import pytest

import synth
from oracle import basis as obasis
from oracle import pipeline
from oracle import subdomains as osub

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mor():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2404_06260_gb300 import _build
    _build.build()
    from paper_2404_06260_gb300 import mor as m
    return m


# slabs > 0: that many slabs, every subdomain with a non-empty B; 0: five k-means parts
@pytest.mark.parametrize("n,slabs,hops", [(5, 2, 1), (6, 3, 1), (7, 3, 1), (9, 2, 1), (9, 3, 1),
                                          (9, 0, 1), (9, 0, 2)])
def test_cholesky_and_explicit_svd(mor, n, slabs, hops):
    mesh = synth.kuhn_cube(n)
    kappa = synth.lognormal_kappa(mesh.n_tets, 17)
    owner = synth.slab_owner(n, slabs) if slabs else synth.kmeans_owner(mesh, 5, 3)
    sd = mor.Subdomains(mor.Mesh(mesh.xyz, mesh.tets, kappa, mesh.dirichlet), owner, hops)
    b = mor.Bases(sd, mor.basis_opts(rank=3, oversample=2, seed=4, precision="fp64",
                                     cg_rtol=1e-13, sketch="paper"))
    for i in range(sd.n_sub):
        loc = obasis.local_system(mesh, kappa, osub.subdomain_sets(mesh, owner, i, hops))
        H = loc["H_plus"].toarray() if hasattr(loc["H_plus"], "toarray") else loc["H_plus"]
        ref = obasis.rbb_cholesky(loc["H_plus"], loc["nI"])
        got = b.rbb(i)
        assert np.all(np.tril(got, -1) == 0.0)
        tol = 4 * len(H) * 2.0 ** -53 * np.linalg.cond(H)
        assert np.linalg.norm(got - ref) <= tol * np.linalg.norm(ref), (i, len(H))
    ref = pipeline.run(mesh, kappa, owner, 3, 0, hops, 4, explicit=True, fe_solution=False)
    e = mor.Bases(sd, mor.basis_opts(rank=3, oversample=0, seed=4, precision="fp64",
                                     explicit_svd=1))
    sig = e.sigma()
    for i, ob in enumerate(ref["bases"]):
        m = min(9, len(ob["sigma"]))
        assert np.max(np.abs(sig[i, :m] - ob["sigma"][:m])) <= 1e-10 * ob["sigma"][0], i
