"""The on-chip CG of small subdomains (mor_resident.cu) against the streaming kernels, which
run whenever kernel timing is on (mor_profile_enable).

Both run the same recursion with the same convergence test (cg_rtol of the largest
right-hand side, by the binary64 residual), so their solutions differ by the solver
tolerance: cg_rtol = 1e-10 moves the singular values by less than 1e-7 of the largest and
the reduced energy, quadratic in a basis error, by less than 1e-8.  Rounding changes the
step at which a column passes its test by a few steps; a replacement interval (40) bounds
what that does to the counts.  Shapes: one row per warp and several rows per thread, one to
eight CTAs per subdomain, uneven subdomains, packs of closed padding columns, no coarse
level, both precisions.
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mor():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2404_06260_gb300 import _build
    _build.build()
    from paper_2404_06260_gb300 import mor as m
    return m


def _run(mor, sd, streaming, **kw):
    mor.profile(streaming)
    mor.profile_reset()
    try:
        n0 = mor.kernel_launches()
        b = mor.Bases(sd, mor.basis_opts(seed=9, cg_rtol=1e-10, **kw))
        n1 = mor.kernel_launches()
    finally:
        mor.profile(False)
    assert b.converged
    return b.sigma(), mor.Reduced(sd, b).solve(rtol=1e-13)[1]["energy"], b.stats(), n1 - n0


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("n,parts,hops,rank,over,rows,kind", [
    (6, 2, 1, 2, 1, -1, "box"), (11, 2, 3, 5, 2, -1, "box"), (16, 2, 4, 8, 5, 0, "box"),
    (20, 3, 4, 9, 7, -1, "box"), (20, 8, -1, 6, 4, 60, "kmeans"), (23, 2, 4, 11, 4, -1, "box"),
    (22, 2, 4, 3, 1, 34, "box")])
def test_resident_against_streaming(mor, prec, n, parts, hops, rank, over, rows, kind):
    mesh = synth.kuhn_cube(n)
    kappa = synth.lognormal_kappa(mesh.n_tets, 31)
    owner = (synth.box_owner(n, parts) if kind == "box" else
             synth.kmeans_owner(mesh, parts, 3))
    sd = mor.Subdomains(mor.Mesh(mesh.xyz, mesh.tets, kappa, mesh.dirichlet), owner, hops)
    kw = dict(rank=rank, oversample=over, precision=prec, coarse_rows=rows)
    s0, e0, st0, l0 = _run(mor, sd, True, **kw)
    s1, e1, st1, l1 = _run(mor, sd, False, **kw)
    # 130 aggregates of 34 rows in binary64 do not fit beside the matrix: that case streams
    # both times
    assert (prec, rows) == ("fp64", 34) or l1 < l0 - 100, "the on-chip path did not run"
    assert np.abs(s1 - s0).max() <= 1e-7 * s0.max()
    assert abs(e1 - e0) <= 1e-8 * e0
    assert np.all(np.abs(st1[:4] - st0[:4]) <= 40), (st0[:4], st1[:4])
    s2, e2, _, _ = _run(mor, sd, False, **kw)
    assert np.abs(s2 - s1).max() <= 1e-7 * s0.max()


def test_iteration_limit(mor):
    mesh = synth.kuhn_cube(14)
    kappa = synth.lognormal_kappa(mesh.n_tets, 8)
    sd = mor.Subdomains(mor.Mesh(mesh.xyz, mesh.tets, kappa, mesh.dirichlet),
                        synth.box_owner(14, 2), 3)
    b = mor.Bases(sd, mor.basis_opts(rank=4, oversample=3, seed=1, max_iter=11))
    assert not b.converged and b.stats()[0] == 11 and np.isfinite(b.sigma()).all()
