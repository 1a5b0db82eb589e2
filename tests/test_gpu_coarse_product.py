"""The coarse product of the local solves in its launch shapes: one CTA per 128 aggregates or
the aggregates split over a cluster, few and many columns, fewer aggregates than CTAs, and
the SIMT products on either side of their line.

The coarse level preconditions, so every shape must reach the same solution: the mixed
path stops each solve at cg_rtol = 1e-9 of the largest right-hand side, and the reduced
energy, quadratic in the errors up to their mean, agrees with binary64 within 1e-6 (the
library's bound for the mixed path).  A wrong product would show in the iterations, which
may exceed the SIMT path's by at most one replacement interval (40).
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


def _plan(mor, n, parts, hops):
    mesh = synth.kuhn_cube(n)
    kappa = synth.lognormal_kappa(mesh.n_tets, 77)
    gm = mor.Mesh(mesh.xyz, mesh.tets, kappa, mesh.dirichlet)
    return mor.Subdomains(gm, synth.box_owner(n, parts), hops)


def _run(mor, sd, **kw):
    b = mor.Bases(sd, mor.basis_opts(seed=5, **kw))
    assert b.converged
    return mor.Reduced(sd, b).solve()[1]["energy"], b.stats()[:4], b.sigma()


# (cells, boxes per axis, hops, rank, oversample, rows per aggregate): 8 subdomains of up to
# 450 aggregates (clusters of 4), 27 of up to 130 (2), 8 of 12 (one), 60 + 1 and 123 + 1
# columns, 1,000 aggregates
@pytest.mark.parametrize("n,parts,hops,rank,over,rows", [
    (32, 2, 8, 6, 4, 35), (24, 3, 4, 17, 6, 35), (12, 2, 3, 5, 2, 100), (20, 2, 5, 50, 10, 35),
    (20, 2, 5, 100, 23, 20), (30, 2, 7, 4, 1, 15)])
def test_tensor_core_product_against_simt(mor, n, parts, hops, rank, over, rows):
    sd = _plan(mor, n, parts, hops)
    kw = dict(rank=rank, oversample=over, coarse_rows=rows)
    E0, it0, s0 = _run(mor, sd, precision="mixed", tc_gram=0, **kw)
    E1, it1, s1 = _run(mor, sd, precision="mixed", tc_gram=1, **kw)
    E2, it2, s2 = _run(mor, sd, precision="fp64", cg_rtol=1e-10, **kw)
    assert abs(E1 - E2) <= 1e-6 * E2 and abs(E0 - E2) <= 1e-6 * E2
    assert np.all(np.abs(it1 - it0) <= 40), (it0, it1)
    assert np.abs(s1 - s2).max() <= 1e-6 * s2.max()


def test_without_a_coarse_level(mor):
    sd = _plan(mor, 16, 2, 4)
    E0, _, _ = _run(mor, sd, rank=6, oversample=4, precision="mixed", coarse_rows=0)
    E1, _, _ = _run(mor, sd, rank=6, oversample=4, precision="fp64", cg_rtol=1e-10)
    assert abs(E0 - E1) <= 1e-6 * E1


# 130 to 222 columns: the SIMT product takes four or eight columns a block (an odd last chunk
# of four), the updates two rows a thread from 196 columns on, the Grams strips of 16
@pytest.mark.parametrize("n,parts,hops,rank,over", [
    (15, 3, 3, 100, 29), (15, 3, 3, 60, 161), (14, 2, 3, 60, 141), (15, 3, 3, 40, 89)])
def test_wide_columns(mor, n, parts, hops, rank, over):
    sd = _plan(mor, n, parts, hops)
    E0, it0, s0 = _run(mor, sd, precision="mixed", rank=rank, oversample=over)
    E1, it1, s1 = _run(mor, sd, precision="fp64", cg_rtol=1e-10, rank=rank, oversample=over)
    assert abs(E0 - E1) <= 1e-6 * E1
    assert np.abs(s0 - s1).max() <= 1e-6 * s1.max()
