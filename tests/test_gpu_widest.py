"""Binary64 builds at the widest sketches (455 to 511 columns, the limit of
mor_build_bases): the local solves' kernels stage rows of all columns in shared memory, in
parts that change with the column count, and every part must fit.

Against the oracle at one width, with the tolerances of the 16^3 parity tests (cg_rtol 1e-13:
singular values within 1e-10 sigma_1, reduced energy and solution within 1e-10).  The other
widths sketch more columns of the same draws; their first `rank` singular values differ from
the oracle's only by what the further columns add to the sketch, so they are compared with
their own mixed-precision build, 1e-6 in relative energy.
"""
import numpy as np
import pytest

import synth
from oracle import pipeline, reduced

pytestmark = pytest.mark.gpu
HOPS, RANK, SEED = 4, 8, 21


@pytest.fixture(scope="module")
def case():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2404_06260_gb300 import _build
    _build.build()
    from paper_2404_06260_gb300 import mor
    mesh = synth.kuhn_cube(20)
    kappa = synth.lognormal_kappa(mesh.n_tets, 31)
    owner = synth.box_owner(20, 2)
    sd = mor.Subdomains(mor.Mesh(mesh.xyz, mesh.tets, kappa, mesh.dirichlet), owner, HOPS)
    return mor, mesh, kappa, owner, sd


def _solve(mor, sd, k, precision, rtol):
    b = mor.Bases(sd, mor.basis_opts(rank=RANK, oversample=k - RANK, seed=SEED,
                                     precision=precision, cg_rtol=rtol))
    assert b.converged and b.k == k and b.stats()[0] > 0
    x, info = mor.Reduced(sd, b).solve(rtol=1e-14)
    assert info["converged"]
    return b, info, mor.lift(sd, b, x)


@pytest.mark.parametrize("k", [455, 456, 467, 468, 503, 511])
def test_widest_sketches_in_binary64(case, k):
    mor, mesh, kappa, owner, sd = case
    b, info, u = _solve(mor, sd, k, "fp64", 1e-13)
    _, _, um = _solve(mor, sd, k, "mixed", 1e-9)
    assert mor.energy_norm(sd, um, u) <= 1e-6 * mor.energy_norm(sd, u)
    if k != 456:
        return
    ref = pipeline.run(mesh, kappa, owner, RANK, k - RANK, HOPS, SEED, fe_solution=False)
    sig = b.sigma()
    for i, ob in enumerate(ref["bases"]):
        want = np.zeros(k)   # the oracle leaves out directions that the draws do not span
        want[:len(ob["sigma"])] = ob["sigma"]
        assert np.max(np.abs(sig[i] - want)) <= 1e-10 * ob["sigma"][0], i
    assert abs(info["energy"] - ref["E"]) <= 1e-10 * ref["E"]
    ug = u.cpu().numpy()
    assert reduced.energy_norm(mesh, kappa, ug - ref["u_red"]) <= \
        1e-10 * reduced.energy_norm(mesh, kappa, ref["u_red"])
