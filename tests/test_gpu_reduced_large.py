"""The reduced solve of more rows than the SMs' shared memory holds (above 739,000 on 152 SMs)
is still one launch with bounded waits.

27^3 subdomains of eight nodes and 40 columns: 787,320 rows.  The solve stops at a relative
residual of 1e-12, so x^T K~ x (the squared energy norm of the lifted solution, from the
elements) and b~^T x differ by at most 1e-12 ||b~|| ||x|| plus rounding.  K~ = Q^T A Q with
identity diagonal blocks: ||x|| <= sqrt(E / lambda_min), and a condition number below 1e4 is
checked by the step count (CG takes about kappa^(1/2) / 2 ln(2 / tol) steps), so 1e-9 covers it.
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


def test_one_launch_above_the_shared_memory_of_the_chip(mor):
    mesh = synth.kuhn_cube(54)
    kappa = synth.lognormal_kappa(mesh.n_tets, 11)
    sd = mor.Subdomains(mor.Mesh(mesh.xyz, mesh.tets, kappa, mesh.dirichlet),
                        synth.box_owner(54, 27), 1)
    b = mor.Bases(sd, mor.basis_opts(rank=39, oversample=1, seed=5, cg_rtol=1e-6))
    r = mor.Reduced(sd, b)
    assert r.dim == 27 ** 3 * 40
    n0 = mor.kernel_launches()
    x, info = r.solve(rtol=1e-12)
    assert mor.kernel_launches() - n0 == 1
    assert info["converged"] and info["iterations"] < 1500
    u = mor.lift(sd, b, x)
    assert abs(mor.energy_norm(sd, u) ** 2 - info["energy"]) <= 1e-9 * info["energy"]
    # the same from a second call, and the limit of the step count
    y, again = r.solve(rtol=1e-12)
    assert again["iterations"] == info["iterations"] and np.array_equal(x.cpu(), y.cpu())
    y, again = r.solve(rtol=1e-12, max_iter=3)
    assert again["iterations"] == 3 and not again["converged"]
