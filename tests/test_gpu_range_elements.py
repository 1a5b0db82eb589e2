"""A build that touches few elements of a large mesh (a range of subdomains of a streamed
plan) keeps no element table of the whole mesh beside the sketch's element factors, and
assembles the same matrices without it.

Memory: the same corner subdomain in a 32^3 and a 48^3 cube.  Its own rows are the same in
both, so the peak of the pooled workspace differs by what is kept per element of the mesh:
the factors' ten float2, 80 bytes (one slab of 1 MB for rounding).  Results: the element
table holds what the direct path computes, so the singular values agree with those of the
whole build (which takes the table) to the solves' tolerance, 1e-10 of the largest.
"""
import ctypes

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


class _Pool:
    """Peak of the default memory pool's use, in bytes."""
    USED_MEM_HIGH = 8   # cudaMemPoolAttrUsedMemHigh

    def __init__(self):
        self.rt = ctypes.CDLL("libcudart.so.13")   # the one libmor.so has loaded
        self.pool = ctypes.c_void_p()
        assert self.rt.cudaDeviceGetDefaultMemPool(ctypes.byref(self.pool), 0) == 0

    def reset(self):
        v = ctypes.c_uint64(0)
        assert self.rt.cudaMemPoolSetAttribute(self.pool, self.USED_MEM_HIGH,
                                               ctypes.byref(v)) == 0

    def high(self):
        v = ctypes.c_uint64(0)
        assert self.rt.cudaMemPoolGetAttribute(self.pool, self.USED_MEM_HIGH,
                                               ctypes.byref(v)) == 0
        return v.value


def _plan(mor, n, wave):
    mesh = synth.kuhn_cube(n)
    kappa = synth.lognormal_kappa(mesh.n_tets, 5)
    gm = mor.Mesh(mesh.xyz, mesh.tets, kappa, mesh.dirichlet)
    return mesh.n_tets, mor.Subdomains(gm, synth.box_owner(n, n // 8), 2, wave=wave)


def _build(mor, sd, **kw):
    return mor.Bases(sd, mor.basis_opts(rank=6, oversample=4, seed=3, precision="fp64",
                                        cg_rtol=1e-13, **kw))


def test_a_range_keeps_no_table_of_the_whole_mesh(mor):
    import torch
    pool, got = _Pool(), []
    for n in (32, 48):
        n_tets, sd = _plan(mor, n, 1)
        torch.cuda.synchronize()
        pool.reset()
        _build(mor, sd, sub_begin=0, sub_end=1)
        got.append((n_tets, pool.high()))
    (t0, b0), (t1, b1) = got
    assert b1 - b0 <= 80 * (t1 - t0) + 2 ** 20


def test_both_assemblies_agree(mor):
    _, one = _plan(mor, 32, 0)
    _, few = _plan(mor, 32, 1)
    a, b = _build(mor, one), _build(mor, few, sub_begin=0, sub_end=2)
    sa, sb = a.sigma(), b.sigma()
    assert np.abs(sa[:2] - sb[:2]).max() <= 1e-10 * sa[:2].max()
    assert np.array_equal(a.kept[:2], b.kept[:2])
