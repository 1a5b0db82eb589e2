"""A refused launch of the on-chip CG (a device or a partition of it that does not grant the
cluster) leaves the solve to the streaming kernels.  The refusal comes from a preloaded fake
of cudaLaunchKernelExC, which turns down the blocks of that kernel's sizes (512 threads in
binary32, 320 in binary64); nothing else launches clusters of those sizes but the reduced
solve, which has its own second choice.

Both runs solve to cg_rtol = 1e-10: singular values within 1e-7 of the largest and the
reduced energy within 1e-8, as for the on-chip and streaming kernels against each other.
"""
import json
import os
import shutil
import subprocess
import sys

import numpy as np
import pytest

from conftest import ROOT

pytestmark = pytest.mark.gpu

FAKE = r"""
#define _GNU_SOURCE
#include <cuda_runtime_api.h>
#include <dlfcn.h>
static int refused = 0;
int fake_refused(void) { return refused; }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** a) {
  static cudaError_t (*real)(const cudaLaunchConfig_t*, const void*, void**);
  if (!real) real = dlsym(RTLD_NEXT, "cudaLaunchKernelExC");
  unsigned i;
  for (i = 0; i < c->numAttrs; ++i)
    if (c->attrs[i].id == cudaLaunchAttributeClusterDimension &&
        (c->blockDim.x == 512 || c->blockDim.x == 320)) {
      ++refused;
      return cudaErrorInvalidConfiguration;
    }
  return real(c, f, a);
}
"""

RUN = r"""
import ctypes, json, sys
sys.path.insert(0, %r)
import synth
from paper_2404_06260_gb300 import mor
mesh = synth.kuhn_cube(16)
kappa = synth.lognormal_kappa(mesh.n_tets, 31)
sd = mor.Subdomains(mor.Mesh(mesh.xyz, mesh.tets, kappa, mesh.dirichlet),
                    synth.box_owner(16, 2), 4)
out = []
for prec in ("mixed", "fp64"):
    n0 = mor.kernel_launches()
    b = mor.Bases(sd, mor.basis_opts(rank=8, oversample=5, seed=9, cg_rtol=1e-10,
                                     precision=prec))
    launches = mor.kernel_launches() - n0
    e = mor.Reduced(sd, b).solve(rtol=1e-13)[1]["energy"]
    out.append(dict(sigma=b.sigma().tolist(), energy=e, converged=bool(b.converged),
                    iters=b.stats()[:4].tolist(), launches=launches))
fake = getattr(ctypes.CDLL(None), "fake_refused", None)
print(json.dumps(dict(runs=out, refused=fake() if fake else 0)))
"""


def _run(env):
    p = subprocess.run([sys.executable, "-c", RUN % ROOT], cwd=ROOT, env=env,
                       capture_output=True, text=True, timeout=300)
    assert p.returncode == 0, p.stderr[-2000:]
    return json.loads(p.stdout.strip().splitlines()[-1])


def test_streaming_steps_take_over(tmp_path):
    cc = shutil.which("gcc")
    if cc is None:
        pytest.skip("no C compiler")
    from paper_2404_06260_gb300 import _build
    _build.build()
    src, lib = tmp_path / "fake.c", tmp_path / "fake.so"
    src.write_text(FAKE)
    subprocess.run([cc, "-shared", "-fPIC", "-I", os.path.join(_build._cuda_home(), "include"),
                    "-o", str(lib), str(src), "-ldl"], check=True)
    want = _run(dict(os.environ))
    got = _run(dict(os.environ, LD_PRELOAD=str(lib)))
    assert want["refused"] == 0 and got["refused"] >= 8   # four solves in each precision
    for a, b in zip(want["runs"], got["runs"]):
        assert a["converged"] and b["converged"]
        assert b["launches"] > a["launches"] + 100, "the streaming kernels did not run"
        sa, sb = np.array(a["sigma"]), np.array(b["sigma"])
        assert np.abs(sa - sb).max() <= 1e-7 * sa.max()
        assert abs(a["energy"] - b["energy"]) <= 1e-8 * a["energy"]
        assert np.all(np.abs(np.array(a["iters"]) - np.array(b["iters"])) <= 40)
