"""The host plan where the process may start no more threads (a container's process limit):
its loops go on with the threads they have, down to the calling one, instead of ending the
process with an uncaught exception.  pthread_create is replaced by a preloaded fake that
refuses after the first `allowed` threads."""
import os
import shutil
import subprocess
import sys

import pytest

from conftest import ROOT

FAKE = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <errno.h>
#include <pthread.h>
static int left = -1, refused = 0;
void fake_allow(int n) { left = n; }
int fake_refused(void) { return refused; }
int pthread_create(pthread_t* t, const pthread_attr_t* a, void* (*f)(void*), void* x) {
  static int (*real)(pthread_t*, const pthread_attr_t*, void* (*)(void*), void*);
  if (!real) real = dlsym(RTLD_NEXT, "pthread_create");
  if (left == 0) { ++refused; return EAGAIN; }
  if (left > 0) --left;
  return real(t, a, f, x);
}
"""

CHECK = r"""
import ctypes, sys
sys.path.insert(0, %r)
import synth
from paper_2404_06260_gb300 import mor
mesh, kappa, owner, p = synth.workload("cube64_p4")
fake = ctypes.CDLL(None)
out = []
for allowed in (-1, int(sys.argv[1])):
    fake.fake_allow(allowed)
    out.append(mor.plan_check(mesh, owner, p["r_hops"], 22))
assert fake.fake_refused() > 0
assert out[0] == out[1] and out[0]["rows"] > 100000 and out[0]["wave_mismatches"] == 0
print("same plan")
"""


@pytest.mark.parametrize("allowed", [0, 3])
def test_plan_with_no_more_threads(tmp_path, allowed):
    cc = shutil.which("gcc")
    if cc is None:
        pytest.skip("no C compiler")
    from paper_2404_06260_gb300 import _build
    _build.build()
    src, lib = tmp_path / "fake.c", tmp_path / "fake.so"
    src.write_text(FAKE)
    subprocess.run([cc, "-shared", "-fPIC", "-o", str(lib), str(src), "-ldl"], check=True)
    p = subprocess.run([sys.executable, "-c", CHECK % ROOT, str(allowed)], cwd=ROOT,
                       env=dict(os.environ, LD_PRELOAD=str(lib), OMP_NUM_THREADS="1"),
                       capture_output=True, text=True, timeout=600)
    assert p.returncode == 0 and "same plan" in p.stdout, (p.returncode, p.stderr[-2000:])
