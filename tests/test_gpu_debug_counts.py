"""The step counts that MOR_DEBUG prints per subdomain, for solves on chip (one launch per
replacement interval of 40 steps) as for the streaming kernels.

The 16^3 workload to 1e-10 takes 40 to 80 steps per solve: a subdomain that is still open in
the second launch has run the whole first interval, so the largest count is the solve's own.
"""
import os
import re
import subprocess
import sys

import pytest

from conftest import ROOT

pytestmark = pytest.mark.gpu

RUN = r"""
import sys
sys.path.insert(0, %r)
import synth
from paper_2404_06260_gb300 import mor
mesh = synth.kuhn_cube(16)
kappa = synth.lognormal_kappa(mesh.n_tets, 31)
sd = mor.Subdomains(mor.Mesh(mesh.xyz, mesh.tets, kappa, mesh.dirichlet),
                    synth.box_owner(16, 2), 4)
b = mor.Bases(sd, mor.basis_opts(rank=8, oversample=5, seed=9, cg_rtol=1e-10))
print("stats", *b.stats()[:4])
"""


def test_counts_add_up_over_the_launches():
    from paper_2404_06260_gb300 import _build
    _build.build()
    p = subprocess.run([sys.executable, "-c", RUN % ROOT], cwd=ROOT, capture_output=True,
                       env=dict(os.environ, MOR_DEBUG="1"), text=True, timeout=300)
    assert p.returncode == 0, p.stderr[-2000:]
    total = [int(v) for v in p.stdout.split("stats")[1].split()]
    per = {int(m[1]): (int(m[2]), int(m[3])) for m in re.finditer(
        r"solve (\d) recursion iterations per subdomain: min (\d+) median \d+ max (\d+)", p.stderr)}
    assert len(per) == 4 and max(total) > 40
    for which, (lo, hi) in per.items():
        assert 0 < lo <= hi == total[which], (which, lo, hi, total)
    # before the last interval ends a solve has open columns, and says so
    rec = [int(m[1]) for m in re.finditer(r"recursive-active (\d+)", p.stderr)]
    assert max(rec) > 0
