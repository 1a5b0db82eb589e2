"""The library holds no kernel variant that its dispatch cannot reach: blocks of 1024 threads
and two rows in flight in the CG steps are choices of the binary32 path alone."""
import shutil
import subprocess

import pytest


def test_binary64_steps_have_one_block_size():
    nm = shutil.which("nm")
    if nm is None:
        pytest.skip("no nm")
    from paper_2404_06260_gb300 import _build
    names = subprocess.run([nm, "-C", _build.build()], capture_output=True, text=True,
                           check=True).stdout
    assert "k_cg_update_p<double, 256, 1>" in names and "k_cg_update_p<float, 1024, 1>" in names
    for kernel in ("k_cg_update_p<double, 1024", "k_cg_update_p<double, 256, 2>",
                   "k_cg_update_xr<double, 1024", "k_cg_update_xr<double, 256, 2>",
                   "k_cg_spmm_pq<double, 2, 1024>"):
        assert kernel not in names, kernel
