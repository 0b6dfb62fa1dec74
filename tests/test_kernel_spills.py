"""One species runs four CTAs of 256 threads per SM, 64 registers a thread: its
step must fit them (a boundary tile's halo once held in registers spilled in
every tile)."""
import os
import re
import subprocess

import pytest

from paper_2006_15932_gb300 import build as B


@pytest.mark.parametrize("unit", ["dbm_step_s1.cu", "dbm_step_acc_s1.cu"])
def test_one_species_step_does_not_spill(unit, tmp_path):
    r = subprocess.run([B.nvcc(), *B.ARCH, *B.NVCC_FLAGS, "-Xptxas", "-v", "-c", os.path.join(B.CSRC, unit), "-o",
                        str(tmp_path / "o.o")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    kernels = re.findall(r"Compiling entry function '(\w*k_step_tma\w*)'.*?(\d+) bytes spill stores, (\d+) bytes spill "
                         r"loads", r.stdout + r.stderr, re.S)
    assert kernels
    assert all(k[1:] == ("0", "0") for k in kernels), kernels
