"""Sweep counts that the V-cycle's restriction and prolongation do not allow for are
refused when the solver is compiled."""
import os
import subprocess

import pytest

from paper_1801_00972_gb300 import build as B


@pytest.mark.parametrize("option", ["PIC_MG_PRE=0", "PIC_MG_POST=0"])
def test_a_cycle_without_sweeps_does_not_compile(tmp_path, option):
    r = subprocess.run([B.nvcc(), *B.ARCH, *B.FLAGS, f"-D{option}", "-c", os.path.join(B.CSRC, "poisson.cu"),
                        "-o", str(tmp_path / "poisson.o")], capture_output=True, text=True)
    assert r.returncode != 0 and "V-cycle needs a sweep" in r.stdout + r.stderr
