"""The compiler's report on the step kernels: every variant is fitted to a number of resident CTAs, and the
default and small-lattice forms do so without spilling registers."""
import os
import re
import subprocess

import pytest

from paper_2202_06516_gb300 import _native


def _report(source, tmp_path):
    """kernel (mangled) -> bytes of spill stores and loads"""
    cmd = [_native._nvcc(), *_native.ARCH, *_native.NVCC_FLAGS, "-Xptxas", "-v", "-cubin",
           os.path.join(_native.CSRC, source), "-o", str(tmp_path / "k.cubin")]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return {m[0]: int(m[1]) + int(m[2]) for m in re.findall(
        r"Compiling entry function '(\S+)'.*?(\d+) bytes spill stores, (\d+) bytes spill loads",
        r.stderr, re.S)}


@pytest.mark.parametrize("source,forms", [
    ("lbm_batch.cu", ["k_batch_stepILi32ELi16ELi5ELi256E", "k_batch_stepILi16ELi8ELi3ELi320E",
                      "k_batch_stepILi32ELi8ELi3ELi384E"]),
    ("lbm_step.cu", ["k_stepIfLi32ELi16ELi256ELb0ELi5ELb0E", "k_stepIfLi32ELi16ELi256ELb0ELi4ELb1E",
                     "k_stepIfLi32ELi16ELi640E", "k_stepIfLi32ELi8ELi384E", "k_stepIfLi16ELi8ELi320E"])])
def test_step_kernels_do_not_spill(source, forms, tmp_path):
    report = _report(source, tmp_path)
    for f in forms:
        found = {k: v for k, v in report.items() if f in k}
        assert found and not any(found.values()), (f, found)
