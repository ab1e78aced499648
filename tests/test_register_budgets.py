"""Registers of kernels whose speed hangs on how many blocks an SM holds, from the
compiler's report for the sources as they are built."""

import os
import re
import subprocess

import pytest

from paper_2505_18519_gb300 import build


def _report(name, tmp_path):
    """{kernel: (registers, bytes spilled)} of one source file."""
    try:
        nvcc = build._nvcc()
    except RuntimeError as e:
        pytest.skip(str(e))
    r = subprocess.run([nvcc, *build.ARCH, *build.FLAGS, "-Xptxas", "-v", "-c", os.path.join(build.CSRC, name), "-o",
                        str(tmp_path / "x.o")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    out, kernel, spill = {}, None, 0
    for line in r.stderr.splitlines():
        if m := re.search(r"Compiling entry function '(\S+)'", line):
            kernel, spill = m[1], 0
        elif kernel and (m := re.search(r"(\d+) bytes spill stores, (\d+) bytes spill loads", line)):
            spill += int(m[1]) + int(m[2])
        elif kernel and (m := re.search(r"Used (\d+) registers", line)):
            out[kernel] = (int(m[1]), spill)
            kernel = None
    return out


@pytest.mark.parametrize("source,kernel,registers", [
    ("trial_df.cu", "chebyshev_expm_df_kernel", 48),        # five blocks of 256 threads
    ("trial_df.cu", "chebyshev_expm_df_list_kernel", 64),   # four, nothing spilled
    ("overlap_tc.cu", "overlap_tc_kernel", 64),
])
def test_registers_and_no_spills(source, kernel, registers, tmp_path):
    found = [v for k, v in _report(source, tmp_path).items() if kernel in k]
    assert found and all(r <= registers and s == 0 for r, s in found), found
