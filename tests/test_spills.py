"""Kernels keep their values in registers: what the compiler reports for every source, built as the library is (CPU, nvcc)."""
import os
import re
import subprocess

import pytest

from paper_2507_04123_b200 import build

REPORT = re.compile(r"Compiling entry function '(\w+)'[^\n]*\n[^\n]*\n\s*(\d+) bytes stack frame, (\d+) bytes spill stores")


@pytest.mark.parametrize("source", [s for s in build.SOURCES if s != "bridge.cu"])       # no kernels there
def test_no_kernel_spills(source, tmp_path):
    full = build.nvcc_command(verbose_ptxas=True)
    flags = [a for a in full if a not in ("-shared", "-o", build.LIB) and not a.endswith(".cu")]
    out = subprocess.run(flags + ["-c", "-o", str(tmp_path / "one.o"), os.path.join(build.CSRC, source)], check=True,
                         capture_output=True, text=True).stderr
    kernels = REPORT.findall(out)
    assert kernels and len(kernels) == out.count("Compiling entry function")
    assert [k for k in kernels if int(k[1]) or int(k[2])] == []
