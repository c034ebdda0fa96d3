"""Shared-memory limits and occupancy of kernels (KernelLimits): kept per
device, without allocation, for several threads - compiled for the host from
the library's header and driven with a fake runtime of two devices.  The
library keeps no such state in any other way."""
import os
import re
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2409_10774_gb300", "csrc")


def test_kernel_limits(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host C++ compiler")
    exe = str(tmp_path / "kernel_limits_check")
    subprocess.run([gxx, "-std=c++17", "-O1", "-pthread", "-x", "c++", f"-I{CSRC}",
                    os.path.join(HERE, "kernel_limits_check.cpp"), "-o", exe], check=True, capture_output=True, text=True)
    out = subprocess.run([exe], capture_output=True, text=True)
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout


def test_one_way_to_raise_a_limit():
    uses = [f for f in sorted(os.listdir(CSRC))
            for _ in re.findall(r"cudaFuncSetAttribute\s*\(", open(os.path.join(CSRC, f)).read())]
    assert uses == ["mp_kernels.cu"]
