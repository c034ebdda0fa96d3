"""Static shared memory of the y / z line kernels against the reserve that the
tile budget leaves for it (no GPU needed: nvcc cross-compiles).

Their tiles may take the opt-in maximum less kSmemStaticReserve; the longest
FP64 column that is accepted takes all of that, and the multi-cell kernels add
a cell descriptor of static memory.  (The single-cell line kernels have none;
test_build_cpu.py covers the kernels of mp_kernels.cu.)"""
import os
import re
import shutil
import subprocess
from concurrent.futures import ThreadPoolExecutor

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2409_10774_gb300", "csrc")
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
# multi-cell units and their kernels: y forward and inverse, or z
UNITS = {f"mp_lines_{u}{p}.cu": n for p in (32, 64) for u, n in (("ym", 2), ("zm", 1))}


def _resources(unit, out):
    # (static shared memory does not depend on ptxas' level, its time does)
    r = subprocess.run([NVCC, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17",
                        "--expt-relaxed-constexpr", "-I", os.path.join(ROOT, "include"), "-Xptxas", "-v,-O0", "-c",
                        os.path.join(CSRC, unit), "-o", os.path.join(out, unit + ".o")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    name, seen = None, {}
    for line in r.stderr.splitlines():
        m = re.search(r"Compiling entry function '([^']+)'", line)
        if m:
            name = m.group(1)
        elif name and re.search(r"Used \d+ registers", line):
            sm = re.search(r"(\d+) bytes smem", line)
            seen[name] = int(sm.group(1)) if sm else 0
            name = None
    return seen


@pytest.mark.skipif(not os.path.exists(NVCC), reason="nvcc not available")
def test_line_kernels_fit_the_reserve(tmp_path):
    text = open(os.path.join(CSRC, "mp_kernels.cu")).read()
    reserve = int(re.search(r"kSmemStaticReserve\s*=\s*(\d+)", text).group(1))
    with ThreadPoolExecutor(max_workers=len(UNITS)) as ex:
        found = dict(zip(UNITS, ex.map(lambda u: _resources(u, str(tmp_path)), UNITS)))
    for unit, count in UNITS.items():
        smem = [v for k, v in found[unit].items() if "k_line_multi" in k]
        assert len(smem) == count and min(smem) > 0, (unit, found[unit])
        assert max(smem) <= reserve, (unit, smem)
    # a single-cell line kernel: dynamic shared memory only
    lines = open(os.path.join(CSRC, "mp_lines.cuh")).read()
    for kernel in ("k_fft_y", "k_green_z"):
        body = re.search(kernel + r"\(CellDev<R> c\) \{(.*?)\n\}", lines, re.S).group(1)
        assert re.findall(r"(\w+\s+)?__shared__", body) == ["extern "], kernel


def test_one_formula_admits_and_launches():
    """sizes_fit asks for the shared memory that a launch of one column takes,
    and the kernels whose tiles may fill the budget are held to the reserve."""
    kernels = open(os.path.join(CSRC, "mp_kernels.cu")).read()
    body = re.search(r"bool sizes_fit\(int n1, int n2, int n3\) \{(.*?)\n\}", kernels, re.S).group(1)
    assert "smem_line<R>(n2, 1, 18)" in body and "smem_line<R>(n3, 1, 18)" in body and "* (size_t)n" not in body
    lines = open(os.path.join(CSRC, "mp_lines.cuh")).read()
    calls = re.findall(r"resident_blocks\((.*?)\) \* nsm", lines)
    assert len(calls) == 2 and all(c.endswith(", true") for c in calls)
