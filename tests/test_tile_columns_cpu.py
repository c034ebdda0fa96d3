"""Columns per y / z tile (tile_columns, compiled for the host from the
kernels' header) against the rule it states, over short and long axes.

An SM holds at most 32 blocks: a lone FP32 cell's tiles must be the ones that
end soonest under that limit (to the rule's 3 %), also where a column is a few
points long and narrower tiles would only queue."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2409_10774_gb300", "csrc")
NSM = 152


@pytest.fixture(scope="module")
def columns(tmp_path_factory):
    gxx = shutil.which("g++")
    inc = [d for d in ("/usr/local/cuda/include", os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include"))
           if os.path.isdir(d)]
    if gxx is None or not inc:
        pytest.skip("no host C++ compiler or CUDA headers")
    exe = str(tmp_path_factory.mktemp("tiles") / "tile_columns_check")
    subprocess.run([gxx, "-std=c++17", "-O1", "-x", "c++", f"-I{CSRC}", f"-I{inc[0]}",
                    os.path.join(HERE, "tile_columns_check.cpp"), "-o", exe], check=True, capture_output=True, text=True)

    def run(cases):
        text = "".join("%d %d %d %d %d\n" % (n, c, f, s, NSM) for n, c, f, s in cases)
        out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout
        return [int(v) for v in out.split()]
    return run


def _cost(n, ncols, cols):
    slots = NSM * min(32, max(1, 800 // (cols * n)))
    return -(-(-(-ncols // cols)) // slots) * (cols * n + 100.0)


def test_lone_fp32_cells_take_the_tiles_that_end_soonest(columns):
    cases = [(n, c, 0, 0) for n in (1, 2, 4, 6, 8, 12, 16, 18, 24, 32, 48, 64, 96, 128, 256, 512)
             for c in (1, 5, 64, 1000, 4096, 8192, 16384, 32768, 65536)]
    for (n, ncols, _, _), cols in zip(cases, columns(cases)):
        full = max(1, 256 // n)
        assert 1 <= cols <= full
        best = min(_cost(n, ncols, k) for k in range(1, full + 1))
        assert 0.97 * _cost(n, ncols, cols) <= best, (n, ncols, cols)


def test_shared_and_fp64_tiles(columns):
    cases = [(16, 4096, 0, 1), (54, 100, 0, 1), (512, 9, 0, 1), (16, 4096, 1, 1), (384, 9, 1, 1),
             (16, 128, 1, 0), (16, 1216, 1, 0), (16, 65536, 1, 0)]
    assert columns(cases) == [16, 4, 1, 8, 1, 1, 4, 8]
