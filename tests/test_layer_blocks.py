"""Host logic of the CPML layer's launch (no GPU): a host program compiled with
nvcc from the library's own source walks the clusters and checks that every
line end is taken once, inside the grid, and that wherever the lines of two
axes meet in a point one cluster takes both, the lower axis first, with a
barrier between.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
GRIDS = [(10, 10, 10, 1), (11, 13, 10, 1), (24, 24, 24, 8), (25, 31, 24, 8), (28, 29, 47, 10),
         (64, 28, 33, 10), (32, 70, 35, 12), (41, 40, 44, 16), (72, 41, 57, 16), (48, 51, 66, 20),
         (56, 57, 60, 24), (19, 77, 21, 5), (100, 14, 23, 3)]


@pytest.fixture(scope="module")
def walker(tmp_path_factory):
    nvcc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    if not os.path.exists(nvcc):
        nvcc = shutil.which("nvcc")
    if not nvcc:
        pytest.skip("nvcc not available")
    exe = str(tmp_path_factory.mktemp("blocks") / "layer_blocks")
    subprocess.run([nvcc, "-std=c++17", "-O2", "-gencode", "arch=compute_103a,code=sm_103a",
                    os.path.join(ROOT, "tests", "host", "layer_blocks.cu"), "-o", exe],
                   check=True, capture_output=True)
    return exe


@pytest.mark.parametrize("grid", GRIDS)
def test_blocks_cover_the_layer_in_order(walker, grid):
    out = subprocess.run([walker], input="%d %d %d %d\n" % grid, capture_output=True, text=True,
                         check=True).stdout
    assert out.strip() == "ok"
