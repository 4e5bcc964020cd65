"""split_layers (no GPU): a plan's layers are halved together, in place and in
order, while every half keeps two planes, the launch at most `limit` CTAs and the
plan at most 64 layers; otherwise the plan stays as it is."""
import itertools
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
MAX_LAYERS = 64


@pytest.fixture(scope="module")
def split(tmp_path_factory):
    nvcc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    if not os.path.exists(nvcc):
        nvcc = shutil.which("nvcc")
    if not nvcc:
        pytest.skip("nvcc not available")
    exe = str(tmp_path_factory.mktemp("split") / "split_layers")
    subprocess.run([nvcc, "-std=c++17", "-O2", os.path.join(ROOT, "tests", "host",
                                                            "split_layers.cu"), "-o", exe],
                   check=True, capture_output=True)

    def run(cases):
        text = "".join("%d %d %s\n" % (t, l, " ".join(map(str, ch))) for t, l, ch in cases)
        out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout
        return [[int(v) for v in l.split()] for l in out.splitlines()]
    return run


PLANS = [[1], [2], [3], [4], [5], [7], [8], [64], [4] * 16, [8] * 16, [16] * 16, [17] * 15 + [3],
         [272, 216, 24], [64] * 4, [9, 4], [9, 3], [33, 33, 31], [4096 // 16] * 16, [130] * 2]


@pytest.mark.parametrize("ntiles", [1, 2, 3, 5, 8, 24, 57, 304])
def test_halves(split, ntiles):
    limits = [1, 2, 3, 16, 303, 304, 455, 456, 457, 100000]
    cases = [(ntiles, l, ch) for l, ch in itertools.product(limits, PLANS)]
    for (t, limit, ch), got in zip(cases, split(cases)):
        want = list(ch)
        while 2 * len(want) <= MAX_LAYERS and 2 * len(want) * t <= limit and min(want) >= 4:
            want = [h for c in want for h in ((c + 1) // 2, c // 2)]
        assert got == want
        assert sum(got) == sum(ch) and len(got) <= MAX_LAYERS
        assert got == ch or (min(got) >= 2 and len(got) * t <= limit)
