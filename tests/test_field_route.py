"""Which memory a field's rows reach by kernel (no GPU): only the context device's
own, and only with that device current. A kernel cannot be launched into a stream
of a device that is not current; a copy can, so wave_get_field and
wave_set_state of FP32 fields copy there."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_rows_by_kernel_only_on_the_current_device(tmp_path):
    nvcc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    if not os.path.exists(nvcc):
        nvcc = shutil.which("nvcc")
    if not nvcc:
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "field_route")
    subprocess.run([nvcc, "-std=c++17", "-O2", os.path.join(ROOT, "tests", "host", "field_route.cu"),
                    "-o", exe], check=True, capture_output=True)
    cases = [(t, m, c, d) for t in range(4) for m in range(2) for c in range(2) for d in range(2)]
    out = subprocess.run([exe], input="".join("%d %d %d %d\n" % c for c in cases),
                         capture_output=True, text=True, check=True).stdout.split()
    assert [int(v) for v in out] == [int(t == 2 and m == c == d) for t, m, c, d in cases]
