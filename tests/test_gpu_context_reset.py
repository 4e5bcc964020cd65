"""cudaDeviceReset with a context left behind: the memory that the library kept
for the next gradient went with the CUDA context, so a gradient of a new context
takes memory of its own and gives what the first one gave, bit for bit.

In a process of its own. It ends before the second gradient if the driver gave
the new CUDA context the id of the old one.
"""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
import ctypes, os, sys
import numpy as np
import paper_2404_04441_gb300 as pkg
import workloads as wl

cuda, rt = ctypes.CDLL("libcuda.so.1"), ctypes.CDLL(sys.argv[1])
nx, ny, nz, steps = 33, 28, 30, 20
vel = wl.layered_volume(nx, ny, nz, 1)
rec = np.ascontiguousarray(wl.receiver_plane(nx, ny, nz // 2, 3), dtype=np.int32)
obs = np.zeros((steps, rec.shape[0]), np.float32)
dt = 0.5 * pkg.wave_cfl_dt((10.0,) * 3, float(vel.max()))
ids, grads, left = [], [], []
for _ in range(3):
    s = pkg.WaveSolver((nx, ny, nz), (10.0,) * 3, dt, vel, stream=0)
    left.append(s)
    n = ctypes.c_ulonglong(0)
    assert cuda.cuCtxGetId(None, ctypes.byref(n)) == 0
    assert n.value not in ids, "a new CUDA context took an old one's id"
    ids.append(n.value)
    for _ in range(2):  # the second takes what the first left
        g = np.full((nz, ny, nx), np.nan, np.float32)
        s.gradient((nx // 2, ny // 2, 3, 15.0, -1.0, 1.0), steps, rec, obs, g, ckpt_every=7)
        grads.append(g)
    assert rt.cudaDeviceReset() == 0
assert np.abs(grads[0]).max() > 0
assert all(np.array_equal(g, grads[0]) for g in grads)
print("ok", flush=True)
os._exit(0)
"""


@pytest.mark.gpu
def test_gradient_after_a_device_reset(wave_lib):
    home = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    runtime = os.path.join(home, "lib64", "libcudart.so")
    if not os.path.exists(runtime):
        pytest.skip("no CUDA runtime library")
    p = subprocess.run([sys.executable, "-c", PROGRAM, runtime], cwd=ROOT, capture_output=True,
                       text=True, timeout=120)
    assert p.returncode == 0 and p.stdout.strip() == "ok", p.stdout + p.stderr
