"""The gradient's kept workspace: calls that reuse it, outgrow it, share it
between contexts or run at once on threads and streams of their own give the
gradient of a call alone, bit for bit, and its memory comes back with the last
context. The misfit is an FP64 sum of at most 4 * 152 * 8 warps' terms added by
atomics in any order: 4864 * 2^-53 relative.
"""
import threading

import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu


def _setup(pkg, shape, npml=0, stream=None):
    import torch
    nx, ny, nz = shape
    vel = torch.from_numpy(wl.layered_volume(nx, ny, nz, nx)).cuda()
    dt = 0.5 * pkg.wave_cfl_dt((10.0,) * 3, float(vel.max()))
    s = pkg.WaveSolver(shape, (10.0,) * 3, dt, vel, stream=stream)
    if npml:
        s.set_cpml(npml)
    rec = torch.from_numpy(wl.receiver_plane(nx, ny, nz // 2, 3)).cuda()
    return s, rec


def _gradient(s, rec, steps, ckpt):
    import torch
    nx, ny, nz = s.grid
    obs = torch.zeros((steps, rec.shape[0]), device="cuda")
    g = torch.full((nz, ny, nx), float("nan"), device="cuda")
    torch.cuda.synchronize()
    m = s.gradient((nx // 2, ny // 2, 3, 15.0, -1.0, 1.0), steps, rec, obs, g, ckpt_every=ckpt)
    return m, g.cpu().numpy()


SPECS = [((33, 28, 30), 0, 30, 7), ((40, 44, 48), 8, 25, 10), ((20, 18, 22), 0, 12, 12)]


def test_reused_grown_and_shared(wave_lib):
    alone = []
    for shape, npml, steps, ckpt in SPECS:
        s, rec = _setup(wave_lib, shape, npml)
        alone.append(_gradient(s, rec, steps, ckpt))
        s.close()
    made = [_setup(wave_lib, shape, npml) for shape, npml, _, _ in SPECS]
    for order in ((2, 0, 1, 1, 2, 0), (1, 0, 2)):
        for i in order:
            m, g = _gradient(*made[i], *SPECS[i][2:])
            assert m == pytest.approx(alone[i][0], rel=4864 * 2.0 ** -53)
            assert np.array_equal(g, alone[i][1])
    for s, _ in made:
        s.close()


def test_threads_and_streams(wave_lib):
    import torch
    spec = SPECS[0]
    s, rec = _setup(wave_lib, spec[0])
    want = _gradient(s, rec, *spec[2:])
    streams = [torch.cuda.Stream() for _ in range(3)]
    made = [_setup(wave_lib, spec[0], stream=st.cuda_stream) for st in streams]
    torch.cuda.synchronize()
    got = [None] * 3

    def work(i):
        for _ in range(4):
            got[i] = _gradient(*made[i], *spec[2:])

    threads = [threading.Thread(target=work, args=(i,)) for i in range(3)]
    for t in threads:
        t.start()
    for t in threads:
        t.join(120)
    for m, g in got:
        assert m == pytest.approx(want[0], rel=4864 * 2.0 ** -53)
        assert np.array_equal(g, want[1])
    for x, _ in made:
        x.close()
    s.close()


def test_memory_comes_back_with_the_last_context(wave_lib):
    import gc
    import torch
    gc.collect()
    s, rec = _setup(wave_lib, (160, 160, 160))
    _gradient(s, rec, 2, 1)
    torch.cuda.synchronize()
    held = torch.cuda.mem_get_info()[0]
    s.close()
    # the workspace is (2 * 2 + 2 + 6) fields of 16 MB, the context 3
    assert torch.cuda.mem_get_info()[0] - held >= 13 * 4 * 160 ** 3
