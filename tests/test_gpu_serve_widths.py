"""Served layered shots of several layer widths and storage types in one batch.

Each width has passes of its own (unrolled for 8, 10, 16 and 20 cells, line
walks for the others and on axes too short for two segments), and the passes of
a step run side by side. Every trace must equal the single-grid path's bit for
bit, and a batch must not take its widths one after another: the longest chain
of launches is that of the line walks (three axes, then the receivers), so the
mix may take no longer than the same shots all at such a width, plus a quarter
for joining the streams.
"""
import time

import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu

SP = (10.0, 10.0, 10.0)
R, FCPS = 1e-3, 15.0
WIDTHS = (8, 10, 16, 20, 12, 6)


def _inputs(grid, npml, seed):
    import torch
    nx, ny, nz = grid
    vel = torch.from_numpy(wl.layered_volume(nx, ny, nz, seed)).cuda()
    rec = np.concatenate([wl.receiver_plane(nx, ny, 3, 5), wl.random_receivers(nx, ny, nz, 30, seed),
                          np.array([[0, 0, 0], [nx - 1, ny - 1, nz - 1]])]).astype(np.int32)
    shot = (nx // 2, ny // 2, min(npml + 1, nz // 2), 15.0, -1.0, 1.0)
    return vel, torch.from_numpy(np.ascontiguousarray(rec)).cuda(), shot


def _submit(srv, made, specs, outs):
    return [srv.submit(grid, SP, vel, shot, steps, rec, tr, storage=storage, cpml=(npml, R, FCPS))
            for (grid, storage, steps, npml), (vel, rec, shot), tr in zip(specs, made, outs)]


def _served_equals_single(wave_lib, specs):
    import torch
    made = [_inputs(grid, npml, i) for i, (grid, _, _, npml) in enumerate(specs)]
    outs = [torch.zeros((sp[2], m[1].shape[0]), device="cuda") for sp, m in zip(specs, made)]
    srv = wave_lib.ShotServer(16 * 10 ** 9, 16)
    dts = []
    for t in _submit(srv, made, specs, outs):
        st, res = srv.wait(t, 120.0)
        assert st == 0, res
        dts.append(res["dt"])
    srv.close()
    for (grid, storage, steps, npml), (vel, rec, shot), tr, dt in zip(specs, made, outs, dts):
        s = wave_lib.WaveSolver(grid, SP, dt, vel, storage=storage)
        s.set_cpml(npml, R, FCPS)
        want = torch.zeros_like(tr)
        s.propagate(shot, steps, rec, want)
        s.synchronize()
        s.close()
        assert torch.equal(tr, want), (grid, storage, npml)
        assert float(want.abs().max()) > 0


@pytest.mark.parametrize("storage", [0, 2])
def test_many_line_ends_take_a_launch_per_axis(wave_lib, storage):
    """1.5 million line ends of a width: one flat shot, or several together."""
    _served_equals_single(wave_lib, [((850, 849, 24), storage, 60, 8), ((61, 50, 44), storage, 70, 8),
                                     ((64, 66, 70), storage, 65, 10)])
    _served_equals_single(wave_lib, [((501 + i, 500 - i, 40), storage, 60 + i, 16) for i in range(3)]
                          + [((60, 66, 42), storage, 65, 16), ((60, 66, 39), storage, 65, 16)])


@pytest.mark.parametrize("storages", [(0,), (2, 0, 1)])
def test_widths_beside_each_other_equal_the_single_grid_path(wave_lib, storages):
    specs = [((48 + 5 * i, 61 - 3 * i, 44 + i), storages[i % len(storages)], 30 + 7 * i, w)
             for i, w in enumerate(WIDTHS + (9, 8))]
    # axes too short for two unrolled segments, one, two and all three of them
    specs += [((70, 66, 2 * w + 2), storages[0], 41, w) for w in (8, 16)]
    specs += [((50, 22, 20), storages[-1], 41, 10), ((41, 43, 40), storages[0], 33, 20)]
    _served_equals_single(wave_lib, specs)


def test_widths_do_not_wait_for_one_another(wave_lib):
    import torch
    grids = [(64 + 4 * i, 64 + 3 * i, 64 + i) for i in range(len(WIDTHS))]
    mixed = [(g, 0, 200, w) for g, w in zip(grids, WIDTHS)]
    walks = [(g, 0, 200, 12) for g in grids]
    made = [_inputs(g, 20, i) for i, g in enumerate(grids)]
    outs = [torch.zeros((200, m[1].shape[0]), device="cuda") for m in made]
    srv = wave_lib.ShotServer(16 * 10 ** 9, 16)
    best = [1e9, 1e9]
    for _ in range(8):
        for i, specs in enumerate((mixed, walks)):
            t0 = time.perf_counter()
            for t in _submit(srv, made, specs, outs):
                st, res = srv.wait(t, 120.0)
                assert st == 0, res
            best[i] = min(best[i], time.perf_counter() - t0)
    srv.close()
    print("\nmixed widths %.2f ms, line walks %.2f ms" % (1e3 * best[0], 1e3 * best[1]))
    assert best[0] <= 1.25 * best[1]
