"""The sweep's z layers at the sizes where its prologue and ring can go wrong:
layers of one to a few planes (fewer stages than the ring has slots), grids of
a few tiles, whose plans are split into up to 64 layers, grids whose layers start at, above and below a receiver plane, receivers at every
depth and repeated, against the FP64 oracle.

FP32: relative L2 <= 1e-5, the bar of the parity tests. FP16: each step rounds
u_next to 11 significant bits (2^-11 of a value, in units of the field), and
the leapfrog carries it on undamped: 6 * 2^-11 * sqrt(steps), as the other
16-bit tests.
"""
import math

import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu

CASES = [((37, 21, nz), 0) for nz in (1, 2, 3, 4, 5, 8, 13, 16, 17, 33, 63)] + \
        [((72, 35, nz), 2) for nz in (1, 3, 4, 5, 9, 17, 40)] + \
        [((37, 21, nz), 0) for nz in (64, 67, 130, 260)] + [((72, 35, nz), 2) for nz in (64, 131)]


def rel_l2(a, b):
    a, b = np.asarray(a, np.float64), np.asarray(b, np.float64)
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("grid,storage", CASES)
def test_short_layers_and_receivers_at_every_depth(wave_lib, oracle_mod, grid, storage):
    import torch
    nx, ny, nz = grid
    sp, nsteps = (10.0, 11.0, 9.0), 35
    vel = wl.layered_volume(nx, ny, nz, 5)
    dt = 0.5 * wave_lib.wave_cfl_dt(sp, float(vel.max()))
    rng = np.random.default_rng(nz)
    column = [[nx // 2, ny // 2, z] for z in range(nz)]
    plane = wl.receiver_plane(nx, ny, nz // 2, 4).tolist()
    some = wl.random_receivers(nx, ny, nz, 40, nz).tolist()
    rec = np.array(column + plane + some + some[:7], np.int32)
    rng.shuffle(rec)
    shot = (nx // 3, ny // 3, nz // 2, 15.0, -1.0, 1.0)
    s = wave_lib.WaveSolver(grid, sp, dt, torch.from_numpy(vel).cuda(), storage=storage)
    u0, up0 = wl.random_state((nz, ny, nx), seed=nz)
    s.set_state(torch.from_numpy(u0).cuda(), torch.from_numpy(up0).cuda(), 3)
    start = [np.empty((nz, ny, nx), np.float32) for _ in range(2)]
    s.get_field(0, start[0])
    s.get_field(1, start[1])
    tr = torch.full((nsteps, rec.shape[0]), float("nan"), device="cuda")
    s.propagate(shot, nsteps, torch.from_numpy(rec).cuda(), tr)
    u = np.empty((nz, ny, nx), np.float32)
    s.get_field(0, u)
    s.synchronize()
    s.close()
    ou, _, otr = oracle_mod.propagate(vel, sp, dt, nsteps, u=start[0], u_prev=start[1], step0=3,
                                      source=shot, receivers=rec)
    tol = 1e-5 if storage == 0 else 6 * 2.0 ** -11 * math.sqrt(nsteps)
    assert rel_l2(u, ou) <= tol
    assert rel_l2(tr.cpu().numpy(), otr) <= tol


@pytest.mark.parametrize("storage", [0, 1, 2])
@pytest.mark.parametrize("chunks", [[1] * 5, [1, 32, 2], [33, 1, 1], [64, 3], [2, 65]])
def test_shell_receivers_of_every_call(wave_lib, chunks, storage):
    """With an absorbing layer a step records the shell receivers of the step
    before it, and the call's end those of its last: rows of calls split any way
    (one step, a captured chunk, a chunk and remainders) equal those of one
    call bit for bit, corners, edges and faces of the shell and repeats."""
    import torch
    nx, ny, nz, npml = 44, 31, 40, 10
    sp = (10.0, 11.0, 9.0)
    vel = wl.layered_volume(nx, ny, nz, 7)
    dt = 0.5 * wave_lib.wave_cfl_dt(sp, float(vel.max()))
    ends = [0, 1, 13, 14, 15]
    rec = [[x, y, z] for x in ends + [nx - 1, nx - 14] for y in (0, 15, ny - 1) for z in ends + [nz - 1]]
    rec = torch.from_numpy(np.array(rec + rec[:9], np.int32)).cuda()
    shot = (nx // 2, ny // 2, 12, 15.0, -1.0, 1.0)
    u0, up0 = wl.random_state((nz, ny, nx), seed=3)

    def run(parts):
        s = wave_lib.WaveSolver((nx, ny, nz), sp, dt, torch.from_numpy(vel).cuda(), storage=storage)
        s.set_cpml(npml)
        s.set_state(torch.from_numpy(u0).cuda(), torch.from_numpy(up0).cuda(), 0)
        rows = []
        for k in parts:
            tr = torch.full((k, rec.shape[0]), float("nan"), device="cuda")
            s.propagate(shot, k, rec, tr)
            rows.append(tr)
        u = torch.empty((nz, ny, nx), device="cuda")
        s.get_field(0, u)
        s.synchronize()
        s.close()
        return torch.cat(rows).cpu(), u.cpu()

    tr, u = run([sum(chunks)])
    tr2, u2 = run(chunks)
    assert torch.equal(tr, tr2) and torch.equal(u, u2)
    # the last row is the field itself at the shell receivers (elsewhere a trace
    # is the update before it is rounded to a 16-bit format)
    r = rec.cpu().long()
    w, n = npml + 4, torch.tensor([nx, ny, nz])
    shell = ((r < w) | (r >= n - w)).any(1)
    assert torch.equal(tr[-1][shell], u[r[:, 2], r[:, 1], r[:, 0]][shell])
