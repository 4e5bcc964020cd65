"""Fields in and out of a context (wave_set_state, wave_get_field) at the row
lengths and alignments where the row kernels can go wrong: rows of whole
vectors and ragged ones, one element, arrays that start 4 bytes past a 16-byte
boundary, host arrays.

FP32 fields come back bit for bit. A 16-bit field holds value / 2^e rounded to
the format once, e from the largest magnitude m: 2^(e+14) >= m > 2^(e+13)
(frexp's exponent less 14), so the expected value is exact in torch.
"""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

GRIDS = [(1, 1, 1), (3, 5, 7), (4, 3, 2), (31, 9, 5), (64, 17, 6), (203, 7, 11), (320, 6, 9),
         (1028, 3, 4), (2050, 2, 3)]


@pytest.mark.parametrize("storage", [0, 1, 2])
@pytest.mark.parametrize("grid", GRIDS)
def test_fields_in_and_out(wave_lib, grid, storage):
    import torch
    nx, ny, nz = grid
    n = nx * ny * nz
    vel = torch.full((nz, ny, nx), 2000.0, device="cuda")
    s = wave_lib.WaveSolver(grid, (10.0, 10.0, 10.0), 1e-3, vel, storage=storage)
    gen = torch.Generator().manual_seed(n + storage)
    src = [(torch.rand(n + 1, generator=gen) - 0.5) * 10.0 ** k for k in (0, -3)]
    for off in (0, 1):  # aligned, and 4 bytes past a 16-byte boundary
        u = [t.cuda()[off:off + n].view(nz, ny, nx) for t in src]
        want = []
        for t in u:
            if storage:
                e = math.frexp(float(t.abs().max()))[1] - 14
                kind = torch.bfloat16 if storage == 1 else torch.float16
                t = (t * 2.0 ** -e).to(kind).float() * 2.0 ** e
            want.append(t.cpu())
        s.set_state(u[0], u[1], 5)
        for which in (0, 1):
            for o in (0, 1):
                out = torch.full((n + 2,), -7.0, device="cuda")
                s.get_field(which, out[o:o + n])
                assert torch.equal(out[o:o + n].view(nz, ny, nx).cpu(), want[which])
                assert (out[:o] == -7).all() and (out[o + n:] == -7).all()
            host = np.empty((nz, ny, nx), np.float32)
            s.get_field(which, host)
            assert np.array_equal(host, want[which].numpy())
        s.set_state(u[0].cpu().numpy(), u[1].cpu().numpy(), 5)
        host = np.empty((nz, ny, nx), np.float32)
        s.get_field(0, host)
        assert np.array_equal(host, want[0].numpy())
    s.close()
