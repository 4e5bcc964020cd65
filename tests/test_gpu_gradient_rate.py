"""A layered gradient of several segments runs its recompute beside its adjoint, so
it should move its bytes about as fast as a forward run moves its own.

Bytes a step (each array once): forward 16 a point and, at the 2 w points of a
line end (w = npml + 4), 16, at the 2 npml cells of the layer 16; gradient 72 a
point (forward 16, recompute 20, adjoint 36), on the lines the forward's twice, 8
a point for D, and the adjoint's 16 a point and a cell. For 256^3 and 16 cells
that is 3.94 times the forward's; a twentieth is left for the rest of the call.
"""
import time

import pytest

pytestmark = pytest.mark.gpu


def test_layered_gradient_keeps_the_forward_rate(wave_lib):
    import torch
    n, npml, steps, ckpt = 256, 16, 240, 40
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    vel = 1500 + 2500 * torch.rand((n, n, n), generator=g, device="cuda")
    s = wave_lib.WaveSolver((n, n, n), (10.0,) * 3, 0.5 * wave_lib.wave_cfl_dt((10.0,) * 3, 4000.0), vel)
    s.set_cpml(npml)
    ax = torch.arange(0, n, 4, dtype=torch.int32, device="cuda")
    rec = torch.cartesian_prod(ax, ax, torch.tensor([24], dtype=torch.int32, device="cuda")).contiguous()
    obs = torch.zeros((steps, rec.shape[0]), device="cuda")
    tr, grad = torch.zeros_like(obs), torch.empty_like(vel)
    shot = (n // 2, n // 2, 26, 15.0, -1.0, 1.0)

    def best(run):
        t = []
        for _ in range(5):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            run()
            torch.cuda.synchronize()
            t.append(time.perf_counter() - t0)
        return min(t)

    fwd = best(lambda: (s.reset(), s.propagate(shot, steps, rec, tr)))
    full = best(lambda: s.gradient(shot, steps, rec, obs, grad, ckpt_every=ckpt))
    s.close()
    points, lines, w = n ** 3, 3 * n * n, npml + 4
    layer = 16 * (2 * w + 2 * npml) * lines
    ratio = (72 * points + 3 * layer + 16 * w * lines) / (16 * points + layer)
    print("\nforward %.2f ms, gradient %.2f ms, bytes %.2f x" % (1e3 * fwd, 1e3 * full, ratio))
    assert full <= 1.05 * ratio * fwd
