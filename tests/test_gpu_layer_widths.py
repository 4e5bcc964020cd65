"""The unrolled layer passes of every width (8, 10, 16, 20 cells) against the line
walks (GBWAVE_CPML_GENERIC=1), bit for bit: both round each operation alike and
add the axes' terms in the same order.

In a gradient of several segments the axes take a launch each from 2.8 million
points of line ends on; a gradient of one segment keeps the single launch there.

Grids: the smallest of two disjoint segments on each axis (2 (npml + 4)); x rows
that are whole vectors of 4 and not; x too short for the near cells to be rounded
up to 8, just long enough, and longer; and flat ones of more than 1.5 million
line ends, whose axes take a launch each.
"""
import pytest

pytestmark = pytest.mark.gpu

WIDTHS = (8, 10, 16, 20)
SP = (10.0, 12.0, 9.0)
R, FCPS = 1e-3, 15.0


def _shapes(npml):
    n = 2 * (npml + 4)
    r8 = 2 * ((npml + 4 + 7) // 8 * 8)
    return [(n, n, n), (n + 1, n + 3, n), (n + 3, n, n + 5), (r8, n + 2, n + 1),
            (r8 + 9, n + 30, n + 7)]


def _flat(npml, nx=850):
    return nx, 850, 2 * (npml + 4)


def _model(shape, seed):
    import torch
    nx, ny, nz = shape
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    vel = 1500 + 2500 * torch.rand((nz, ny, nx), generator=g, device="cuda")
    state = [torch.randn((nz, ny, nx), generator=g, device="cuda") for _ in range(2)]
    lim = torch.tensor([nx, ny, nz], device="cuda")
    rec = (torch.rand((400, 3), generator=g, device="cuda") * lim).int()
    # corners of the grid and of the layer's shell
    c = torch.tensor([[x, y, z] for x in (0, nx - 1) for y in (0, ny - 1) for z in (0, nz - 1)],
                     dtype=torch.int32, device="cuda")
    return vel, state, torch.cat([rec, c, rec[:9]]).contiguous()


def _run(pkg, shape, npml, storage, chunks, model):
    import torch
    vel, (u0, up0), rec = model
    nx, ny, nz = shape
    dt = 0.5 * pkg.wave_cfl_dt(SP, 4000.0)
    s = pkg.WaveSolver(shape, SP, dt, vel, storage=storage)
    s.set_cpml(npml, R, FCPS)
    s.set_state(u0, up0, 2)
    out = []
    for k in chunks:
        out.append(torch.full((k, rec.shape[0]), float("nan"), device="cuda"))
        s.propagate((nx // 3, ny - 5, 3, 20.0, -1.0, 1e3), k, rec, out[-1])
    for which in (0, 1):
        out.append(torch.empty((nz, ny, nx), device="cuda"))
        s.get_field(which, out[-1])
    s.synchronize()
    s.close()
    return out


def _gradient(pkg, shape, npml, steps, ckpt, model):
    """Two shots in opposite corners of the layer, each with receivers around its
    source: in a few steps the field goes no further, and the gradient with it.
    Each point once: residuals at one point are added in any order."""
    import torch
    vel, _, rec = model
    nx, ny, nz = shape
    dt = 0.5 * pkg.wave_cfl_dt(SP, 4000.0)
    s = pkg.WaveSolver(shape, SP, dt, vel)
    s.set_cpml(npml, R, FCPS)
    near = torch.cartesian_prod(*[torch.arange(9, dtype=torch.int32, device="cuda")] * 3)
    far = torch.tensor([nx - 1, ny - 1, nz - 1], dtype=torch.int32, device="cuda") - near
    out = []
    for src, box in (((5, ny - 5, 3), torch.stack([near[:, 0], far[:, 1], near[:, 2]], 1)),
                     ((nx - 5, 4, nz - 4), torch.stack([far[:, 0], near[:, 1], far[:, 2]], 1))):
        r = torch.unique(torch.cat([rec, box]), dim=0).contiguous()
        gen = torch.Generator(device="cuda")
        gen.manual_seed(npml)
        obs = torch.randn((steps, r.shape[0]), generator=gen, device="cuda")
        g = torch.full((nz, ny, nx), float("nan"), device="cuda")
        tr = torch.full((steps, r.shape[0]), float("nan"), device="cuda")
        s.gradient((*src, 25.0, 0.0, 1e3), steps, r, obs, g, ckpt_every=ckpt, traces=tr)
        out += [g, tr]
    s.close()
    return out


def _same(monkeypatch, run):
    import torch
    got = run()
    monkeypatch.setenv("GBWAVE_CPML_GENERIC", "1")
    want = run()
    for a, b in zip(got, want):
        assert torch.isfinite(a).all() and float(a.abs().max()) > 0
        assert torch.equal(a, b)


@pytest.mark.parametrize("storage", [0, 1, 2])
@pytest.mark.parametrize("npml", WIDTHS)
def test_forward(wave_lib, monkeypatch, npml, storage):
    for i, shape in enumerate(_shapes(npml)):
        model = _model(shape, npml + i)
        _same(monkeypatch, lambda: _run(wave_lib, shape, npml, storage, [1, 34, 2], model))
        monkeypatch.delenv("GBWAVE_CPML_GENERIC")


@pytest.mark.parametrize("npml,storage,nx", [(8, 0, 850), (10, 0, 851), (16, 2, 852), (20, 0, 850),
                                             (20, 1, 851), (10, 2, 852)])
def test_forward_by_axis(wave_lib, monkeypatch, npml, storage, nx):
    shape = _flat(npml, nx)
    model = _model(shape, npml)
    _same(monkeypatch, lambda: _run(wave_lib, shape, npml, storage, [1, 6], model))


@pytest.mark.parametrize("npml", WIDTHS)
def test_gradient(wave_lib, monkeypatch, npml):
    for i, shape in enumerate(_shapes(npml)):
        model = _model(shape, npml + i)
        _same(monkeypatch, lambda: _gradient(wave_lib, shape, npml, 25, 7, model))
        monkeypatch.delenv("GBWAVE_CPML_GENERIC")


@pytest.mark.parametrize("npml,nx,ckpt", [(8, 850, 3), (10, 851, 8), (16, 852, 3), (20, 850, 3)])
def test_gradient_by_axis(wave_lib, monkeypatch, npml, nx, ckpt):
    shape = _flat(npml, nx)
    model = _model(shape, npml)
    _same(monkeypatch, lambda: _gradient(wave_lib, shape, npml, 8, ckpt, model))


@pytest.mark.parametrize("npml,shape", [(16, (161, 150, 152)), (8, (204, 200, 192))])
@pytest.mark.parametrize("ckpt", [4, 10])
def test_gradient_beside_its_recompute(wave_lib, monkeypatch, npml, shape, ckpt):
    nx, ny, nz = shape
    ends = 2 * (nx * ny + ny * nz + nx * nz)
    assert ends * (npml + 4) >= 2800000 and ends < 1500000
    model = _model(shape, npml)
    _same(monkeypatch, lambda: _gradient(wave_lib, shape, npml, 10, ckpt, model))
