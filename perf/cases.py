"""The work that a user of this framework has it do, as timed cases.

Every case goes through the package's public entry points as a program calls
them: a shot of a survey (reset, propagate, read the field back), a restart
from saved fields, the gradient of a trace misfit, a differentiable forward
model in a torch graph, and a set of shots through the shot server.

Models are random layered velocities of 1500-4500 m/s with 5 % smooth lateral
variation, sources 15 Hz Ricker wavelets near the surface, receivers every
4th point of a plane: the recipes of workloads/__init__.py, built on the GPU.
"""
import math

import torch

import paper_2404_04441_gb300 as gw

STORAGE = {"f32": 0, "bf16": 1, "f16": 2}
W2 = (-205.0 / 72.0, 8.0 / 5.0, -1.0 / 5.0, 8.0 / 315.0, -1.0 / 560.0)
W1 = (0.0, 4.0 / 5.0, -1.0 / 5.0, 4.0 / 105.0, -1.0 / 280.0)
F_PEAK = 15.0
REFLECTION = 1e-3
SERVE_SIZES = tuple(range(128, 513, 32))


def _case(name, kind, nx, ny, nz, nsteps, **more):
    c = {"name": name, "kind": kind, "nx": nx, "ny": ny, "nz": nz, "dz": 10.0,
         "nsteps": nsteps, "storage": "f32", "npml": 0}
    c.update(more)
    return c


def listed():
    return [
        # A small model in an inversion's inner loop or a teaching run: steps of
        # a few microseconds, so launches and load latency are what counts.
        _case("shot_64", "shot", 64, 64, 64, 100),
        # A model cut to its area of interest: no size a multiple of a tile, rows
        # that are not a whole number of 16-byte words.
        _case("shot_ragged", "shot", 203, 157, 131, 150),
        # An ordinary single shot.
        _case("shot_256", "shot", 256, 256, 256, 200),
        # The survey-size model, where memory bandwidth is all there is.
        _case("shot_1024", "shot", 1024, 1024, 512, 40),
        # The same model held in half precision.
        _case("shot_1024_f16", "shot", 1024, 1024, 512, 40, storage="f16"),
        # A run continued from saved fields, in half precision: both fields
        # loaded, stepped with no source, and saved again.
        _case("restart_f16", "restart", 320, 352, 288, 60, storage="f16"),
        # Shots with absorbing boundaries, the usual way to run a survey: a wide
        # layer on a mid-size model, a 10-cell layer on a ragged one, and half
        # precision.
        _case("layer16_512", "shot", 512, 512, 256, 100, npml=16),
        _case("layer10_ragged", "shot", 150, 141, 133, 100, npml=10),
        _case("layer16_f16", "shot", 320, 256, 192, 100, npml=16, storage="f16"),
        # One misfit gradient of full-waveform inversion: forward, residual,
        # checkpointed recompute and adjoint.
        _case("gradient_256", "gradient", 256, 256, 256, 160, ckpt=40),
        # A forward model inside a torch graph, with the absorbing layer: new
        # context, traces, loss gradient back to the squared velocity.
        _case("autograd_layer16", "autograd", 160, 144, 128, 100, npml=16, ckpt=25),
        # Shots of uneven sizes handed to the shot server at once, a third of
        # them with absorbing boundaries.
        _case("serve_mix", "serve", 0, 0, 0, 0, shots=10, steps_lo=40, steps_hi=100, mix=1,
              layer_every=3),
    ]


def draw(rng):
    def size(lo, hi):
        n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        return n if rng.random() < 0.5 else max(lo, n // 32 * 32)

    kind = rng.choice(["shot", "shot", "shot", "shot", "restart", "gradient", "autograd", "serve"])
    dz = rng.choice([10.0, 10.0, 8.0, 5.0])
    if kind == "serve":
        return {"kind": "serve", "nx": 0, "ny": 0, "nz": 0, "dz": dz, "nsteps": 0,
                "storage": rng.choice(["f32", "f32", "f16"]), "npml": 0,
                "shots": rng.randint(3, 8), "steps_lo": 40, "steps_hi": rng.randint(60, 160),
                "mix": rng.randint(2, 1 << 20), "layer_every": rng.choice([0, 2, 3])}
    top = {"shot": 800, "restart": 400, "gradient": 256, "autograd": 200}[kind]
    nx, ny, nz = size(48, top), size(48, top), size(48, min(top, 512))
    npml = 0 if kind == "restart" else rng.choice([0, 0, 8, 10, 16, 20])
    # steps: at most 2e10 point updates, the work of the largest listed case
    most = {"shot": 2e10, "restart": 1e10, "gradient": 3e9, "autograd": 2e9}[kind]
    nsteps = max(8, min(rng.randint(40, 300), int(most / (nx * ny * nz))))
    c = {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "dz": dz, "nsteps": nsteps,
         "storage": "f32", "npml": npml}
    if kind in ("shot", "restart"):
        c["storage"] = rng.choice(["f32", "f32", "f16", "bf16"])
        if c["storage"] == "bf16":  # 8 significant bits: good for short runs
            c["nsteps"] = max(8, nsteps % 20)
    else:
        c["ckpt"] = rng.randint(10, 40)
    return c


# ---------------------------------------------------------------------------
# Inputs.

def _smooth(gen, nx, ny, nz, cells):
    """Smooth noise in [-1, 1] of about `cells` points per bump, on the GPU."""
    coarse = torch.rand((1, 1, nz // cells + 2, ny // cells + 2, nx // cells + 2), generator=gen)
    coarse = (2.0 * coarse - 1.0).cuda()
    return torch.nn.functional.interpolate(coarse, size=(nz, ny, nx), mode="trilinear",
                                           align_corners=True)[0, 0]


def _model(gen, nx, ny, nz):
    """Random layered velocities with smooth lateral variation; (nz, ny, nx) float32."""
    depth = torch.sort(torch.randint(1, max(2, nz), (7,), generator=gen)).values
    vel = torch.sort(1500.0 + 3000.0 * torch.rand(8, generator=gen)).values
    vz = vel[torch.bucketize(torch.arange(nz), depth, right=True)].cuda()
    eta = _smooth(gen, nx, ny, nz, 24)
    return eta.mul_(0.05).add_(1.0).mul_(vz[:, None, None]).contiguous()


def _dt(h, vmax):
    """Half the leapfrog stability limit of the 25-point stencil."""
    s = abs(W2[0]) + 2.0 * sum(abs(w) for w in W2[1:])
    return 0.5 * 2.0 / (vmax * math.sqrt(s * sum(1.0 / (a * a) for a in h)))


def _plane(nx, ny, z):
    xs = torch.arange(0, nx, 4, dtype=torch.int32)
    ys = torch.arange(0, ny, 4, dtype=torch.int32)
    yy, xx = torch.meshgrid(ys, xs, indexing="ij")
    return torch.stack([xx.reshape(-1), yy.reshape(-1),
                        torch.full((xx.numel(),), z, dtype=torch.int32)], 1).contiguous()


def _survey(c, gen):
    """Model, spacing, time step, source and receivers of one grid."""
    nx, ny, nz, npml = c["nx"], c["ny"], c["nz"], c["npml"]
    h = (10.0, 10.0, c["dz"])
    vel = _model(gen, nx, ny, nz)
    sx = int(torch.randint(nx // 4, max(nx // 4 + 1, 3 * nx // 4), (1,), generator=gen))
    sy = int(torch.randint(ny // 4, max(ny // 4 + 1, 3 * ny // 4), (1,), generator=gen))
    # source and receivers below the top layer, as a survey places them
    shot = (sx, sy, min(npml + 10, nz - 1), F_PEAK, -1.0, 1.0)
    rec = _plane(nx, ny, min(npml + 8, nz - 1))
    return vel, h, _dt(h, float(vel.max())), shot, rec


def _observed(gen, nsteps, nrec, dt):
    """Observed traces: on each receiver three Ricker arrivals at random times."""
    t = torch.arange(nsteps, dtype=torch.float32)[:, None].cuda() * dt
    out = torch.zeros((nsteps, nrec), device="cuda")
    for _ in range(3):
        t0 = (torch.rand(nrec, generator=gen) * nsteps * dt).cuda()
        amp = (0.1 * (2.0 * torch.rand(nrec, generator=gen) - 1.0)).cuda()
        a = (math.pi * F_PEAK) ** 2 * (t - t0) ** 2
        out += amp * (1.0 - 2.0 * a) * torch.exp(-a)
    return out


def _shots(c):
    """The shots of a serve case: a case each, by the case's own numbers."""
    gen = torch.Generator().manual_seed(int(c["mix"]))
    out = []
    for i in range(int(c["shots"])):
        n = [SERVE_SIZES[int(torch.randint(len(SERVE_SIZES), (1,), generator=gen))]
             for _ in range(3)]
        if n[0] * n[1] * n[2] > 1 << 26:
            n[2] = 128
        steps = int(torch.randint(c["steps_lo"], c["steps_hi"] + 1, (1,), generator=gen))
        layered = c["layer_every"] > 0 and i % c["layer_every"] == 0
        out.append({"kind": "shot", "nx": n[0], "ny": n[1], "nz": n[2], "dz": c["dz"],
                    "nsteps": steps, "storage": c["storage"], "npml": 16 if layered else 0})
    return out


def _solver(c, vel, h, dt):
    s = gw.WaveSolver((c["nx"], c["ny"], c["nz"]), h, dt, vel, storage=STORAGE[c["storage"]])
    if c["npml"]:
        s.set_cpml(c["npml"], REFLECTION, F_PEAK)
    return s


def prepare(case, seed):
    gen = torch.Generator().manual_seed(int(seed))
    s = {"case": case}
    if case["kind"] == "serve":
        s["server"] = gw.ShotServer(40 * 10 ** 9, 32)
        s["shots"] = []
        for c in _shots(case):
            vel, h, dt, shot, rec = _survey(c, gen)
            rec = rec.cuda()
            s["shots"].append((c, vel, h, dt, shot, rec,
                               torch.empty((c["nsteps"], rec.shape[0]), device="cuda")))
        return s
    vel, h, dt, shot, rec = _survey(case, gen)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    s.update(h=h, dt=dt, shot=shot, rec=rec.cuda())
    if case["kind"] == "autograd":
        s["m"] = (vel * vel).requires_grad_(True)
        s["observed"] = _observed(gen, case["nsteps"], rec.shape[0], dt)
        return s
    s["solver"] = _solver(case, vel, h, dt)
    s["u"] = torch.empty((nz, ny, nx), device="cuda")
    if case["kind"] == "restart":
        s["u0"] = _smooth(gen, nx, ny, nz, 6).contiguous()
        s["up0"] = (0.98 * s["u0"] + 0.02 * _smooth(gen, nx, ny, nz, 6)).contiguous()
        s["up"] = torch.empty((nz, ny, nx), device="cuda")
    else:
        s["traces"] = torch.empty((case["nsteps"], rec.shape[0]), device="cuda")
    if case["kind"] == "gradient":
        s["observed"] = _observed(gen, case["nsteps"], rec.shape[0], dt)
    return s


def run(s):
    c = s["case"]
    if c["kind"] == "shot":
        s["solver"].reset()
        s["solver"].propagate(s["shot"], c["nsteps"], s["rec"], s["traces"])
        return {"traces": s["traces"], "u": s["solver"].get_field(0, s["u"])}
    if c["kind"] == "restart":
        s["solver"].set_state(s["u0"], s["up0"], 7)
        s["solver"].step(c["nsteps"])
        return {"u": s["solver"].get_field(0, s["u"]), "up": s["solver"].get_field(1, s["up"])}
    if c["kind"] == "gradient":
        misfit = s["solver"].gradient(s["shot"], c["nsteps"], s["rec"], s["observed"], s["u"],
                                      ckpt_every=c["ckpt"], traces=s["traces"])
        return {"misfit": misfit, "grad": s["u"], "traces": s["traces"]}
    if c["kind"] == "autograd":
        layer = (c["npml"], REFLECTION, F_PEAK) if c["npml"] else None
        traces = gw.wave_traces(s["m"], s["h"], s["dt"], s["shot"], c["nsteps"], s["rec"],
                                ckpt_every=c["ckpt"], cpml=layer)
        loss = 0.5 * (traces - s["observed"]).square().sum()
        grad, = torch.autograd.grad(loss, s["m"])
        return {"traces": traces.detach(), "grad": grad}
    tickets = []
    for k, vel, h, dt, shot, rec, traces in s["shots"]:
        layer = (k["npml"], REFLECTION, F_PEAK) if k["npml"] else None
        tickets.append(s["server"].submit((k["nx"], k["ny"], k["nz"]), h, vel, shot, k["nsteps"],
                                          rec, traces, storage=STORAGE[k["storage"]], dt=dt,
                                          cpml=layer))
    for t in tickets:
        status, _ = s["server"].wait(t)
        if status != 0:
            raise RuntimeError("shot %d failed with status %d" % (t, status))
    return [x[-1] for x in s["shots"]]


def work(case):
    """Each step reads u, u_prev and v^2 dt^2 and writes u_next once (the fields
    4 or 2 bytes, v^2 dt^2 always 4), and with the layer reads and writes psi
    and zeta once in the slabs. A gradient takes three such passes (forward,
    recompute, adjoint), writes and reads the stored increment and reads and
    writes the time sum. About 40 operations a point and pass."""
    if case["kind"] == "serve":
        parts = [work(c) for c in _shots(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    nx, ny, nz, n, p = case["nx"], case["ny"], case["nz"], case["nsteps"], case["npml"]
    pts = nx * ny * nz
    slab = 16.0 * 2 * p * (ny * nz + nz * nx + nx * ny)
    step = pts * (16.0 if case["storage"] == "f32" else 10.0) + slab
    nrec = (-(-nx // 4)) * (-(-ny // 4))
    if case["kind"] in ("gradient", "autograd"):
        return {"bytes": n * (3 * step + pts * 16.0) + 4.0 * pts + 8.0 * n * nrec,
                "flops": 3 * 40.0 * pts * n}
    out = 4.0 * pts + 4.0 * n * nrec if case["kind"] == "shot" else 16.0 * pts
    return {"bytes": n * step + out, "flops": 40.0 * pts * n}


# ---------------------------------------------------------------------------
# The same results in 64 bits, in plain torch.

class _Grid64:
    """Eq. 1 and the layer's first derivatives on one grid, with a zero halo."""

    def __init__(self, shape, h, c, dt, npml, vmax):
        self.shape, self.h, self.c, self.npml = shape, h, c, npml
        nz, ny, nx = shape
        self.a, self.b = [None] * 3, [None] * 3
        for ax, n in ((0, nx), (1, ny), (2, nz)):
            if not npml:
                continue
            d0 = 3.0 * vmax * math.log(1.0 / REFLECTION) / (2.0 * npml * h[ax])
            a, b = torch.zeros(n, dtype=torch.float64), torch.ones(n, dtype=torch.float64)
            for i in range(n):
                xi = max((npml - i) / npml, (i - (n - npml - 1)) / npml)
                if xi > 0:
                    d, al = d0 * xi * xi, math.pi * F_PEAK * (1.0 - xi)
                    b[i] = math.exp(-(d + al) * dt)
                    a[i] = d / (d + al) * (float(b[i]) - 1.0)
            view = [1, 1, 1]
            view[2 - ax] = n
            self.a[ax], self.b[ax] = a.cuda().view(view), b.cuda().view(view)

    def deriv(self, f, ax, order, out=None):
        """Adds the derivative of f along axis ax (0 = x) to out."""
        dim, n, h = 2 - ax, f.shape[2 - ax], self.h[ax]
        out = torch.zeros_like(f) if out is None else out
        if order == 2:
            out.add_(f, alpha=W2[0] / (h * h))
        for m in range(1, 5):
            if m >= n:
                break
            w = W2[m] / (h * h) if order == 2 else W1[m] / h
            lo, hi = (x.narrow(dim, y, n - m) for x, y in ((out, 0), (f, m)))
            lo.add_(hi, alpha=w)
            hi, lo = (x.narrow(dim, y, n - m) for x, y in ((out, m), (f, 0)))
            hi.add_(lo, alpha=w if order == 2 else -w)
        return out

    def lap(self, f):
        out = torch.zeros_like(f)
        for ax in range(3):
            self.deriv(f, ax, 2, out)
        return out

    def slabs(self):
        return [torch.zeros(self.shape, dtype=torch.float64, device="cuda") if self.npml else None
                for _ in range(3)]

    def increment(self, u, psi, zeta):
        """C (L u + the layer's terms), psi and zeta stepped in place."""
        s = self.lap(u)
        for ax in range(3 if self.npml else 0):
            psi[ax].mul_(self.b[ax]).add_(self.a[ax] * self.deriv(u, ax, 1))
            d1 = self.deriv(psi[ax], ax, 1)
            zeta[ax].mul_(self.b[ax]).add_(self.a[ax] * (self.deriv(u, ax, 2) + d1))
            s.add_(d1).add_(zeta[ax])
        return s.mul_(self.c)

    def adjoint(self, p, nu, mu):
        """C (L p + the layer's transposed terms), nu and mu stepped in place."""
        s = self.lap(p)
        for ax in range(3 if self.npml else 0):
            inside = (self.a[ax] != 0).to(torch.float64)
            nu[ax].mul_(self.b[ax]).add_(p).mul_(inside)
            an = self.a[ax] * nu[ax]
            mu[ax].mul_(self.b[ax]).sub_(self.deriv(p + an, ax, 1)).mul_(inside)
            self.deriv(an, ax, 2, s)
            s.sub_(self.deriv(self.a[ax] * mu[ax], ax, 1))
        return s.mul_(self.c)


def _ricker(t):
    a = (math.pi * F_PEAK * (t - 1.0 / F_PEAK)) ** 2
    return (1.0 - 2.0 * a) * math.exp(-a)


def _forward64(g, dt, shot, rec, nsteps, u=None, up=None, keep=None):
    psi, zeta = g.slabs(), g.slabs()
    u = torch.zeros(g.shape, dtype=torch.float64, device="cuda") if u is None else u
    up = torch.zeros_like(u) if up is None else up
    traces = []
    if rec is not None:
        rx, ry, rz = (rec[:, i].long().cuda() for i in range(3))
    for n in range(nsteps):
        d = g.increment(u, psi, zeta)
        if shot is not None:
            sx, sy, sz = shot[:3]
            d[sz, sy, sx] += g.c[sz, sy, sx] * _ricker(n * dt)
        if keep is not None:
            keep.append(d)
        u, up = up.neg_().add_(u, alpha=2.0).add_(d), u
        if rec is not None:
            traces.append(u[rz, ry, rx].clone())
    return u, up, torch.stack(traces) if traces else None


def _gradient64(g, m, dt, shot, rec, nsteps, observed):
    kept = []
    _, _, traces = _forward64(g, dt, shot, rec, nsteps, keep=kept)
    resid = traces - observed.double()
    rx, ry, rz = (rec[:, i].long().cuda() for i in range(3))
    nu, mu = g.slabs(), g.slabs()
    p1 = torch.zeros(g.shape, dtype=torch.float64, device="cuda")
    p2, total = torch.zeros_like(p1), torch.zeros_like(p1)
    for k in range(nsteps, 0, -1):  # p^k, paired with the increment of step k - 1
        p = 2.0 * p1 - p2 + g.adjoint(p1, nu, mu)
        p.index_put_((rz, ry, rx), g.c[rz, ry, rx] * resid[k - 1], accumulate=True)
        total += p * kept[k - 1]
        p1, p2 = p, p1
    return traces, 0.5 * float(resid.square().sum()), total / (g.c * m)


def _exact_shot(c, gen):
    vel, h, dt, shot, rec = _survey(c, gen)
    v = vel.double()
    g = _Grid64(v.shape, h, v * v * (dt * dt), dt, c["npml"], float(vel.max()))
    return vel, dt, shot, rec, g


def exact(case, seed):
    gen = torch.Generator().manual_seed(int(seed))
    if case["kind"] == "serve":
        out = []
        for c in _shots(case):
            _, dt, shot, rec, g = _exact_shot(c, gen)
            out.append(_forward64(g, dt, shot, rec, c["nsteps"])[2])
        return out
    vel, dt, shot, rec, g = _exact_shot(case, gen)
    nx, ny, nz, nsteps = case["nx"], case["ny"], case["nz"], case["nsteps"]
    if case["kind"] == "shot":
        u, _, traces = _forward64(g, dt, shot, rec, nsteps)
        return {"traces": traces, "u": u}
    if case["kind"] == "restart":
        u0 = _smooth(gen, nx, ny, nz, 6).contiguous()
        up0 = (0.98 * u0 + 0.02 * _smooth(gen, nx, ny, nz, 6)).contiguous()
        u, up, _ = _forward64(g, dt, None, None, nsteps, u0.double(), up0.double())
        return {"u": u, "up": up}
    observed = _observed(gen, nsteps, rec.shape[0], dt)
    m = vel.double().square()
    if case["kind"] == "autograd":  # the model handed over is the rounded square
        m = (vel * vel).double()
        g = _Grid64(g.shape, g.h, m * (dt * dt), dt, case["npml"], math.sqrt(float(m.max())))
    traces, misfit, grad = _gradient64(g, m, dt, shot, rec, nsteps, observed)
    if case["kind"] == "autograd":
        return {"traces": traces, "grad": grad}
    return {"misfit": misfit, "grad": grad, "traces": traces}
