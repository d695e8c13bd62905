"""The work that users of this framework have it do, as measurable cases.

A case is a dict of plain values.  prepare() makes its inputs and the handle a
program keeps, run() is one pass through the public entry points, work() the
bytes and operations a pass cannot do without, exact() the same outputs in
plain float64 torch.

Kinds of work:
- "run": a forward run.  Load the fields, take `steps` steps, read the
  macroscopic fields and the conservation sums.  With `every` > 0 the sums are
  also read every so many steps (the time series of melted fraction and
  Nusselt number that a melting study plots).
- "batch": several cavities of uneven size advanced together.
- "adjoint": the conduction step's objective and gradients.
- "coupled": the coupled step's objective and gradients (flow on).

Everything is drawn from the seed on the device: porosity and permeability
fields as smoothed noise, fronts at a seeded place near the case's `melted`.
"""
import math

import numpy as np
import torch

from paper_1503_08406_gb300 import Batch, Lattice


def listed():
    return [
        # Conduction melting of a porous slab, 256 x 4, periodic in y, no flow: the smallest
        # standard configuration; each step is far below a microsecond of memory traffic, so
        # launches and latency are what it costs.
        dict(name="slab_256x4", kind="run", shape="slab", nx=256, ny=4, steps=200, every=0,
             St=1.0, nu=0.0, Da=1e-2, melted=0.2, storage="fp32"),
        # A first look at a small cavity: a few steps, the sums read along the way.
        dict(name="cavity_48", kind="run", shape="cavity", nx=48, ny=48, steps=30, every=10,
             St=1.0, nu=0.026, Da=1e-3, melted=0.33, storage="fp32"),
        # Convection melting in the 256 x 256 cavity (Ra = 1e5), a stretch of a long run with
        # its time series.
        dict(name="cavity_256", kind="run", shape="cavity", nx=256, ny=256, steps=256, every=64,
             St=1.0, nu=0.14, Da=1e-4, melted=0.4, storage="fp32"),
        # The gallium / glass-bead cavity, 200 x 200 (ragged tiles), with a mushy band, both
        # heat-capacity ratios, extrapolated no-slip on the walls and on the moving front.
        dict(name="gallium_200", kind="run", shape="gallium", nx=200, ny=200, steps=100, every=0,
             St=0.1241, nu=0.0054, Da=1.37e-5, melted=0.5, storage="fp32"),
        # The headline: heterogeneous 2048 x 2048 cavity, seven eighths melted.
        dict(name="cavity_2048", kind="run", shape="cavity", nx=2048, ny=2048, steps=64, every=0,
             St=1.0, nu=0.2, Da=1e-4, melted=0.875, storage="fp32"),
        # A cavity whose rows are no multiple of anything.
        dict(name="cavity_1001x701", kind="run", shape="cavity", nx=1001, ny=701, steps=64,
             every=0, St=0.5, nu=0.1, Da=1e-4, melted=0.6, storage="fp32"),
        # A doubly periodic box: a melted inclusion convecting in a closed porous medium.
        dict(name="box_768x640", kind="run", shape="box", nx=768, ny=640, steps=65, every=0,
             St=0.5, nu=0.06, Da=1e-2, melted=0.3, storage="fp32"),
        # 16-bit population storage: half the memory per node.
        dict(name="cavity_1024_fp16", kind="run", shape="cavity", nx=1024, ny=1024, steps=64,
             every=0, St=1.0, nu=0.1, Da=1e-4, melted=0.6, storage="fp16"),
        # The largest: a wide tank in bf16.
        dict(name="cavity_4096x2048_bf16", kind="run", shape="cavity", nx=4096, ny=2048, steps=48,
             every=0, St=1.0, nu=0.12, Da=1e-4, melted=0.7, storage="bf16"),
        # A parameter study: cavities of sides 64 to 512 advanced together.
        dict(name="batch_24", kind="batch", count=24, least=64, most=512, steps=64, melted=0.3),
        # Gradient of the melted fraction through the conduction step, in porosity and the wall
        # profile, the front a few nodes from the wall (where it is for most of such a run).
        dict(name="adjoint_2048x512", kind="adjoint", nx=2048, ny=512, steps=96,
             objective="melt", front=8),
        # The inverse problem (gradients in porosity, ln K and the wall profile) with
        # checkpoints every 10 steps, as its long runs need.
        dict(name="coupled_256", kind="coupled", nx=256, ny=256, steps=100, checkpoint=10,
             objective="melt", front=12),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    """One more case of the same ranges.  Sizes are spread over their logarithm."""
    kind = rng.choice(("run", "run", "run", "run", "run", "batch", "adjoint", "coupled"))
    melted = round(rng.uniform(0.15, 0.85), 3)
    if kind == "batch":
        most = rng.choice((128, 192, 256, 384, 512))
        return dict(kind=kind, count=rng.randint(4, 24), least=64, most=most,
                    steps=rng.choice((32, 48, 64, 65)), melted=round(rng.uniform(0.1, 0.6), 3))
    if kind == "adjoint":
        nx, ny, front = int(_log(rng, 40, 2048)), int(_log(rng, 4, 512)), rng.randint(4, 10)
        return dict(kind=kind, nx=nx, ny=ny, steps=rng.randint(48, 96),
                    objective="melt" if front > 6 else "nusselt", front=front)
    if kind == "coupled":
        nx, ny, front = int(_log(rng, 40, 256)), int(_log(rng, 40, 256)), rng.randint(4, 14)
        return dict(kind=kind, nx=nx, ny=ny, steps=rng.randint(48, 100),
                    checkpoint=rng.choice((0, 7, 10)),
                    objective="melt" if front > 6 else "nusselt", front=front)
    shape = rng.choice(("slab", "cavity", "cavity", "cavity", "gallium", "box"))
    storage = rng.choice(("fp32", "fp32", "fp32", "fp16", "bf16")) if shape == "cavity" else "fp32"
    if shape == "slab":
        nx, ny = int(_log(rng, 100, 2048)), int(_log(rng, 4, 64))
    elif shape == "gallium":
        nx = ny = int(_log(rng, 64, 400))
    else:
        nx, ny = int(_log(rng, 48, 3000)), int(_log(rng, 48, 2400))
        if rng.random() < 0.6:   # most users take round widths
            nx = max(48, nx // 8 * 8)
    steps = max(24, min(256, int(2.0e8 / (nx * ny))))
    steps = rng.randint(steps // 2, steps)
    if shape == "gallium":
        steps += steps & 1
    return dict(kind=kind, shape=shape, nx=nx, ny=ny, steps=steps,
                every=rng.choice((0, 0, max(1, steps // 4))), St=round(rng.uniform(0.3, 1.0), 3)
                if shape != "gallium" else 0.1241, nu={"slab": 0.0, "gallium": 0.0054}.get(
                    shape, round(_log(rng, 0.03, 0.14), 4)),
                Da={"slab": 1e-2, "gallium": 1.37e-5, "box": 1e-2}.get(
                    shape, round(_log(rng, 1e-5, 1e-3), 7)),
                melted=0.3 if shape == "box" else melted, storage=storage)


# ---- inputs -------------------------------------------------------------------------------

def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _smooth(gen, ny, nx, cells):
    """Unit-variance, zero-mean noise smoothed by a periodic Gaussian of `cells` cells."""
    dev = gen.device
    g = torch.randn((ny, nx), generator=gen, device=dev, dtype=torch.float32)
    ky = torch.fft.fftfreq(ny, device=dev)[:, None]
    kx = torch.fft.rfftfreq(nx, device=dev)[None, :]
    kern = torch.exp(-2.0 * math.pi ** 2 * cells ** 2 * (kx ** 2 + ky ** 2))
    s = torch.fft.irfft2(torch.fft.rfft2(g) * kern, s=(ny, nx))
    s = s - s.mean()
    return s / s.std().clamp_min(1e-12)


def _kozeny(phi, mean_k):
    """K = phi^3 d^2 / (175 (1 - phi)^2) with the particle diameter that gives its mean."""
    shape = phi ** 3 / (1.0 - phi) ** 2
    return shape * (mean_k / shape.mean())


def _fields(case, gen):
    """(params, phi, K, T0, fl0, wall profile or None) of one lattice."""
    nx, ny, dev = case["nx"], case["ny"], gen.device
    x = torch.arange(nx, device=dev, dtype=torch.float32)[None, :].expand(ny, nx)
    y = torch.arange(ny, device=dev, dtype=torch.float32)[:, None].expand(ny, nx)
    u = float(torch.rand((), generator=gen, device=dev))
    front = case["front"] + u if "front" in case else case["melted"] * nx + 0.04 * (u - 0.5) * nx
    front = max(2.0, min(nx - 3.0, front))
    liquid = (x < front).float()
    kind = case["kind"]
    wall = None
    if kind == "adjoint":
        params = dict(bc=("dirichlet", "dirichlet", "periodic", "periodic"),
                      T_bc=(1.0, -1.0, 0.0, 0.0), flow=0, St=1.0, sigma=1.0, dT=1.0, T_s=-0.3,
                      T_l=0.3, tau_T=0.6, H=float(nx))
        phi = 0.6 + 0.2 * torch.rand((ny, nx), generator=gen, device=dev)
        K = torch.full((ny, nx), 1e3, device=dev)
        T0 = torch.where(x < front, 1.0 - 2.0 * x / front, torch.full_like(x, -1.0))
        fl0 = ((T0 + 0.3) / 0.6).clamp(0.0, 1.0)
        yy = torch.arange(ny, device=dev, dtype=torch.float32)
        wall = 1.0 + 0.2 * torch.sin(2.0 * math.pi * (yy / ny + u))
        T0[:, 0] = 1.0
        fl0[:, 0] = 1.0
        return params, phi, K, T0, fl0, wall
    if kind == "coupled":
        nu = 0.1   # tau_nu - 1/2
        params = dict(bc=("dirichlet", "dirichlet", "adiabatic", "adiabatic"),
                      T_bc=(1.0, -0.05, 0.0, 0.0), flow=1, Ra=3.0 * (0.1 * ny / nu) ** 2, Pr=1.0,
                      Ma=0.1, J=1.0, lambda_=1.0, sigma=1.0, St=1.0, dT=1.0, H=float(ny),
                      T_ref=0.0, T_s=0.0, T_l=0.05)
        phi = (0.45 + 0.15 * _smooth(gen, ny, nx, 8.0)).clamp(0.3, 0.6)
        K = torch.exp(0.5 * _smooth(gen, ny, nx, 11.0))
        K = K * (1e-5 * ny * ny / K.mean())
        T0 = torch.where(x < front, 1.0 - 0.95 * x / front, torch.full_like(x, -0.05))
        T0[:, 0] = 1.0
        return params, phi, K, T0, liquid, torch.ones(ny, device=dev)
    shape = case["shape"]
    if shape == "slab":
        params = dict(bc=("dirichlet", "dirichlet", "periodic", "periodic"),
                      T_bc=(1.0, 0.0, 0.0, 0.0), flow=0, St=case["St"], sigma=1.0, dT=1.0,
                      T_s=0.0, T_l=0.0, tau_T=0.6, H=float(nx))
        phi = torch.full((ny, nx), 0.4 + 0.2 * u, device=dev)
        K = torch.full((ny, nx), case["Da"] * nx * nx, device=dev)
        T0 = torch.where(x < front, 1.0 - x / front, torch.zeros_like(x))
    elif shape == "gallium":
        T_m = (29.78 - 20.0) / 25.0
        params = dict(bc=("dirichlet", "dirichlet", "adiabatic", "adiabatic"),
                      T_bc=(1.0, 0.0, 0.0, 0.0), flow=1, Pr=0.0208, Ma=0.1, J=1.0,
                      Ra=3.0 * 0.0208 * (0.1 * ny / case["nu"]) ** 2, lambda_=0.2719,
                      sigma=0.8604, sigma_solid=0.8352, St=case["St"], dT=1.0, H=float(ny),
                      T_ref=0.0, T_s=T_m - 0.02, T_l=T_m + 0.02, flow_walls=1, flow_front=1)
        phi = torch.full((ny, nx), 0.385, device=dev)
        K = torch.full((ny, nx), case["Da"] * ny * ny * (0.9 + 0.2 * u), device=dev)
        T0 = torch.where(x < front, 1.0 - (0.98 - T_m) * x / front, torch.zeros_like(x))
    elif shape == "box":
        params = dict(bc=("periodic",) * 4, T_bc=(0.0,) * 4, flow=1, Pr=1.0, Ma=0.1, J=1.0,
                      Ra=3.0 * (0.1 * ny / case["nu"]) ** 2, lambda_=1.0, sigma=1.0,
                      St=case["St"], dT=1.0, H=float(ny), T_ref=0.0, T_s=0.0, T_l=0.0)
        phi = (0.45 + 0.1 * _smooth(gen, ny, nx, 6.0)).clamp(0.3, 0.6)
        K = _kozeny(phi, case["Da"] * ny * ny)
        r = torch.hypot(x - nx * (0.3 + 0.1 * u), y - ny / 2.0)
        T0 = torch.where(r < case["melted"] * min(nx, ny), 0.8, -0.2)
        T0 = T0 + 0.02 * _smooth(gen, ny, nx, 6.0)
        liquid = (T0 > 0.0).float()
    else:
        params = dict(bc=("dirichlet", "dirichlet", "adiabatic", "adiabatic"),
                      T_bc=(1.0, 0.0, 0.0, 0.0), flow=1, Ra=3.0 * (0.1 * ny / case["nu"]) ** 2,
                      Pr=1.0, Ma=0.1, J=1.0, lambda_=1.0, sigma=1.0, St=case["St"], dT=1.0,
                      H=float(ny), T_ref=0.0, T_s=0.0, T_l=0.0)
        phi = (0.45 + 0.15 * _smooth(gen, ny, nx, 16.0 if min(nx, ny) > 128 else 6.0)).clamp(0.3,
                                                                                            0.6)
        K = _kozeny(phi, case["Da"] * ny * ny)
        T0 = torch.where(x < front, 1.0 - x / front, torch.zeros_like(x))
    if shape != "box":
        T0[:, 0], liquid[:, 0] = 1.0, 1.0
    return params, phi, K, T0, liquid, wall


def _members(case, gen):
    """The cavities of a batch: side, tau and St drawn per cavity, each a "run" case."""
    n = case["count"]
    u = torch.rand((n, 3), generator=gen, device=gen.device).cpu().numpy()
    sides = [s for s in (64, 96, 128, 192, 256, 384, 512) if case["least"] <= s <= case["most"]]
    out = []
    for k in range(n):
        # every size in turn, so that the work does not hang on the seed
        side = sides[k % len(sides)]
        out.append(dict(kind="run", shape="cavity", nx=side, ny=side, steps=case["steps"], every=0,
                        St=round(0.3 + 0.7 * float(u[k, 0]), 3),
                        nu=round(0.03 + 0.1 * float(u[k, 1]), 4),
                        Da=1e-4 * 10.0 ** round(float(u[k, 2]), 2),
                        melted=case["melted"], storage="fp32"))
    return out


def _inputs(case, seed):
    gen = torch.Generator(device=_device()).manual_seed(int(seed) % (1 << 62))
    if case["kind"] != "batch":
        return [(case, *_fields(case, gen))]
    return [(m, *_fields(m, gen)) for m in _members(case, gen)]


def prepare(case, seed):
    lats = []
    for m, params, *fields in _inputs(case, seed):
        lat = Lattice(m["nx"], m["ny"], **params, storage=m.get("storage", "fp32"))
        lats.append((lat, [None if t is None else t.contiguous() for t in fields]))
    state = dict(case=case, lats=lats)
    if case["kind"] == "batch":
        state["batch"] = Batch([lat for lat, _ in lats])
    return state


def run(state):
    case = state["case"]
    for lat, (phi, K, T0, fl0, wall) in state["lats"]:
        lat.set_fields(phi, K, T0, fl0, wall)
    if case["kind"] == "batch":
        state["batch"].step(case["steps"])
        return _together([lat.macros(numpy=False) for lat, _ in state["lats"]])
    lat = state["lats"][0][0]
    if case["kind"] == "adjoint":
        J, dphi, dwall = lat.adjoint(case["steps"], case["objective"], device=True)
        return dict(J=J, dphi=dphi, dwall=dwall)
    if case["kind"] == "coupled":
        J, dphi, dlnK, dwall = lat.adjoint_coupled(case["steps"], case["objective"],
                                                   checkpoint_every=case["checkpoint"],
                                                   device=True)
        return dict(J=J, dphi=dphi, dlnK=dlnK, dwall=dwall)
    sums, left = [], case["steps"]
    while case["every"] and left > case["every"]:
        lat.step(case["every"])
        left -= case["every"]
        sums.append(lat.reduce())
    lat.step(left)
    sums.append(lat.reduce())
    out = lat.macros(numpy=False)
    return dict(out, sums=[[s[k] for k in _sums(case)] for s in sums])


def _together(fields):
    """The members' fields one after another, field by field."""
    return {k: torch.cat([f[k].reshape(-1) for f in fields]) for k in fields[0]}


def _sums(case):
    """The sums a case reads: a doubly periodic box has no hot wall, and 16-bit storage does
    not resolve the wall gradient of a large lattice over a few steps."""
    hot = case["shape"] != "box" and case["storage"] == "fp32"
    return ("mass", "enthalpy", "melt_frac") + (("nu_hot",) if hot else ())


# ---- work ---------------------------------------------------------------------------------

def work(case):
    """Per step, a node that carries flow reads and writes 14 populations and reads f_l, phi and
    K; another one 5 populations and f_l.  The flow collision takes about 330 operations, the
    thermal one about 70.  The fields are loaded and the macroscopic fields written once.  A
    gradient also runs the step's transpose: the populations of the state and the adjoints
    before and after it."""
    if case["kind"] == "batch":
        gen = torch.Generator(device="cpu").manual_seed(0)
        parts = [work(m) for m in _members(case, gen)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    n = case["nx"] * case["ny"]
    if case["kind"] == "adjoint":   # forward 44 B; reverse: adjoints 5 + 1 in and out, f_l twice
        return dict(bytes=n * (case["steps"] * (44 + 56) + 16 + 4),
                    flops=n * case["steps"] * (70 + 90))
    liquid = case["front"] / case["nx"] if "front" in case else case["melted"]
    liquid = liquid if case.get("shape") != "box" else math.pi * 0.3 ** 2 * 0.8
    flow = 0.0 if case.get("shape") == "slab" else liquid
    if case["kind"] == "coupled":   # reverse: the state 15, adjoints 15 in and 15 out, sums 2 + 2
        return dict(bytes=n * (case["steps"] * (124 * flow + 44 * (1 - flow) + 4 * 49) + 16 + 8),
                    flops=n * case["steps"] * (flow * (400 + 1100) + 240))
    size = 4 if case["storage"] == "fp32" else 2
    step = flow * (28 * size + 12) + (1 - flow) * (10 * size + 4)
    return dict(bytes=n * (case["steps"] * step + 16 + 20),
                flops=n * case["steps"] * (330 * flow + 70))


# ---- the same in float64 ------------------------------------------------------------------

_EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
_EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
_OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
_M = np.array([[1, 1, 1, 1, 1, 1, 1, 1, 1], [-4, -1, -1, -1, -1, 2, 2, 2, 2],
               [4, -2, -2, -2, -2, 1, 1, 1, 1], [0, 1, 0, -1, 0, 1, -1, -1, 1],
               [0, -2, 0, 2, 0, 1, -1, -1, 1], [0, 0, 1, 0, -1, 1, 1, -1, -1],
               [0, 0, -2, 0, 2, 1, 1, -1, -1], [0, 1, -1, 1, -1, 0, 0, 0, 0],
               [0, 0, 0, 0, 0, 1, -1, 1, -1]], dtype=np.float64)
_N = np.array([[1, 1, 1, 1, 1], [0, 1, 0, -1, 0], [0, 0, 1, 0, -1], [-4, 1, 1, 1, 1],
               [0, 1, -1, 1, -1]], dtype=np.float64)


def _from(t, i):
    """The value at x - e_i (the last two axes are y, x)."""
    return torch.roll(t, (_EY[i], _EX[i]), (-2, -1)) if i else t


class _Enthalpy(torch.autograd.Function):
    """f_l(n+1): f = clamp((T* + sum_i w_i s(x - e_i) + a f - T_s) / (T_l - T_s + a), 0, 1) with
    s = -a (f - f_n), by sweeps to convergence; backward by the implicit function theorem."""

    @staticmethod
    def forward(ctx, tstar, a, fn, model):
        w0, w1, ts, dt, inside = model.w0, model.w1, model.T_s, model.dTm, model.inside
        av = torch.where(inside, a, torch.zeros_like(a))
        base, inv = tstar + w0 * a * fn - ts, 1.0 / (dt + w0 * a)
        f = fn.clone()
        for k in range(400):
            q = av * (f - fn)
            nb = _from(q, 1) + _from(q, 2) + _from(q, 3) + _from(q, 4)
            new = torch.where(inside, ((base - w1 * nb) * inv).clamp(0.0, 1.0), fn)
            last = k % 8 == 7 and float((new - f).abs().max()) < 1e-14
            f = new
            if last:
                break
        ctx.model = model
        ctx.save_for_backward(a, fn, f)
        return f

    @staticmethod
    def backward(ctx, lam):
        a, fn, f = ctx.saved_tensors
        w0, w1, inside = ctx.model.w0, ctx.model.w1, ctx.model.inside
        mushy = inside & (f > 0.0) & (f < 1.0)
        c = torch.where(mushy, 1.0 / (ctx.model.dTm + a), torch.zeros_like(a))
        # mu = lam + a c mu - a sum_i w_i (c mu)(y + e_i); nu = c mu
        den = 1.0 - a * (1.0 - w0) * c
        mu = torch.zeros_like(lam)
        for k in range(400):
            nu = c * mu
            nb = _from(nu, 1) + _from(nu, 2) + _from(nu, 3) + _from(nu, 4)
            new = (lam - a * w1 * nb) / den
            last = k % 8 == 7 and float((new - mu).abs().max()) <= 1e-14 * float(new.abs().max())
            mu = new
            if last:
                break
        nu = c * mu
        s = w0 * nu + w1 * (_from(nu, 1) + _from(nu, 2) + _from(nu, 3) + _from(nu, 4))
        s = torch.where(inside, s, torch.zeros_like(s))
        return nu, -(f - fn) * s, torch.where(inside, a * s, lam), None


class _Model:
    """One lattice of the double-MRT method in float64: two buffers, collide then stream."""

    def __init__(self, nx, ny, p, dev):
        g = lambda k, v: float(p.get(k, v))  # noqa: E731
        self.nx, self.ny, self.flow, self.dev = nx, ny, bool(p["flow"]), dev
        self.H, self.dT, self.sigma, self.St = g("H", ny), g("dT", 1), g("sigma", 1), g("St", 1)
        self.sigma_s = g("sigma_solid", self.sigma)
        self.T_s, self.T_l = g("T_s", 0), g("T_l", 0)
        self.dTm = self.T_l - self.T_s
        self.varpi, self.f_act = -2.0, 1e-3
        self.cs2t = (4.0 + self.varpi) / 10.0
        self.w0, self.w1 = (1.0 - self.varpi) / 5.0, (4.0 + self.varpi) / 20.0
        self.lat = self.dT / (self.sigma * self.St)
        if self.flow:
            ma, j, lam = g("Ma", 0.1), g("J", 1), g("lambda_", 1)
            nu = ma * j * self.H * math.sqrt(3.0 * p["Pr"]) / math.sqrt(p["Ra"])
            self.tau_nu = 0.5 + nu
            self.tau_T = 0.5 + lam * nu / 3.0 / (j * self.sigma * self.cs2t * p["Pr"])
            self.nu_l = nu / 3.0 / j
            self.g_beta = p["Ra"] * self.nu_l * (self.nu_l / p["Pr"]) / (self.dT * self.H ** 3)
        else:
            self.tau_T = g("tau_T", 1)
        self.bc, self.T_bc, self.T_ref = p["bc"], [float(t) for t in p["T_bc"]], g("T_ref", 0)
        self.walls, self.front = bool(p.get("flow_walls")), bool(p.get("flow_front"))
        px, py = self.bc[0] == "periodic", self.bc[2] == "periodic"
        self.px, self.py = px, py
        x = torch.arange(nx, device=dev)[None, :].expand(ny, nx)
        y = torch.arange(ny, device=dev)[:, None].expand(ny, nx)
        no = torch.zeros((ny, nx), dtype=torch.bool, device=dev)
        self.side = [no if px else x == 0, no if px else x == nx - 1, no if py else y == 0,
                     no if py else y == ny - 1]
        self.inside = ~(self.side[0] | self.side[1] | self.side[2] | self.side[3])
        ix = x if px else x.clamp(1, nx - 2)
        iy = y if py else y.clamp(1, ny - 2)
        self.inward = (iy, ix)
        # links that leave the lattice through a wall's outer face
        self.reach = [torch.ones_like(no)]
        for i in range(1, 9):
            sx, sy = x - _EX[i], y - _EY[i]
            self.reach.append((torch.ones_like(no) if px else (sx >= 0) & (sx < nx)) &
                              (torch.ones_like(no) if py else (sy >= 0) & (sy < ny)))
        t = lambda a: torch.tensor(a, dtype=torch.float64, device=dev)  # noqa: E731
        self.M, self.Minv = t(_M), t(np.linalg.inv(_M))
        self.N, self.Ninv = t(_N), t(np.linalg.inv(_N))
        if self.flow:
            s = 1.0 / self.tau_nu
            self.lam9 = t([1.0, 1.1, 1.1, 1.0, 1.2, 1.0, 1.2, s, s])[:, None, None]
        self.w9 = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4

    def start(self, T0, fl0):
        f = torch.zeros((9, self.ny, self.nx), dtype=torch.float64, device=self.dev)
        g = torch.stack([self.w0 * T0] + [self.w1 * T0] * 4)
        return f, g, fl0

    def velocity(self, f, T, fl, phi, K):
        """Eq. (24)-(28), (4)-(6): u, the force and varphi of populations f (deviations)."""
        e = [sum(c[i] * f[i] for i in range(1, 9) if c[i]) for c in (_EX, _EY)]
        vp = phi * fl
        G = self.g_beta * (T - self.T_ref)
        Ke = K * fl ** 3 * ((1.0 - phi) / (1.0 - vp)) ** 2
        cf = 1.75 / torch.sqrt(175.0 * vp ** 3)
        a1, a2 = vp * self.nu_l / Ke, vp * cf / torch.sqrt(Ke)
        vx, vy = e[0], e[1] + 0.5 * vp * G
        l0, l1 = 0.5 * (1.0 + 0.5 * a1), 0.5 * a2
        den = l0 + torch.sqrt(l0 ** 2 + l1 * torch.sqrt(vx ** 2 + vy ** 2 + 1e-300))
        ux, uy = vx / den, vy / den
        drag = a1 + a2 * torch.sqrt(ux ** 2 + uy ** 2 + 1e-300)
        return ux, uy, -drag * ux, -drag * uy + vp * G, vp

    def collide(self, f, T, fl, phi, K):
        """Eq. (16)-(23): the post-collision deviations and the velocity."""
        ux, uy, Fx, Fy, vp = self.velocity(f, T, fl, phi, K)
        m = torch.einsum("ki,iyx->kyx", self.M, f)
        uu, uF = (ux ** 2 + uy ** 2) / vp, (ux * Fx + uy * Fy) / vp
        eq = torch.stack([m[0], -2 * m[0] + 3 * uu, m[0] - 3 * uu, ux, -ux, uy, -uy,
                          (ux ** 2 - uy ** 2) / vp, ux * uy / vp])
        S = torch.stack([torch.zeros_like(ux), 6 * uF, -6 * uF, Fx, -Fx, Fy, -Fy,
                         2 * (ux * Fx - uy * Fy) / vp, (ux * Fy + uy * Fx) / vp])
        dm = -self.lam9 * (m - eq) + (1.0 - 0.5 * self.lam9) * S
        return f + torch.einsum("ik,kyx->iyx", self.Minv, dm), ux, uy

    def at_rest(self, f, ux, uy, vp):
        """f minus the velocity part of f^eq, Eq. (29): the extrapolated boundary node."""
        uu = (ux ** 2 + uy ** 2) / vp
        out = []
        for i in range(9):
            eu = _EX[i] * ux + _EY[i] * uy
            out.append(f[i] - self.w9[i] * (3 * eu + 4.5 * eu * eu / vp - 1.5 * uu))
        return torch.stack(out)

    def step(self, f, g, fl, phi, K, wall):
        zero = torch.zeros_like(fl)
        T = g.sum(0)
        ux = uy = zero
        f2 = f
        if self.flow:
            act = self.inside & (fl >= self.f_act)
            fs = torch.where(act, fl, torch.ones_like(fl))
            fp, ux, uy = self.collide(f, T, fs, phi, K)
            ux, uy = torch.where(act, ux, zero), torch.where(act, uy, zero)
            ext = None
            if self.walls or self.front:
                ext = self.collide(self.at_rest(f, ux, uy, phi * fs), T, fs, phi, K)[0]
            carries = act
            if self.walls:   # a wall node carries flow with its inward node, as a copy at rest
                iy, ix = self.inward
                carries = act | (~self.inside & act[iy, ix])
                fp = torch.where(self.inside, fp, ext[:, iy, ix])
            new = [fp[0]]
            for i in range(1, 9):
                back = fp[_OPP[i]]
                if self.front:   # a link into a lattice node without flow
                    back = torch.where(act & _from(self.inside, i), ext[i], back)
                src = _from(carries, i) & self.reach[i]
                new.append(torch.where(src, _from(fp[i], i), back))
            f2 = torch.where(carries, torch.stack(new), f)
        ratio = (self.sigma / (self.sigma_s + fl * (self.sigma - self.sigma_s))
                 if self.sigma_s != self.sigma else 1.0)
        za = 1.0 / (0.5 + (self.tau_T - 0.5) * ratio)
        n = torch.einsum("ki,iyx->kyx", self.N, g)
        k = (1.0 / self.sigma) * ratio if self.flow else 0.0
        dn = torch.stack([zero, -za * (n[1] - k * ux * T), -za * (n[2] - k * uy * T),
                          -1.5 * (n[3] - self.varpi * T), -1.5 * n[4]])
        gp = list(g + torch.einsum("ik,kyx->iyx", self.Ninv, dn))
        # thermal walls, in post-collision form: the inward population of each wall node
        for s, (i, u, sg) in enumerate(((1, ux, 1), (3, ux, -1), (2, uy, 1), (4, uy, -1))):
            if self.bc[s] == "periodic":
                continue
            j = _OPP[i]   # the inward node is at x + e_i
            Tf, uf = _from(T, j), _from(u, j)
            c = k / self.cs2t if not torch.is_tensor(k) else _from(k, j) / self.cs2t
            Tw = Tf if self.bc[s] == "adiabatic" else wall[:, None] if s == 0 else self.T_bc[s]
            gp[i] = torch.where(self.side[s], self.w1 * Tw + _from(gp[i], j) -
                                self.w1 * Tf * (1.0 + sg * c * uf), gp[i])
        gs = torch.stack([_from(gp[i], i) for i in range(5)])
        a = phi * self.lat * ratio
        fn = _Enthalpy.apply(gs.sum(0), a, fl, self)
        src = torch.where(self.inside, -a * (fn - fl), zero)
        gs = torch.stack([gs[i] + (self.w0 if i == 0 else self.w1) * _from(src, i)
                          for i in range(5)])
        return f2, torch.where(self.inside, gs, g), fn

    def temperature(self, g, wall):
        """T with the imposed values on wall nodes (corners follow their vertical wall, then
        the horizontal one, then the diagonal node)."""
        iy, ix = self.inward
        Tn = g.sum(0)
        T = torch.where(self.inside, Tn, Tn[iy, ix])
        for s in (3, 2, 1, 0):
            if self.bc[s] == "dirichlet":
                T = torch.where(self.side[s], wall[:, None] if s == 0 else
                                torch.full_like(T, self.T_bc[s]), T)
        return T

    def nusselt(self, g, wall):
        T = self.temperature(g, wall)
        T = T if self.py else T[1:-1]
        return (-(-3.0 * T[:, 0] + 4.0 * T[:, 1] - T[:, 2]) * 0.5).mean() * self.H / self.dT

    def sums(self, f, g, fl, phi, wall, keys):
        iv = self.inside
        ratio = (self.sigma / (self.sigma_s + fl * (self.sigma - self.sigma_s))
                 if self.sigma_s != self.sigma else 1.0)
        out = dict(mass=lambda: (1.0 + f.sum(0))[iv].sum(), melt_frac=lambda: fl[iv].mean(),
                   enthalpy=lambda: (g.sum(0) + phi * self.lat * ratio * fl)[iv].sum(),
                   nu_hot=lambda: self.nusselt(g, wall))
        return [float(out[k]()) for k in keys]

    def macros(self, f, g, fl, phi, K, wall):
        T = self.temperature(g, wall)
        ux = uy = torch.zeros_like(fl)
        if self.flow:
            act = self.inside & (fl >= self.f_act)
            fs = torch.where(act, fl, torch.ones_like(fl))
            ux, uy = (torch.where(act, v, torch.zeros_like(fl))
                      for v in self.velocity(f, T, fs, phi, K)[:2])
        return dict(ux=ux, uy=uy, rho=1.0 + f.sum(0), T=T, fl=fl)


def _exact_run(m, params, phi, K, T0, fl0):
    """Macroscopic fields and sums of one forward run in float64."""
    model = _Model(m["nx"], m["ny"], params, phi.device)
    phi, K, T0, fl0 = (t.double() for t in (phi, K, T0, fl0))
    wall = torch.full((m["ny"],), float(params["T_bc"][0]), dtype=torch.float64, device=phi.device)
    st = model.start(T0, fl0)
    sums = []
    for k in range(1, m["steps"] + 1):
        st = model.step(*st, phi, K, wall)
        if k == m["steps"] or (m["every"] and k % m["every"] == 0):
            sums.append(model.sums(*st, phi, wall, _sums(m)))
    return dict(model.macros(*st, phi, K, wall), sums=sums)


def _exact_gradient(case, params, phi, K, T0, fl0, wall):
    """Objective and gradients in float64: one checkpoint per step, autograd through each."""
    model = _Model(case["nx"], case["ny"], params, phi.device)
    phi, lnK, wall = (t.double().clone().requires_grad_(True) for t in (phi, torch.log(K.double()),
                                                                        wall))
    melt = case["objective"] == "melt"
    states = [model.start(T0.double(), fl0.double())]

    def forward(st):
        out = model.step(*st, phi, torch.exp(lnK), wall)
        return out, torch.zeros((), dtype=torch.float64, device=phi.device) if melt else \
            model.nusselt(out[1], wall) / case["steps"]

    J = 0.0
    with torch.no_grad():
        for _ in range(case["steps"]):
            st, nu = forward(states[-1])
            states.append(st)
            J += float(nu)
    last = states.pop()[2].clone().requires_grad_(True)
    grads = [torch.zeros_like(t) for t in (phi, lnK, wall)]
    lam = [torch.zeros_like(states[0][0]), torch.zeros_like(states[0][1]), torch.zeros_like(last)]
    if melt:
        obj = last[model.inside].mean()
        J = float(obj.detach())
        lam[2] = torch.autograd.grad(obj, last)[0]
    while states:
        st = [t.clone().requires_grad_(True) for t in states.pop()]
        out, nu = forward(st)
        value = sum((o * w).sum() for o, w in zip(out, lam)) + nu
        got = torch.autograd.grad(value, [*st, phi, lnK, wall], allow_unused=True)
        got = [torch.zeros_like(t) if v is None else v for v, t in zip(got, [*st, phi, lnK, wall])]
        lam, grads = got[:3], [a + b for a, b in zip(grads, got[3:])]
    return dict(J=J, dphi=grads[0], dlnK=grads[1], dwall=grads[2])


def exact(case, seed):
    inputs = _inputs(case, seed)
    if case["kind"] in ("adjoint", "coupled"):
        _, params, phi, K, T0, fl0, wall = inputs[0]
        out = _exact_gradient(case, params, phi, K, T0, fl0, wall)
        return out if case["kind"] == "coupled" else {k: out[k] for k in ("J", "dphi", "dwall")}
    with torch.no_grad():
        outs = [_exact_run(m, params, *fields[:4]) for m, params, *fields in inputs]
    if case["kind"] == "run":
        return outs[0]
    return _together([{k: o[k] for k in ("ux", "uy", "rho", "T", "fl")} for o in outs])
