"""What the framework's speed is measured on: calls of its public entry points as programs make them.

A case is a dict of plain values.  ``listed()`` gives the fixed ones, ``draw(rng)`` another of
the same ranges; ``prepare(case, seed)`` builds what a program has in hand before the call,
``run(state)`` is one pass, ``work(case)`` the bytes and operations that pass cannot do without
and ``exact(case, seed)`` its outputs in float64 from plain torch and numpy.

Inputs are matter fields of the workloads' cosmology: Gaussian white noise filtered by the BBKS
spectrum, 2LPT displacements, and for evolved states a share of the lattice collapsed into
isothermal clumps of 4^3 to 16^3 particles (the virial radius of 178 times the mean density), as
the particles of a run sit at late times.
"""
import functools
import math

import numpy as np
import torch

import paper_1301_0322_gb300 as cola

OM, OL, H, SIGMA8, NS, NLPT = 0.27, 0.73, 0.7, 0.8, 0.96, -2.5
A_INIT, A_FINAL = 0.1, 1.0
DEVICE = "cuda"

# ng / np / box of the ensemble's box sizes (0.78 Mpc/h mesh cells, as the 48-box mock ensemble)
ENSEMBLE_SIZES = ((32, 64, 50.0), (48, 96, 75.0), (64, 128, 100.0), (96, 192, 150.0), (128, 256, 200.0))
NG = (32, 48, 64, 96, 128, 192, 256, 384, 512, 768, 1024)
NP = (32, 48, 64, 96, 128, 192, 256, 384, 512)


def listed():
    return [
        # the smallest whole simulation (noise in, 2LPT, 11 force evaluations): launches and latency
        dict(name="run_32p_64g", kind="run", np=32, ng=64, box=100.0, deconv=1, bits=16, scheme="cola"),
        # gradient of a loss of the final density with respect to the noise: forward and backward
        # of a whole run, as reconstruction from a density field does it
        dict(name="gradient_128p_256g", kind="gradient", np=128, ng=256, box=200.0, deconv=1, bits=16),
        # one time step of a small box at the resolution of the paper's run
        dict(name="step_64p_192g", kind="step", np=64, ng=192, box=25.0, deconv=1, bits=16, scheme="cola", step=6),
        # one time step of the paper's run (Sec. 2: mesh three times finer than the lattice)
        dict(name="step_256p_768g", kind="step", np=256, ng=768, box=100.0, deconv=1, bits=16, scheme="cola", step=8),
        # one time step of a large box, mesh twice finer than the lattice
        dict(name="step_512p_1024g", kind="step", np=512, ng=1024, box=500.0, deconv=1, bits=16, scheme="cola", step=5),
        # the bare force on a mesh that is no multiple of the lattice, deconvolved twice
        dict(name="force_192p_256g", kind="force", np=192, ng=256, box=200.0, deconv=2, bits=16),
        # 2LPT initial conditions of the paper's lattice
        dict(name="ic_256p", kind="ic", np=256, ng=256, box=100.0, scheme="cola"),
        # P(k) of a snapshot without a density mesh in between, every shell to the Nyquist frequency
        dict(name="density_power_256p_768g", kind="density_power", np=256, ng=768, box=100.0, bits=16, nbins=384),
        # integer and float density of a snapshot, mesh as fine as the lattice
        dict(name="density_512p_512g", kind="density", np=512, ng=512, box=500.0, bits=16),
        # cross-correlation of two runs' densities (Sec. 3.1)
        dict(name="cross_power_384g", kind="cross_power", np=128, ng=384, box=50.0, nbins=192),
        # halos of an evolved snapshot of the paper's run, b = 0.2 (a plan that also holds the adjoint's buffers)
        dict(name="fof_256p_768g", kind="fof", np=256, ng=768, box=100.0, bits=16, num=1, den=5, nmin=25),
        # one time step of the mock ensemble: 48 boxes of three sizes, per-box launches on two
        # streams (what the autotuner picks for it)
        dict(name="ensemble_48_step", kind="ensemble", n64=0, n96=0, n128=16, n192=16, n256=16, threads=128, launch=2,
             streams=0, step=5),
    ]


def draw(rng):
    kind = rng.choice(("step", "step", "step", "force", "run", "gradient", "step_adjoint", "ic", "density",
                       "density_power", "power", "cross_power", "fft", "fof", "ensemble"))
    if kind == "ensemble":
        case = dict(kind=kind, n64=rng.randint(1, 12), n96=rng.randint(0, 12), n128=rng.randint(0, 12),
                    n192=rng.randint(0, 8), n256=rng.randint(0, 8), threads=rng.choice((128, 256)))
        mode = rng.choice(("multi-box", "per-box", "hybrid"))
        return dict(case, launch=rng.choice((1, 2)) if mode == "per-box" else 0,
                    streams=rng.choice((1, 2)) if mode == "hybrid" else 0, step=rng.randint(0, 10))
    # whole runs up to mid size; backward passes to the differentiable workload's mesh
    most = {"run": 192, "gradient": 192, "step_adjoint": 384, "fof": 768}.get(kind, 1024)
    ng = rng.choice([n for n in NG if n <= most])
    nps = [n for n in NP if n <= ng <= 4 * n and (kind != "fof" or (ng % n == 0 and n <= 256))]
    n = rng.choice(nps or [max(NP[0], min(512, ng // 2))])
    cell = round(10.0 ** rng.uniform(-1.0, 0.0), 4)
    case = dict(kind=kind, np=n, ng=ng, box=round(ng * cell, 3))
    if kind in ("power", "cross_power", "density_power"):
        case["nbins"] = rng.randint(max(4, ng // 8), ng // 2)
    if kind not in ("ic", "power", "cross_power", "fft"):
        # (finer positions than 2^-16 cell leave no room for the clumps' cells in 62 bits)
        case["bits"] = rng.choice((16, 16, 16, 14, 12)) if kind != "fof" else 16
    if kind in ("step", "force", "run", "gradient", "step_adjoint"):
        case["deconv"] = rng.choice((1, 1, 0, 2))
    if kind in ("step", "run", "ic"):
        case["scheme"] = rng.choice(("cola", "cola", "cola_std", "pm_std", "cola_u1"))
    if kind in ("step", "step_adjoint"):
        case["step"] = rng.randint(0, 10)
    if kind == "fof":
        case.update(num=1, den=rng.choice((4, 5, 6)), nmin=rng.choice((20, 25, 50)))
    if kind == "fft":
        case["which"] = rng.choice((0, 1))
    return case


# ---- inputs ---------------------------------------------------------------------------------
def _generator(seed):
    return torch.Generator(device=DEVICE).manual_seed(int(seed))


def _randn(shape, gen):
    return torch.randn(shape, generator=gen, device=DEVICE, dtype=torch.float32)


def _plan(case):
    """The plan a program keeps for this mesh (memory of its workspace included)."""
    return cola.Plan(np_side=case["np"], ng=case["ng"], box=case["box"], deconv=case.get("deconv", 1),
                     fixed_bits=case.get("bits", 16), scheme=case.get("scheme", "cola"),
                     adjoint=case["kind"] in ("gradient", "step_adjoint", "fof"), device=DEVICE)


def _matter(n, box, a, gen, collapsed):
    """(s, v, s1, s2), float32 [3][n^3]: a state at scale factor a of which a share `collapsed`
    sits in clumps."""
    s1, s2 = _lpt64(_randn((n, n, n), gen), n, box)
    row = _growth_at(a)
    s = row["D1"] * s1 + row["D2"] * s2
    spacing = box / n
    idx = torch.arange(n, device=DEVICE, dtype=torch.float64)
    for b in (16, 8, 4):
        m = n // b
        if m < 2 or collapsed <= 0:
            continue
        pick = torch.rand((m, m, m), generator=gen, device=DEVICE) < collapsed / 3
        pick = pick.repeat_interleave(b, 0).repeat_interleave(b, 1).repeat_interleave(b, 2).reshape(-1)
        mean = s.view(3, m, b, m, b, m, b).mean(dim=(2, 4, 6), keepdim=True).expand(3, m, b, m, b, m, b).reshape(3, -1)
        to_centre = ((torch.div(idx, b, rounding_mode="floor") + 0.5) * b - 0.5 - idx) * spacing
        d = torch.stack([to_centre.view(1, 1, n).expand(n, n, n), to_centre.view(1, n, 1).expand(n, n, n),
                         to_centre.view(n, 1, 1).expand(n, n, n)]).reshape(3, -1)
        way = _randn((3, n**3), gen)
        r = 0.11 * b * spacing * torch.rand(n**3, generator=gen, device=DEVICE)
        d = d + mean + way * (r / way.norm(dim=0).clamp_min(1e-6))
        s = torch.where(pick, d, s)
    v = 0.2 * (s1 * row["D1"]) + 0.3 * _randn((3, n**3), gen)
    return [x.to(torch.float32).contiguous() for x in (s, v, s1, s2)]


def _density_field(ng, box, gen):
    """A float32 density contrast [ng^3]: filtered noise through an exponential, mean 0."""
    k = _k64(ng, box, torch.float32)
    k[0, 0, 0] = 1.0
    f = torch.fft.irfftn(torch.fft.rfftn(_randn((ng,) * 3, gen)) / k, s=(ng,) * 3)
    d = torch.exp(f / f.std())
    return (d / d.mean() - 1.0).reshape(-1).contiguous()


def _boxes(case):
    return [ENSEMBLE_SIZES[i] for i, n in enumerate((64, 96, 128, 192, 256)) for _ in range(case["n%d" % n])]


def _step_a(step):
    return A_INIT + (A_FINAL - A_INIT) * step / 10


def _inputs(case, seed):
    """The call's input tensors, from the seed alone."""
    gen, kind = _generator(seed), case["kind"]
    if kind == "ensemble":
        a = _step_a(case["step"])
        parts = [_matter(n, box, a, gen, 0.4 * a) for n, _, box in _boxes(case)]
        return dict(zip(("s", "v", "s1", "s2"), (torch.cat([p[j].reshape(-1) for p in parts]) for j in range(4))))
    n, ng, box = case["np"], case["ng"], case["box"]
    if kind in ("run", "ic"):
        return dict(noise=_randn(n**3, gen))
    if kind == "gradient":
        return dict(noise=_randn(n**3, gen), target=_density_field(ng, box, gen))
    if kind == "power":
        return dict(delta=_density_field(ng, box, gen))
    if kind == "cross_power":
        a = _density_field(ng, box, gen)
        return dict(a=a, b=(0.8 * a + 0.5 * _density_field(ng, box, gen)).contiguous())
    if kind == "fft":
        return dict(x=_density_field((ng, n)[case["which"]], box, gen))
    a = _step_a(case["step"]) if "step" in case else 1.0
    s, v, s1, s2 = _matter(n, box, a, gen, 0.4 * a)
    if kind in ("step",):
        return dict(s=s, v=v, s1=s1, s2=s2)
    if kind == "step_adjoint":
        return dict(s=s, lam=[_randn((3, n**3), gen) for _ in range(4)])
    return dict(s=s)


def prepare(case, seed):
    state = _inputs(case, seed)
    if case["kind"] == "ensemble":
        ens = cola.Ensemble(_boxes(case), device=DEVICE)
        ens.tuning = (case["threads"], 0, 0, 0, case["launch"], case["streams"])
        state["ens"] = ens
    else:
        state["plan"] = _plan(case)
    if case["kind"] in ("step", "ensemble"):  # the buffers a step works on in place
        state["work"] = [torch.empty_like(state["s"]), torch.empty_like(state["v"])]
    if case["kind"] == "step_adjoint":
        state["work"] = [torch.empty_like(x) for x in state["lam"]]
    if case["kind"] == "gradient":
        state["noise"].requires_grad_()
    state["case"] = dict(case)
    return state


# ---- one pass -------------------------------------------------------------------------------
def run(state):
    case = state["case"]
    kind, plan = case["kind"], state.get("plan")
    if kind == "run":
        return list(plan.run(state["noise"]))
    if kind == "gradient":
        state["noise"].grad = None
        delta = cola.cola_density_from_noise(state["noise"], plan)
        ((delta - state["target"]) ** 2).sum().backward()
        return [delta.detach(), state["noise"].grad]
    if kind in ("step", "ensemble"):  # the state before the step is kept, as a checkpointed run keeps it
        s, v = state["work"]
        s.copy_(state["s"])
        v.copy_(state["v"])
        (plan or state["ens"]).step(case["step"], s, v, state["s1"], state["s2"])
        return [s, v]
    if kind == "step_adjoint":
        for w, x in zip(state["work"], state["lam"]):
            w.copy_(x)
        plan.step_adjoint(case["step"], state["s"], *state["work"])
        return list(state["work"])
    if kind == "force":
        return plan.force(state["s"])
    if kind == "ic":
        return list(plan.ic_2lpt(state["noise"]))
    if kind == "density":
        return list(plan.density(state["s"]))
    if kind == "density_power":
        return list(plan.density_power(state["s"], case["nbins"]))
    if kind == "power":
        return list(plan.power(state["delta"], case["nbins"]))
    if kind == "cross_power":
        return list(plan.cross_power(state["a"], state["b"], case["nbins"]))
    if kind == "fft":
        return plan.fft_r2c(state["x"], case["which"])
    if kind == "fof":
        return list(plan.fof(state["s"], nmin=case["nmin"], b=(case["num"], case["den"]),
                             thresholds=[25, 50, 100, 200, 400, 800, 1600, 3200]))
    raise ValueError(kind)


# ---- work -----------------------------------------------------------------------------------
def _fft_flops(n):
    """One three-dimensional real transform of side n (half of 5 N log2 N)."""
    return 2.5 * n**3 * 3 * math.log2(n)


def _step_work(n, ng):
    # state in and out, first- and second-order displacements in; the deposit, four transforms,
    # the Green's function with its gradient, the gather and the update
    return 72.0 * n**3, 4 * _fft_flops(ng) + 8 * ng**3 + (16 + 48 + 30) * n**3


def work(case):
    kind = case["kind"]
    if kind == "ensemble":
        parts = [_step_work(n, ng) for n, ng, _ in _boxes(case)]
        return dict(bytes=sum(p[0] for p in parts), flops=sum(p[1] for p in parts))
    n, ng = case["np"], case["ng"]
    force = _step_work(n, ng)[1]
    n3, g3 = float(n**3), float(ng**3)
    ic = 14 * _fft_flops(n) + 60 * n3
    if kind == "step":
        return dict(bytes=72 * n3, flops=force)
    if kind == "run":
        return dict(bytes=52 * n3, flops=ic + 11 * force)
    if kind == "gradient":
        return dict(bytes=12 * n3 + 8 * g3, flops=3 * (ic + 11 * force))
    if kind == "step_adjoint":
        return dict(bytes=108 * n3, flops=2 * force)
    if kind == "force":
        return dict(bytes=24 * n3, flops=force)
    if kind == "ic":
        return dict(bytes=52 * n3, flops=ic)
    if kind == "density":
        return dict(bytes=12 * n3 + 12 * g3, flops=16 * n3 + 2 * g3)
    if kind == "density_power":
        return dict(bytes=12 * n3, flops=16 * n3 + _fft_flops(ng) + 4 * g3)
    if kind == "power":
        return dict(bytes=4 * g3, flops=_fft_flops(ng) + 4 * g3)
    if kind == "cross_power":
        return dict(bytes=8 * g3, flops=2 * _fft_flops(ng) + 8 * g3)
    if kind == "fft":
        m = (ng, n)[case["which"]]
        return dict(bytes=4.0 * m**3 + 8.0 * m * m * (m // 2 + 1), flops=_fft_flops(m))
    if kind == "fof":
        return dict(bytes=20 * n3, flops=27 * 8 * n3)
    raise ValueError(kind)


# ---- the same in float64 --------------------------------------------------------------------
def _Q(a):
    return np.sqrt(OM * a**3 + (1 - OM - OL) * a**4 + OL * a**6)


@functools.lru_cache(maxsize=None)
def _growth_table():
    """ln a grid and D1, T[D1], D2u, T[D2u] (unnormalised) by Runge-Kutta 4 from a = 1e-8."""
    x0, m = math.log(1e-8), 16000
    h = -x0 / m

    def rhs(x, y):
        a = math.exp(x)
        q = math.sqrt(OM * a**3 + (1 - OM - OL) * a**4 + OL * a**6)
        src = 1.5 * OM * a
        return (a * y[1] / q, a * src * y[0] / q, a * y[3] / q, a * src * (y[2] - y[0] * y[0]) / q)

    q0 = float(_Q(1e-8))
    y = (1e-8, q0, -3.0 / 7.0 * 1e-16, -6.0 / 7.0 * 1e-8 * q0)
    rows = [y]
    for i in range(m):
        x = x0 + i * h
        k1 = rhs(x, y)
        k2 = rhs(x + h / 2, tuple(p + h / 2 * k for p, k in zip(y, k1)))
        k3 = rhs(x + h / 2, tuple(p + h / 2 * k for p, k in zip(y, k2)))
        k4 = rhs(x + h, tuple(p + h * k for p, k in zip(y, k3)))
        y = tuple(p + h / 6 * (a + 2 * b + 2 * c + d) for p, a, b, c, d in zip(y, k1, k2, k3, k4))
        rows.append(y)
    return x0, h, np.array(rows)


def _growth_at(a):
    """D1, D2 and their first and second T derivatives at a, with D1(1) = D2(1) = 1."""
    x0, h, t = _growth_table()
    p = (math.log(a) - x0) / h
    i = int(min(max(math.floor(p) - 3, 0), len(t) - 8))
    y = np.zeros(4)
    for j in range(8):  # Lagrange interpolation through eight points
        w = 1.0
        for k in range(8):
            if k != j:
                w *= (p - i - k) / (j - k)
        y = y + w * t[i + j]
    d1, norm2 = t[-1][0], t[-1][0] ** 2
    d2u1 = t[-1][2] / norm2
    D1, D2u = y[0] / d1, y[2] / norm2
    return dict(D1=D1, D2=D2u / d2u1, TD1=y[1] / d1, TD2=y[3] / norm2 / d2u1, T2D1=1.5 * OM * a * D1,
                T2D2=1.5 * OM * a * (D2u - D1 * D1) / d2u1, d2u1=d2u1)


def _bbks(k):
    q = k / (OM * H)
    poly = 1 + 3.89 * q + (16.1 * q) ** 2 + (5.46 * q) ** 3 + (6.71 * q) ** 4
    m = np if isinstance(k, np.ndarray) else torch
    return m.log1p(2.34 * q) / (2.34 * q) * poly**-0.25


@functools.lru_cache(maxsize=None)
def _amplitude():
    """A of P = A k^ns T^2 for the given sigma8."""
    x = np.linspace(math.log(1e-7), math.log(1e4), 131073)
    k = np.exp(x)
    y = 8.0 * k
    w = np.where(y < 1e-2, 1 - y * y / 10 + y**4 / 280, 3 * (np.sin(y) - y * np.cos(y)) / y**3)
    f = k ** (3 + NS) * _bbks(k) ** 2 * w * w
    c = np.full(len(x), 2.0)
    c[1::2], c[0], c[-1] = 4.0, 1.0, 1.0
    return SIGMA8**2 * 2 * math.pi**2 / (float((c * f).sum()) * (x[1] - x[0]) / 3)


def _modes(n):
    f = torch.arange(n, device=DEVICE)
    f = torch.where(f < n // 2, f, f - n)
    return f.view(n, 1, 1), f.view(1, n, 1), torch.arange(n // 2 + 1, device=DEVICE).view(1, 1, -1)


def _k64(n, box, dtype=torch.float64):
    z, y, x = _modes(n)
    return torch.sqrt((x * x + y * y + z * z).to(dtype)) * (2 * math.pi / box)


def _gradient_factors(n, box):
    """k_x, k_y, k_z of the first derivatives, zero on their Nyquist plane."""
    z, y, x = _modes(n)
    return [torch.where(m.abs() == n // 2, 0, m).to(torch.float64) * (2 * math.pi / box) for m in (x, y, z)]


def _lpt64(noise, n, box):
    """First- and second-order displacements at a = 1 for white noise, [3][n^3] float64."""
    k = _k64(n, box)
    k[0, 0, 0] = 1.0
    f = torch.sqrt(_amplitude() * k**NS * n**3 / box**3) * _bbks(k)
    f[0, 0, 0] = 0.0
    d = torch.fft.rfftn(noise.to(torch.float64).view(n, n, n)) * f / k**2
    g = _gradient_factors(n, box)

    def back(x):
        return torch.fft.irfftn(x, s=(n, n, n))

    s1 = torch.stack([back(1j * g[j] * d) for j in range(3)]).reshape(3, -1)
    diag = [back(-g[j] * g[j] * d) for j in range(3)]
    mu = diag[0] * diag[1] + diag[0] * diag[2] + diag[1] * diag[2]
    del diag
    for i, j in ((0, 1), (0, 2), (1, 2)):
        mu = mu - back(-g[i] * g[j] * d) ** 2
    m = torch.fft.rfftn(mu) / k**2
    d2u1 = _growth_at(1.0)["d2u1"]
    return s1, torch.stack([back(-1j * g[j] * m) for j in range(3)]).reshape(3, -1) * d2u1


def _coordinates(s, n, ng, box, bits):
    """Cells (int64) and upper weights (float64) of the positions rounded down to 2^-bits cell, as
    the interface states them; the weights keep the positions' derivative."""
    one = 1 << bits
    scale = np.float32(ng / box)
    w = (s.detach().to(torch.float32) * float(scale)).to(torch.float64) * one
    p = torch.arange(n**3, device=s.device)
    cells, weights = [], []
    for d, i in enumerate((p % n, (p // n) % n, p // (n * n))):
        f = (torch.div(i * ng * one, n, rounding_mode="floor") + torch.floor(w[d]).to(torch.int64)) % (ng * one)
        c = f // one
        t = (f - c * one).to(torch.float64) / one
        if s.requires_grad:
            t = t + (s[d] - s[d].detach()) * (ng / box)
        cells.append(c)
        weights.append(t)
    return cells, weights


def _corners(cells, weights, ng):
    for dz in (0, 1):
        for dy in (0, 1):
            for dx in (0, 1):
                i = (((cells[2] + dz) % ng) * ng + (cells[1] + dy) % ng) * ng + (cells[0] + dx) % ng
                w = 1.0
                for t, up in zip(weights, (dx, dy, dz)):
                    w = w * (t if up else 1 - t)
                yield i, w


def _delta64(cells, weights, n, ng):
    rho = torch.zeros(ng**3, device=DEVICE, dtype=torch.float64)
    for i, w in _corners(cells, weights, ng):
        rho = rho.index_add(0, i, w) if w.requires_grad else rho.index_add_(0, i, w)
    return rho * (ng**3 / n**3) - 1


def _window(ng):
    x = torch.arange(ng, device=DEVICE, dtype=torch.float64)
    x = torch.sinc(torch.where(x < ng // 2, x, x - ng) / ng) ** 2
    return x.view(-1, 1, 1) * x.view(1, -1, 1) * torch.sinc(torch.arange(ng // 2 + 1, device=DEVICE,
                                                                         dtype=torch.float64) / ng) ** 2


def _force64(s, n, ng, box, bits, deconv):
    cells, weights = _coordinates(s, n, ng, box, bits)
    dk = torch.fft.rfftn(_delta64(cells, weights, n, ng).view(ng, ng, ng))
    k = _k64(ng, box)
    k[0, 0, 0] = 1.0
    green = 1 / k**2
    green[0, 0, 0] = 0.0
    if deconv:
        green = green / _window(ng) ** deconv
    dk = dk * green
    del k, green
    out = []
    for kj in _gradient_factors(ng, box):
        f = torch.fft.irfftn(1j * kj * dk, s=(ng,) * 3).reshape(-1)
        out.append(sum(w * f[i] for i, w in _corners(cells, weights, ng)))
        del f
    return torch.stack(out)


def _simpson(f, a, b):
    x = np.linspace(math.log(a), math.log(b), 4097)
    c = np.full(len(x), 2.0)
    c[1::2], c[0], c[-1] = 4.0, 1.0, 1.0
    e = np.exp(x)
    return float((c * f(e) * e).sum()) * (x[1] - x[0]) / 3


def _step64(s, v, s1, s2, step, n, ng, box, bits, deconv, scheme):
    """Force evaluation `step` of ten: kick, then drift (or the return to the lab frame)."""
    a = [_step_a(i) for i in range(11)]
    now = _growth_at(a[step])
    ka = a[0] if step == 0 else (a[step - 1] + a[step]) / 2
    kb = a[10] if step == 10 else (a[step] + a[step + 1]) / 2
    frame = 0.0 if scheme == "pm_std" else 1.0
    if scheme in ("cola", "cola_u1"):
        kick = (kb**NLPT - ka**NLPT) / (float(_Q(a[step])) * NLPT * a[step] ** (NLPT - 1))
    else:
        kick = _simpson(lambda x: x / _Q(x), ka, kb) / a[step]
    g = _force64(s, n, ng, box, bits, deconv)
    v = v + kick * (1.5 * OM * a[step] * g - frame * (now["T2D1"] * s1 + now["T2D2"] * s2))
    if step == 10:
        return s, v + frame * (now["TD1"] * s1 + now["TD2"] * s2)
    to, mid = _growth_at(a[step + 1]), (a[step] + a[step + 1]) / 2
    if scheme == "cola":
        drift = _simpson(lambda x: x**NLPT / _Q(x), a[step], a[step + 1]) / mid**NLPT
    else:
        drift = _simpson(lambda x: 1 / _Q(x), a[step], a[step + 1])
    return s + drift * v + frame * ((to["D1"] - now["D1"]) * s1 + (to["D2"] - now["D2"]) * s2), v


def _ic64(noise, n, box, scheme):
    s1, s2 = _lpt64(noise, n, box)
    g = _growth_at(A_INIT)
    s = g["D1"] * s1 + g["D2"] * s2
    v = g["TD1"] * s1 + g["TD2"] * s2 if scheme == "pm_std" else torch.zeros_like(s)
    return s, v, s1, s2


def _shells(ng, box, nbins, *fields):
    """Shell numbers, mode weights and window-corrected spectra of the pairs of `fields`."""
    z, y, x = _modes(ng)
    m = x * x + y * y + z * z
    r = torch.floor(torch.sqrt(m.to(torch.float64))).to(torch.int64)
    b = torch.where(m <= r * (r + 1), r, r + 1)
    w = torch.where((x == 0) | (x == ng // 2), 1.0, 2.0).to(torch.float64).expand(b.shape)
    keep = (b >= 1) & (b <= nbins)
    at, w = b[keep] - 1, w[keep]
    count = torch.bincount(at, weights=w, minlength=nbins)

    def mean(q):
        return torch.bincount(at, weights=w * q[keep], minlength=nbins) / count

    norm = box**3 / float(ng) ** 6 / _window(ng) ** 2
    k = mean(torch.sqrt(m.to(torch.float64)) * (2 * math.pi / box))
    return [k] + [mean((p * q.conj()).real * norm) for p, q in fields] + [count.to(torch.int64)]


def exact(case, seed):
    kind = case["kind"]
    if kind == "fof":  # whole numbers
        return None
    x = _inputs(case, seed)
    d = lambda t: t.to(torch.float64)  # noqa: E731
    if kind == "ensemble":
        at, out = 0, []
        for n, ng, box in _boxes(case):
            part = [d(x[key][at:at + 3 * n**3]).view(3, -1) for key in ("s", "v", "s1", "s2")]
            out.append(_step64(*part, case["step"], n, ng, box, 16, 1, "cola"))
            at += 3 * n**3
        return [torch.cat([o[j].reshape(-1) for o in out]) for j in range(2)]
    n, ng, box, bits, deconv = case["np"], case["ng"], case["box"], case.get("bits", 16), case.get("deconv", 1)
    mesh = (n, ng, box, bits, deconv)
    if kind == "ic":
        return list(_ic64(x["noise"], n, box, case["scheme"]))
    if kind == "run":
        s, v, s1, s2 = _ic64(x["noise"], n, box, case["scheme"])
        for i in range(11):
            s, v = _step64(s, v, s1, s2, i, *mesh, case["scheme"])
        return [s, v, s1, s2]
    if kind == "gradient":
        noise = d(x["noise"]).requires_grad_()
        s, v, s1, s2 = _ic64(noise, n, box, "cola")
        for i in range(11):
            s, v = _step64(s, v, s1, s2, i, *mesh, "cola")
        delta = _delta64(*_coordinates(s, n, ng, box, bits), n, ng)
        ((delta - d(x["target"])) ** 2).sum().backward()
        return [delta.detach(), noise.grad]
    if kind == "step":
        return list(_step64(*[d(x[key]) for key in ("s", "v", "s1", "s2")], case["step"], *mesh, case["scheme"]))
    if kind == "force":
        return _force64(d(x["s"]), *mesh)
    if kind == "step_adjoint":
        # s in its float32 value; v, s1 and s2 enter linearly, so any values give their adjoints
        ins = [d(x["s"]).requires_grad_()] + [torch.zeros((3, n**3), device=DEVICE, dtype=torch.float64,
                                                          requires_grad=True) for _ in range(3)]
        s, v = _step64(*ins, case["step"], *mesh, "cola")
        lam = [d(t) for t in x["lam"]]
        grads = torch.autograd.grad((lam[0] * s).sum() + (lam[1] * v).sum(), ins)
        return [grads[0], grads[1], lam[2] + grads[2], lam[3] + grads[3]]
    if kind == "density":
        return [None, _delta64(*_coordinates(d(x["s"]), n, ng, box, bits), n, ng)]
    if kind == "fft":
        m = (ng, n)[case["which"]]
        return torch.fft.rfftn(d(x["x"]).view(m, m, m))
    back = lambda t: torch.fft.rfftn(d(t).view(ng, ng, ng))  # noqa: E731
    if kind in ("power", "density_power"):
        delta = x["delta"] if kind == "power" else _delta64(*_coordinates(d(x["s"]), n, ng, box, bits), n, ng)
        f = back(delta)
        k, p, count = _shells(ng, box, case["nbins"], (f, f))
        return [k, p, None]
    f, g = back(x["a"]), back(x["b"])
    k, pa, pb, pab, count = _shells(ng, box, case["nbins"], (f, f), (g, g), (f, g))
    rho = pab / torch.sqrt(pa * pb)
    return [k, pa, pb, pab, rho, 2.0 / 3.0 * rho / torch.sqrt(1 - rho * rho), None]
