"""What is timed: the solver's public entry points on the work its users give it.

A case is a dict of plain values.  ``kind`` names the call sequence:

  solve     initial planes in device memory, n outer steps, the observers'
            waveforms and the final state read out on the device: one evolution
            with the grid and the coefficients kept
  scan      a new black hole on a kept grid: coefficient precompute, generated
            initial pulse, n outer steps, waveforms and final state
  gradient  waveforms() under autograd: forward evolution, then the gradient of
            a waveform loss with respect to the initial planes
  adjoint   the adjoint sweep alone, for a trajectory taken beforehand
  param     waveforms_with_params() under autograd: forward evolution, then the
            gradients with respect to the spin and to the initial planes
  batch     several evolutions advanced together by one Batch

Sizes, time steps and substeps are those of the repository's workloads
(``inputs``: Schwarzschild 1601 x 32, Kerr 25601 x 64, the batched set of 4001
to 16001 x 32 to 128, the adjoint set 16001 x 128), with the number of outer
steps cut so that one pass takes at most a few tens of milliseconds, and ragged
sizes in between.  ``exact`` evolves the same initial data with the scheme of
arXiv 1010.3816, Sec. 3, written here in plain torch in double precision.
"""
import math

import numpy as np
import torch

import paper_1010_3816_gb300 as tk

DEV = "cuda"
SUBSTEPS = {32: 2, 64: 4, 128: 8}   # per outer step of dt = 1/32, by theta rows


def _case(name, kind, Nr, Nth, n, *, drs, dt, k, a=0.9, s=-2, m=2, variable=1, precision=0,
          noise=1e-3, nobs=1, rs_min=-50.0, members=1):
    return {"name": name, "kind": kind, "Nr": Nr, "Nth": Nth, "n": n, "drs": drs, "dt": dt, "k": k,
            "a": a, "s": s, "m": m, "variable": variable, "precision": precision, "noise": noise,
            "nobs": nobs, "rs_min": rs_min, "members": members}


def listed():
    return [
        # a control loop that advances a small grid a little and reads everything
        # back: launch and synchronisation latency
        _case("small_401x32_f64", "solve", 401, 32, 4, drs=0.25, dt=0.125, k=1, rs_min=-40.0, nobs=2),
        # the Schwarzschild workload (no noise, L2-resident), a tenth of its length
        _case("schwarzschild_1601x32_f64", "solve", 1601, 32, 200, drs=0.125, dt=1 / 16, k=1, a=0.0,
              noise=0.0),
        # the flagship Kerr workload, 60 of its 38400 outer steps
        _case("kerr_25601x64_f64", "solve", 25601, 64, 60, drs=1 / 32, dt=1 / 64, k=2, rs_min=-100.0, nobs=2),
        # the same grid in single precision
        _case("kerr_25601x64_f32", "solve", 25601, 64, 300, drs=1 / 32, dt=1 / 64, k=2, rs_min=-100.0,
              nobs=2, precision=1),
        # the finest angular grid of the batched set
        _case("kerr_8001x128_f64", "solve", 8001, 128, 8, drs=1 / 16, dt=1 / 32, k=8, a=0.5, m=3),
        # ragged sizes, the literal variable and the scalar field
        _case("scalar_literal_4999x45_f64", "solve", 4999, 45, 12, drs=1 / 16, dt=1 / 32, k=8, a=0.7, s=0,
              m=1, variable=0),
        # a ragged single-precision grid too small for the four-step sweep
        _case("kerr_2999x50_f32", "solve", 2999, 50, 100, drs=1 / 16, dt=1 / 32, k=4, a=0.99, m=-2,
              precision=1),
        # a parameter scan: every pass precomputes the coefficients of its own black hole
        _case("scan_4001x64_f64", "scan", 4001, 64, 16, drs=1 / 16, dt=1 / 32, k=4),
        # fitting the initial pulse: forward and backward through autograd
        _case("gradient_4001x64_f64", "gradient", 4001, 64, 16, drs=1 / 16, dt=1 / 32, k=4, a=0.5),
        # the adjoint workload's backward sweep
        _case("adjoint_16001x128_f64", "adjoint", 16001, 128, 4, drs=1 / 16, dt=1 / 32, k=8, a=0.7,
              rs_min=-100.0, noise=0.0),
        # fitting the spin and the pulse: checkpointed recomputation and the adjoint
        _case("param_gradient_1601x32_f64", "param", 1601, 32, 30, drs=1 / 8, dt=1 / 16, k=2, a=0.7,
              noise=0.0),
        # a small ensemble in one batch
        _case("batch_6x1601x32_f64", "batch", 1601, 32, 32, drs=1 / 16, dt=1 / 32, k=2, members=6),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "solve", "scan", "gradient", "adjoint", "param", "batch"])
    precision = rng.choice([0, 0, 1]) if kind in ("solve", "batch") else 0
    Nth = rng.choice([16, 27, 32, 45, 64, 64, 90, 128])
    drs, dt = 1 / 16, 1 / 32
    k = SUBSTEPS[32 if Nth <= 32 else 64 if Nth <= 64 else 128]
    a = rng.choice([0.0, 0.3, 0.5, 0.7, 0.9, 0.99]) if kind != "param" else rng.uniform(0.1, 0.9)
    s = rng.choice([-2, -2, -2, 0])
    m = rng.choice([0, 1, 2, 3, 4, -2])
    variable = rng.choice([1, 1, 1, 0]) if (kind == "solve" and precision == 0) else 1
    if variable == 0:
        s, m, k = 0, rng.choice([0, 1, 2]), 2 * k
    members = rng.randint(2, 6) if kind == "batch" else 1
    hi = {"solve": 25601, "scan": 6001, "gradient": 8001, "adjoint": 16001, "param": 2001, "batch": 4001}[kind]
    Nr = _log(rng, 801 if kind != "solve" else 401, hi)
    # at most the largest listed case's work
    budget = {"solve": 1.6e8, "scan": 1.6e7, "gradient": 3e7, "adjoint": 6e7, "param": 6e6, "batch": 3e7}[kind]
    if precision == 1:
        budget *= 4
    n_hi = max(1, int(budget / (Nr * Nth * k * members)))
    n_lo = 2 if kind in ("solve", "batch") else 4
    n = _log(rng, n_lo, max(n_lo, min(n_hi, 400)))
    return _case("drawn", kind, Nr, Nth, n, drs=drs, dt=dt, k=k, a=a, s=s, m=m, variable=variable,
                 precision=precision, noise=rng.choice([0.0, 1e-3]) if kind in ("solve", "batch") else 0.0,
                 nobs=rng.choice([1, 2]), members=members) | {"name": ""}


# --- inputs -----------------------------------------------------------------------
def _rmax(c):
    return c["rs_min"] + (c["Nr"] - 1) * c["drs"]


def _pulse(c, rng):
    """(amplitude, centre, width) of the initial Gaussian."""
    L = _rmax(c) - c["rs_min"]
    return (rng.uniform(0.5, 2.0), c["rs_min"] + L * rng.uniform(0.35, 0.5),
            min(rng.uniform(2.0, 8.0), L / 20.0))


def _observers(c):
    """Observers near the pulse, so that every sample sees the field."""
    L = _rmax(c) - c["rs_min"]
    pts = [(c["rs_min"] + 0.45 * L, math.pi / 2), (c["rs_min"] + 0.52 * L + 0.37 * c["drs"], math.pi / 4)]
    return pts[:c["nobs"]]


def _planes(c, seed):
    rng = np.random.default_rng(seed)
    amp, cen, wid = _pulse(c, rng)
    rs = c["rs_min"] + torch.arange(c["Nr"], dtype=torch.float64, device=DEV) * c["drs"]
    th = (torch.arange(c["Nth"], dtype=torch.float64, device=DEV) + 0.5) * (math.pi / c["Nth"])
    re = amp * torch.exp(-(rs - cen) ** 2 / (2 * wid * wid))[None, :] * torch.sin(th)[:, None] ** 2
    im = 0.25 * re if c["noise"] > 0 or c["kind"] in ("gradient", "adjoint", "param") else torch.zeros_like(re)
    if c["noise"] > 0:
        g = torch.Generator(device=DEV)
        g.manual_seed(int(rng.integers(1 << 62)))
        re = re + c["noise"] * (2 * torch.rand(re.shape, generator=g, dtype=torch.float64, device=DEV) - 1)
        im = im + c["noise"] * (2 * torch.rand(re.shape, generator=g, dtype=torch.float64, device=DEV) - 1)
    return re.contiguous(), im.contiguous()


def _cotangent(c, seed):
    """Loss gradient of the waveform samples, [nobs][n][2]."""
    rng = np.random.default_rng(seed + 77)
    return torch.from_numpy(rng.standard_normal((c["nobs"], c["n"], 2))).to(DEV)


def _scan_params(c, seed):
    rng = np.random.default_rng(seed)
    amp, cen, wid = _pulse(c, rng)
    return {"a": float(rng.uniform(0.0, 0.95)), "amp": amp, "cen": cen, "wid": wid,
            "noise": 1e-3, "seed": int(rng.integers(1 << 30))}


def _solver(c, a=None):
    s = tk.Solver(rstar_min=c["rs_min"], rstar_max=_rmax(c), Nr=c["Nr"], Ntheta=c["Nth"], dt=c["dt"],
                  substeps=c["k"], variable=c["variable"], precision=c["precision"])
    s.precompute(c["a"] if a is None else a, 1.0, c["s"], c["m"])
    return s


def _outputs(c):
    wave = torch.empty((c["nobs"], 2, c["n"]), dtype=torch.float64, device=DEV)
    return wave, torch.empty((4, c["Nth"], c["Nr"]), dtype=torch.float64, device=DEV)


def _spins(c):
    return [0.9 * j / max(1, c["members"] - 1) for j in range(c["members"])]


def prepare(case, seed):
    c = case
    kind = c["kind"]
    if kind == "batch":
        solvers, planes = [], []
        for j, a in enumerate(_spins(c)):
            s = _solver(c, a)
            planes.append(_planes(c, seed + 1000 * j))
            s.set_initial(*planes[-1])
            for p in _observers(c):
                s.add_observer(*p)
            solvers.append(s)
        return {"c": c, "batch": tk.Batch(solvers), "solvers": solvers, "planes": planes,
                "out": [_outputs(c) for _ in solvers]}
    s = _solver(c)
    st = {"c": c, "s": s, "out": _outputs(c)}
    if kind == "scan":
        st["p"] = _scan_params(c, seed)
        s.set_initial_gaussian(1.0, st["p"]["cen"], st["p"]["wid"])
    else:
        st["planes"] = _planes(c, seed)
        s.set_initial(*st["planes"])
    for p in _observers(c):
        s.add_observer(*p)
    if kind == "adjoint":
        s.step(c["n"])
    if kind in ("gradient", "adjoint", "param"):
        st["g"] = _cotangent(c, seed)
    return st


def _read(s, c, out):
    wave, state = out
    for j in range(c["nobs"]):
        tk.tk_extract(s.h, j, wave[j, 0], wave[j, 1])
    return [wave, s.state(out=state)]


def run(state):
    c = state["c"]
    kind = c["kind"]
    if kind == "batch":
        for s, p in zip(state["solvers"], state["planes"]):
            s.set_initial(*p)
        state["batch"].step(c["n"])
        return [x for s, o in zip(state["solvers"], state["out"]) for x in _read(s, c, o)]
    s = state["s"]
    if kind == "solve":
        s.set_initial(*state["planes"])
        s.step(c["n"])
        return _read(s, c, state["out"])
    if kind == "scan":
        p = state["p"]
        s.precompute(p["a"], 1.0, c["s"], c["m"])
        s.set_initial_gaussian(p["amp"], p["cen"], p["wid"], p["noise"], p["seed"])
        s.step(c["n"])
        return _read(s, c, state["out"])
    if kind == "gradient":
        re, im = (x.detach().requires_grad_(True) for x in state["planes"])
        y = tk.waveforms(s, re, im, c["n"])
        gr, gi = torch.autograd.grad(y, [re, im], grad_outputs=state["g"])
        return [y.detach(), gr, gi]
    if kind == "adjoint":
        grad = torch.empty((2, c["Nth"], c["Nr"]), dtype=torch.float64, device=DEV)
        return [s.adjoint(grad, dL_dwave=state["g"])]
    a = torch.tensor(c["a"], dtype=torch.float64, device=DEV, requires_grad=True)
    M = torch.tensor(1.0, dtype=torch.float64, device=DEV)
    re, im = (x.detach().requires_grad_(True) for x in state["planes"])
    y = tk.waveforms_with_params(s, a, M, c["s"], c["m"], re, im, c["n"])
    ga, gr, gi = torch.autograd.grad(y, [a, re, im], grad_outputs=state["g"])
    return [y.detach(), ga, gr, gi]


def work(case):
    """Every plane read or written once, and the scheme's operations: 98 per
    grid point and Lax-Wendroff step, 108 per transposed step."""
    c = case
    P = c["Nr"] * c["Nth"]
    steps = c["n"] * c["k"] * c["members"]
    wave = 16 * c["nobs"] * c["n"]
    kind = c["kind"]
    if kind == "scan":
        return {"bytes": 32 * P + wave, "flops": 98 * P * steps + 400 * P}
    if kind == "gradient":
        return {"bytes": 32 * P + 2 * wave, "flops": (98 + 108) * P * steps}
    if kind == "adjoint":
        return {"bytes": 16 * P + wave, "flops": 108 * P * steps}
    if kind == "param":
        # forward, and backward the tangent of the step beside its transpose
        return {"bytes": 32 * P + 2 * wave, "flops": (98 + 98 + 108) * P * steps + 400 * P}
    return {"bytes": c["members"] * (48 * P + wave), "flops": 98 * P * steps}


# --- the scheme in plain torch, double precision ---------------------------------------
def _invert(rstar, M, a):
    """x = r - r+ of every r* (bisection in ln x, then one Newton step that
    carries the derivative in a)."""
    d = torch.sqrt(M * M - a * a)
    rp, rm = M + d, M - d
    Ap, Am = 2 * M * rp / (rp - rm), 2 * M * rm / (rp - rm)

    def f(y, rp, rm, Ap, Am):
        x = torch.exp(y)
        return rp + x + Ap * (y - math.log(2 * M)) - Am * torch.log((rp + x - rm) / (2 * M))

    fixed = tuple(v.detach() for v in (rp, rm, Ap, Am))
    lo, hi = torch.full_like(rstar, -700.0), torch.full_like(rstar, 12.0)
    for _ in range(80):
        mid = 0.5 * (lo + hi)
        below = f(mid, *fixed) < rstar
        lo, hi = torch.where(below, mid, lo), torch.where(below, hi, mid)
    y = 0.5 * (lo + hi)
    x = torch.exp(y)
    r = rp + x
    dfdy = (r * r + a * a) / (r - rm)
    y = y - (f(y, rp, rm, Ap, Am) - rstar) / dfdy
    return torch.exp(y)


def _weight(c, th):
    if c["variable"] == 0:
        return torch.ones_like(th)
    al, be = 0.5 * abs(c["m"] + c["s"]), 0.5 * abs(c["m"] - c["s"])
    return (2 * torch.sin(th / 2) ** 2) ** al * (2 * torch.cos(th / 2) ** 2) ** be


def _face_weights(c):
    """Self-adjoint angular stencil: P at the faces over the cell mean of P."""
    Nth, dth = c["Nth"], math.pi / c["Nth"]
    xg, wg = np.polynomial.legendre.leggauss(24)
    lo = torch.arange(Nth, dtype=torch.float64) * dth
    th = lo[:, None] + 0.5 * dth * (1 + torch.from_numpy(xg))[None, :]
    P = torch.sin(th) * _weight(c, th) ** 2
    Q = (P * torch.from_numpy(wg)).sum(1) * 0.5
    face = torch.arange(Nth + 1, dtype=torch.float64) * dth
    Pf = torch.sin(face) * _weight(c, face) ** 2
    Pf[0] = 0.0
    Pf[-1] = 0.0
    return ((Pf[1:] / (Q * dth * dth)).to(DEV)[:, None], (Pf[:-1] / (Q * dth * dth)).to(DEV)[:, None])


def _coefficients(c, rstar, a):
    """b, c1, c2, c3, c4 of the first-order system on [Nth][len(rstar)]."""
    M, s, m = 1.0, c["s"], c["m"]
    x = _invert(rstar, M, a)[None, :]
    th = ((torch.arange(c["Nth"], dtype=torch.float64, device=DEV) + 0.5) * (math.pi / c["Nth"]))[:, None]
    d = torch.sqrt(M * M - a * a)
    rp, rm = M + d, M - d
    r = rp + x
    Dl, dD = x * (r - rm), 2 * (r - M)
    vp = r * r + a * a
    sn, cs = torch.sin(th), torch.cos(th)
    S2 = vp * vp - a * a * Dl * sn * sn
    S = torch.sqrt(S2)
    b = vp / S
    # Delta factored out of the terms that cancel at the horizon
    b_s = Dl / vp * a * a * sn * sn * (vp * dD - 4 * r * Dl) / (2 * S2 * S)
    cross = 2 * s * vp / S2 * (2 * r * Dl / vp
                               + a * a * Dl * sn * sn * (r * Dl - M * (r * r - a * a)) / (S * vp * (S + vp)))
    fs = 3 * Dl / (r * vp)
    fss = Dl / vp * ((6 * r * Dl + 3 * r * r * dD) / vp - 6 * r ** 3 * Dl / vp ** 2) / r ** 3
    CtR = 2 * s * (r * Dl - M * (r * r - a * a)) / S2
    CtI = (4 * M * a * m * r + 2 * s * a * Dl * cs) / S2
    E0 = (2 * r * Dl + s * dD * vp) / S2
    c4 = Dl / S2
    if c["variable"] == 0:
        V = -(m + s * cs) ** 2 / (sn * sn) + s
    else:
        l0 = max(abs(m), abs(s))
        V = -float((l0 - s) * (l0 + s + 1))
    c1 = torch.complex(cross + 2 * r * Dl / S2 + 2 * b * b * fs - b * b_s, b * CtI)
    c2 = torch.complex(-CtR, -CtI)
    c3 = torch.complex(b * b * fss + E0 * fs + (m * a) ** 2 / S2 + c4 * V, 2 * m * s * a * (r - M) / S2)
    return b, c1, c2, c3, c4


class _Plain:
    def __init__(self, c, a=None):
        self.c = c
        a = torch.tensor(float(c["a"] if a is None else a), dtype=torch.float64, device=DEV) \
            if not torch.is_tensor(a) else a
        rs = c["rs_min"] + torch.arange(c["Nr"], dtype=torch.float64, device=DEV) * c["drs"]
        rh = c["rs_min"] + (torch.arange(c["Nr"] - 1, dtype=torch.float64, device=DEV) + 0.5) * c["drs"]
        self.node, self.half = _coefficients(c, rs, a), _coefficients(c, rh, a)
        self.dt = c["dt"] / c["k"]
        th = ((torch.arange(c["Nth"], dtype=torch.float64, device=DEV) + 0.5) * (math.pi / c["Nth"]))[:, None]
        self.w = _weight(c, th)
        self.dth = math.pi / c["Nth"]
        if c["variable"]:
            self.Ap, self.Am = _face_weights(c)
        else:
            self.cot = torch.cos(th) / torch.sin(th)
            self.parity = 1.0 if c["m"] % 2 == 0 else -1.0

    def angular(self, F):
        if self.c["variable"]:
            up = torch.cat([F[1:], F[-1:]])
            dn = torch.cat([F[:1], F[:-1]])
            return self.Ap * (up - F) - self.Am * (F - dn)
        up = torch.cat([F[1:], self.parity * F[-1:]])
        dn = torch.cat([self.parity * F[:1], F[:-1]])
        return (up - 2 * F + dn) / self.dth ** 2 + self.cot * (up - dn) / (2 * self.dth)

    def rates(self, co, lo, hi):
        """Right-hand side from the values left and right of a point."""
        b, c1, c2, c3, c4 = co
        (fl, pl), (fh, ph) = lo, hi
        h = 1.0 / self.c["drs"]
        f, p = 0.5 * (fl + fh), 0.5 * (pl + ph)
        df, dp = h * (fh - fl), h * (ph - pl)
        return (f, p, p - b * df, b * dp + c1 * df + c2 * p + c3 * f + c4 * self.angular(f))

    def step(self, f, p):
        fm, pm, rf, rp = self.rates(self.half, (f[:, :-1], p[:, :-1]), (f[:, 1:], p[:, 1:]))
        hf, hp = fm + 0.5 * self.dt * rf, pm + 0.5 * self.dt * rp
        inner = tuple(x[:, 1:-1] for x in self.node)
        _, _, rf, rp = self.rates(inner, (hf[:, :-1], hp[:, :-1]), (hf[:, 1:], hp[:, 1:]))
        pad = torch.nn.functional.pad
        return (pad(f[:, 1:-1] + self.dt * rf, (1, 1)), pad(p[:, 1:-1] + self.dt * rp, (1, 1)))

    def initial(self, re, im):
        z = torch.complex(re, im)
        pad = torch.nn.functional.pad
        dz = (z[:, 2:] - z[:, :-2]) / (2 * self.c["drs"])
        return pad(z[:, 1:-1], (1, 1)), pad(self.node[0][:, 1:-1] * dz, (1, 1))

    def sample(self, f):
        c, out = self.c, []
        for rs, th in _observers(c):
            x, y = (rs - c["rs_min"]) / c["drs"], th / self.dth - 0.5
            i, j = min(int(x), c["Nr"] - 2), min(int(y), c["Nth"] - 2)
            u, v = x - i, y - j
            g = f[j:j + 2, i:i + 2] * self.w[j:j + 2]
            out.append((1 - u) * ((1 - v) * g[0, 0] + v * g[1, 0]) + u * ((1 - v) * g[0, 1] + v * g[1, 1]))
        return torch.stack(out)

    def evolve(self, f, p):
        """Final fields and the samples, [nobs][n] complex."""
        waves = []
        for _ in range(self.c["n"]):
            for _ in range(self.c["k"]):
                f, p = self.step(f, p)
            waves.append(self.sample(f))
        return f, p, torch.stack(waves, 1)


def _whole(E, re, im):
    f, p, w = E.evolve(*E.initial(re, im))
    return [torch.stack([w.real, w.imag], 1), torch.stack([f.real, f.imag, p.real, p.imag])]


def _splitmix01(seed, n):
    """Uniform doubles of SplitMix64, the generator of the generated pulse."""
    with np.errstate(over="ignore"):
        z = np.uint64(seed) + np.arange(1, n + 1, dtype=np.uint64) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    return torch.from_numpy((z >> np.uint64(11)).astype(np.float64) * 2.0 ** -53).to(DEV)


def exact(case, seed):
    c = case
    kind = c["kind"]
    with torch.no_grad():
        if kind == "solve":
            return _whole(_Plain(c), *_planes(c, seed))
        if kind == "batch":
            out = []
            for j, a in enumerate(_spins(c)):
                out += _whole(_Plain(c, a), *_planes(c, seed + 1000 * j))
            return out
        if kind == "scan":
            p = _scan_params(c, seed)
            rs = c["rs_min"] + torch.arange(c["Nr"], dtype=torch.float64, device=DEV) * c["drs"]
            th = (torch.arange(c["Nth"], dtype=torch.float64, device=DEV) + 0.5) * (math.pi / c["Nth"])
            P = c["Nr"] * c["Nth"]
            u = p["noise"] * (2 * _splitmix01(p["seed"], 2 * P) - 1)
            re = p["amp"] * torch.exp(-(rs - p["cen"]) ** 2 / (2 * p["wid"] ** 2))[None, :] * torch.sin(th)[:, None] ** 2
            return _whole(_Plain(c, p["a"]), re + u[:P].view(c["Nth"], c["Nr"]), u[P:].view(c["Nth"], c["Nr"]))
    # gradients in the initial planes: the steps are linear, so each is
    # transposed at the zero state
    E = _Plain(c)
    g = _cotangent(c, seed)
    shape = (c["Nth"], c["Nr"])
    z = lambda: torch.zeros(shape, dtype=torch.complex128, device=DEV, requires_grad=True)
    lf = torch.zeros(shape, dtype=torch.complex128, device=DEV)
    lp = torch.zeros_like(lf)
    for t in range(c["n"] - 1, -1, -1):
        f = z()
        lf = lf + torch.autograd.grad(E.sample(f), f, torch.complex(g[:, t, 0], g[:, t, 1]))[0]
        for _ in range(c["k"]):
            f, p = z(), z()
            lf, lp = torch.autograd.grad(E.step(f, p), [f, p], [lf, lp])
    re = torch.zeros(shape, dtype=torch.float64, device=DEV, requires_grad=True)
    im = torch.zeros(shape, dtype=torch.float64, device=DEV, requires_grad=True)
    gr, gi = torch.autograd.grad(E.initial(re, im), [re, im], [lf, lp])
    if kind == "adjoint":
        return [torch.stack([gr, gi])]
    with torch.no_grad():
        _, _, w = E.evolve(*E.initial(*_planes(c, seed)))
    y = torch.stack([w.real, w.imag], 2)
    if kind == "param":
        return [y, _exact_spin(c, seed), gr, gi]
    return [y, gr, gi]


def _exact_spin(c, seed):
    """dL/da by automatic differentiation of the whole evolution, segment by
    segment (checkpointed)."""
    from torch.utils.checkpoint import checkpoint
    a = torch.tensor(c["a"], dtype=torch.float64, device=DEV, requires_grad=True)
    E = _Plain(c, a)
    re, im = _planes(c, seed)
    g = _cotangent(c, seed)
    f, p = E.initial(re, im)

    def segment(f, p):
        for _ in range(c["k"]):
            f, p = E.step(f, p)
        return f, p

    loss = torch.zeros((), dtype=torch.float64, device=DEV)
    for t in range(c["n"]):
        f, p = checkpoint(segment, f, p, use_reentrant=False)
        w = E.sample(f)
        loss = loss + (g[:, t, 0] * w.real + g[:, t, 1] * w.imag).sum()
    return torch.autograd.grad(loss, a)[0]
