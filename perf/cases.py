"""Performance cases: the work that users of this library have it do, through its Python
binding (Propagator and Batch), over the range of dimensions, sizes, arithmetic forms,
potentials and step counts that its workloads, tests and benchmark use.

A case is a dict of plain values:

  kind   "run"   a propagation job: the initial state (complex128, on the GPU) goes in, nt
                 steps with an observable record every nprint, the final state and the
                 records come out (Algorithm 1 of the paper as wp_run offers it);
         "step"  the next chunk of nt steps of a propagation under way (what the server and
                 a caller with its own loop issue), starting again from the initial state;
         "live"  nt steps and one observable record: a caller that looks at every record;
         "batch" count uneven driven-trap instances advanced nt steps together.
  prec   "c128" native FP64, "c128f" float-float, "c64" FP32 with high + low tables
  n      extents of the grid, "x"-separated
  pot    "trap"    driven trap: quadratic + oscillating linear term (1-D workload, batch)
         "laser"   anisotropic trap + linear term under a Gaussian envelope (2-D workload)
         "barrier" time-dependent spherical Gaussian barrier (3-D workload)
         "moving"  moving Gaussian barrier over a weak trap (served requests)
         "morse"   Morse well + sin^2-enveloped dipole (the paper's CO molecule)
         "paul"    the paper's Ba+ ion trap in SI units
  order  "vkv" or "kvk" (the paper's order)

The potential's parameters and the packet come from the workloads' recipes, spread by the
seed. complex64 results are returned in their own precision (complex64 state, float32
records), the other forms' as complex128 and float64.
"""
import math

import numpy as np
import torch

from paper_1306_3247_gb300 import wavepacket as WPK

HALF_PI = math.pi / 2
HBAR_SI, E_SI = 1.054571726e-34, 1.602176565e-19
COLS = ("t", "norm", "x0", "x1", "x2", "p0", "p1", "p2", "xx0", "xx1", "xx2", "energy", "ekin", "epot")


def listed():
    return [
        # the 1-D driven-trap workload: 1000-step jobs with a record every 10 steps (a fifth
        # of the job)
        {"name": "trap_1d_1024_c128", "kind": "run", "prec": "c128", "n": "1024", "pot": "trap", "order": "vkv",
         "nt": 200, "nprint": 10},
        # the paper's CO molecule on its 4096-point line, in the middle of the pulse: half a
        # million steps in the paper, records far apart
        {"name": "morse_1d_4096_c128", "kind": "run", "prec": "c128", "n": "4096", "pot": "morse", "order": "vkv",
         "nt": 100, "nprint": 100},
        # a served 1-D request at the longest line, one scheduling chunk
        {"name": "chunk_1d_16384_c64", "kind": "step", "prec": "c64", "n": "16384", "pot": "trap", "order": "vkv",
         "nt": 50, "nprint": 50},
        # the smallest call: a small grid with unequal axes, a record after every step
        {"name": "live_2d_64x256_c64", "kind": "live", "prec": "c64", "n": "64x256", "pot": "moving", "order": "vkv",
         "nt": 1, "nprint": 1},
        # the 2-D laser workload in native FP64 (50 of its 500 steps, its record interval)
        {"name": "laser_2d_1024_c128", "kind": "run", "prec": "c128", "n": "1024x1024", "pot": "laser",
         "order": "vkv", "nt": 50, "nprint": 50},
        # the same grid in complex64, the paper's operator order
        {"name": "laser_2d_1024_c64", "kind": "run", "prec": "c64", "n": "1024x1024", "pot": "laser",
         "order": "kvk", "nt": 100, "nprint": 50},
        # a mid-sized uneven 2-D grid in the float-float form
        {"name": "moving_2d_512x128_c128f", "kind": "run", "prec": "c128f", "n": "512x128", "pot": "moving",
         "order": "kvk", "nt": 40, "nprint": 20},
        # a served 3-D request at the smallest extent, one scheduling chunk
        {"name": "chunk_3d_64_c64", "kind": "step", "prec": "c64", "n": "64x64x64", "pot": "moving", "order": "vkv",
         "nt": 50, "nprint": 50},
        # the 3-D barrier workload in native FP64, one record interval: the benchmark's headline
        {"name": "barrier_3d_256_c128", "kind": "run", "prec": "c128", "n": "256x256x256", "pot": "barrier",
         "order": "vkv", "nt": 20, "nprint": 20},
        # the same job in complex64, two record intervals
        {"name": "barrier_3d_256_c64", "kind": "run", "prec": "c64", "n": "256x256x256", "pot": "barrier",
         "order": "vkv", "nt": 40, "nprint": 20},
        # the paper's ion trap on its 512^3 grid, one record interval, float-float: the largest
        {"name": "paul_3d_512_c128f", "kind": "run", "prec": "c128f", "n": "512x512x512", "pot": "paul",
         "order": "vkv", "nt": 10, "nprint": 10},
        # the uneven batch of 1-D and 2-D instances (an eighth of the benchmark's), one chunk
        {"name": "batch_512_c64", "kind": "batch", "prec": "c64", "n": "mixed", "pot": "trap", "order": "vkv",
         "nt": 20, "nprint": 20, "count": 512},
    ]


def draw(rng):
    # at most the cost of the 512^3 float-float job: points x steps weighted by the form
    weight = {"c64": 1.0, "c128f": 4.0, "c128": 16.0}
    budget = 2.0 ** 27 * 10 * weight["c128f"]
    prec = rng.choice(("c64", "c64", "c128", "c128", "c128f"))
    order = rng.choice(("vkv", "vkv", "kvk"))
    if rng.random() < 0.1:
        return {"kind": "batch", "prec": prec, "n": "mixed", "pot": "trap", "order": "vkv",
                "nt": rng.randint(5, 25), "nprint": 1, "count": int(round(2 ** rng.uniform(4, 9)))}
    nd = rng.choice((1, 1, 2, 2, 3, 3))
    if nd == 1:
        n = [2 ** rng.randint(8, 14 if prec == "c64" else 13)]
        pot = rng.choice(("trap", "trap", "morse", "moving"))
        nt = int(round(2 ** rng.uniform(0, 8)))
    elif nd == 2:
        n = [2 ** rng.randint(6, 11) for _ in range(2)]
        pot = rng.choice(("laser", "moving", "trap"))
        nt = int(round(2 ** rng.uniform(0, 6.5)))
    else:
        base = rng.randint(5, 9 if prec != "c128" else 8)
        n = [2 ** max(5, base - rng.randint(0, 2)) for _ in range(2)] + [2 ** base]
        rng.shuffle(n)
        pot = rng.choice(("barrier", "moving", "paul"))
        nt = int(round(2 ** rng.uniform(0, 5.5)))
    # the record passes cost about as much as two steps
    most = int(budget / (math.prod(n) * weight[prec])) - 4
    nt = max(1, min(nt, most))
    kind = rng.choice(("run", "run", "step", "live"))
    nprint = nt if kind != "run" else rng.choice((nt, max(1, nt // 2), max(1, nt // 5)))
    return {"kind": kind, "prec": prec, "n": "x".join(str(v) for v in n), "pot": pot, "order": order, "nt": nt,
            "nprint": nprint}


# ---------------------------------------------------------------- inputs
def _spread(rng, v, by=0.1):
    return v * float(rng.uniform(1.0 - by, 1.0 + by))


def _inputs(case, seed):
    """Problem, potential terms and packet of a single propagation (workloads.py's schema)."""
    rng = np.random.default_rng([1306, int(seed)])
    n = [int(v) for v in case["n"].split("x")]
    nd = len(n)
    box, mass, hbar, dt, t0 = [40.0] * nd, 1.0, 1.0, 0.005, 0.0
    rest = [0.0] * (nd - 1)
    xmin = None
    pot = case["pot"]
    if pot == "trap":
        w = float(rng.uniform(0.5, 2.0))
        terms = [{"shape": "quad", "a": [w * w] * nd, "coef": {"A0": 1.0}},
                 {"shape": "linear", "a": [1.0] + rest, "coef": {"A": float(rng.uniform(0.02, 0.2)), "omega": 0.9 * w}}]
        init = {"x0": [_spread(rng, 2.0)] + rest, "p0": [0.0] * nd, "sigma": [math.sqrt(2.0 / w)] * nd}
        dt = 0.01 if nd == 1 else 0.005
    elif pot == "laser":
        box = [80.0] * nd
        terms = [{"shape": "quad", "a": [_spread(rng, 1.0), _spread(rng, 4.0)], "coef": {"A0": 1.0}},
                 {"shape": "linear", "a": [1.0, 0.0],
                  "coef": {"A": _spread(rng, 0.05), "omega": _spread(rng, 0.5), "phi": HALF_PI, "env": "gauss",
                           "t0": 10.0, "tau": 4.0}}]
        init = {"x0": [0.0, 0.0], "p0": [_spread(rng, 1.0), 0.0], "sigma": [1.0, _spread(rng, 0.7)]}
        t0 = 8.0  # the envelope is on
    elif pot == "barrier":
        box = [60.0] * nd
        terms = [{"shape": "gauss", "a": [1.0] * nd,
                  "coef": {"A0": _spread(rng, 1.5), "A": _spread(rng, 0.45), "omega": _spread(rng, 2.0)}}]
        init = {"x0": [_spread(rng, -3.0)] + rest, "p0": [_spread(rng, 2.0)] + rest,
                "sigma": [_spread(rng, 1.5) for _ in range(nd)]}
        dt = 0.002
    elif pot == "moving":
        terms = [{"shape": "quad", "a": [0.01] * nd, "coef": {"A0": 1.0}},
                 {"shape": "gauss", "a": [float(rng.uniform(0.5, 1.5))] + rest, "c0": [2.0] + rest,
                  "v": [float(rng.uniform(-1.0, 1.0))] + rest, "coef": {"A0": float(rng.uniform(0.5, 3.0))}}]
        init = {"x0": [_spread(rng, -4.0)] + rest, "p0": [_spread(rng, 2.0)] + rest, "sigma": [1.5] * nd}
    elif pot == "morse":
        lo, hi = 1.5e-3, 6.0
        box, xmin = [n[0] * (hi - lo) / (n[0] - 1)], [lo]
        mass, dt, t0 = 12498.10, 0.1, 20000.0
        xe = 2.1322214
        pulse = {"omega": 9.8864e-3, "phi": HALF_PI, "env": "sin2", "t0": 0.0, "tau": 41341.37}
        terms = [{"shape": "morse", "a": [0.4076, 1.230211, 0.0], "c0": [xe], "coef": {"A0": 1.0}},
                 {"shape": "linear", "a": [-0.948], "c0": [xe], "coef": dict(pulse, A=_spread(rng, 1.69e-3))},
                 {"shape": "const", "coef": dict(pulse, A=-0.1466 * 1.69e-3)}]
        init = {"x0": [_spread(rng, xe, 0.02)], "p0": [0.0], "sigma": [_spread(rng, 0.1)]}
    else:  # paul
        lo, hi = -1e-6, 1e-6
        box, xmin = [v * (hi - lo) / (v - 1) for v in n], [lo] * nd
        mass, hbar, dt = 2.28997005e-25, HBAR_SI, 2e-9
        r0 = 1.6e-3
        kappa = E_SI / (2.0 * r0 * r0)  # d^2 = r0^2 + 2 z0^2 with z0 = r0 / sqrt(2)
        terms = [{"shape": "quad", "a": [kappa, kappa, -2.0 * kappa],
                  "coef": {"A0": 0.0, "A": _spread(rng, 200.0), "omega": 2 * math.pi * 18e6, "phi": HALF_PI}}]
        init = {"x0": [_spread(rng, 2e-8), _spread(rng, 1e-8), _spread(rng, 2e-8)],
                "p0": [_spread(rng, 1e-27), 0.0, 0.0], "sigma": [_spread(rng, 7.342e-8), 7.342e-8, 5.192e-8]}
    if xmin is None:
        xmin = [-v / 2 for v in box]
    problem = {"ndim": nd, "n": n, "xmin": xmin, "L": box, "mass": mass, "hbar": hbar, "dt": dt, "t0": t0,
               "order": case["order"]}
    return problem, terms, init


def _batch_inputs(case, seed):
    """The uneven instances: 1-D or 2-D by a fair coin, 1-D lengths 2^8..2^13, 2-D axes of 64,
    128 or 256, driven traps. The shapes do not depend on the seed; the parameters do."""
    shapes, rng = np.random.default_rng(1306), np.random.default_rng([3247, int(seed)])
    out = []
    for _ in range(case["count"]):
        if shapes.random() < 0.5:
            n = [int(shapes.choice([64, 128, 256])), int(shapes.choice([64, 128, 256]))]
        else:
            n = [int(2 ** shapes.integers(8, 14))]
        nd = len(n)
        w = float(rng.uniform(0.5, 2.0))
        sig = math.sqrt(2.0 / w) * float(rng.uniform(0.7, 1.3))
        box = [max(20.0, 16.0 * sig * v / 256.0) for v in n]
        problem = {"ndim": nd, "n": n, "xmin": [-v / 2 for v in box], "L": box, "dt": 0.005, "order": case["order"]}
        terms = [{"shape": "quad", "a": [w * w] * nd, "coef": {"A0": 1.0}},
                 {"shape": "linear", "a": [1.0] + [0.0] * (nd - 1),
                  "coef": {"A": float(rng.uniform(0.0, 0.2)), "omega": 0.9 * w}}]
        out.append((problem, terms, {"x0": [0.0] * nd, "p0": [0.0] * nd, "sigma": [sig] * nd}))
    return out


def _axes(problem):
    for d in range(problem["ndim"]):
        n, step = problem["n"][d], problem["L"][d] / problem["n"][d]
        yield d, problem["xmin"][d] + torch.arange(n, dtype=torch.float64, device="cuda") * step


def _along(v, d, nd):
    return v.reshape([-1 if k == d else 1 for k in range(nd)])


def _packet(problem, init):
    """The normalised Gaussian packet on the grid, complex128."""
    nd, hbar = problem["ndim"], problem.get("hbar", 1.0)
    psi = None
    for d, x in _axes(problem):
        u, s = x - init["x0"][d], init["sigma"][d]
        f = torch.polar((2.0 / math.pi) ** 0.25 / math.sqrt(s) * torch.exp(-(u / s) ** 2), init["p0"][d] * u / hbar)
        psi = _along(f, d, nd) if psi is None else psi * _along(f, d, nd)
    return psi.contiguous()


class _View:
    """A handle's complex64 state, for torch's array interface; keeps its owner alive."""

    def __init__(self, owner, handle, shape):
        self.owner = owner
        self.__cuda_array_interface__ = {"data": (WPK.wp_state_ptr(handle), False), "shape": tuple(shape),
                                         "typestr": "<c8", "version": 3}


def _state_view(owner, handle, shape):
    return torch.as_tensor(_View(owner, handle, shape), device="cuda")


class _Single:
    """A propagator, its initial state and the buffer its results go to."""

    def __init__(self, case, seed):
        problem, terms, init = _inputs(case, seed)
        self.case, self.stream = case, torch.cuda.Stream()
        self.prop = WPK.Propagator(problem, terms, case["prec"], stream=self.stream.cuda_stream)
        self.psi0 = _packet(problem, init)
        # complex64 states are read in place, the other forms as complex128
        self.out = (_state_view(self.prop, self.prop.h, self.prop.shape) if case["prec"] == "c64"
                    else torch.empty_like(self.psi0))
        torch.cuda.synchronize()


class _Many:
    def __init__(self, case, seed):
        self.case, self.stream = case, torch.cuda.Stream()
        self.batch = WPK.Batch(case["prec"], stream=self.stream.cuda_stream)
        self.psi0, self.views = [], []
        for problem, terms, init in _batch_inputs(case, seed):
            k = self.batch.add(problem, terms)
            h = self.batch.handle(k)
            psi = _packet(problem, init)
            self.psi0.append((h, psi))
            if case["prec"] == "c64":
                self.views.append(_state_view(self.batch, h, problem["n"]).reshape(-1))
        self.out = torch.empty(sum(p.numel() for _, p in self.psi0), dtype=torch.complex128, device="cuda")
        torch.cuda.synchronize()
        for h, psi in self.psi0:
            WPK.wp_set_state(h, psi.data_ptr(), True)
        torch.cuda.synchronize()


def prepare(case, seed):
    return _Many(case, seed) if case["kind"] == "batch" else _Single(case, seed)


def _records(prec, rec):
    m = np.stack([np.atleast_1d(rec)[c] for c in COLS], axis=-1)
    return m.astype(np.float32) if prec == "c64" else m


def run(state):
    case = state.case
    if case["kind"] == "batch":
        # the next chunk of every instance; the states come back as one flat array
        state.batch.step(case["nt"])
        if case["prec"] == "c64":
            with torch.cuda.stream(state.stream):
                return torch.cat(state.views)
        at = 0
        for h, psi in state.psi0:
            WPK.wp_get_state(h, state.out.data_ptr() + 16 * at, True)
            at += psi.numel()
        return state.out
    P = state.prop
    WPK.wp_set_state(P.h, state.psi0.data_ptr(), True)
    P.step_index = 0
    rec = None
    if case["kind"] == "run":
        rec = P.run(case["nt"], case["nprint"])
    else:
        P.step(case["nt"])
        if case["kind"] == "live":
            rec = P.observe()
    out = state.out if case["prec"] == "c64" else P.get_state_device(state.out)
    return out if rec is None else [out, _records(case["prec"], rec)]


# ---------------------------------------------------------------- what a pass cannot do without
def work(case):
    """Bytes: the initial state in and the final state out (and the records), once each.
    FLOPs: per step a forward and an inverse FFT at 5 log2 N per point and two products with
    a unit factor at 6 (one potential, one kinetic), and 10 log2 N per record for its
    momentum sums."""
    if case["kind"] == "batch":
        sizes = [math.prod(p["n"]) for p, _, _ in _batch_inputs(case, 0)]
        elem = 8 if case["prec"] == "c64" else 16
        return {"bytes": float(sum(2 * elem * v for v in sizes)),
                "flops": float(sum(case["nt"] * v * (10 * math.log2(v) + 12) for v in sizes))}
    npts = math.prod(int(v) for v in case["n"].split("x"))
    records = {"run": 1 + case["nt"] // case["nprint"], "step": 0, "live": 1}[case["kind"]]
    out = 8 if case["prec"] == "c64" else 16
    return {"bytes": float(npts * (16 + out) + 128 * records),
            "flops": float(npts * (case["nt"] * (10 * math.log2(npts) + 12) + records * (5 * math.log2(npts) + 20)))}


# ---------------------------------------------------------------- the same in 64 bits, plainly
def _coef(tm, t):
    c = tm.get("coef", {})
    env, tau, at = c.get("env", "none"), c.get("tau", 1.0), c.get("t0", 0.0)
    e = 1.0
    if env == "gauss":
        e = math.exp(-((t - at) / tau) ** 2)
    elif env == "sin2":
        e = math.sin(math.pi * t / tau) ** 2 if at <= t <= at + tau else 0.0
    return c.get("A0", 0.0) + c.get("A", 0.0) * e * math.sin(c.get("omega", 0.0) * t + c.get("phi", 0.0))


def _potential(problem, terms, t):
    """V(x, t) on the grid, FP64."""
    nd = problem["ndim"]
    V = torch.zeros([1] * nd, dtype=torch.float64, device="cuda")
    axes = dict(_axes(problem))
    for tm in terms:
        f, a = _coef(tm, t), list(tm.get("a", [])) + [0.0] * 3
        c0, v = list(tm.get("c0", [])) + [0.0] * 3, list(tm.get("v", [])) + [0.0] * 3
        if tm["shape"] == "const":
            V = V + f
            continue
        if tm["shape"] == "morse":
            k = int(a[2])
            u = axes[k] - (c0[k] + v[k] * t)
            V = V + f * _along(a[0] * (1.0 - torch.exp(-a[1] * u)) ** 2, k, nd)
            continue
        prod = None
        for d in range(nd):
            u = axes[d] - (c0[d] + v[d] * t)
            if tm["shape"] == "quad":
                V = V + f * _along(0.5 * a[d] * u * u, d, nd)
            elif tm["shape"] == "linear":
                V = V + f * _along(a[d] * u, d, nd)
            elif a[d] > 0.0:
                g = _along(torch.exp(-(u / a[d]) ** 2), d, nd)
                prod = g if prod is None else prod * g
        if tm["shape"] == "gauss":
            V = V + f * (1.0 if prod is None else prod)
    return V.expand(problem["n"])


def _wavenumbers(problem):
    for d in range(problem["ndim"]):
        n = problem["n"][d]
        j = torch.arange(n, dtype=torch.float64, device="cuda")
        yield d, 2.0 * math.pi / problem["L"][d] * torch.where(j < n // 2, j, j - n)


def _kinetic(problem, tau):
    nd, hbar, mass = problem["ndim"], problem.get("hbar", 1.0), problem.get("mass", 1.0)
    f = None
    for d, k in _wavenumbers(problem):
        th = -hbar * k * k * tau / (2.0 * mass)
        g = _along(torch.complex(torch.cos(th), torch.sin(th)), d, nd)
        f = g if f is None else f * g
    return f


def _advance(problem, terms, psi, s, m):
    """m steps from step index s, adjacent half-steps not merged."""
    hbar, dt, t0 = problem.get("hbar", 1.0), problem["dt"], problem.get("t0", 0.0)

    def pot(x, t, tau):
        th = _potential(problem, terms, t) * (-tau / hbar)
        return x * torch.complex(torch.cos(th), torch.sin(th))

    vkv = problem["order"] == "vkv"
    full = _kinetic(problem, dt if vkv else 0.5 * dt)

    def kin(x):
        return torch.fft.ifftn(torch.fft.fftn(x) * full)

    for k in range(s, s + m):
        if vkv:
            psi = pot(kin(pot(psi, t0 + k * dt, 0.5 * dt)), t0 + (k + 1) * dt, 0.5 * dt)
        else:
            psi = kin(pot(kin(psi), t0 + k * dt + 0.5 * dt, dt))
    return psi


def _record(problem, terms, psi, s):
    nd, hbar, mass = problem["ndim"], problem.get("hbar", 1.0), problem.get("mass", 1.0)
    dv = math.prod(problem["L"][d] / problem["n"][d] for d in range(nd))
    t = problem.get("t0", 0.0) + s * problem["dt"]
    rho = psi.real ** 2 + psi.imag ** 2
    hat = torch.fft.fftn(psi)
    rhok = hat.real ** 2 + hat.imag ** 2
    dvk = dv / psi.numel()
    x, xx, p, ek = [0.0] * 3, [0.0] * 3, [0.0] * 3, 0.0
    for (d, g), (_, k) in zip(_axes(problem), _wavenumbers(problem)):
        others = [e for e in range(nd) if e != d]
        m = rho.sum(dim=others) if others else rho
        mk = rhok.sum(dim=others) if others else rhok
        x[d], xx[d] = float((g * m).sum()) * dv, float((g * g * m).sum()) * dv
        p[d] = hbar * float((k * mk).sum()) * dvk
        ek += hbar * hbar / (2.0 * mass) * float((k * k * mk).sum()) * dvk
    ev = float((_potential(problem, terms, t) * rho).sum()) * dv
    return [t, math.sqrt(float(rho.sum()) * dv)] + x + p + xx + [ek + ev, ek, ev]


def exact(case, seed):
    if case["kind"] == "batch":
        return torch.cat([_advance(p, tm, _packet(p, i), 0, case["nt"]).reshape(-1)
                          for p, tm, i in _batch_inputs(case, seed)])
    problem, terms, init = _inputs(case, seed)
    psi, rec = _packet(problem, init), []
    nt, each = case["nt"], case["nprint"]
    if case["kind"] == "run":
        rec.append(_record(problem, terms, psi, 0))
        for s in range(0, nt - nt % each, each):
            psi = _advance(problem, terms, psi, s, each)
            rec.append(_record(problem, terms, psi, s + each))
        psi = _advance(problem, terms, psi, nt - nt % each, nt % each)
    else:
        psi = _advance(problem, terms, psi, 0, nt)
        if case["kind"] == "live":
            rec.append(_record(problem, terms, psi, nt))
    return [psi, np.array(rec)] if rec else psi
