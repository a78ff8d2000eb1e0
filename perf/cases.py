"""Performance cases of the stepper: what a user's program has the library do, through
its public Python entry points (``Simulation`` and ``Server``).

A case is a dict of plain values.  ``prepare`` makes what a program has in hand before
the call (a simulation with its seeded initial condition, or a running server and its
requests), ``run`` is one pass (a number of time steps and the fields they leave; or a
burst of served requests), ``work`` the bytes and operations a pass cannot do without,
and ``exact`` the same pass in plain FP64 torch.

BF16 storage is left out: the library refuses it unless a program opts out of every
accuracy bound.
"""
import math
import random

import torch

import paper_2511_10508_gb300 as sp

MODELS = {"ac": sp.ALLEN_CAHN, "ch": sp.CAHN_HILLIARD, "gs": sp.GRAY_SCOTT, "mc": sp.MODEL_C, "mh": sp.MODEL_H}
STENCILS = {"5": sp.LAP_5, "9box": sp.LAP_9BOX, "9cross": sp.LAP_9CROSS4, "7": sp.LAP_7, "27": sp.LAP_27,
            "13cross": sp.LAP_13CROSS4, "gen": sp.LAP_GENERATED}
DTYPES = {"f64": sp.F64, "f32": sp.F32}
# floating-point operations of one application (sums of neighbour classes, one multiply
# or multiply-add per class and one for the centre)
STENCIL_OPS = {"5": 4, "9box": 6, "9cross": 8, "7": 6, "27": 12, "13cross": 12}
# central second differences of accuracy 2, 4, 6, 8: weights of f0, f(+-1), ...
CENTRAL = {2: (-2.0, 1.0), 4: (-5 / 2, 4 / 3, -1 / 12), 6: (-49 / 18, 3 / 2, -3 / 20, 1 / 90),
           8: (-205 / 72, 8 / 5, -1 / 5, 8 / 315, -1 / 560)}


def _case(name, model, dtype, nx, ny, nz, steps, stencil, **kw):
    """A simulation case: nz = 0 is a 2D grid; order only counts for generated stencils."""
    c = {"kind": "step", "model": model, "dtype": dtype, "nx": nx, "ny": ny, "nz": nz, "steps": steps,
         "stencil": stencil, "order": 0, "spectral": False, "tune": False, "monitor": False,
         "mean": 0.0, "amp": 0.01, "patches": 0, "patch": 0}
    c.update(kw)
    if name:
        c = {"name": name, **c}
    return c


def _serve(name, requests, mix, max2d, max3d, max_steps):
    c = {"kind": "serve", "requests": requests, "mix": mix, "max2d": max2d, "max3d": max3d, "max_steps": max_steps}
    return {"name": name, **c} if name else c


def listed():
    return [
        # The smallest benchmark configuration: a grid that fits on chip, stepped between
        # two snapshots; the cost of a launch is what counts.
        _case("ac2d-256-f64", "ac", "f64", 256, 256, 0, 100, "5", tune=True, amp=0.1),
        # The benchmark's default workload: FP64 Cahn-Hilliard at production size.
        _case("ch2d-4096-f64", "ch", "f64", 4096, 4096, 0, 70, "5", tune=True),
        # A domain sized by physics rather than by powers of two, with the 4th-order stencil.
        _case("ch2d-1503x1001-f32", "ch", "f32", 1503, 1001, 0, 20, "9cross"),
        # Two-field reaction-diffusion patterns on a grid far larger than any cache.
        _case("gs2d-16384-f32", "gs", "f32", 16384, 16384, 0, 10, "5", patches=64, patch=20),
        # Off-critical 3D coarsening with mass and free energy watched after every block of steps.
        _case("ch3d-512-f32-monitored", "ch", "f32", 512, 512, 512, 10, "7", monitor=True, mean=0.1),
        # The isotropic 27-point stencil, which 3D coarsening studies use to avoid grid anisotropy.
        _case("ch3d-384-f32-27", "ch", "f32", 384, 384, 384, 10, "27"),
        # Solidification (Model C) in a box with odd sides.
        _case("mc3d-250x198x301-f32", "mc", "f32", 250, 198, 301, 10, "7", amp=0.1),
        # Model H (a scalar and a three-component current): the most fields per point.
        _case("mh3d-256-f32", "mh", "f32", 256, 256, 256, 10, "7", amp=0.1),
        # High-accuracy generated stencil.
        _case("ch2d-8192-f32-order8", "ch", "f32", 8192, 8192, 0, 5, "gen", order=8),
        # The semi-implicit spectral scheme with large steps, 2D single precision.
        _case("ch2d-8192-f32-spectral", "ch", "f32", 8192, 8192, 0, 5, "5", spectral=True, amp=0.1),
        # The same in 3D, double precision.
        _case("ch3d-256-f64-spectral", "ch", "f64", 256, 256, 256, 5, "7", spectral=True, amp=0.1),
        # A burst of simulations of differing model, dimension, size and precision, served together.
        _serve("served-burst", 10, 4, 2048, 256, 300),
    ]


def _side(rng, lo, hi):
    """Log-uniform; about a third of the sides odd, the others multiples of 2 to 16."""
    s = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    g = rng.choice((1, 1, 2, 4, 8, 16))
    return max(lo, int(round(s / g)) * g) | (1 if g == 1 and rng.random() < 0.7 else 0)


def _smooth_side(rng, lo, hi):
    """A transform length: a power of two half of the time, else a product of 2, 3, 5, 7."""
    if rng.random() < 0.5:
        return 1 << rng.randint(int(math.log2(lo)), int(math.log2(hi)))
    while True:
        n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        m = n
        for p in (2, 3, 5, 7):
            while m % p == 0:
                m //= p
        if m == 1:
            return n


def draw(rng):
    what = rng.choice(("2d", "2d", "3d", "3d", "spectral", "spectral", "serve"))
    if what == "serve":
        return _serve(None, rng.randint(3, 8), rng.randint(0, 10 ** 6), 1024, 128, 300)
    dims = 2 if what == "2d" or (what == "spectral" and rng.random() < 0.5) else 3
    dtype = rng.choice(("f32", "f32", "f64"))
    if what == "spectral":
        model = rng.choice(("ac", "ch"))
        # lengths every side may have: 2048 (FP64) or 4096 (FP32), twice that for powers of two
        lo, hi = (64, 2048 if dtype == "f64" else 4096) if dims == 2 else (32, 256)
        sides = [_smooth_side(rng, lo, hi) for _ in range(dims)]
        stencil, order = ("5" if dims == 2 else "7"), 0
    else:
        model = rng.choice(("ac", "ch", "ch", "gs", "mc", "mh"))
        lo, hi = (64, 8192) if dims == 2 else (32, 400)
        sides = [_side(rng, lo, hi) for _ in range(dims)]
        stencil = rng.choice((("5", "9box", "9cross") if dims == 2 else ("7", "27", "13cross")) +
                             (("gen",) if model != "mh" else ()))
        order = rng.choice((2, 4, 6, 8)) if stencil == "gen" else 0
    n = math.prod(sides)
    steps = max(4, min(100, int(1e9 / n) // 4))
    if what == "spectral":
        steps = max(3, steps // 4)
    amp = 0.01 if model == "gs" else math.exp(rng.uniform(math.log(0.01), math.log(0.3)))
    return _case(None, model, dtype, sides[0], sides[1], sides[2] if dims == 3 else 0, steps, stencil, order=order,
                 spectral=what == "spectral", tune=what != "spectral" and steps >= 70 and rng.random() < 0.5,
                 monitor=what != "spectral" and rng.random() < 0.25, mean=0.1 if model != "gs" else 0.0,
                 amp=round(amp, 4), patches=8 if model == "gs" else 0, patch=min(20, min(sides) // 4) if model == "gs" else 0)


# ------------------------------------------------------------------ what a case means --

def _dims(c):
    return 3 if c["nz"] else 2


def _shape(c):
    return (c["nz"], c["ny"], c["nx"]) if c["nz"] else (c["ny"], c["nx"])


def _nfields(model, dims):
    return 1 + dims if model == "mh" else 2 if model in ("gs", "mc") else 1


def _dt(c):
    """Inside the stability bound of every stencil the model is drawn with."""
    two = not c["nz"]
    if c["spectral"]:
        return 0.5
    if c["stencil"] == "gen":
        return {"ac": 0.05, "ch": 0.002 if two else 0.001, "gs": 0.5, "mc": 0.02}[c["model"]]
    return {"ac": 0.05, "ch": 0.01 if two else 0.005, "gs": 1.0 if two and c["stencil"] != "9cross" else 0.5,
            "mc": 0.02, "mh": 0.01 if two else 0.005}[c["model"]]


def _requests(c):
    """The burst's simulations as cases (their model, size, precision and coefficients follow from the case alone)."""
    rng = random.Random(c["mix"])
    out = []
    for _ in range(c["requests"]):
        model = rng.choice(("ac", "ch", "gs"))
        two = rng.random() < 0.5
        lo, hi = (64, c["max2d"]) if two else (32, c["max3d"])
        side = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        r = _case(None, model, rng.choice(("f32", "f64")), side, side, 0 if two else side,
                  rng.randint(100, c["max_steps"]), "5" if two else "7", amp=0.01 if model == "gs" else 0.05,
                  mean=0.0, patches=4 if model == "gs" else 0, patch=8 if model == "gs" else 0)
        out.append(r)
    return out


def _kw(c, seed):
    kw = {"seed": int(seed), "dtype": DTYPES[c["dtype"]], "ic_mean": c["mean"], "ic_amp": c["amp"]}
    if c["spectral"]:
        kw["scheme"] = sp.SCHEME_SPECTRAL
    else:
        kw["stencil"] = STENCILS[c["stencil"]]
        if c["order"]:
            kw["stencil_order"] = c["order"]
    if c["model"] == "gs":
        kw.update(gs_patches=c["patches"], gs_patch=c["patch"])
    if c["tune"]:
        kw["flags"] = sp.FLAG_AUTOTUNE
    return kw


def prepare(case, seed):
    if case["kind"] == "serve":
        todo = [((MODELS[r["model"]], _shape(r)), dict(dt=_dt(r), nsteps=r["steps"], return_fields=True, **_kw(r, seed + 1000 * i)))
                for i, r in enumerate(_requests(case))]
        return {"server": sp.Server(120 << 30, max_slots=512, quantum_steps=50), "todo": todo}
    sim = sp.Simulation(MODELS[case["model"]], _shape(case), dt=_dt(case), **_kw(case, seed))
    return {"sim": sim, "steps": case["steps"], "monitor": case["monitor"]}


def run(state):
    if "server" in state:
        srv = state["server"]
        tickets = [srv.submit(*a, **k) for a, k in state["todo"]]
        done = [srv.wait(t) for t in tickets]
        for t in tickets:
            srv.release(t)
        return [{"fields": r.fields, "steps": r.steps_done} for r in done]
    sim = state["sim"]
    sim.step(state["steps"])
    out = {}
    if state["monitor"]:
        out["mass"] = sim.reduce(sp.MASS)
        out["free_energy"] = sim.reduce(sp.FREE_ENERGY)
    out["fields"] = []
    for f in range(sim.nfields):
        t = sim.field_tensor(f)
        t.owner = sim  # the view is the simulation's own memory: the tensor keeps it alive
        out["fields"].append(t)
    return out


def _step_work(c):
    """Bytes and operations of one time step: every field read once and written once
    (spectral: one pass per transform axis), the counted operations of the update."""
    dims, p = _dims(c), 8 if c["dtype"] == "f64" else 4
    n = math.prod(_shape(c))
    if c["spectral"]:
        return (7 if dims == 2 else 11) * p * n, (5.0 * math.log2(n) + 9.5) * n
    if c["stencil"] == "gen":
        r = c["order"] // 2
        s = r * (2 * dims - 1) + r + 1
    else:
        s = STENCIL_OPS[c["stencil"]]
    dc = 3 if c["stencil"] in ("9cross", "13cross") else 1
    ops = {"ac": s + 5, "ch": 2 * s + 5, "gs": 2 * s + 9, "mc": 2 * s + 9,
           "mh": (2 + dims) * s + dims * (7 + 2 * dc) + 6}[c["model"]]
    return 2 * _nfields(c["model"], dims) * p * n, ops * n


def work(case):
    if case["kind"] == "serve":
        b = f = 0
        for r in _requests(case):
            rb, rf = _step_work(r)
            b += rb * r["steps"] + 8 * _nfields(r["model"], _dims(r)) * math.prod(_shape(r))
            f += rf * r["steps"]
        return {"bytes": b, "flops": f}
    b, f = _step_work(case)
    b, f = b * case["steps"], f * case["steps"]
    if case["monitor"]:  # the fields read once more, a few operations per value
        n = math.prod(_shape(case))
        b += n * _nfields(case["model"], _dims(case)) * (8 if case["dtype"] == "f64" else 4)
        f += 10 * n
    return {"bytes": b, "flops": f}


# --------------------------------------------------------------- the same in FP64 torch --

def _i64(x):
    x &= (1 << 64) - 1
    return x - (1 << 64) if x >> 63 else x


_GAMMA, _M1, _M2 = 0x9E3779B97F4A7C15, 0xBF58476D1CE4E5B9, 0x94D049BB133111EB


def _noise(seed, first, n, amp, dev):
    """amp (2 U - 1) for outputs first .. first + n - 1 of SplitMix64(seed)."""
    z = torch.arange(n, dtype=torch.int64, device=dev).mul_(_i64(_GAMMA)).add_(_i64(seed + (first + 1) * _GAMMA))
    for sh, m in ((30, _M1), (27, _M2), (31, None)):
        z = z ^ ((z >> sh) & ((1 << (64 - sh)) - 1))
        if m is not None:
            z = z * _i64(m)
    u = ((z >> 11) & ((1 << 53) - 1)).double().mul_(2.0 ** -53)
    return u.mul_(2.0).sub_(1.0).mul_(amp)


def _splitmix(seed, n):
    m = (1 << 64) - 1
    z = (seed + (n + 1) * _GAMMA) & m
    z = ((z ^ (z >> 30)) * _M1) & m
    z = ((z ^ (z >> 27)) * _M2) & m
    return z ^ (z >> 31)


def _initial(c, seed, dev):
    """The seeded start in the storage precision, widened to FP64."""
    shape, dims = _shape(c), _dims(c)
    n = math.prod(shape)
    fields = []
    for f in range(_nfields(c["model"], dims)):
        base = 0.0 if c["model"] == "mh" and f else c["mean"]
        if c["model"] == "gs":
            sides = (c["nx"], c["ny"], c["nz"])[:dims]
            base = torch.full(shape, 1.0 - f, dtype=torch.float64, device=dev)
            for p in range(c["patches"]):
                at = [(torch.arange(c["patch"], device=dev) + (_splitmix(seed, 2 * n + 3 * p + a) % s - c["patch"] // 2) % s) % s
                      for a, s in enumerate(sides)]
                base[torch.meshgrid(*at[::-1], indexing="ij")] = 0.25 if f else 0.5
        x = _noise(seed, f * n, n, c["amp"], dev).reshape(shape).add_(base)
        fields.append(x.float().double() if c["dtype"] == "f32" else x)
    return fields


def _pairs(f, axis, d=1):
    return torch.roll(f, d, axis).add_(torch.roll(f, -d, axis))


def _laplacian(f, c):
    axes, st = range(f.dim()), c["stencil"]
    if st in ("5", "7"):
        s = f * (-2.0 * f.dim())
        for a in axes:
            s += _pairs(f, a)
        return s
    if st in ("9cross", "13cross", "gen"):
        w = CENTRAL[c["order"] or 4]
        s = f * (w[0] * f.dim())
        for a in axes:
            for d in range(1, len(w)):
                s.add_(_pairs(f, a, d), alpha=w[d])
        return s
    if st == "9box":
        p = _pairs(f, 1)
        return ((p + _pairs(f, 0)).mul_(4.0).add_(_pairs(p, 0)).add_(f, alpha=-20.0)).div_(6.0)
    faces, px, py = torch.zeros_like(f), _pairs(f, 2), _pairs(f, 1)  # 27 points
    faces += px
    faces += py
    faces += _pairs(f, 0)
    pxy = _pairs(px, 1)
    s = f * -128.0
    s.add_(faces, alpha=14.0)
    s.add_(pxy.add(_pairs(px.add_(py), 0)), alpha=3.0)
    return s.add_(_pairs(pxy, 0)).div_(30.0)


def _gradient(f, axis, c):
    d1 = torch.roll(f, -1, axis) - torch.roll(f, 1, axis)
    if c["stencil"] not in ("9cross", "13cross"):
        return d1 / 2.0
    return (8.0 * d1 - (torch.roll(f, -2, axis) - torch.roll(f, 2, axis))) / 12.0


def _fd_step(q, c):
    dt, m = _dt(c), c["model"]
    if m == "ac":
        return [q[0] + dt * (_laplacian(q[0], c) + q[0] - q[0] ** 3)]
    if m == "ch":
        mu = (q[0] ** 3).sub_(q[0]).sub_(_laplacian(q[0], c))
        return [q[0] + dt * _laplacian(mu, c)]
    if m == "gs":
        u, v = q
        r = u * v * v
        return [u + dt * (0.16 * _laplacian(u, c) - r + 0.035 * (1.0 - u)),
                v + dt * (0.08 * _laplacian(v, c) + r - (0.035 + 0.065) * v)]
    if m == "mc":
        p, r = q
        return [p + dt * (_laplacian(p, c) + p - p ** 3 + p * r), r + dt * _laplacian(r - 0.5 * p * p, c)]
    phi, j = q[0], q[1:]
    mu = (phi ** 3).sub_(phi).sub_(_laplacian(phi, c))
    axes = [phi.dim() - 1 - a for a in range(phi.dim())]  # component a of j points along axis a of (x, y, z)
    div = sum(_gradient(phi * ja, ax, c) for ja, ax in zip(j, axes))
    return [phi + dt * (_laplacian(mu, c) - 0.5 * div)] + \
        [ja + dt * (_laplacian(ja, c) - 0.5 * phi * _gradient(mu, ax, c)) for ja, ax in zip(j, axes)]


def _spectral_run(phi, c):
    dt, shape = _dt(c), phi.shape
    k2 = torch.zeros((), dtype=torch.float64, device=phi.device)
    for a, n in enumerate(shape):
        fr = torch.fft.rfftfreq if a == len(shape) - 1 else torch.fft.fftfreq
        k = 2.0 * math.pi * fr(n, dtype=torch.float64, device=phi.device)
        k2 = k2 + (k * k).reshape([-1 if b == a else 1 for b in range(len(shape))])
    denom = 1.0 - dt * (1.0 - k2 if c["model"] == "ac" else k2 * (1.0 - k2))
    weight = -1.0 if c["model"] == "ac" else -k2
    uh = torch.fft.rfftn(phi)
    for _ in range(c["steps"]):
        uh = (uh + dt * weight * torch.fft.rfftn(phi ** 3)) / denom
        phi = torch.fft.irfftn(uh, s=shape)
    return phi


def _free_energy(q, c):
    phi = q[0]
    e = (phi ** 4).mul_(0.25).sub_(0.5 * phi * phi)
    for a in range(phi.dim()):
        e.add_((torch.roll(phi, -1, a) - phi).square_(), alpha=0.5)
    if c["model"] == "mc":
        e += 0.5 * q[1] * q[1] - 0.5 * phi * phi * q[1]
    for j in q[1:] if c["model"] == "mh" else ():
        e.add_(j * j, alpha=0.5)
    return float(e.sum())


def _exact_fields(c, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    q = _initial(c, int(seed), dev)
    if c["spectral"]:
        return [_spectral_run(q[0], c)]
    for _ in range(c["steps"]):
        q = _fd_step(q, c)
    return q


def exact(case, seed):
    if case["kind"] == "serve":
        out = []
        for i, r in enumerate(_requests(case)):
            out.append({"fields": torch.stack(_exact_fields(r, seed + 1000 * i)), "steps": None})
        return out
    q = _exact_fields(case, seed)
    out = {}
    if case["monitor"]:
        out["mass"] = float(q[1 if case["model"] == "mc" else 0].sum())
        out["free_energy"] = _free_energy(q, case)
    out["fields"] = q
    return out
