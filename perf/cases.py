"""Workloads of the split-step Crank-Nicolson propagator, as a user's program runs them.

Every case is one call sequence through the public Python entry points: a state
is put on a handle, propagated, and read back together with what the paper's
programs report (norm, energy, chemical potential, rms sizes).  The handle (grid
tables, kernel shapes, captured step blocks) is made once in ``prepare`` and kept,
as a program that runs many states on one grid keeps it.
"""
import math

import numpy as np
import torch

from paper_1709_04423_gb300 import gpe

OBS = ("norm", "energy", "mu", "rms_x", "rms_y", "rms_z", "rms_r")
SIM = "grid"        # one grid: Propagator
BATCH = "batch"     # many 2d grids: Batch
ADJOINT = "adjoint"  # gradient of a final-state objective: real_time_evolution


def _grid(name, n, prec, imag, steps, dx, dt, g, geom="cartesian", nkl=(1.0, 1.4, 1.8), potential=False,
          strang=False, real=False, tune=False, every=0):
    c = {"kind": SIM, "dim": len(n), "prec": prec, "imag": imag, "steps": steps, "dt": dt, "g": g, "geom": geom,
         "potential": potential, "strang": strang, "real": real, "tune": tune, "every": every}
    for d in range(3):
        c["n%d" % d] = n[d] if d < len(n) else 1
        c["dx%d" % d] = dx[d] if d < len(n) else 1.0
        c["nu%d" % d] = nkl[d] if d < len(n) else 1.0
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # The smallest calls: the radial line of a spherical trap (513 points, FP32) advanced by a
        # short block of steps and looked at, as an interactive run or an outer fit does.
        _grid("radial_f32_short", [513], "f32", True, 100, [0.02], 1e-4, 100.0, geom="spherical"),
        # The paper's 1d imaginary-time program: a ground state on 256 points in FP64.
        _grid("line256_f64_imag", [256], "f64", True, 2000, [0.05], 1e-4, 10.0),
        # A finely resolved 1d dynamics run: a line longer than a block's segments, FP64.
        _grid("line4001_f64_real", [4001], "f64", False, 100, [0.01], 2e-4, 60.0),
        # 2d dynamics in a trap with a rough potential on an odd grid, rms(t) recorded on the way.
        _grid("plane_series_f64", [257, 201], "f64", False, 200, [0.07, 0.09], 5e-4, 40.0, potential=True, every=20),
        # The paper's largest 2d grid (its NX = NY scan ends at 1000), imaginary time, FP64.
        _grid("plane1000_f64_imag", [1000, 1000], "f64", True, 20, [0.02, 0.02], 1e-4, 80.0),
        # An axially symmetric trap (rho x z = 256 x 512), Strang splitting, FP32.
        _grid("axial_strang_f32", [256, 512], "f32", True, 100, [0.04, 0.04], 5e-4, 100.0, geom="axisym",
              nkl=(1.0, 2.0), strang=True),
        # The 3d ground-state job: 128^3, FP32, shapes tuned once, a block of 100 steps and its observables.
        _grid("cube128_f32_imag", [128, 128, 128], "f32", True, 100, [0.1, 0.1, 0.1], 1e-3, 50.0, tune=True),
        # 3d dynamics on a ragged FP64 grid.
        _grid("box_f64_real", [120, 101, 90], "f64", False, 40, [0.1, 0.12, 0.12], 5e-4, 50.0),
        # 3d ground state in the double-float form (FP64-class results).
        _grid("cube128_df64_imag", [128, 128, 128], "df64", True, 40, [0.1, 0.1, 0.1], 1e-3, 50.0),
        # The 3d quench: 256^3 real time, FP32, larger than the L2 cache, shapes tuned once.
        _grid("cube256_f32_real", [256, 256, 256], "f32", False, 60, [0.08, 0.08, 0.08], 2e-4, 40.0,
              nkl=(1.0, 1.0, 1.0), tune=True),
        # A parameter scan: 64 independent 2d runs of uneven size stepped together, launch form tuned once.
        {"name": "batch64_f32_real", "kind": BATCH, "prec": "f32", "runs": 64, "lo": 128, "hi": 512, "unit": 64,
         "steps": 100, "dt": 5e-4, "dx": 0.1},
        # Optimal control: gradient of a final overlap with respect to the state, V(r) and g.
        {"name": "adjoint96_f32", "kind": ADJOINT, "prec": "f32", "n0": 96, "n1": 96, "n2": 96, "dx": 0.13, "dt": 5e-4,
         "g": 30.0, "steps": 50, "every": 25},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["line", "line", "long line", "plane", "plane", "long plane", "axial", "box", "box", "large box",
                       "batch", "adjoint"])
    prec = rng.choice(["f64", "f32", "df64"])
    imag = rng.random() < 0.5
    g = round(rng.uniform(0.0, 100.0), 2)
    if kind == "line":
        geom = rng.choice(["cartesian", "spherical", "axisym"])
        n = _log_int(rng, 33, 514)
        return _grid(None, [n], prec, imag, _log_int(rng, 20, 2000), [round(12.0 / n, 4)], 1e-4, g, geom=geom,
                     strang=rng.random() < 0.25)
    if kind == "long line":
        n = _log_int(rng, 515, 8000)
        return _grid(None, [n], rng.choice(["f64", "f32"]), imag, rng.randint(20, max(21, 400000 // n)),
                     [round(24.0 / n, 5)], 1e-4, g, geom=rng.choice(["cartesian", "spherical"]))
    if kind == "plane":
        n = [_log_int(rng, 33, 514) for _ in range(2)]
        return _grid(None, n, prec, imag, rng.randint(20, 150), [round(16.0 / v, 4) for v in n], 5e-4, g,
                     potential=rng.random() < 0.4, strang=rng.random() < 0.25, every=rng.choice([0, 0, 10]))
    if kind == "long plane":
        n = [rng.randint(515, 1000), rng.randint(400, 1000)]
        rng.shuffle(n)
        return _grid(None, n, rng.choice(["f64", "f32"]), imag, 20, [round(20.0 / v, 5) for v in n], 1e-4, g)
    if kind == "axial":
        n = [rng.randint(64, 512), rng.randint(64, 512)]
        return _grid(None, n, prec, imag, rng.randint(20, 100), [round(10.0 / n[0], 4), round(20.0 / n[1], 4)], 5e-4, g,
                     geom="axisym", nkl=(1.0, 2.0), strang=rng.random() < 0.5)
    if kind == "box":
        n = [_log_int(rng, 32, 144) for _ in range(3)]
        real = imag and prec != "df64" and n[0] % 2 == 0 and rng.random() < 0.5
        return _grid(None, n, prec, imag, rng.randint(10, 40), [round(12.8 / v, 4) for v in n], 5e-4, g,
                     potential=rng.random() < 0.3, strang=not real and rng.random() < 0.25, real=real,
                     tune=rng.random() < 0.5)
    if kind == "large box":
        n = [16 * rng.randint(10, 16), rng.randint(150, 256), rng.randint(150, 256)]
        return _grid(None, n, "f32", imag, rng.randint(10, 50), [round(20.5 / v, 4) for v in n], 2e-4, g, tune=True)
    if kind == "batch":
        return {"kind": BATCH, "prec": prec, "runs": rng.randint(8, 64), "lo": 96, "hi": 448, "unit": rng.choice([1, 32]),
                "steps": 20 if prec != "f32" else rng.randint(20, 80), "dt": 5e-4, "dx": 0.1}
    n = [_log_int(rng, 32, 96) for _ in range(3)]
    return {"kind": ADJOINT, "prec": "f32", "n0": n[0], "n1": n[1], "n2": n[2], "dx": 0.13, "dt": 5e-4, "g": g,
            "steps": rng.randint(10, 40), "every": rng.randint(5, 25)}


# ------------------------------------------------------------------ inputs

def _lens(c):
    return [c["n%d" % d] for d in range(c.get("dim", 3))]


def _coords(n, dx, geom, axis):
    i = torch.arange(n, dtype=torch.float64, device="cuda")
    if geom == "spherical":
        return i * dx
    if geom == "axisym" and axis == 0:
        return (i - 0.5) * dx
    return -0.5 * n * dx + i * dx


def _outer(parts):
    """x fastest: the last axis of the result is axis 0."""
    out = parts[0]
    for p in parts[1:]:
        out = p.reshape(-1, *([1] * out.dim())) * out
    return out


def _state(n, dx, nkl, geom, gen, noise=1e-3):
    """A trapped condensate: a displaced, squeezed Gaussian plus seeded noise."""
    r = torch.rand(2 * len(n), generator=gen, dtype=torch.float64)
    parts = []
    for d in range(len(n)):
        x = _coords(n[d], dx[d], geom, d)
        radial = geom != "cartesian" and d == 0
        w = nkl[d] * (0.5 + 0.5 * float(r[2 * d]))
        x0 = 0.0 if radial else float(r[2 * d + 1]) - 0.5
        f = (w / math.pi) ** 0.25 * torch.exp(-0.5 * w * (x - x0) ** 2)
        parts.append(math.sqrt(4 * math.pi) * x * f if geom == "spherical" else f)
    psi = _outer(parts)
    dev = torch.Generator(device="cuda").manual_seed(int(torch.randint(1 << 31, (1,), generator=gen)))
    return torch.complex(psi + noise * torch.rand(psi.shape, generator=dev, dtype=torch.float64, device="cuda"),
                         torch.zeros_like(psi))


def _rough(n, dx, nkl, gen):
    """The trap plus a smooth random potential (eight Gaussian bumps)."""
    xs = [_coords(n[d], dx[d], "cartesian", d) for d in range(len(n))]
    shape = [[-1 if e == d else 1 for e in reversed(range(len(n)))] for d in range(len(n))]
    V = sum((0.5 * (nkl[d] * xs[d]) ** 2).reshape(shape[d]) for d in range(len(n)))
    r = torch.rand(8, 2 + len(n), generator=gen, dtype=torch.float64)
    for b in r.tolist():
        s = 0.5 + b[1]
        V = V + (b[0] - 0.5) * _outer([torch.exp(-(xs[d] - 6.0 * (b[2 + d] - 0.5)) ** 2 / (2 * s * s))
                                       for d in range(len(n))])
    return V.contiguous()


def _batch_runs(c, gen):
    """Sizes, nonlinearities and traps of a batch.  The sizes belong to the case (its seed does not move them)."""
    own = torch.Generator().manual_seed(1712 + c["runs"] + c["lo"])
    steps = (c["hi"] - c["lo"]) // c["unit"] + 1
    sizes = (c["lo"] + c["unit"] * torch.randint(steps, (c["runs"], 2 if c["unit"] == 1 else 1), generator=own)).tolist()
    r = torch.rand(c["runs"], 2, generator=gen, dtype=torch.float64).tolist()
    return [(s[0], s[-1]) for s in sizes], [50.0 * v[0] for v in r], [(1.0, 1.0 + v[1]) for v in r]


def _ctype(prec):
    return torch.complex64 if prec == "f32" else torch.complex128


def _inputs(c, seed):
    """Everything a case's pass takes: states, potential, parameters."""
    gen = torch.Generator().manual_seed(seed)
    if c["kind"] == BATCH:
        sizes, gs, nkl = _batch_runs(c, gen)
        flat = torch.cat([_state(s, [c["dx"]] * 2, k, "cartesian", gen).reshape(-1) for s, k in zip(sizes, nkl)])
        return {"sizes": sizes, "g": gs, "nkl": nkl, "psi": flat.to(_ctype(c["prec"]))}
    n = _lens(c)
    if c["kind"] == ADJOINT:
        dx, nkl = [c["dx"]] * 3, [1.0] * 3
        return {"psi": _state(n, dx, nkl, "cartesian", gen).to(_ctype(c["prec"])),
                "target": _state(n, dx, nkl, "cartesian", gen).to(_ctype(c["prec"])),
                "V": _rough(n, dx, nkl, gen).to(torch.float32),
                "g": torch.tensor(c["g"], dtype=torch.float32)}
    dx = [c["dx%d" % d] for d in range(c["dim"])]
    nkl = [c["nu%d" % d] for d in range(c["dim"])]
    return {"psi": _state(n, dx, nkl, c["geom"], gen).to(_ctype(c["prec"])).contiguous(),
            "V": _rough(n, dx, nkl, gen) if c["potential"] else None}


def prepare(case, seed):
    c = case
    s = {"case": c, **_inputs(c, seed)}
    if c["kind"] == BATCH:
        s["b"] = gpe.Batch(s["sizes"], [(c["dx"], c["dx"])] * c["runs"], c["dt"], s["nkl"], s["g"], precision=c["prec"])
        if c["prec"] == "f32":
            s["b"].set_all(s["psi"])
            s["b"].autotune(32)
        return s
    n = _lens(c)
    if c["kind"] == ADJOINT:
        s["p"] = gpe.Propagator(3, n, [c["dx"]] * 3, c["dt"], [1.0] * 3, c["g"], precision=c["prec"])
        return s
    p = gpe.Propagator(c["dim"], n, [c["dx%d" % d] for d in range(c["dim"])], c["dt"],
                       [c["nu%d" % d] for d in range(c["dim"])], c["g"], precision=c["prec"],
                       spherical=c["geom"] == "spherical", axisym=c["geom"] == "axisym")
    if s["V"] is not None:
        p.set_potential(s["V"])
    if c["strang"]:
        p.set_splitting("strang")
    if c["real"]:
        p.set_real_state(True)
    if c["tune"]:
        p.set_state(s["psi"])
        p.autotune(c["imag"], cache=False)
    s["p"] = p
    return s


# ------------------------------------------------------------------ one pass

def _reported(c, rows):
    """The reported values as one array, in the state's precision."""
    return np.array([[o[k] for k in OBS] for o in rows], dtype=np.float32 if c["prec"] == "f32" else np.float64)


def run(state):
    c = state["case"]
    if c["kind"] == BATCH:
        b = state["b"]
        b.set_all(state["psi"])
        b.step_real(c["steps"])
        obs = b.observables()
        return {"observables": _reported(c, obs), "states": [b.get_state(r, device=True) for r in range(0, c["runs"], 8)]}
    if c["kind"] == ADJOINT:
        psi = state["psi"].clone().requires_grad_(True)
        V = state["V"].clone().requires_grad_(True)
        g = state["g"].clone().requires_grad_(True)
        out = gpe.real_time_evolution(state["p"], psi, V, g, c["steps"], c["every"])
        overlap = torch.sum(torch.conj(state["target"]) * out) * c["dx"] ** 3
        J = overlap.real ** 2 + overlap.imag ** 2
        J.backward()
        return {"state": out.detach(), "J": J.detach(), "psi": psi.grad, "V": V.grad, "g": g.grad}
    p = state["p"]
    p.set_state(state["psi"])
    res = {}
    if c["every"]:
        series = p.step_series(c["imag"], c["steps"], c["every"])
        res["series"] = series.to(torch.float32) if c["prec"] == "f32" else series
    elif c["imag"]:
        p.step_imag(c["steps"])
    else:
        p.step_real(c["steps"])
    res["state"] = p.get_state()
    res["observables"] = _reported(c, [p.observables()])
    return res


def work(case):
    """Bytes: the state in and out, the potential and the gradients once.  Operations: per point and step the
    sub-step N and, per axis, one increment-form Crank-Nicolson solve (real coefficients in imaginary time)."""
    c = case
    if c["kind"] == BATCH:
        np_ = sum(a * b for a, b in _batch_runs(c, torch.Generator().manual_seed(0))[0])
        dim, imag, halves = 2, False, 1
    else:
        np_ = math.prod(_lens(c))
        dim = c.get("dim", 3)
        imag, halves = c.get("imag", False), 2 if c.get("strang") else 1
    size = 8 if c["prec"] == "f32" else 16
    per_step = dim * (16 if imag else 22) + halves * (12 if imag else 20)
    if c.get("real"):
        size, per_step = size // 2, per_step // 2
    byts = 2 * size * np_ + (8 * np_ if c.get("potential") else 0)
    if c["kind"] == ADJOINT:   # the gradients of state and V; a recomputed step and a reverse step each
        byts += (2 * size + 4 + 4) * np_
        per_step *= 3
    return {"bytes": byts, "flops": np_ * c["steps"] * per_step}


# ------------------------------------------------------------------ the same in 64 bits, from dense matrices

def _cn_matrix(n, dx, dt, imag, rho=False):
    """2 (1 + A)^-1 A with A = r T, T the (n-2)-point second difference (a rho axis: its conservative form)."""
    M = n - 2
    r = dt / (4 * dx * dx) * (1.0 if imag else 1j)
    k = torch.arange(1, M + 1, dtype=torch.float64, device="cuda")
    h = 1.0 / (2 * k - 1) if rho else torch.zeros_like(k)
    T = 2 * torch.eye(M, dtype=torch.float64, device="cuda")
    T = T - torch.diag((1 - h)[1:], -1) - torch.diag((1 + h)[:-1], 1)
    A = r * T if imag else torch.complex(torch.zeros_like(T), r.imag * T)
    return 2 * torch.linalg.solve(torch.eye(M, dtype=A.dtype, device="cuda") + A, A)


def _apply(B, u, axis):
    """u - B u along an axis (0 = x, the last dimension), the two end points zero."""
    t = u.movedim(-1 - axis, -1)
    inner = t[..., 1:-1]
    if B.is_complex():
        z = inner @ B.T
    else:
        z = torch.complex(inner.real @ B.T, inner.imag @ B.T)
    t = torch.nn.functional.pad(inner - z, (1, 1))
    return t.movedim(-1, -1 - axis)


def _weights(n, dx, geom, axis):
    if geom == "axisym" and axis == 0:
        w = 2 * math.pi * dx * _coords(n, dx, geom, axis)
        w[0] = w[-1] = 0.0
        return w
    m = n if n % 2 else n - 1
    w = torch.zeros(n, dtype=torch.float64, device="cuda")
    w[1:m - 1:2] = 4.0
    w[2:m - 1:2] = 2.0
    w[0] = w[m - 1] = 1.0
    return w * dx / 3


def _slope(u, axis, dx, geom):
    t = u.movedim(-1 - axis, -1)
    n = t.shape[-1]
    first = geom != "cartesian" and axis == 0
    if first and geom == "axisym":   # even across the axis: point 0 mirrors point 1
        t = torch.cat([t[..., 1:2], t[..., 1:]], -1)
    d = torch.zeros_like(t)
    d[..., 1] = (t[..., 2] - t[..., 0]) / (2 * dx)
    d[..., n - 2] = (t[..., n - 1] - t[..., n - 3]) / (2 * dx)
    if n > 4:
        d[..., 2:n - 2] = (t[..., :n - 4] - 8 * t[..., 1:n - 3] + 8 * t[..., 3:n - 1] - t[..., 4:]) / (12 * dx)
    if first and geom == "spherical":
        d[..., 0] = t[..., 1] / dx
    return d.movedim(-1, -1 - axis)


class _Exact:
    def __init__(self, n, dx, dt, imag, geom, V, g):
        dim = len(n)
        self.dt, self.imag, self.geom, self.V, self.dx = dt, imag, geom, V, dx
        self.B = [_cn_matrix(n[d], dx[d], dt, imag, geom == "axisym" and d == 0) for d in range(dim)]
        self.w = _outer([_weights(n[d], dx[d], geom, d) for d in range(dim)])
        self.x = [_coords(n[d], dx[d], geom, d) for d in range(dim)]
        self.g = g
        if geom == "spherical":
            r = _coords(n[0], dx[0], geom, 0)
            self.g = torch.where(r > 0, g / (4 * math.pi * r.clamp(min=dx[0]) ** 2), torch.zeros_like(r))

    def phase(self, u, dt):
        th = dt * (self.V + self.g * (u.real ** 2 + u.imag ** 2))
        return u * (torch.exp(-th) if self.imag else torch.polar(torch.ones_like(th), -th))

    def norm(self, u):
        return (self.w * (u.real ** 2 + u.imag ** 2)).sum((-1,) if u.dim() == 1 else tuple(range(-len(self.B), 0)))

    def step(self, u, strang=False):
        u = self.phase(u, 0.5 * self.dt if strang else self.dt)
        for d, B in enumerate(self.B):
            u = _apply(B, u, d)
        if strang:
            u = self.phase(u, 0.5 * self.dt)
        return u / torch.sqrt(self.norm(u)) if self.imag else u

    def observables(self, u):
        dim = len(self.B)
        dens = u.real ** 2 + u.imag ** 2
        N = float((self.w * dens).sum())
        kin = sum(float((self.w * (s.real ** 2 + s.imag ** 2)).sum()) / 2
                  for s in (_slope(u, d, self.dx[d], self.geom) for d in range(dim)))
        pot = float((self.w * dens * self.V).sum())
        four = float((self.w * dens * dens * self.g).sum())
        r2 = [float((self.w * dens * self.x[d].reshape([-1] + [1] * d) ** 2).sum()) / N for d in range(dim)]
        r2 += [0.0] * (3 - dim)
        return [N, (kin + pot) / N + 0.5 * four / N ** 2, (kin + pot) / N + four / N ** 2,
                *(math.sqrt(v) for v in r2), math.sqrt(sum(r2))]


def _trap(n, dx, nkl, geom):
    xs = [_coords(n[d], dx[d], geom, d) for d in range(len(n))]
    shape = [[-1 if e == d else 1 for e in reversed(range(len(n)))] for d in range(len(n))]
    return sum((0.5 * (nkl[d] * xs[d]) ** 2).reshape(shape[d]) for d in range(len(n)))


def exact(case, seed):
    c = case
    s = _inputs(c, seed)
    if c["kind"] == BATCH:
        return _exact_batch(c, s)
    n = _lens(c)
    if c["kind"] == ADJOINT:
        psi = s["psi"].to(torch.complex128).requires_grad_(True)
        V = s["V"].double().requires_grad_(True)
        g = s["g"].double().cuda().requires_grad_(True)
        E = _Exact(n, [c["dx"]] * 3, c["dt"], False, "cartesian", V, g)
        u = psi
        for _ in range(c["steps"]):
            u = E.step(u)
        overlap = torch.sum(torch.conj(s["target"].to(torch.complex128)) * u) * c["dx"] ** 3
        J = overlap.real ** 2 + overlap.imag ** 2
        J.backward()
        return {"state": u.detach(), "J": J.detach(), "psi": psi.grad, "V": V.grad, "g": g.grad}
    dx = [c["dx%d" % d] for d in range(c["dim"])]
    nkl = [c["nu%d" % d] for d in range(c["dim"])]
    V = s["V"] if s["V"] is not None else _trap(n, dx, nkl, c["geom"])
    E = _Exact(n, dx, c["dt"], c["imag"], c["geom"], V, c["g"])
    u = s["psi"].to(torch.complex128)
    res, series = {}, []
    for t in range(c["steps"]):
        u = E.step(u, c["strang"])
        if c["every"] and (t + 1) % c["every"] == 0:
            series.append(E.observables(u))
    if c["every"]:
        res["series"] = torch.tensor(series, dtype=torch.float64).reshape(-1, 7)
    res["state"] = u
    res["observables"] = np.array([E.observables(u)], dtype=np.float64)
    return res


def _exact_batch(c, s):
    """The runs of one size together: they share the matrices."""
    off, groups = 0, {}
    for r, size in enumerate(s["sizes"]):
        groups.setdefault(size, []).append((r, off))
        off += size[0] * size[1]
    obs, states = [None] * c["runs"], [None] * c["runs"]
    for size, members in groups.items():
        nx, ny = size
        dx = [c["dx"]] * 2
        u = torch.stack([s["psi"][o:o + nx * ny].reshape(ny, nx) for _, o in members]).to(torch.complex128)
        V = torch.stack([_trap(size, dx, s["nkl"][r], "cartesian") for r, _ in members])
        g = torch.tensor([s["g"][r] for r, _ in members], dtype=torch.float64, device="cuda").reshape(-1, 1, 1)
        E = _Exact(list(size), dx, c["dt"], False, "cartesian", V, g)
        for _ in range(c["steps"]):
            u = E.step(u)
        for i, (r, _) in enumerate(members):
            E.V, E.g = V[i], g[i]
            obs[r], states[r] = E.observables(u[i]), u[i]
    return {"observables": np.array(obs, dtype=np.float64), "states": states[::8]}
