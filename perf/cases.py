"""The work that users of this package have it do, as cases that can be timed and checked.

Four kinds of pass, each through the public binding (paper_1607_01105_gb300.ppml):
* "grid": K timesteps of a uniform grid (1D, 2D or 3D; float, double-float or double
  states): the first with a given step size, the rest with the device-resident CFL step, as
  a run loop that never waits for the host;
* "disk": one self-gravitating step: the periodic Poisson solve, the fixed halo potential
  added to it, the step with gravity;
* "batch": K steps of many independent 1D problems of uneven lengths in one launch;
* "iso": one isolated-boundary Poisson solve.

exact() is the same scheme written with plain torch operations in 64 bits.
"""
import math

import numpy as np
import torch

from paper_1607_01105_gb300 import ppml

DEV = "cuda"
F64 = torch.float64
BC = {"o": ppml.OUTFLOW, "p": ppml.PERIODIC, "r": ppml.REFLECT}


# ----------------------------------------------------------------------------- the cases

def _grid(name, n, prec, shape, bc="oooooo", steps=2, diag=False):
    return {"name": name, "kind": "grid", "nx": n[0], "ny": n[1], "nz": n[2], "prec": prec,
            "shape": shape, "bc": bc, "steps": steps, "diag": diag}


def listed():
    return [
        # the plain FP64 method on the 256-cell Sod tube: the smallest grid anyone runs, bound
        # by launches and latency; its loop reads the diagnostics every few steps
        _grid("sod_256_f64", (256, 1, 1), "f64", "tube", steps=8, diag=True),
        # a 2D shear-layer run (nz = 1), the size class of the paper's 2D experiments
        _grid("shear_256x256_f32", (256, 256, 1), "f32", "smooth", bc="ppppoo", steps=4),
        # an odd box with reflecting walls: ragged tiles on every axis, mirrored halos
        _grid("walls_97x83x61_f32", (97, 83, 61), "f32", "smooth", bc="rrppor", steps=4),
        # the planar 128^3 shock tube, periodic across
        _grid("planar_128_f32", (128, 128, 128), "f32", "tube", bc="oopppp"),
        # the point blast on a double-float state (totals held as float pairs)
        _grid("blast_128_ff", (128, 128, 128), "ff", "blast"),
        # the 256^3 point blast, the package's headline run, in FP32 ...
        _grid("blast_256_f32", (256, 256, 256), "f32", "blast"),
        # ... and in FP64
        _grid("blast_256_f64", (256, 256, 256), "f64", "blast", steps=1),
        # the galactic disk: a 512^3 step with self-gravity, the largest run
        {"name": "disk_512_f32", "kind": "disk", "nx": 512, "ny": 512, "nz": 512, "prec": "f32"},
        # one 1D problem through the batch path: the lowest-latency way to run a tube
        {"name": "batch_1x256_f32", "kind": "batch", "inst": 1, "nmin": 256, "nmax": 256,
         "prec": "f32", "steps": 128},
        # the 512 Riemann problems of 128 to 4096 cells, between two snapshots
        {"name": "batch_512_f32", "kind": "batch", "inst": 512, "nmin": 128, "nmax": 4096,
         "prec": "f32", "steps": 128},
        # the same kind of batch in FP64
        {"name": "batch_192_f64", "kind": "batch", "inst": 192, "nmin": 128, "nmax": 2048,
         "prec": "f64", "steps": 16},
        # isolated-boundary self-gravity of a compact blob
        {"name": "iso_128_f32", "kind": "iso", "nx": 128, "ny": 128, "nz": 128, "prec": "f32"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["grid1", "grid2", "grid3", "grid3", "grid3", "disk", "batch", "batch", "iso"])
    prec = rng.choice(["f32", "f32", "f64", "ff"])
    if kind == "grid1":
        c = _grid("", (_log(rng, 64, 4096), 1, 1), prec, rng.choice(["tube", "smooth"]),
                  bc=rng.choice(["oooooo", "rroooo", "ppoooo"]), steps=8, diag=rng.random() < 0.5)
    elif kind == "grid2":
        c = _grid("", (_log(rng, 32, 700), _log(rng, 32, 700), 1), prec, "smooth",
                  bc=rng.choice(["ppppoo", "oooooo", "rrppoo", "orrooo"]), steps=4)
    elif kind == "grid3":
        top = 160 if prec == "f64" else 300
        n = [_log(rng, 20, top) for _ in range(3)]
        if rng.random() < 0.5:
            n = [n[0]] * 3
        c = _grid("", n, prec, rng.choice(["smooth", "blast", "tube"]),
                  bc=rng.choice(["oooooo", "oopppp", "pppppp", "rrppor", "rrrrrr"]), steps=2)
    elif kind == "disk":
        n = 2 * _log(rng, 16, 160)
        c = {"kind": "disk", "nx": n, "ny": n, "nz": n, "prec": "f64" if prec == "f64" and n <= 160 else "f32"}
    elif kind == "batch":
        lo = _log(rng, 64, 1024)
        prec = "f32" if prec == "ff" and rng.random() < 0.5 else prec
        c = {"kind": "batch", "inst": _log(rng, 1, 160 if prec == "f64" else 640), "nmin": lo,
             "nmax": min(4 * lo, 2048 if prec == "f64" else 4096), "prec": prec,
             "steps": 16 if prec == "f64" else rng.choice([32, 96, 160])}
    else:
        n = [_log(rng, 40, 200) for _ in range(3)]
        c = {"kind": "iso", "nx": n[0], "ny": n[1], "nz": n[2], "prec": "f64" if prec == "f64" else "f32"}
    c.pop("name", None)
    return c


# ---------------------------------------------------------------------------- the inputs

def _uni(g, lo, hi, n=None):
    x = torch.rand(n or 1, generator=g, dtype=F64, device="cpu") * (hi - lo) + lo
    return x.tolist() if n else float(x)


def _axes(c, lo):
    n = (c["nx"], c["ny"], c["nz"])
    h = 1.0 / max(n)
    x = [(torch.arange(m, dtype=F64, device=DEV) + 0.5 - 0.5 * m * (lo != 0)) * h for m in n]
    return n, h, x[0].view(1, 1, -1), x[1].view(1, -1, 1), x[2].view(-1, 1, 1)


def _conserved(rho, v, p, gamma, shape):
    rho, p = rho.expand(shape), p.expand(shape)
    v = [torch.as_tensor(a, dtype=F64, device=DEV).expand(shape) for a in v]
    ei = p / (gamma - 1.0)
    en = ei + 0.5 * rho * (v[0] * v[0] + v[1] * v[1] + v[2] * v[2])
    return [a.contiguous() for a in (rho, rho * v[0], rho * v[1], rho * v[2], en, ei)]


def _tube(c, g):
    """A shock tube part-way through its run, uniform across: rarefaction, contact and shock."""
    n, h, x, _, _ = _axes(c, 0)
    xs, t, k = _uni(g, 0.45, 0.55), _uni(g, 0.08, 0.15), _uni(g, 0.9, 1.1)
    s = (x / (n[0] * h) - xs) / t  # similarity coordinate; Sod's states, scaled in density
    ramp = ((s + 1.183) / (1.183 - 0.07)).clamp(0.0, 1.0)
    rho = torch.where(s < 0.93, 1.0 + ramp * (0.426 - 1.0), torch.where(s < 1.752, 0.2656, 0.125) + 0 * s)
    p = torch.where(s < 1.752, 1.0 + ramp * (0.303 - 1.0), 0.1 + 0 * s)
    v = torch.where(s < 1.752, 0.927 * ramp, 0 * s)
    return _conserved(k * rho, (v, 0.0, 0.0), k * p, 1.4, (n[2], n[1], n[0])), 1.4, h


def _blast(c, g):
    """A point blast part-way through its run: a thin shell, a hot centre, cold gas ahead."""
    n, h, x, y, z = _axes(c, -0.5)
    gamma, R = 5.0 / 3.0, _uni(g, 0.25, 0.38) * min(n) / max(n)
    cx = _uni(g, -1.0, 1.0, 3)
    x, y, z = x - cx[0] * h, y - cx[1] * h, z - cx[2] * h
    r = torch.sqrt(x * x + y * y + z * z)
    xi = (r / R).clamp(max=1.0)
    speed = 0.4 * R / math.sqrt((R / 1.15) ** 5)
    wob = 1.0 + 0.02 * torch.sin(9.0 * x + 7.0 * y + 5.0 * z + _uni(g, 0.0, 6.0))
    inside = r < R
    rho = torch.where(inside, (4.0 * xi ** 4.5 + 0.02) * wob, 1.0 + 0 * r)
    p = torch.where(inside, 0.75 * speed ** 2 * (0.31 + 0.69 * xi ** 8) * wob, 1e-5 + 0 * r)
    vr = torch.where(inside, 0.75 * speed * xi, 0 * r) / r.clamp(min=1e-12)
    return _conserved(rho, (vr * x, vr * y, vr * z), p, gamma, (n[2], n[1], n[0])), gamma, h


def _smooth(c, g):
    """Waves in every field and a sheared interface."""
    n, h, x, y, z = _axes(c, 0)
    tw = 2.0 * math.pi

    def waves(base, amp):
        f = torch.full((n[2], n[1], n[0]), base, dtype=F64, device=DEV)
        for _ in range(3):
            k = [round(q) for q in _uni(g, -2.4, 2.4, 3)]
            ph, a = _uni(g, 0.0, tw), amp * _uni(g, -1.0, 1.0) / 3.0
            f += a * torch.sin(tw * (k[0] * x / (n[0] * h) + k[1] * y / (n[1] * h) * (n[1] > 1)
                                     + k[2] * z / (n[2] * h) * (n[2] > 1)) + ph)
        return f

    lower = (y / (n[1] * h) < 0.5) if n[1] > 1 else (x / (n[0] * h) < 0.5)
    rho = waves(1.0, 0.3) * torch.where(lower, 1.0, 2.0)
    v = [waves(0.0, 0.5) for _ in range(3)]
    for a in range(3):
        if n[a] == 1:
            v[a] = 0 * v[a]
    v[0] = v[0] + torch.where(lower, 0.5, -0.5)
    return _conserved(rho, v, waves(2.0, 0.3), 1.4, (n[2], n[1], n[0])), 1.4, h


def _disk(c, g):
    """An exponential, sech^2-thin gas disk in a fixed halo, 1 % density noise, G = 1."""
    n, h, x, y, z = _axes(c, -0.5)
    gamma, r0, rd, z0 = 5.0 / 3.0, 0.05, 0.125, 2.0 * h
    R = torch.sqrt(x * x + y * y)

    def vc2(q):  # halo circular speed squared / (4 pi rho0 r0^2)
        return 1.0 - torch.atan(q / r0) / (q / r0)

    amp = 1.0 / float(vc2(torch.tensor(rd, dtype=F64)))
    q = torch.sqrt(R * R + z * z) / r0
    phi = amp * (0.5 * torch.log1p(q * q) + torch.atan(q) / q)
    cs = _uni(g, 0.45, 0.55)
    rho = torch.exp(-R / rd) / (2.0 * z0) / torch.cosh(z / z0) ** 2
    low = 1e-6 * float(rho.max())
    inside = rho > low
    p = rho.clamp(min=low) * cs * cs / gamma
    vp = torch.sqrt((amp * vc2(R) - cs * cs / gamma * R / rd).clamp(min=0.0)) * inside
    noise = torch.randn(rho.shape, generator=torch.Generator(device=DEV).manual_seed(int(_uni(g, 0, 2 ** 31))),
                        device=DEV, dtype=torch.float32)
    rho = (rho * (1.0 + 0.01 * noise * inside)).clamp(min=low)
    return _conserved(rho, (-vp * y / R, vp * x / R, 0.0), p, gamma, rho.shape), gamma, h, phi


def _batch(c, g):
    """Riemann problems of even lengths in [nmin, nmax] (the same for every seed), each with
    a little structure.  Draws within two fifths of a vacuum, or whose kinetic energy is over
    three times the internal (there float rounding decides the internal energy), are redrawn."""
    I, gamma = c["inst"], 1.4
    n = [2 * (int(q) // 2) for q in _uni(_gen(1607), c["nmin"], c["nmax"] + 1.999, I + 1)[:I]]
    rows = []
    for _ in range(I):
        while True:
            r, p, u = _uni(g, 0.1, 10.0, 2), [10.0 ** q for q in _uni(g, -2.0, 2.0, 2)], _uni(g, -2.0, 2.0, 2)
            if (u[1] - u[0] < 2.0 * sum(math.sqrt(gamma * a / b) for a, b in zip(p, r))
                    and all(0.5 * a * b * b < 3.0 * q / (gamma - 1.0) for a, b, q in zip(r, u, p))):
                break
        rows.append(r + p + u + _uni(g, 0.0, 6.28, 1))
    s = torch.tensor(rows, dtype=F64, device=DEV)
    nt = torch.tensor(n, device=DEV)
    inst = torch.repeat_interleave(torch.arange(I, device=DEV), nt)
    off = torch.cumsum(nt, 0) - nt
    x = (torch.arange(int(nt.sum()), device=DEV) - off[inst] + 0.5) / nt[inst]
    left, s = x < 0.5, s[inst]
    wave = 1.0 + 0.05 * torch.sin(25.0 * x + s[:, 6])
    rho, p, u = torch.where(left, s[:, 0], s[:, 1]) * wave, torch.where(left, s[:, 2], s[:, 3]), torch.where(left, s[:, 4], s[:, 5])
    ei = p / (gamma - 1.0)
    return n, [rho, rho * u, ei + 0.5 * rho * u * u, ei], gamma


def _blob(c, g):
    n, h, x, y, z = _axes(c, -0.5)
    a = _uni(g, 0.6, 1.4, 3)
    o = [q * h for q in _uni(g, -3.0, 3.0, 3)]
    R = 0.35 * min(n) * h
    r = torch.sqrt(((x - o[0]) / a[0]) ** 2 + ((y - o[1]) / a[1]) ** 2 + ((z - o[2]) / a[2]) ** 2) / R
    return torch.where(r < 1.0, 2.0 * r ** 3 - 3.0 * r ** 2 + 1.0, 0 * r) * (1.0 + 0.1 * torch.sin(20.0 * x + 15.0 * y)), h


def _gen(seed):
    return torch.Generator(device="cpu").manual_seed(int(seed))


def _inputs(c, seed):
    """(fields in 64 bits, gamma, h) of a grid case, with phi for the disk."""
    g = _gen(seed)
    return _disk(c, g) if c["kind"] == "disk" else {"tube": _tube, "blast": _blast, "smooth": _smooth}[c["shape"]](c, g)


def _stored(u, prec):
    """The values that a state of this precision holds: a list of tensors, hi then lo."""
    if prec == "f64":
        return list(u)
    hi = [a.float() for a in u]
    return hi if prec == "f32" else hi + [(a - b.double()).float() for a, b in zip(u[:-1], hi[:-1])]


def _held(t, nf):
    """What _stored holds, in 64 bits."""
    return [t[f].double() + (t[nf + f].double() if len(t) > nf and f < len(t) - nf else 0.0) for f in range(nf)]


def _code(prec):
    return ppml.PPML_F64 if prec == "f64" else ppml.PPML_F32


def _cfl(c):
    return 0.4 if c["ny"] == 1 else 0.2


def _first_dt(u, gamma, h, cfl):
    v = torch.sqrt(u[1] ** 2 + u[2] ** 2 + u[3] ** 2) / u[0]
    return cfl * h / float(v.max() + torch.sqrt(gamma * (gamma - 1.0) * u[5] / u[0]).max())


# ------------------------------------------------------------------------- one pass of each

def prepare(case, seed):
    c = case
    prec = c["prec"]
    if c["kind"] == "batch":
        n, u, gamma = _batch(c, _gen(seed))
        t = _stored(u, prec)
        # an end time that is never reached: a pass can be repeated on one handle
        b = ppml.Batch(n, [1.0 / q for q in n], [1e9] * len(n), gamma, 0.4, _code(prec))
        return {"c": c, "b": b, "u": t, "w": [torch.empty_like(a) for a in t]}
    if c["kind"] == "iso":
        rho, h = _blob(c, _gen(seed))
        rho = _stored([rho], prec)[0].reshape(-1).contiguous()
        u = [torch.ones_like(rho) for _ in range(6)]
        grid = ppml.Grid((c["nx"], c["ny"], c["nz"]), (h,) * 3, 5.0 / 3.0, 0.2, dtype=_code(prec), u0=u)
        return {"c": c, "g": grid, "rho": rho, "phi": torch.empty_like(rho)}
    u, gamma, h, *phi = _inputs(c, seed)
    dt = _first_dt(u, gamma, h, _cfl(c))
    t = [a.reshape(-1).contiguous() for a in _stored(u, prec)]
    del u
    bc = tuple(BC[q] for q in c.get("bc", "oooooo"))
    grid = ppml.Grid((c["nx"], c["ny"], c["nz"]), (h,) * 3, gamma, _cfl(c), bc, _code(prec), u0=t)
    s = {"c": c, "g": grid, "dt": dt, "u": t, "a": [torch.empty_like(q) for q in t]}
    if phi:
        s["halo"] = _stored(phi, prec)[0].reshape(-1).contiguous()
        s["phi"] = torch.empty_like(s["halo"])
    elif c["steps"] > 1:
        s["b"] = [torch.empty_like(q) for q in t]
    return s


def run(state):
    s, c = state, state["c"]
    if c["kind"] == "batch":
        for w, u in zip(s["w"], s["u"]):
            w.copy_(u)
        s["b"].step(s["w"][:4], c["steps"], lo=s["w"][4:] or None)
        return s["w"]
    if c["kind"] == "iso":
        s["g"].poisson_isolated(s["rho"], s["phi"], 1.0)
        return s["phi"]
    if c["kind"] == "disk":
        s["g"].poisson_periodic(s["u"][0], s["phi"], 1.0)
        s["phi"].add_(s["halo"])
        s["g"].step_phi(s["u"], s["a"], s["phi"], s["dt"])
        return s["a"]
    s["g"].step(s["u"], s["a"], s["dt"])
    src, dst = s["a"], s.get("b")
    for _ in range(c["steps"] - 1):
        s["g"].step(src, dst)
        src, dst = dst, src
    if c["diag"]:
        d = s["g"].diag()
        return {"u": src, "diag": [d["dt_next"], d["vmax"], d["cmax"]] + d["sums"], "n": [d["n_vacuum"], d["n_bad"]]}
    return src


def work(case):
    """Fields read and written once per pass; additions and multiplications of the scheme
    (18 line updates of a field, the template, the face solves, the energy correction)."""
    c = case
    e = {"f32": 4, "ff": 4, "f64": 8}[c["prec"]]
    if c["kind"] == "batch":
        cells = c["inst"] * (c["nmin"] + c["nmax"]) / 2.0
        return {"bytes": cells * 2 * e * (7 if c["prec"] == "ff" else 4), "flops": cells * c["steps"] * 250.0}
    cells = float(c["nx"] * c["ny"] * c["nz"])
    if c["kind"] == "iso":  # six sine transforms of 5 N log2 N / 2 operations
        return {"bytes": 2 * e * cells, "flops": 15.0 * cells * math.log2(cells)}
    axes = sum(c[q] > 1 for q in ("nx", "ny", "nz"))
    per = 45.0 + axes * 250.0
    if c["kind"] == "disk":
        return {"bytes": cells * 4 * 14, "flops": cells * (per + 20.0 + 5.0 * math.log2(cells))}
    return {"bytes": cells * e * 2 * (11 if c["prec"] == "ff" else 6), "flops": cells * per * c["steps"]}


# ---------------------------------------------------- the scheme in plain 64-bit torch

def _cut(q, d, lo, n):
    return q.narrow(d, lo, n)


def _parabolas(q, d):
    """(q_L, q_R, D, q6) of the cells 2 .. L-3 along dimension d."""
    L = q.shape[d]
    r = _cut(q, d, 1, L - 1) - _cut(q, d, 0, L - 1)
    a, b = _cut(r, d, 0, L - 2), _cut(r, d, 1, L - 2)
    dq = 0.5 * (_cut(q, d, 2, L - 2) - _cut(q, d, 0, L - 2))
    m = torch.minimum(dq.abs(), 2.0 * torch.minimum(a.abs(), b.abs()))
    s = torch.where(a * b > 0, torch.copysign(m, dq), 0.0)  # cells 1 .. L-2
    f = 0.5 * (_cut(q, d, 1, L - 3) + _cut(q, d, 2, L - 3)) - (_cut(s, d, 1, L - 3) - _cut(s, d, 0, L - 3)) / 6.0
    q0, l, r = _cut(q, d, 2, L - 4), _cut(f, d, 0, L - 4), _cut(f, d, 1, L - 4)
    D, S = r - l, 6.0 * (q0 - 0.5 * (l + r))
    flat = (l - q0) * (q0 - r) <= 0
    nl = torch.where(flat, q0, torch.where(D * S > D * D, 3.0 * q0 - 2.0 * r, l))
    nr = torch.where(flat, q0, torch.where(D * S < -(D * D), 3.0 * q0 - 2.0 * l, r))
    return nl, nr, nr - nl, 6.0 * (q0 - 0.5 * (nl + nr))


def _sides(P, y, d):
    """Characteristic averages at the faces: of the left cell and of the right cell."""
    n = P[0].shape[d] - 1
    L, R, D, S = P
    w = 1.0 - 2.0 * y / 3.0
    left = _cut(R, d, 0, n) - 0.5 * y * (_cut(D, d, 0, n) - _cut(S, d, 0, n) * w)
    right = _cut(L, d, 1, n) + 0.5 * y * (_cut(D, d, 1, n) + _cut(S, d, 1, n) * w)
    return left, right


def _diff(q, d):
    n = q.shape[d] - 1
    return _cut(q, d, 1, n) - _cut(q, d, 0, n)


def _face_solve(v, p, rho, gamma, th, d):
    """(V, P) at the faces 0 .. n from values at the cells -3 .. n+2."""
    n = v.shape[d] - 6
    rl, rr, pl, pr = _cut(rho, d, 2, n + 1), _cut(rho, d, 3, n + 1), _cut(p, d, 2, n + 1), _cut(p, d, 3, n + 1)
    sl, sr = rl.sqrt(), rr.sqrt()
    A, B = rl * sl + rr * sr, pl * sl + pr * sr
    lam, Z = (gamma * B / A).sqrt(), (gamma * A * B).sqrt() / (sl + sr)
    y = lam * th
    vl, vr = _sides(_parabolas(v, d), y, d)
    ql, qr = _sides(_parabolas(p, d), y, d)
    return 0.5 * (vl + vr) + (ql - qr) / (2.0 * Z), 0.5 * (ql + qr) + 0.5 * Z * (vl - vr)


def _flux(q, vh, th, d):
    left, right = _sides(_parabolas(q, d), vh.abs() * th, d)
    return vh * torch.where(vh >= 0, left, right)


def _correct(u, rho_vac):
    """Energy consistency; u = rho, m components, rho E, rho eps."""
    rho, m, en, ei = u[0], u[1:-2], u[-2], u[-1]
    m2 = sum(a * a for a in m)
    vac = (rho < rho_vac) & (m2 > 0)
    e = en - m2 / (2.0 * rho)
    de = en - ei
    s = torch.where(vac, torch.where(de < 0, 0.0, (2.0 * de.clamp(min=0.0) * rho / m2.clamp(min=1e-300)).sqrt()), 1.0)
    ei = torch.where(vac, torch.where(de < 0, en, ei), torch.where(e > 0, e, ei))
    return [rho] + [a * s for a in m] + [en, ei]


def _pad(q, n, bc, comp=None, dims=(0, 1, 2)):
    """Three ghost cells on the active axes in dims; comp: the momentum component q is."""
    for a in dims:
        if n[a] == 1:
            continue
        d = 2 - a
        i = np.arange(-3, n[a] + 3)
        j, sign = i.copy(), np.ones(n[a] + 6)
        for side, out in ((0, i < 0), (1, i >= n[a])):
            b = bc[2 * a + side]
            if b == "p":
                j[out] = i[out] % n[a]
            elif b == "r":
                j[out] = -1 - i[out] if side == 0 else 2 * n[a] - 1 - i[out]
                if comp == a:
                    sign[out] = -1.0
            else:
                j[out] = np.clip(i[out], 0, n[a] - 1)
        q = q.index_select(d, torch.as_tensor(j, device=DEV))
        if (sign < 0).any():
            shape = [1, 1, 1]
            shape[d] = -1
            q = q * torch.as_tensor(sign, device=DEV).view(shape)
    return q


def _inner(q, n, dims):
    for a in dims:
        if n[a] > 1:
            q = _cut(q, 2 - a, 3, n[a])
    return q


def _grid_step(u, n, bc, gamma, h, dt, rho_vac, phi=None):
    th = dt / h
    act = [a for a in range(3) if n[a] > 1]
    star = list(u)
    for a in act:  # Eulerian stage
        d = 2 - a
        rho = _pad(u[0], n, bc, None, (a,))
        V, P = _face_solve(_pad(u[1 + a], n, bc, a, (a,)) / rho, (gamma - 1.0) * _pad(u[5], n, bc, None, (a,)), rho, gamma, th, d)
        del rho
        star[1 + a] = star[1 + a] - th * _diff(P, d)
        star[4] = star[4] - th * _diff(P * V, d)
        star[5] = star[5] - (gamma - 1.0) * u[5] * th * _diff(V, d)
        del V, P
        if phi is not None:
            f = _pad(phi, n, "oooooo", None, (a,))
            grad = (_cut(f, d, 4, n[a]) - _cut(f, d, 2, n[a])) / (2.0 * h)
            star[1 + a] = star[1 + a] - dt * u[0] * grad
            star[4] = star[4] - dt * u[1 + a] * grad
            del f, grad
    out = list(star)
    rho = _pad(star[0], n, bc)
    for a in act:  # Lagrangian stage
        d = 2 - a
        v = _pad(star[1 + a], n, bc, a) / rho
        for t in act:
            if t != a:  # (1/4, 1/2, 1/4) across each other axis: the 9-point template
                L = v.shape[2 - t]
                v = 0.25 * _cut(v, 2 - t, 2, L - 6) + 0.5 * _cut(v, 2 - t, 3, L - 6) + 0.25 * _cut(v, 2 - t, 4, L - 6)
        s = _inner(rho, n, [t for t in act if t != a]).sqrt()
        v, s = _cut(v, d, 2, n[a] + 2), _cut(s, d, 2, n[a] + 2)
        m = n[a] + 1
        vh = (_cut(v * s, d, 0, m) + _cut(v * s, d, 1, m)) / (_cut(s, d, 0, m) + _cut(s, d, 1, m))
        del v, s
        for f in range(6):
            q = _pad(star[f], n, bc, f - 1 if 1 <= f <= 3 else None, (a,))
            out[f] = out[f] - th * _diff(_flux(q, vh, th, d), d)
    return _correct(out, rho_vac)


def _exact_grid(c, seed):
    u, gamma, h, *phi = _inputs(c, seed)
    dt = _first_dt(u, gamma, h, _cfl(c))
    u = _held(_stored(u, c["prec"]), 6)
    n, bc = (c["nx"], c["ny"], c["nz"]), c.get("bc", "oooooo")
    rho_vac = 1e-5 * float(u[0].mean())
    if phi:
        halo = _held(_stored(phi, c["prec"]), 1)[0]
        k = [torch.sin(math.pi * torch.arange(m, dtype=F64, device=DEV) / m) ** 2 for m in n]
        sym = [1.0 - (2.0 / 3.0) * q for q in k]
        den = 1.0 - sym[2].view(-1, 1, 1) * sym[1].view(1, -1, 1) * sym[0][: n[0] // 2 + 1].view(1, 1, -1)
        den[0, 0, 0] = 1.0
        spec = torch.fft.rfftn(u[0]) * (-(2.0 / 3.0) * math.pi * h * h) / den
        spec[0, 0, 0] = 0.0
        phi = torch.fft.irfftn(spec, s=(n[2], n[1], n[0])) + halo
        del spec, den, halo
        u = _grid_step(u, n, bc, gamma, h, dt, rho_vac, phi)
        return _laid_out(u, c)
    for k in range(c["steps"]):
        u = _grid_step(u, n, bc, gamma, h, dt, rho_vac)
        dt = _first_dt(u, gamma, h, _cfl(c))
    fields = _laid_out(u, c)
    if c["diag"]:
        v = torch.sqrt(u[1] ** 2 + u[2] ** 2 + u[3] ** 2) / u[0]
        cs = torch.sqrt(gamma * (gamma - 1.0) * u[5] / u[0])
        return {"u": fields, "diag": [dt, float(v.max()), float(cs.max())] + [float(q.sum()) * h ** 3 for q in u], "n": [None, None]}
    return fields


def _laid_out(u, c):
    """The fields as run() returns them; a double-float state's high parts are the values."""
    return [q.reshape(-1) for q in u] + [None] * (len(u) - 1 if c["prec"] == "ff" else 0)


def _exact_batch(c, seed):
    n, u, gamma = _batch(c, _gen(seed))
    t = _stored(u, c["prec"])
    u = _held(t, 4)
    I, top = len(n), max(n)
    nt = torch.tensor(n, device=DEV)
    off = (torch.cumsum(nt, 0) - nt).view(-1, 1)
    last = (nt - 1).view(-1, 1)
    at = torch.arange(-3, top + 3, device=DEV).view(1, -1)
    at = torch.minimum(at.clamp(min=0), last)  # outflow ghosts: the instance's end cells
    u = [q[off + at] for q in u]
    h = 1.0 / nt.double().view(-1, 1)
    own = torch.arange(top, device=DEV).view(1, -1) <= last
    rho_vac = 1e-5 * ((u[0][:, 3:-3] * own).sum(1, keepdim=True) / nt.view(-1, 1))

    def fill(q):  # cells 0 .. top-1 -> with ghosts
        return q.gather(1, at)

    for _ in range(c["steps"]):
        v = u[1] / u[0]
        cs = (gamma * (gamma - 1.0) * u[3] / u[0]).sqrt()
        th = 0.4 / (v.abs().amax(1, keepdim=True) + cs.amax(1, keepdim=True))
        V, P = _face_solve(v, (gamma - 1.0) * u[3], u[0], gamma, th, 1)
        mid = [q[:, 3:-3] for q in u]
        star = [mid[0], mid[1] - th * _diff(P, 1), mid[2] - th * _diff(P * V, 1),
                mid[3] - (gamma - 1.0) * mid[3] * th * _diff(V, 1)]
        u = [fill(q) for q in star]
        v, s = (u[1] / u[0])[:, 2:-2], u[0].sqrt()[:, 2:-2]
        vh = (v[:, :-1] * s[:, :-1] + v[:, 1:] * s[:, 1:]) / (s[:, :-1] + s[:, 1:])
        star = _correct([q[:, 3:-3] - th * _diff(_flux(q, vh, th, 1), 1) for q in u], rho_vac)
        u = [fill(q) for q in star]
    got = [q[:, 3:-3][own] for q in u]
    return got + [None] * (3 if c["prec"] == "ff" else 0)


def _exact_iso(c, seed):
    rho, h = _blob(c, _gen(seed))
    rho = _held(_stored([rho], c["prec"]), 1)[0]
    n = (c["nx"], c["ny"], c["nz"])
    x = [(torch.arange(-1, m + 1, dtype=F64, device=DEV) + 0.5 - 0.5 * m) * h for m in n]
    X, Y, Z = x[0].view(1, 1, -1), x[1].view(1, -1, 1), x[2].view(-1, 1, 1)
    i = (slice(1, -1),) * 3
    x1, y1, z1 = X[:, :, 1:-1], Y[:, 1:-1], Z[1:-1]
    m = rho * h ** 3
    M, Ix, Iy, Iz = m.sum(), ((z1 * z1 + y1 * y1) * m).sum(), ((x1 * x1 + z1 * z1) * m).sum(), ((x1 * x1 + y1 * y1) * m).sum()
    Ixy, Ixz, Iyz = (x1 * y1 * m).sum(), (x1 * z1 * m).sum(), (y1 * z1 * m).sum()
    r2 = X * X + Y * Y + Z * Z
    r = r2.sqrt()
    I0 = (X * X * Ix + Y * Y * Iy + Z * Z * Iz - 2.0 * (X * Y * Ixy + X * Z * Ixz + Y * Z * Iyz)) / r2
    shell = -M / r - 0.5 * (Ix + Iy + Iz - 3.0 * I0) / (r2 * r)
    shell[i] = 0.0
    q = torch.zeros_like(shell)
    q[i] = rho
    lap = -6.0 * q[i]
    for d in range(3):
        for o in (0, 2):
            s = list(i)
            s[d] = slice(o, o + rho.shape[d])
            lap = lap + q[tuple(s)]
    rhs = 4.0 * math.pi * h * h * (rho + lap / 12.0)
    for dz in range(3):
        for dy in range(3):
            for dx in range(3):
                k = (dz != 1) + (dy != 1) + (dx != 1)
                if k:
                    rhs = rhs - (0.0, 4.0 / 9.0, 1.0 / 9.0, 1.0 / 36.0)[k] * shell[dz:dz + n[2], dy:dy + n[1], dx:dx + n[0]]
    F, sym = [], []
    for k in n:
        j = torch.arange(1, k + 1, dtype=F64, device=DEV)
        F.append(torch.sin(math.pi * j.view(-1, 1) * j.view(1, -1) / (k + 1)))
        sym.append(1.0 - (2.0 / 3.0) * torch.sin(0.5 * math.pi * j / (k + 1)) ** 2)

    def sine(w):
        w = w @ F[0]
        w = (w.transpose(1, 2) @ F[1]).transpose(1, 2)
        return (w.permute(1, 2, 0) @ F[2]).permute(2, 0, 1)

    lam = 6.0 * (sym[2].view(-1, 1, 1) * sym[1].view(1, -1, 1) * sym[0].view(1, 1, -1) - 1.0)
    scale = math.prod(2.0 / (k + 1) for k in n)
    return sine(sine(rhs) / lam * scale).reshape(-1)


def exact(case, seed):
    if case["kind"] == "batch":
        return _exact_batch(case, seed)
    if case["kind"] == "iso":
        return _exact_iso(case, seed)
    return _exact_grid(case, seed)
