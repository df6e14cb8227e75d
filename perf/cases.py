"""Performance cases: the calls a user of the library makes, over the sizes and options it is used with.

A case is a dict of plain values; "op" names the public entry point of paper_1612_00474_gb300.rpb it
goes through:

  product     Context.mobility_apply: U = M_tt F (+ M_tr T)
  lanczos     Context.lanczos_sqrt_apply: M^{1/2} W
  drift       Context.rfd_drift
  forces      Context.forces
  step        Context.ab_step, one Adams-Bashforth step driven from the host
  run         Context.run, several steps in one call
  batch_run   BatchContext.run, many suspensions, several steps in one call
  batch_step  BatchContext.ab_step, one step of a served mix of requests

Suspensions are roller monolayers: area fraction phi in a square, heights a + Exp(0.5a), gravity -1 z,
torque +1 y, U0 = 1, b = 0.1a, a = eta = kT = 1, time step 0.01.  The spheres stand on a jittered lattice
in random order (close pairs and a few slight overlaps, as a suspension in motion has), which is
quick to make at any size.  The drift's delta is the one each precision is used with: 1e-6 in float64,
5e-3 in float32.
"""
import math
import random

import numpy as np
import torch

from paper_1612_00474_gb300 import rpb

DT, TOL, MAX_ITER = 0.01, 1e-3, 64
DELTA = {"fp64": 1e-6, "fp32": 5e-3}
WEIGHT, U0, B, TORQUE = 1.0, 1.0, 0.1, (0.0, 1.0, 0.0)


def listed():
    return [
        # a handful of spheres, the reference precision: the smallest product, launch latency
        dict(name="product_f64_n64", op="product", n=64, precision="fp64", torque=True),
        # trajectory of the small plain configuration: 256 spheres, float64
        dict(name="run_f64_n256", op="run", n=256, precision="fp64", steps=20, periodic=False),
        # equilibrium sampling in the pseudo-periodic cell: 256 spheres, 20 steps between samples
        dict(name="run_periodic_f32_n256", op="run", n=256, precision="fp32", steps=20, periodic=True),
        # the accuracy configuration, one step of 4096 spheres in either precision
        dict(name="step_f64_n4096", op="step", n=4096, precision="fp64"),
        dict(name="step_f32_n4096", op="step", n=4096, precision="fp32"),
        # the large monolayer, one step
        dict(name="step_f32_n65536", op="step", n=65536, precision="fp32"),
        # the deterministic velocity of a roller strip's worth of spheres: forces and torques
        dict(name="product_f32_n32768", op="product", n=32768, precision="fp32", torque=True),
        # the drift of an odd-sized suspension
        dict(name="drift_f32_n10007", op="drift", n=10007, precision="fp32"),
        # the Brownian velocity without the wall's screening (iteration count against size)
        dict(name="lanczos_free_f32_n3001", op="lanczos", n=3001, precision="fp32", wall=False),
        # the steric forces of the large monolayer
        dict(name="forces_n65536", op="forces", n=65536, precision="fp32"),
        # many small suspensions of different sizes, advanced together
        dict(name="batch_run_512", op="batch_run", count=512, lo=64, hi=2048, mix=0, steps=2),
        # one tick of the trajectory server: requests of very different sizes
        dict(name="batch_step_serving", op="batch_step", count=24, lo=128, hi=32768, mix=1),
    ]


def _log_int(rng, lo, hi):
    return min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))


def draw(rng):
    op = rng.choice(["product", "product", "lanczos", "drift", "forces", "step", "step", "run", "run", "batch_run",
                     "batch_step"])
    precision = rng.choice(["fp64", "fp32"])
    f64 = precision == "fp64"
    if op == "product":
        return dict(op=op, n=_log_int(rng, 16, 8192 if f64 else 32768), precision=precision,
                    torque=rng.random() < 0.5)
    if op == "lanczos":
        wall = rng.random() < 0.5
        return dict(op=op, n=_log_int(rng, 100, 3000 if f64 else 16384), precision=precision, wall=wall)
    if op == "drift":
        return dict(op=op, n=_log_int(rng, 256, 32768), precision="fp32")
    if op == "forces":
        return dict(op=op, n=_log_int(rng, 256, 65536), precision=precision)
    if op == "step":
        return dict(op=op, n=_log_int(rng, 64, 4096 if f64 else 40000), precision=precision)
    if op == "run":
        return dict(op=op, n=_log_int(rng, 48, 700), precision=precision, steps=_log_int(rng, 4, 24),
                    periodic=not f64 and rng.random() < 0.5)
    if op == "batch_run":
        return dict(op=op, count=_log_int(rng, 64, 512), lo=64, hi=2048, mix=rng.randrange(2, 1000),
                    steps=rng.randint(1, 3))
    return dict(op=op, count=_log_int(rng, 2, 24), lo=128, hi=16384, mix=rng.randrange(2, 1000))


# ---------------------------------------------------------------- inputs
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) % (1 << 62))


def _cell(n, phi=0.4):
    return math.sqrt(n * math.pi / phi)


def _monolayer(n, gen, phi=0.4):
    """3n positions [x | y | z] on the GPU."""
    side = _cell(n, phi)
    m = math.ceil(math.sqrt(n))
    h = side / m
    site = torch.randperm(m * m, generator=gen, device="cuda")[:n]
    u = torch.rand(3, n, generator=gen, device="cuda", dtype=torch.float64)
    pos = torch.empty(3 * n, dtype=torch.float64, device="cuda")
    pos[:n] = (site % m + 0.5) * h + (u[0] - 0.5) * 0.5 * h
    pos[n:2 * n] = (site // m + 0.5) * h + (u[1] - 0.5) * 0.5 * h
    pos[2 * n:] = 1.0 - 0.5 * torch.log1p(-u[2])
    return pos


def _normal(n, gen):
    return torch.randn(n, generator=gen, device="cuda", dtype=torch.float64)


def _sizes(case):
    rng = random.Random(case["mix"])
    return [_log_int(rng, case["lo"], case["hi"]) for _ in range(case["count"])]


def _phi(case):
    return 0.25 if case.get("periodic") else 0.4


def prepare(case, seed):
    gen = _generator(seed)
    op = case["op"]
    s = dict(op=op, case=case, seed=int(seed) & 0xffffffff)
    if op.startswith("batch"):
        sizes = _sizes(case)
        q = [_monolayer(n, gen) for n in sizes]
        s["start"] = torch.cat(q)
        s["q"] = torch.empty_like(s["start"])
        s["u"] = torch.empty_like(s["start"])
        ends = [3 * n for n in sizes]
        s["qs"], s["us"] = list(torch.split(s["q"], ends)), list(torch.split(s["u"], ends))
        s["seeds"] = [s["seed"] + k for k in range(len(sizes))]
        s["zeros"] = [0] * len(sizes)
        s["bt"] = rpb.BatchContext(max_total_N=sum(sizes), max_B=len(sizes), precision="fp32", max_iter=MAX_ITER)
        return s
    n, precision = case["n"], case["precision"]
    s["ctx"] = rpb.Context(max_N=n, precision=precision, max_iter=MAX_ITER, wall=case.get("wall", True))
    s["delta"] = DELTA[precision]
    if case.get("periodic"):
        s["ctx"].set_periodic(_cell(n, 0.25), _cell(n, 0.25))
    s["start"] = _monolayer(n, gen, _phi(case))
    if op == "product":
        s["f"] = _normal(3 * n, gen)
        s["t"] = _normal(3 * n, gen) if case["torque"] else None
    elif op in ("lanczos", "drift"):
        s["w"] = _normal(3 * n, gen)
    elif op in ("step", "run"):
        s["q"] = torch.empty_like(s["start"])
        s["u"] = torch.empty_like(s["start"])
    return s


# ---------------------------------------------------------------- the calls
def run(s):
    op, case = s["op"], s["case"]
    if op == "product":
        return s["ctx"].mobility_apply(s["start"], s["f"], s["t"])
    if op == "lanczos":
        g, m, _, _ = s["ctx"].lanczos_sqrt_apply(s["start"], s["w"], tol=TOL)
        return {"g": g, "m": m}
    if op == "drift":
        return s["ctx"].rfd_drift(s["start"], s["w"], delta=s["delta"])
    if op == "forces":
        return s["ctx"].forces(s["start"], weight=WEIGHT, U0=U0, b=B)
    # trajectories start from the given configuration
    s["q"].copy_(s["start"])
    s["u"].zero_()
    if op == "step":
        st = s["ctx"].ab_step(s["q"], s["u"], 0, s["seed"], dt=DT, delta=s["delta"], tol=TOL, weight=WEIGHT, U0=U0,
                              b=B, torque=TORQUE)
        return {"q": s["q"], "u": s["u"], "m": st["m"]}
    if op == "run":
        st, _ = s["ctx"].run(s["q"], s["u"], 0, s["seed"], case["steps"], dt=DT, delta=s["delta"], tol=TOL,
                             weight=WEIGHT, U0=U0, b=B, torque=TORQUE)
        return {"q": s["q"], "u": s["u"], "m": st["m"]}
    if op == "batch_run":
        st, _ = s["bt"].run(s["qs"], s["us"], s["zeros"], s["seeds"], case["steps"], dt=DT, delta=DELTA["fp32"],
                            tol=TOL, weight=WEIGHT, U0=U0, b=B, torque=TORQUE)
    else:
        st = s["bt"].ab_step(s["qs"], s["us"], s["zeros"], s["seeds"], dt=DT, delta=DELTA["fp32"], tol=TOL,
                             weight=WEIGHT, U0=U0, b=B, torque=TORQUE)
    return {"q": s["q"], "u": s["u"], "m": np.array([x["m"] for x in st])}


# ---------------------------------------------------------------- the work a pass cannot do without
# flops of one unordered pair, both directions (a fused multiply-add is two): translation-translation,
# with the rotation coupling, and what a second right-hand side adds; without the wall terms the
# free-space part alone
PAIR_TT, PAIR_TR, PAIR_RHS2, PAIR_FREE = 135, 210, 57, 58


def _products(n, case, m):
    """flops of the products of one step: fused with the first Lanczos product, m - 1 others, 2 of the drift."""
    pairs = n * (n - 1) / 2 * (9 if case.get("periodic") else 1)
    return pairs * (PAIR_TR + PAIR_RHS2 + PAIR_TT * (m + 1))


def work(case):
    op = case["op"]
    if op.startswith("batch"):
        sizes, steps = _sizes(case), case.get("steps", 1)
        return {"bytes": 24 * 3 * sum(sizes), "flops": steps * sum(_products(n, case, 8) for n in sizes)}
    n = case["n"]
    v = 24 * n  # bytes of one vector
    pairs = n * (n - 1) / 2
    if op == "product":
        return {"bytes": v * (4 if case["torque"] else 3), "flops": pairs * (PAIR_TR if case["torque"] else PAIR_TT)}
    if op == "lanczos":
        m = 8 if case["wall"] else max(10, round(15 + 1.7 * math.log2(n / 2048)))
        return {"bytes": v * 3, "flops": m * pairs * (PAIR_TT if case["wall"] else PAIR_FREE)}
    if op == "drift":
        return {"bytes": v * 3, "flops": 2 * pairs * PAIR_TT}
    if op == "forces":
        return {"bytes": v * 2, "flops": n * 20 * 20}  # about 20 spheres within the cutoff of each
    return {"bytes": v * 3, "flops": case.get("steps", 1) * _products(n, case, 8)}


# ---------------------------------------------------------------- the same in plain 64-bit torch
MU = 1.0 / (8.0 * math.pi)


def _pair_terms(rx, ry, zi, zj, f, t, wall):
    """Velocity (units 1/(8 pi eta)) of the targets from the sources, elementwise over a (rows, n) block."""
    rz = zi - zj
    rho2 = rx * rx + ry * ry
    r = torch.sqrt(rho2 + rz * rz)
    near = r < 2.0
    ir = 1.0 / torch.where(r > 0, r, torch.ones_like(r))
    c1 = torch.where(near, 4.0 / 3.0 * (1.0 - 9.0 / 32.0 * r), ir * (1.0 + 2.0 / 3.0 * ir * ir))
    c2 = torch.where(near, 0.125 * ir, ir ** 3 * (1.0 - 2.0 * ir * ir))
    c2 = torch.where(r > 0, c2, torch.zeros_like(c2))
    k = c2 * (rx * f[0] + ry * f[1] + rz * f[2])
    u = [c1 * f[0] + k * rx, c1 * f[1] + k * ry, c1 * f[2] + k * rz]
    if t is not None:
        ct = torch.where(near, 0.5 * (1.0 - 0.375 * r), ir ** 3)
        u[0] = u[0] + ct * (t[1] * rz - t[2] * ry)
        u[1] = u[1] + ct * (t[2] * rx - t[0] * rz)
        u[2] = u[2] + ct * (t[0] * ry - t[1] * rx)
    if not wall:
        return u
    # image of the source below the wall: R = x_i - x_j*, e = R/|R|, h = z_j/|R|, s = 1/|R|^2
    Rz = zi + zj
    iR = torch.rsqrt(rho2 + Rz * Rz)
    ex, ey, ez, h, s = rx * iR, ry * iR, Rz * iR, zj * iR, iR * iR
    e2, eh, h2, s2 = ez * ez, ez * h, h * h, s * s
    A = -1 - 2 * eh + 2 * h2 + s * (2 * e2 - 2 / 3) + s2 * (2 / 3 - 10 / 3 * e2)
    Bc = -1 + 6 * eh - 6 * h2 + s * (2 - 10 * e2) + s2 * (70 / 3 * e2 - 10 / 3)
    C = 2 * h - 12 * e2 * h + 12 * ez * h2 + s * (20 * ez * e2 - 4 * ez) + s2 * (40 / 3 * ez - 140 / 3 * ez * e2)
    D = 2 * h - 20 / 3 * s2 * ez
    E = -4 * h2 - 4 * s * e2 + s2 * (20 * e2 - 8 / 3)
    eF = ex * f[0] + ey * f[1] + ez * f[2]
    ke, kz = (Bc * eF + C * f[2]) * iR, (D * eF + E * f[2]) * iR
    u = [u[0] + A * iR * f[0] + ke * ex, u[1] + A * iR * f[1] + ke * ey, u[2] + A * iR * f[2] + ke * ez + kz]
    if t is not None:
        cz, ce, w = 2 * (h + s * ez), 6 * (ez - h) - 10 * s * ez, ex * t[1] - ey * t[0]
        u[0] = u[0] + s * (-(t[1] * ez - t[2] * ey) + cz * t[1] + ce * w * ex)
        u[1] = u[1] + s * (-(t[2] * ex - t[0] * ez) - cz * t[0] + ce * w * ey)
        u[2] = u[2] + s * (-(t[0] * ey - t[1] * ex) + (ce * ez + 2 * s) * w)
    return u


def _mobility(q, f, t=None, wall=True, period=0.0):
    """M_tt f + M_tr t of q, f, t of shape (3, n)."""
    n = q.shape[1]
    z = torch.clamp(q[2], min=1.0) if wall else q[2]
    w = torch.clamp(q[2], 0.0, 1.0) if wall else torch.ones_like(q[2])
    f = f * w
    t = None if t is None else t * w
    out = torch.empty_like(q)
    rows = max(1, (1 << 22) // n)
    shifts = [(a * period, b * period) for a in (-1, 0, 1) for b in (-1, 0, 1)] if period else [(0.0, 0.0)]
    for i0 in range(0, n, rows):
        i1 = min(n, i0 + rows)
        dx, dy = q[0, i0:i1, None] - q[0], q[1, i0:i1, None] - q[1]
        if period:
            dx, dy = dx - period * torch.round(dx / period), dy - period * torch.round(dy / period)
        for a, b in shifts:
            u = _pair_terms(dx + a, dy + b, z[i0:i1, None], z, f, t, wall)
            for c in range(3):
                v = u[c].sum(1)
                out[c, i0:i1] = v if (a, b) == shifts[0] else out[c, i0:i1] + v
    return MU * w * out


def _steric(q, period=0.0):
    n = q.shape[1]
    out = torch.empty_like(q)
    rows = max(1, (1 << 22) // n)
    f0 = U0 / B
    for i0 in range(0, n, rows):
        i1 = min(n, i0 + rows)
        d = [q[c, i0:i1, None] - q[c] for c in range(3)]
        if period:
            d = [x - period * torch.round(x / period) if c < 2 else x for c, x in enumerate(d)]
        r = torch.sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2])
        k = torch.where(r > 0, f0 * torch.exp(-torch.clamp(r - 2.0, min=0.0) / B) / torch.where(r > 0, r, 1.0), 0.0)
        for c in range(3):
            out[c, i0:i1] = (k * d[c]).sum(1)
    out[2] += f0 * torch.exp(-torch.clamp(q[2] - 1.0, min=0.0) / B) - WEIGHT
    return out


def _sqrt_product(apply, w):
    """Lanczos approximation of M^{1/2} w of shape (3, n), to the relative change TOL; and its dimension."""
    norm = torch.linalg.vector_norm(w)
    V, alpha, beta, last = [(w / norm).reshape(-1)], [], [], None
    for _ in range(MAX_ITER):
        x = apply(V[-1].reshape(w.shape)).reshape(-1)
        basis = torch.stack(V)
        c = basis @ x
        alpha.append(float(c[-1]))
        x = x - c @ basis
        c = basis @ x
        alpha[-1] += float(c[-1])
        x = x - c @ basis
        beta.append(float(torch.linalg.vector_norm(x)))
        lam, Q = np.linalg.eigh(np.diag(alpha) + np.diag(beta[:-1], 1) + np.diag(beta[:-1], -1))
        y = Q @ (np.sqrt(np.maximum(lam, 0.0)) * Q[0])
        if last is not None and np.linalg.norm(y - np.append(last, 0.0)) <= TOL * np.linalg.norm(last):
            break
        last = y
        V.append(x / beta[-1])
    return norm * (torch.as_tensor(y, device=w.device) @ basis).reshape(w.shape), len(y)


def _philox(n, seed, step, stream):
    """3n standard normals as (3, n): Philox4x32-10 with counter (k / 2, step, stream, 0), two 53-bit
    uniforms and a Box-Muller pair per counter, normal k = 3 i + c of sphere i."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    lo = 0xffffffff
    p = torch.arange((3 * n + 1) // 2, dtype=torch.int64, device=dev)
    c = [p, torch.full_like(p, step), torch.full_like(p, stream), torch.zeros_like(p)]
    k0, k1 = seed & lo, (seed >> 32) & lo
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & lo, (k1 + 0xBB67AE85) & lo
        a, b = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57  # wrap modulo 2^64: the low and high words are right
        c = [((b >> 32) & lo) ^ c[1] ^ k0, b & lo, ((a >> 32) & lo) ^ c[3] ^ k1, a & lo]
    u1 = ((c[0] >> 5).double() * 2.0 ** 26 + (c[1] >> 6).double() + 1.0) * 2.0 ** -53
    u2 = ((c[2] >> 5).double() * 2.0 ** 26 + (c[3] >> 6).double() + 1.0) * 2.0 ** -53
    rad = torch.sqrt(-2.0 * torch.log(u1))
    out = torch.stack([rad * torch.cos(2 * math.pi * u2), rad * torch.sin(2 * math.pi * u2)], 1).reshape(-1)
    return out[:3 * n].reshape(n, 3).T.contiguous()


def _steps(q, seed, steps, delta, period):
    q = q.reshape(3, -1).clone()
    n = q.shape[1]
    t = torch.tensor(TORQUE, dtype=torch.float64, device=q.device)[:, None].expand(3, n)
    prev = None
    for k in range(steps):
        u = _mobility(q, _steric(q, period), t, period=period)
        g, m = _sqrt_product(lambda v: _mobility(q, v, period=period), _philox(n, seed, k, 0))
        wt = _philox(n, seed, k, 1)
        d = (_mobility(q + 0.5 * delta * wt, wt, period=period) -
             _mobility(q - 0.5 * delta * wt, wt, period=period)) / delta
        q = q + DT * (1.5 * u - 0.5 * (u if prev is None else prev)) + math.sqrt(2 * DT) * g + DT * d
        prev = u
    return q.reshape(-1), prev.reshape(-1), m


def exact(case, seed):
    op, steps = case["op"], case.get("steps", 1)
    sizes = _sizes(case) if op.startswith("batch") else [case["n"]]
    passes = {"product": 1, "lanczos": 24, "drift": 2, "forces": 0.3}.get(op, 11 * steps)
    # about 0.6 ns a pair and 1.5 ms of launches a product
    if passes * sum(6e-10 * n * n * (9 if case.get("periodic") else 1) + 1.5e-3 for n in sizes) > 12.0:
        return None
    s = prepare(case, seed)
    if op.startswith("batch"):
        parts = [_steps(x, sd, steps, DELTA["fp32"], 0.0)
                 for x, sd in zip(torch.split(s["start"], [3 * n for n in sizes]), s["seeds"])]
        return {"q": torch.cat([p[0] for p in parts]), "u": torch.cat([p[1] for p in parts]),
                "m": np.array([p[2] for p in parts])}
    n = case["n"]
    q = s["start"].reshape(3, n)
    v = {k: s[k].reshape(3, n) for k in ("f", "t", "w") if s.get(k) is not None}
    if op == "product":
        return _mobility(q, v["f"], v.get("t")).reshape(-1)
    if op == "lanczos":
        g, m = _sqrt_product(lambda x: _mobility(q, x, wall=case["wall"]), v["w"])
        return {"g": g.reshape(-1), "m": m}
    if op == "drift":
        w, h = v["w"], 0.5 * s["delta"]
        return ((_mobility(q + h * w, w) - _mobility(q - h * w, w)) / s["delta"]).reshape(-1)
    if op == "forces":
        return _steric(q).reshape(-1)
    q, u, m = _steps(s["start"], s["seed"], steps, s["delta"], _cell(n, 0.25) if case.get("periodic") else 0.0)
    return {"q": q, "u": u, "m": m}
