"""What a program does with this library, as cases that can be timed.

Five kinds of pass, all through the binding's public calls:

  advance   resume a stored state and integrate it to t_end (hg_set_state, hg_advance,
            hg_get_state): graph-replayed block steps of every size that occurs
  batch     the same for many independent clusters in one context (hg_init_batch)
  evaluate  predict every particle and evaluate m listed ones (hg_predict, hg_evaluate)
  block     the explicit calls of one block step: hg_next_block, hg_predict, hg_evaluate
  energy    the conservation check at a synchronisation time: hg_energy and
            hg_angular_momentum

Inputs are Plummer spheres in Henon units (G = M = 1, E = -1/4), with equal masses or masses
from a Salpeter IMF on [0.1, 100], drawn on the GPU.  States of the evaluate, block and
energy kinds are as read from a checkpoint: the sphere's mean-field derivatives and a
hierarchy of power-of-two steps.  advance and batch start from the library's own start-up.
"""
import math

import numpy as np
import torch

from paper_1207_2367_gb300 import binding as hg

B_HENON = 3.0 * math.pi / 16.0   # Plummer radius in Henon units
ETA, ETA_INIT = 0.45, 0.01
DT_MIN, DT_MAX = 2.0 ** -25, 2.0 ** -4
FLOPS_PER_PAIR = 77              # adds and multiplications of the pair law, the root not counted
STATE_BYTES = 176                # FP64 fields of a particle: mass, t, dt, its tend, six vectors

VECTORS = ("pos", "vel", "acc", "jerk", "snap", "crackle")


def _case(name, kind, n, precision="mixed", eps=1e-4, imf="equal", order=6, m=0, t_log2=0, clusters=0, n_lo=0):
    return {"name": name, "kind": kind, "n": n, "precision": precision, "eps": eps, "imf": imf, "order": order,
            "m": m, "t_log2": t_log2, "clusters": clusters, "n_lo": n_lo}


def listed():
    return [
        # The smallest calls: one explicit block step of a small system, a few particles due.
        _case("block_mixed_n1024", "block", 1024, eps=1e-3),
        # Whole integrations.  A small FP64 system: nothing but short block steps.
        _case("advance_fp64_n1024", "advance", 1024, "fp64", eps=1e-3, t_log2=-2),
        # FP64 throughout at scale: the evaluation's FP64 arithmetic.
        _case("advance_fp64_n65536", "advance", 65536, "fp64", t_log2=-10),
        # The main path, mixed precision: thousands of small blocks and a few large ones.
        _case("advance_mixed_n65536", "advance", 65536, t_log2=-7),
        # A mass spectrum at a larger, odd N.
        _case("advance_mixed_n200001", "advance", 200001, imf="salpeter", t_log2=-10),
        # The 4th-order scheme.
        _case("advance_order4_n16384", "advance", 16384, order=4, t_log2=-6),
        # Independent clusters of 256 to 16384 particles in one context.
        _case("batch_mixed_64", "batch", 16384, eps=1e-3, t_log2=-8, clusters=64, n_lo=256),
        # Start-up and synchronised blocks: every particle active.
        _case("evaluate_mixed_n131072", "evaluate", 131072, m=131072),
        _case("evaluate_fp64_n32768", "evaluate", 32768, "fp64", m=32768),
        # A few hundred of many particles, both precisions; odd sizes.
        _case("evaluate_mixed_n8388608", "evaluate", 8388608, imf="salpeter", m=301),
        _case("evaluate_fp64_n65537", "evaluate", 65537, "fp64", m=333),
        # Conservation check.
        _case("energy_fp64_n65536", "energy", 65536, "fp64"),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["advance", "advance", "batch", "evaluate", "evaluate", "block", "energy"])
    precision = rng.choice(["mixed", "mixed", "fp64"]) if kind in ("advance", "evaluate", "block") else "mixed"
    eps = rng.choice([1e-4, 1e-4, 1e-3, 1e-2])
    imf = rng.choice(["equal", "salpeter"])
    if kind == "advance":
        if precision == "fp64":
            n = _log_uniform(rng, 256, 40000)
            t = -4 if n < 2000 else (-7 if n < 10000 else -9)
        else:
            n = _log_uniform(rng, 256, 200000)
            t = -4 if n < 4000 else (-6 if n < 20000 else (-8 if n < 80000 else -10))
        c = _case("", kind, n, precision, max(eps, 1e-3) if n < 4000 else eps, imf, rng.choice([6, 6, 4]), t_log2=t)
    elif kind == "batch":
        c = _case("", kind, _log_uniform(rng, 2000, 16384), eps=1e-3, t_log2=-8, clusters=rng.randint(8, 64),
                  n_lo=_log_uniform(rng, 100, 1000))
    elif kind == "evaluate":
        pairs = 1.0e9 if precision == "fp64" else 1.5e10
        n = _log_uniform(rng, 100, 130000 if precision == "fp64" else 4000000)
        c = _case("", kind, n, precision, eps, imf, m=_log_uniform(rng, 1, max(1, min(n, int(pairs / n)))))
    elif kind == "block":
        c = _case("", kind, _log_uniform(rng, 64, 300000), precision, eps, imf)
    else:
        c = _case("", kind, _log_uniform(rng, 256, 65536), "fp64", eps, imf)
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# Inputs.
# ---------------------------------------------------------------------------
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _uniform(g, *shape):
    return torch.rand(*shape, dtype=torch.float64, device="cuda", generator=g)


def _directions(g, n):
    z = 2.0 * _uniform(g, n) - 1.0
    phi = 2.0 * math.pi * _uniform(g, n)
    s = torch.sqrt((1.0 - z * z).clamp_min(0.0))
    return torch.stack([s * torch.cos(phi), s * torch.sin(phi), z], dim=1)


def _plummer(n, g, imf):
    """Masses, positions and velocities of a Plummer sphere in Henon units."""
    r = 1.0 / torch.sqrt((0.999 * (1.0 - _uniform(g, n))) ** (-2.0 / 3.0) - 1.0)
    q = torch.zeros(n, dtype=torch.float64, device="cuda")
    todo = torch.ones(n, dtype=torch.bool, device="cuda")
    while bool(todo.any()):          # von Neumann rejection on q^2 (1 - q^2)^3.5
        a, b = _uniform(g, n), 0.1 * _uniform(g, n)
        ok = todo & (b < a * a * (1.0 - a * a) ** 3.5)
        q = torch.where(ok, a, q)
        todo &= ~ok
    pos = r[:, None] * _directions(g, n)
    vel = (q * math.sqrt(2.0) * (1.0 + r * r) ** -0.25)[:, None] * _directions(g, n)
    if imf == "salpeter":
        lo, hi = 0.1 ** -1.35, 100.0 ** -1.35
        mass = (lo + _uniform(g, n) * (hi - lo)) ** (-1.0 / 1.35)
        mass = mass / mass.sum()
    else:
        mass = torch.full((n,), 1.0 / n, dtype=torch.float64, device="cuda")
    pos = (pos - (mass[:, None] * pos).sum(0)) * B_HENON
    vel = (vel - (mass[:, None] * vel).sum(0)) / math.sqrt(B_HENON)
    return mass, pos.contiguous(), vel.contiguous()


def _sizes(case):
    """Cluster sizes, spread over the logarithm between n_lo and n, small and large ones in turn."""
    c, ratio = case["clusters"], case["n"] / case["n_lo"]
    order = [k // 2 if k % 2 == 0 else c - 1 - k // 2 for k in range(c)]
    return [int(round(case["n_lo"] * ratio ** ((k + 0.5) / c))) for k in order]


def _power_of_two(e):
    """2^e, exactly, for a tensor of whole exponents."""
    return ((e.long() + 1023) << 52).view(torch.float64)


def _deepest(n):
    """Level of the shortest steps in _checkpoint, which 8 to 16 particles have."""
    return max(2, int(math.log2(n)) - 3)


def _checkpoint(case, seed):
    """A stored state at t = 0: a sphere with its mean-field acceleration, jerk and snap, and
    steps of which half the particles have the longest, a quarter the next, and so on."""
    g = _generator(seed)
    n = case["n"]
    mass, x, v = _plummer(n, g, case["imf"])
    d2 = ((x * x).sum(1) + B_HENON ** 2)[:, None]
    xv = (x * v).sum(1)[:, None]
    acc = -x / d2 ** 1.5
    jerk = -(v - 3.0 * xv / d2 * x) / d2 ** 1.5
    snap = -(acc - 6.0 * xv / d2 * v - 3.0 * (((v * v).sum(1) + (x * acc).sum(1))[:, None] / d2
                                              - 5.0 * xv * xv / (d2 * d2)) * x) / d2 ** 1.5
    share = (torch.randperm(n, device="cuda", generator=g) + 0.5) / n
    level = torch.floor(-torch.log2(share)).clamp_max(_deepest(n))
    return {"mass": mass, "pos": x, "vel": v, "acc": acc, "jerk": jerk, "snap": snap,
            "crackle": torch.zeros_like(x), "t": torch.zeros_like(mass), "dt": DT_MAX * _power_of_two(-level)}


def _listed_particles(case, seed):
    g = _generator(seed + (1 << 40))
    return torch.randperm(case["n"], device="cuda", generator=g)[:case["m"]].sort().values.int()


# ---------------------------------------------------------------------------
# Passes.
# ---------------------------------------------------------------------------
class _State:
    """A context and the arrays a program holds beside it."""

    def __init__(self, case):
        self.case, self.ctx = case, None

    def __del__(self):
        if self.ctx is not None:
            hg.hg_free(self.ctx)
            self.ctx = None


def _options(case, start_mode):
    return hg.hg_default_opts(precision=hg.HG_FP64 if case["precision"] == "fp64" else hg.HG_MIXED,
                              energy_precision=hg.HG_FP64, dt_min=DT_MIN, dt_max=DT_MAX, eta_init=ETA_INIT,
                              order=case["order"], start_mode=start_mode)


def prepare(case, seed):
    s = _State(case)
    n, eps = case["n"], case["eps"]
    if case["kind"] in ("advance", "batch"):
        g = _generator(seed)
        if case["kind"] == "batch":
            sizes = _sizes(case)
            offsets = np.cumsum([0] + sizes)
            parts = [_plummer(k, g, "equal") for k in sizes]
            mass, pos, vel = (torch.cat([p[f] for p in parts]) for f in range(3))
            n = sum(sizes)
            torch.cuda.synchronize()
            s.ctx = hg.hg_init_batch(offsets, mass, pos, vel, eps, ETA, _options(case, 0))
        else:
            mass, pos, vel = _plummer(n, g, case["imf"])
            torch.cuda.synchronize()
            s.ctx = hg.hg_init(mass, pos, vel, eps, ETA, _options(case, 0))
        s.start = hg.new_state(n, like="cuda")
        s.t_start = hg.hg_get_state(s.ctx, s.start)
        s.out = hg.new_state(n, like="cuda")
        return s
    st = _checkpoint(case, seed)
    torch.cuda.synchronize()
    s.ctx = hg.hg_init(st["mass"], st["pos"], st["vel"], eps, ETA, _options(case, 1))
    hg.hg_set_state(s.ctx, st, 0.0)
    if case["kind"] == "evaluate":
        s.idx = _listed_particles(case, seed)
        s.out = [torch.empty(case["m"], 3, dtype=torch.float64, device="cuda") for _ in range(3)]
        torch.cuda.synchronize()
    elif case["kind"] == "block":
        s.idx = torch.empty(n, dtype=torch.int32, device="cuda")
        s.out = [torch.empty(n, 3, dtype=torch.float64, device="cuda") for _ in range(3)]
    return s


T_EVALUATE = 2.0 ** -9   # the evaluate kind predicts this far


def run(s):
    case = s.case
    kind = case["kind"]
    if kind in ("advance", "batch"):
        hg.hg_set_state(s.ctx, s.start, s.t_start)
        hg.hg_advance(s.ctx, 2.0 ** case["t_log2"])
        t = hg.hg_get_state(s.ctx, s.out)
        return {"t_sys": t, **{f: s.out[f] for f in hg.STATE_FIELDS}}
    if kind == "energy":
        K, W = hg.hg_energy(s.ctx)
        return {"kinetic": K, "potential": W, "angular_momentum": hg.hg_angular_momentum(s.ctx)}
    if kind == "block":
        t, m = hg.hg_next_block(s.ctx, s.idx)
        hg.hg_predict(s.ctx, t)
        hg.hg_evaluate(s.ctx, None, m, *s.out)
        return {"t": t, "idx": s.idx[:m], "acc": s.out[0][:m], "jerk": s.out[1][:m], "snap": s.out[2][:m]}
    hg.hg_predict(s.ctx, T_EVALUATE)
    hg.hg_evaluate(s.ctx, s.idx, case["m"], *s.out)
    return {"acc": s.out[0], "jerk": s.out[1], "snap": s.out[2]}


def work(case):
    n, kind = float(case["n"]), case["kind"]
    if kind == "energy":
        return {"bytes": n * 128 + 40, "flops": 0.5 * n * n * 11}
    if kind in ("evaluate", "block"):
        m = float(case["m"]) if kind == "evaluate" else max(1.0, n * 2.0 ** -_deepest(case["n"]))
        return {"bytes": n * 160 + m * 76, "flops": FLOPS_PER_PAIR * m * n}
    # Integrations: 350 n^2 pair evaluations per unit of time is what block steps take on these spheres.
    t = 2.0 ** case["t_log2"]
    if kind == "batch":
        sizes = _sizes(case)
        return {"bytes": 2 * STATE_BYTES * sum(sizes),
                "flops": FLOPS_PER_PAIR * 350 * t * sum(k * k for k in sizes)}
    return {"bytes": 2 * STATE_BYTES * n, "flops": FLOPS_PER_PAIR * 350 * t * n * n}


# ---------------------------------------------------------------------------
# The same in plain torch, 64 bits.
# ---------------------------------------------------------------------------
def _pairs(mass, x, v, a, eps, idx):
    """Acceleration, jerk and snap of the listed particles from all n."""
    n = mass.numel()
    out = [torch.empty(idx.numel(), 3, dtype=torch.float64, device="cuda") for _ in range(3)]
    rows = max(1, (1 << 25) // n)
    for k in range(0, idx.numel(), rows):
        i = idx[k:k + rows].long()
        r, w, da = (f[None, :, :] - f[i][:, None, :] for f in (x, v, a))
        r2 = (r * r).sum(2) + eps * eps
        q = mass / (r2 * torch.sqrt(r2))
        q[torch.arange(i.numel(), device="cuda"), i] = 0.0
        alpha = ((r * w).sum(2) / r2)[:, :, None]
        beta = (((w * w).sum(2) + (r * da).sum(2)) / r2)[:, :, None] + alpha * alpha
        w = w - 3.0 * alpha * r
        u = da - 6.0 * alpha * w - 3.0 * beta * r
        for o, f in zip(out, (r, w, u)):
            o[k:k + rows] = torch.einsum("ij,ijk->ik", q, f)
    return out


def _taylor(st, t):
    h = (t - st["t"])[:, None]
    x, v, a, j, s, c = (st[f] for f in VECTORS)
    return (x + h * (v + h / 2 * (a + h / 3 * (j + h / 4 * (s + h / 5 * c)))),
            v + h * (a + h / 2 * (j + h / 3 * (s + h / 4 * c))), a + h * (j + h / 2 * (s + h / 3 * c)))


def _aarseth(eta, p, d):
    nr = [f.norm(dim=1) for f in d]
    big = torch.sqrt(nr[0] * nr[2] + nr[1] ** 2)
    small = torch.sqrt(nr[p - 3] * nr[p - 1] + nr[p - 2] ** 2)
    return eta * (big / small) ** (1.0 / (p - 3))


def _integrate(mass, x, v, eps, t_end):
    """6th-order Hermite block steps from the start-up at t = 0 to t_end."""
    n = mass.numel()
    zero = torch.zeros_like(x)
    a, j, s = _pairs(mass, x, v, zero, eps, torch.arange(n, device="cuda"))
    crit = _aarseth(ETA_INIT, 4, [a, j, s, zero])
    dt = _power_of_two(torch.floor(torch.log2(crit))).clamp(DT_MIN, DT_MAX)
    st = {"mass": mass, "pos": x, "vel": v, "acc": a, "jerk": j, "snap": s, "crackle": zero.clone(),
          "t": torch.zeros_like(mass), "dt": dt}
    t_sys = 0.0
    while True:
        tend = st["t"] + st["dt"]
        t = float(tend.min())
        if t > t_end:
            return {"t_sys": t_sys, **st}
        t_sys = t
        i = (tend == t).nonzero()[:, 0]
        xp, vp, ap = _taylor(st, t)
        a1, j1, s1 = _pairs(mass, xp, vp, ap, eps, i)
        x0, v0, a0, j0, s0 = (st[f][i] for f in VECTORS[:5])
        h1 = st["dt"][i]
        h = h1[:, None]
        v1 = v0 + h / 2 * (a1 + a0) - h * h / 10 * (j1 - j0) + h ** 3 / 120 * (s1 + s0)
        x1 = x0 + h / 2 * (v1 + v0) - h * h / 10 * (a1 - a0) + h ** 3 / 120 * (j1 + j0)
        A, J, S = a1 - a0 - j0 * h - s0 * h * h / 2, (j1 - j0 - s0 * h) * h, (s1 - s0) * h * h
        c3 = (60 * A - 36 * J + 9 * S) / h ** 3
        c4 = (360 * A - 192 * J + 36 * S) / h ** 4
        c5 = (720 * A - 360 * J + 60 * S) / h ** 5
        for f, value in zip(VECTORS, (x1, v1, a1, j1, s1, c3)):
            st[f][i] = value
        crit = _aarseth(ETA, 6, [a1, j1, s1, c3, c4, c5])
        grow = (crit >= 2 * h1) & (2 * h1 <= DT_MAX) & (torch.remainder(torch.full_like(h1, t), 2 * h1) == 0)
        st["dt"][i] = torch.where(crit < h1, _power_of_two(torch.floor(torch.log2(crit))),
                                  torch.where(grow, 2 * h1, h1)).clamp(DT_MIN, DT_MAX)
        st["t"][i] = t


def exact(case, seed):
    kind, n, eps = case["kind"], case["n"], case["eps"]
    if kind == "batch" or (kind == "advance" and (case["precision"] == "mixed" or case["order"] == 4 or n > 4096)):
        return None   # mixed: its step rule has a noise floor of its own; large FP64: over 20 seconds
    if kind == "advance":
        return _integrate(*_plummer(n, _generator(seed), case["imf"]), eps, 2.0 ** case["t_log2"])
    st = _checkpoint(case, seed)
    if kind == "energy":
        mass, x, v = st["mass"], st["pos"], st["vel"]
        phi = torch.zeros_like(mass)
        rows = max(1, (1 << 27) // n)
        for k in range(0, n, rows):
            r = x[None, :, :] - x[k:k + rows, None, :]
            q = mass / torch.sqrt((r * r).sum(2) + eps * eps)
            i = torch.arange(q.shape[0], device="cuda")
            q[i, i + k] = 0.0
            phi[k:k + rows] = q.sum(1)
        L = (mass[:, None] * torch.linalg.cross(x, v)).sum(0)
        return {"kinetic": float(0.5 * (mass * (v * v).sum(1)).sum()), "potential": float(-0.5 * (mass * phi).sum()),
                "angular_momentum": L}
    t = T_EVALUATE if kind == "evaluate" else float(st["dt"].min())
    idx = _listed_particles(case, seed) if kind == "evaluate" else (st["dt"] == t).nonzero()[:, 0].int()
    xp, vp, ap = _taylor(st, t)
    out = dict(zip(("acc", "jerk", "snap"), _pairs(st["mass"], xp, vp, ap, eps, idx)))
    return out if kind == "evaluate" else {"t": t, "idx": idx, **out}
