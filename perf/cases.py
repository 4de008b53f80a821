"""The workloads this framework is timed on, through its public entry points.

Each case is one unit of a P3M simulation's work: a single force evaluation, a
kick-drift-kick step with every particle active, a substep of the rung scheme with
some rungs due, the periodic reordering with its rung update, kick and drift, the
adjoint, the differentiable leapfrog, and the long-range mesh force.  Particle sets
are the clustered recipe of the ``synth`` workloads (a uniform fraction plus Plummer
spheres), drawn here on the GPU; the physical parameters are the P3M defaults
(n_phi = 2 cbrt(N), x_s = 1.25 / n_phi, x_r = 4.5 x_s, eps = 0.03 / cbrt(N), G m = 1/N).

  accel     ``autograd.short_range_accel`` in the caller's order: sort, work list,
            forces, back to the caller's order
  step      out-of-place sort with the momenta, work list, forces of all particles,
            kick, drift
  substep   the same with the receivers on rungs >= rung_min and their rung's kick
  vjp       out-of-place sort, work list, forces and their adjoint
  reorder   out-of-place sort with four carried arrays, then Eq. rung, kick and drift
            in one pass for accelerations in hand
  leapfrog  ``autograd.leapfrog`` with checkpoints, and the backward pass
  mesh      ``LongRange.accel`` on positions in tile order
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2112_01508_gb300 import LongRange, ShortRange
from paper_2112_01508_gb300.autograd import leapfrog, short_range_accel

N_RUNG = 8
ETA = 0.025  # accuracy parameter of Eq. rung


# ---------------------------------------------------------------------------
# The cases.
# ---------------------------------------------------------------------------

def listed():
    clustered = {"frac_uniform": 0.3, "per_sphere": 358, "b_lo": 0.128, "b_hi": 1.28}  # the 128^3 set's recipe
    return [
        # the smallest useful call: forces of a few thousand particles (a test problem, a
        # tracer set), where launches and the longest serial chain count
        {"name": "accel_4k", "kind": "accel", "n": 4096, "precision": 32, "softening": "bspline", "n_sub": 2,
         "symmetric": True, "frac_uniform": 0.5, "per_sphere": 256, "b_lo": 0.16, "b_hi": 0.16},
        # a small simulation: one all-active step of the 32^3 set
        {"name": "step_32k", "kind": "step", "n": 32768, "precision": 32, "softening": "bspline", "n_sub": 2,
         "symmetric": True, "frac_uniform": 0.5, "per_sphere": 256, "b_lo": 0.32, "b_hi": 0.32},
        # the benchmark's set: one all-active step at 128^3
        {"name": "step_2m", "kind": "step", "n": 128 ** 3, "precision": 32, "softening": "bspline", "n_sub": 2,
         "symmetric": True, **clustered},
        # a production-sized box, more strongly clustered, an odd particle count
        {"name": "step_15m", "kind": "step", "n": 249 ** 3 + 7, "precision": 32, "softening": "bspline", "n_sub": 2,
         "symmetric": True, "frac_uniform": 0.2, "per_sphere": 410, "b_lo": 0.128, "b_hi": 1.28},
        # a middle substep of a global time step: the rungs due hold about a third of the particles
        {"name": "substep_2m_mid", "kind": "substep", "n": 128 ** 3, "precision": 32, "softening": "bspline", "n_sub": 2,
         "rung_min": 5, "symmetric": True, **clustered},
        # every other substep: only the deepest rung, in the cluster cores
        {"name": "substep_2m_deep", "kind": "substep", "n": 128 ** 3, "precision": 32, "softening": "bspline",
         "n_sub": 2, "rung_min": 7, "symmetric": True, **clustered},
        # reference-precision forces (the fake kick that starts a run, convergence checks)
        {"name": "accel_262k_fp64", "kind": "accel", "n": 64 ** 3, "precision": 64, "softening": "bspline", "n_sub": 2,
         "symmetric": True, **clustered},
        # gradients through a short integration in the default (double) precision, Plummer
        # softened, as an inference loop over initial conditions runs it
        {"name": "leapfrog_9k_fp64", "kind": "leapfrog", "n": 21 ** 3, "precision": 64, "softening": "plummer",
         "n_sub": 2, "n_steps": 4, "checkpoint_every": 2, "symmetric": True, **clustered},
        # forces and their adjoint at the benchmark's size in single precision
        {"name": "vjp_2m", "kind": "vjp", "n": 128 ** 3, "precision": 32, "softening": "bspline", "n_sub": 2,
         "symmetric": True, **clustered},
        # the passes over all particles between force calls, at a size that fills no tile evenly
        {"name": "reorder_2m", "kind": "reorder", "n": 127 ** 3, "n_sub": 2, **clustered},
        # the mesh half of the benchmark's set: 256^3 mesh, CIC, D_4
        {"name": "mesh_2m", "kind": "mesh", "n": 128 ** 3, "n_phi": 256, "p_i": 2, "p_d": 4, "precision": 32,
         "accumulate": False, **clustered},
        # a small mesh in double precision with higher orders, added onto other accelerations
        {"name": "mesh_36k_fp64", "kind": "mesh", "n": 33 ** 3, "n_phi": 66, "p_i": 3, "p_d": 6, "precision": 64,
         "accumulate": True, **clustered},
    ]


def draw(rng):
    kind = rng.choice(["accel", "step", "step", "substep", "substep", "vjp", "reorder", "leapfrog", "mesh"])
    top = {"accel": 128, "step": 200, "substep": 160, "vjp": 140, "reorder": 200, "leapfrog": 20, "mesh": 160}[kind]
    low = 14
    precision = 32 if kind == "step" else rng.choice([32, 32, 64])
    if kind == "substep":
        precision = 32 if rng.random() < 0.8 else 64
    if kind == "leapfrog":
        precision = 64
    if precision == 64 and kind in ("accel", "substep", "vjp"):
        top = {"accel": 60, "substep": 60, "vjp": 44}[kind]
    side = math.exp(rng.uniform(math.log(low), math.log(top)))
    n = int(side ** 3) + rng.randrange(0, 50)
    spread = rng.choice([1.0, 10.0])
    b_lo = rng.uniform(0.1, 0.32)
    case = {"kind": kind, "n": n, "frac_uniform": round(rng.uniform(0.1, 0.6), 3),
            "per_sphere": rng.randrange(150, 420), "b_lo": round(b_lo, 4), "b_hi": round(b_lo * spread, 4)}
    if kind == "mesh":
        n_phi = 2 * max(8, int(side * rng.choice([0.5, 1.0, 1.0])))
        case |= {"n_phi": n_phi, "p_i": rng.choice([1, 2, 2, 2, 3, 4]), "p_d": rng.choice([2, 4, 4, 6, 8]),
                 "precision": precision, "accumulate": rng.random() < 0.5}
        return case
    case["n_sub"] = rng.choice([1, 2, 2, 2, 3])
    if kind == "reorder":
        return case
    # point particles only in double precision, and not integrated: single precision does not
    # resolve their closest pairs
    point = ["none"] if precision == 64 and kind != "leapfrog" else []
    case |= {"precision": precision, "softening": rng.choice(["bspline", "bspline", "bspline", "plummer"] + point),
             "symmetric": rng.random() < 0.75}
    if kind == "substep":
        case["rung_min"] = rng.randrange(1, N_RUNG)
    if kind == "leapfrog":
        case |= {"n_steps": rng.randrange(2, 5), "checkpoint_every": rng.choice([0, 1, 2])}
    return case


# ---------------------------------------------------------------------------
# Inputs.
# ---------------------------------------------------------------------------

def _device():
    return torch.device("cuda") if torch.cuda.is_available() else torch.device("cpu")


def _params(case):
    """The P3M defaults for n particles in the unit box."""
    n = case["n"]
    side = n ** (1.0 / 3.0)
    x_s = 1.25 / (2.0 * side)
    return {"x_s": x_s, "x_r": 4.5 * x_s, "G_m": 1.0 / n, "eps": 0.03 / side}


def _generator(seed):
    g = torch.Generator(device=_device())
    g.manual_seed(int(seed))
    return g


def _particles(case, seed):
    """Positions (3, n) float64 in [0, 1) in random order, and an estimate of each
    particle's acceleration (its own sphere's enclosed mass plus a background), from
    which rungs and time steps are taken without evaluating a force."""
    n, dev, g = case["n"], _device(), _generator(seed)

    def u(*shape):
        return torch.rand(*shape, generator=g, device=dev, dtype=torch.float64)

    side = n ** (1.0 / 3.0)
    n_u = int(round(case["frac_uniform"] * n))
    m = n - n_u
    k = max(1, m // case["per_sphere"])
    lo, hi = case["b_lo"] / side, case["b_hi"] / side  # Plummer scales, in units of the mean spacing
    centre = u(3, k)
    b_all = lo * torch.exp(u(k) * math.log(hi / lo)) if hi > lo else torch.full((k,), lo, dtype=torch.float64, device=dev)
    which = (u(m) * k).to(torch.int64).clamp_(max=k - 1)
    b = b_all[which]
    r_max = 0.25
    w = 1e-12 + u(m) * (r_max ** 3 / (r_max ** 2 + b * b) ** 1.5 - 1e-12)  # M(<r) / M, cut at r_max
    r = b / torch.sqrt(w.pow(-2.0 / 3.0) - 1.0)
    cz, phi = 2.0 * u(m) - 1.0, 2.0 * math.pi * u(m)
    st = torch.sqrt((1.0 - cz * cz).clamp_(min=0.0))
    off = torch.stack((r * st * torch.cos(phi), r * st * torch.sin(phi), r * cz))
    pos = torch.cat((u(3, n_u), centre[:, which] + off), dim=1)
    mass = (m / n) / k
    a = torch.cat((torch.full((n_u,), 1.0 / n / _params(case)["x_r"] ** 2, dtype=torch.float64, device=dev),
                   mass * r / (r * r + b * b) ** 1.5))
    order = torch.argsort(u(n))
    pos = pos[:, order]
    pos = pos - torch.floor(pos)
    pos = torch.where(pos >= 1.0, torch.zeros_like(pos), pos)
    return pos.contiguous(), a[order].contiguous()


def _time_step(case, a):
    """dt for which 99% of the particles sit on rung 0, from the acceleration estimate."""
    q99 = torch.sort(a).values[int(0.99 * (a.numel() - 1))]
    return math.sqrt(2.0 * ETA * _params(case)["eps"] / float(q99))


def _momenta(case, seed, dt, dtype):
    """Thermal momenta that move a particle by a tenth of the softening length per step."""
    g = _generator(seed * 7919 + 17)
    q = torch.randn(3, case["n"], generator=g, device=_device(), dtype=torch.float64)
    return (q * (0.1 * _params(case)["eps"] / dt)).to(dtype).contiguous()


def _subtile_ids(case, pos):
    """Subtile ids in walk order: tiles of side >= x_r, n_sub subtiles per tile and dimension."""
    n_t, ns = int(math.floor(1.0 / _params(case)["x_r"])), case["n_sub"]
    m = n_t * ns
    gx, gy, gz = (pos * float(m)).floor().to(torch.int64).clamp_(max=m - 1)
    tile = (gx // ns * n_t + gy // ns) * n_t + gz // ns
    return (tile * ns ** 3) + ((gx % ns) * ns + gy % ns) * ns + gz % ns


def _inputs(case, seed):
    """Everything a case's program has in hand, as tensors, from the seed alone."""
    kind, n, dev = case["kind"], case["n"], _device()
    pos, a = _particles(case, seed)
    g = _generator(seed * 104729 + 3)
    x = {"pos": pos}
    if kind in ("step", "substep"):
        dt = _time_step(case, a)
        x["mom"] = _momenta(case, seed, dt, torch.float32 if case["precision"] == 32 else torch.float64)
        if kind == "substep":  # a global step that puts 1% of the particles on the deepest rung
            dt *= 64.0
            s = dt * torch.sqrt(a / (2.0 * ETA * _params(case)["eps"]))
            x["rung"] = torch.ceil(torch.log2(s)).clamp_(0, N_RUNG - 1).to(torch.int8)
        x["dt"] = dt
    elif kind == "vjp":
        dt = torch.float32 if case["precision"] == 32 else torch.float64
        x["acc_bar"] = torch.randn(3, n, generator=g, device=dev, dtype=torch.float64).to(dt)
    elif kind == "reorder":
        x["dt"] = _time_step(case, a) * 64.0
        x["mom"] = _momenta(case, seed, x["dt"], torch.float64)
        d = torch.randn(3, n, generator=g, device=dev, dtype=torch.float64)
        x["acc"] = (d / d.norm(dim=0) * a).to(torch.float32).contiguous()
        x["rung"] = torch.randint(0, N_RUNG, (n,), generator=g, device=dev, dtype=torch.int32).to(torch.int8)
        x["ids"] = torch.arange(n, device=dev, dtype=torch.int64)
    elif kind == "leapfrog":
        x["dt"] = _time_step(case, a)
        x["mom"] = _momenta(case, seed, x["dt"], torch.float64)
        x["x_bar"] = torch.randn(3, n, generator=g, device=dev, dtype=torch.float64)
        x["q_bar"] = torch.randn(3, n, generator=g, device=dev, dtype=torch.float64)
    elif kind == "mesh":
        x["pos"] = pos[:, torch.argsort(_subtile_ids({**case, "n_sub": 2}, pos), stable=True)].contiguous()
        dt = torch.float32 if case["precision"] == 32 else torch.float64
        if case["accumulate"]:
            x["acc"] = torch.randn(3, n, generator=g, device=dev, dtype=torch.float64).to(dt)
    return x


def prepare(case, seed):
    st = {"case": case, **_inputs(case, seed)}
    p, kind, n = _params(case), case["kind"], case["n"]
    if kind == "mesh":
        st["lr"] = LongRange(n, case["n_phi"], 1.25 / case["n_phi"], p["G_m"], p_i=case["p_i"], p_d=case["p_d"],
                             precision=case["precision"])
        st["out"] = torch.empty(3, n, dtype=st["lr"].dtype, device=st["pos"].device)
        return st
    st["sr"] = ShortRange(n, p["x_s"], p["x_r"], p["G_m"], softening=case.get("softening", "bspline"), eps=p["eps"],
                          n_sub=case["n_sub"], n_rung=N_RUNG, symmetric=case.get("symmetric", True))
    for name in ("pos", "mom", "rung", "ids", "acc"):  # the second set of arrays the sort writes into
        if kind in ("step", "substep", "vjp", "reorder") and name in st:
            st[name + "_sorted"] = torch.empty_like(st[name])
    if kind in ("step", "substep", "vjp"):
        st["out"] = torch.zeros(3, n, dtype=torch.float32 if case["precision"] == 32 else torch.float64,
                                device=st["pos"].device)
    if kind == "vjp":
        st["acc_bar_sorted"] = torch.empty_like(st["acc_bar"])
        st["pos_bar"] = torch.empty_like(st["out"])
    if kind == "substep":
        st["kick"] = [st["dt"] / 2.0 ** l for l in range(N_RUNG)]
    if kind == "reorder":
        st["kick"] = [st["dt"] / 2.0 ** l for l in range(N_RUNG)]
        st["rung_new"] = torch.empty_like(st["rung"])
    if kind == "leapfrog":
        st["pos"].requires_grad_(True)
        st["mom"].requires_grad_(True)
    return st


# ---------------------------------------------------------------------------
# One pass.
# ---------------------------------------------------------------------------

def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "mesh":
        if case["accumulate"]:
            st["out"].copy_(st["acc"])
        return st["lr"].accel(st["pos"], st["out"], accumulate=case["accumulate"])
    sr = st["sr"]
    if kind == "accel":
        return short_range_accel(st["pos"], sr, case["precision"])
    if kind == "leapfrog":
        x, q = leapfrog(st["pos"], st["mom"], sr, st["dt"], n_steps=case["n_steps"],
                        checkpoint_every=case["checkpoint_every"], precision=case["precision"])
        gx, gq = torch.autograd.grad((x, q), (st["pos"], st["mom"]), (st["x_bar"], st["q_bar"]))
        return {"x": x, "q": q, "x_grad": gx, "q_grad": gq}
    pos = st["pos_sorted"]
    if kind == "reorder":
        carried = ("mom", "acc", "rung", "ids")
        sr.sort_into(st["pos"], pos, [st[c] for c in carried], [st[c + "_sorted"] for c in carried])
        sr.kick_drift(pos, st["mom_sorted"], st["acc_sorted"], st["rung_new"], st["dt"], ETA, _params(case)["eps"],
                      st["kick"], st["dt"])
        return {"pos": pos, "rung_new": st["rung_new"], **{c: st[c + "_sorted"] for c in carried}}
    if kind == "vjp":
        sr.sort_into(st["pos"], pos, [st["acc_bar"]], [st["acc_bar_sorted"]])
        sr.build_pairs()
        sr.forces(pos, case["precision"], st["out"])
        sr.vjp(pos, st["acc_bar_sorted"], case["precision"], st["pos_bar"])
        return {"pos": pos, "acc": st["out"], "pos_bar": st["pos_bar"]}
    if kind == "step":
        sr.sort_into(st["pos"], pos, [st["mom"]], [st["mom_sorted"]])
        sr.build_pairs()
        sr.forces(pos, case["precision"], st["out"])
        sr.kick(st["mom_sorted"], st["out"], [st["dt"]])
        sr.drift(pos, st["mom_sorted"], st["dt"])
        return {"pos": pos, "mom": st["mom_sorted"], "acc": st["out"]}
    sr.sort_into(st["pos"], pos, [st["mom"], st["rung"]], [st["mom_sorted"], st["rung_sorted"]])
    sr.build_pairs(st["rung_sorted"], case["rung_min"])
    sr.forces(pos, case["precision"], st["out"])
    sr.kick(st["mom_sorted"], st["out"], st["kick"], st["rung_sorted"], case["rung_min"])
    sr.drift(pos, st["mom_sorted"], st["dt"] / 2.0 ** (N_RUNG - 1))
    return {"pos": pos, "mom": st["mom_sorted"], "rung": st["rung_sorted"], "acc": st["out"]}


# ---------------------------------------------------------------------------
# What a pass cannot do without.
# ---------------------------------------------------------------------------

def _pairs_per_particle(case):
    """Interacting ordered pairs per particle, from the recipe: the mean density, plus the
    partners in a clustered particle's own sphere (a fixed sample of pair distances)."""
    n, x_r = case["n"], _params(case)["x_r"]
    rng = np.random.default_rng(0)
    side = n ** (1.0 / 3.0)
    m = 4000

    def points():
        w = rng.uniform(1e-12, 1.0, m)
        r = 1.0 / np.sqrt(w ** (-2.0 / 3.0) - 1.0)
        d = rng.normal(size=(3, m))
        return r * d / np.linalg.norm(d, axis=0)

    b = case["b_lo"] / side * np.exp(rng.uniform(size=m) * math.log(case["b_hi"] / case["b_lo"]))
    near = np.mean(np.linalg.norm(points() - points(), axis=0) * b < x_r)
    f = 1.0 - case["frac_uniform"]
    per_sphere = f * n / max(1, int(f * n) // case["per_sphere"])
    return n * 4.0 / 3.0 * math.pi * x_r ** 3 + f * per_sphere * near


def work(case):
    kind, n = case["kind"], case["n"]
    real = 8 if case.get("precision", 64) == 64 else 4
    if kind == "mesh":
        p, mesh = case["p_i"], case["n_phi"] ** 3
        flops = n * (p ** 3 * 2 + 3 * p * p * (p + case["p_d"]) * 2) + 2 * 2.5 * mesh * math.log2(mesh) + 4 * mesh
        return {"bytes": n * (24 + 3 * real * (2 if case["accumulate"] else 1)), "flops": flops}
    if kind == "reorder":
        return {"bytes": n * (2 * (24 + 24 + 12 + 1 + 8) + 1), "flops": n * 24}
    pairs = n * _pairs_per_particle(case)
    forward, adjoint = 26.0, 38.0  # arithmetic operations of one interacting pair
    if kind == "accel":
        return {"bytes": n * (24 + 3 * real), "flops": forward * pairs}
    if kind == "step":
        return {"bytes": n * (2 * (24 + 3 * real) + 3 * real), "flops": forward * pairs + 24 * n}
    if kind == "substep":
        share = (1.0, 0.7, 0.69, 0.67, 0.56, 0.35, 0.16, 0.01)[case["rung_min"]]  # receivers, from the recipe
        return {"bytes": n * (2 * (24 + 3 * real + 1) + 3 * real * share), "flops": forward * pairs * share + 24 * n}
    if kind == "vjp":
        return {"bytes": n * (2 * 24 + 3 * 3 * real), "flops": (forward + adjoint) * pairs}
    evaluations = case["n_steps"] + 1
    return {"bytes": n * 8 * 24, "flops": evaluations * (forward + adjoint) * pairs}


# ---------------------------------------------------------------------------
# The same in 64 bits, in plain torch.
# ---------------------------------------------------------------------------

def _bracket(r2, case):
    """B(r) and B'(r)/r of the short-range force, softening included."""
    p = _params(case)
    x_s, eps, soft = p["x_s"], p["eps"], case.get("softening", "bspline")
    r = torch.sqrt(r2)
    u = r / (2.0 * x_s)
    zero = r2 == 0
    rs = torch.where(zero, torch.ones_like(r), r)
    e = torch.exp(-u * u)
    root_pi = math.sqrt(math.pi)
    B = (torch.erfc(u) + 2.0 / root_pi * u * e) / rs ** 3
    D = -(3.0 * B + e / (2.0 * root_pi * x_s ** 3)) / rs ** 2
    if soft == "none":
        return torch.where(zero, torch.zeros_like(B), B), torch.where(zero, torch.zeros_like(D), D)
    # below 2.8 eps: B = shape - h(u) / (2 x_s)^3 without the cancellation against r^-3
    near = r < 2.8 * eps
    u2 = u * u
    h, hd, fact = torch.zeros_like(u), torch.zeros_like(u), 1.0
    pw = torch.ones_like(u)
    prev = None
    for m in range(19):
        fact *= m + 1
        H = 2.0 / root_pi * (-1.0) ** m * 2.0 * (m + 1) / (fact * (2.0 * m + 3.0))
        if m < 18:
            h = h + H * pw
        if prev is not None:
            hd = hd + 2.0 * m * H * prev
        prev, pw = pw, pw * u2
    w = 2.0 * x_s
    if soft == "plummer":
        s = r2 + eps * eps
        s3, ds = s ** -1.5, -3.0 * s ** -2.5
        far_B, far_D = B + (s3 - rs ** -3), D + (ds + 3.0 * rs ** -5)
    else:
        eb = 2.8 * eps
        x = rs / eb
        c, ce = 32.0 / eb ** 3, 32.0 / eb ** 5
        x0 = torch.where(zero, torch.zeros_like(x), x)
        inner = x0 < 0.5
        xo = torch.where(inner, torch.ones_like(x), x)
        s3 = torch.where(inner, c * (x0 ** 3 - 1.2 * x0 ** 2 + 1.0 / 3.0),
                         c * (-xo ** 3 / 3.0 + 1.2 * xo ** 2 - 1.5 * xo + 2.0 / 3.0 - 1.0 / (480.0 * xo ** 3)))
        ds = torch.where(inner, ce * (3.0 * x0 - 2.4), ce * (-xo + 2.4 - 1.5 / xo + 1.0 / (160.0 * xo ** 5)))
        far_B, far_D = B, D
    return torch.where(near, s3 - h / w ** 3, far_B), torch.where(near, ds - hd / w ** 5, far_D)


def _segment_sums(v, hit, counts):
    """Row sums of the ragged rows of lengths `counts` over the entries where `hit`; v (3, hits)."""
    seen = torch.cat((torch.zeros(1, dtype=torch.int64, device=hit.device), torch.cumsum(hit, 0)))
    ends = torch.cumsum(counts, 0)
    lengths = seen[ends] - seen[ends - counts]
    return torch.segment_reduce(v.t().contiguous(), "sum", lengths=lengths, axis=0).t()


def _pair_sums(case, pos, acc_bar=None, receivers=None, forward=True):
    """Short-range accelerations (3, n) and, with acc_bar, the vector-Jacobian product, in the
    order of pos: every particle against the 27 cells (of side >= x_r) around it."""
    p, n, dev = _params(case), pos.shape[1], pos.device
    x_r = p["x_r"]
    n_t = int(math.floor(1.0 / x_r))
    c = (pos * n_t).floor().to(torch.int64).clamp_(max=n_t - 1)
    order = torch.argsort((c[0] * n_t + c[1]) * n_t + c[2])
    c, xs = c[:, order], pos[:, order].contiguous()
    ab = None if acc_bar is None else acc_bar.to(torch.float64)[:, order].contiguous()
    start = torch.searchsorted((c[0] * n_t + c[1]) * n_t + c[2],
                               torch.arange(n_t ** 3 + 1, device=dev, dtype=torch.int64))
    rows = torch.arange(n, device=dev)
    if receivers is not None:
        rows = rows[receivers[order]]
    acc = torch.zeros(3, n, dtype=torch.float64, device=dev)
    bar = torch.zeros(3, n, dtype=torch.float64, device=dev)
    most = 48_000_000 if dev.type == "cuda" else 1_000_000
    for o in range(27):
        d = (o // 9 - 1, o // 3 % 3 - 1, o % 3 - 1)
        q = [c[k][rows] + d[k] for k in range(3)]
        shift = torch.stack([torch.where(v < 0, -1.0, torch.where(v >= n_t, 1.0, 0.0)) for v in q]).to(torch.float64)
        cell = (q[0] % n_t * n_t + q[1] % n_t) * n_t + q[2] % n_t
        first, counts = start[cell], start[cell + 1] - start[cell]
        total = torch.cumsum(counts, 0).cpu().numpy()
        lo = 0
        while lo < rows.numel():
            base = int(total[lo - 1]) if lo else 0
            hi = max(lo + 1, int(np.searchsorted(total, base + most, side="right")))
            k = counts[lo:hi]
            size = int(total[hi - 1]) - base
            if size > 0:
                row = torch.repeat_interleave(torch.arange(lo, hi, device=dev), k, output_size=size)
                ends = torch.cumsum(k, 0)
                j = first[row] + torch.arange(size, device=dev) - (ends - k)[row - lo]
                i = rows[row]
                dx = torch.stack([xs[m][i] - (xs[m][j] + shift[m][row]) for m in range(3)])
                r2 = dx[0] * dx[0] + dx[1] * dx[1] + dx[2] * dx[2]
                hit = (r2 < x_r * x_r) & (i != j)
                dx, r2, i, j = dx[:, hit], r2[hit], i[hit], j[hit]
                B, D = _bracket(r2, case)
                here = rows[lo:hi]
                if forward:
                    acc[:, here] += _segment_sums(B * dx, hit, k)
                if ab is not None:
                    v = ab[:, i] - ab[:, j]
                    t = B * v + D * (dx * v).sum(0) * dx
                    bar[:, here] += _segment_sums(t, hit, k)
            lo = hi
    back = torch.empty_like(order)
    back[order] = torch.arange(n, device=dev)
    return -p["G_m"] * acc[:, back], -p["G_m"] * bar[:, back]


def _wrapped(x):
    y = x - torch.floor(x)
    return torch.where(y >= 1.0, torch.zeros_like(y), y)


def _exact_leapfrog(case, x):
    """Kick-drift-kick steps and their adjoint, state by state."""
    dt, steps = x["dt"], case["n_steps"]
    pos, mom = x["pos"], x["mom"]
    trail = [pos]
    a, _ = _pair_sums(case, pos)
    for _ in range(steps):
        mom = mom + 0.5 * dt * a
        pos = _wrapped(pos + dt * mom)
        a, _ = _pair_sums(case, pos)
        mom = mom + 0.5 * dt * a
        trail.append(pos)
    x_bar, q_bar = x["x_bar"], x["q_bar"]
    a_bar = torch.zeros_like(q_bar)
    for s in range(steps, 0, -1):
        a_bar = a_bar + 0.5 * dt * q_bar
        x_bar = x_bar + _pair_sums(case, trail[s], a_bar, forward=False)[1]
        q_bar = q_bar + dt * x_bar
        a_bar = 0.5 * dt * q_bar
    x_bar = x_bar + _pair_sums(case, trail[0], a_bar, forward=False)[1]
    return {"x": pos, "q": mom, "x_grad": x_bar, "q_grad": q_bar}


def _exact_mesh(case, x):
    n, pos, p_i, p_d = case["n_phi"], x["pos"], case["p_i"], case["p_d"]
    h, dev = 1.0 / n, pos.device
    s = pos * n - 0.5
    base = torch.floor(s + 0.5) - (p_i - 1) // 2 if p_i % 2 else torch.floor(s) - (p_i // 2 - 1)
    cells = base[:, :, None] + torch.arange(p_i, device=dev, dtype=torch.float64)
    t = (cells - s[:, :, None]).abs()
    if p_i == 1:
        w = torch.ones_like(t)
    elif p_i == 2:
        w = 1.0 - t
    elif p_i == 3:
        w = torch.where(t < 0.5, 0.75 - t * t, (2.0 * t - 3.0) ** 2 / 8.0)
    else:
        w = torch.where(t < 1.0, (3.0 * t ** 3 - 6.0 * t * t + 4.0) / 6.0, (2.0 - t) ** 3 / 6.0)
    cells = cells.to(torch.int64) % n
    places = [(a, b, c) for a in range(p_i) for b in range(p_i) for c in range(p_i)]

    def flat(a, b, c):
        return (cells[0, :, a] * n + cells[1, :, b]) * n + cells[2, :, c]

    rho = torch.zeros(n ** 3, dtype=torch.float64, device=dev)
    for a, b, c in places:
        rho.index_add_(0, flat(a, b, c), w[0, :, a] * w[1, :, b] * w[2, :, c])
    k = 2.0 * math.pi * torch.fft.fftfreq(n, 1.0 / n, dtype=torch.float64, device=dev)
    kz = k[: n // 2 + 1].abs()
    x_s = 1.25 / n

    def factor(v):
        return torch.sinc(v * h / (2.0 * math.pi)) ** (-2 * p_i) * torch.exp(-x_s * x_s * v * v)

    k2 = k[:, None, None] ** 2 + k[None, :, None] ** 2 + kz[None, None, :] ** 2
    k2[0, 0, 0] = 1.0
    green = factor(k)[:, None, None] * factor(k)[None, :, None] * factor(kz)[None, None, :] / k2
    green[0, 0, 0] = 0.0
    phi = torch.fft.irfftn(torch.fft.rfftn(rho.view(n, n, n)) * green, s=(n, n, n))
    weights = {2: [1 / 2], 4: [8 / 12, -1 / 12], 6: [45 / 60, -9 / 60, 1 / 60],
               8: [672 / 840, -168 / 840, 32 / 840, -3 / 840]}[p_d]
    out = []
    for axis in range(3):
        f = torch.zeros_like(phi)
        for q, cq in enumerate(weights, 1):
            f += cq * (torch.roll(phi, -q, axis) - torch.roll(phi, q, axis))
        f = f.reshape(-1)
        out.append(sum(w[0, :, a] * w[1, :, b] * w[2, :, c] * f[flat(a, b, c)] for a, b, c in places))
    acc = 4.0 * math.pi * _params(case)["G_m"] / h ** 4 * torch.stack(out)
    return acc + x["acc"].to(torch.float64) if case["accumulate"] else acc


def exact(case, seed):
    kind = case["kind"]
    x = _inputs(case, seed)
    if kind == "mesh":
        return _exact_mesh(case, x)
    if kind == "leapfrog":
        return _exact_leapfrog(case, x)
    if kind == "accel":
        return _pair_sums(case, x["pos"])[0]
    order = torch.argsort(_subtile_ids(case, x["pos"]), stable=True)
    pos = x["pos"][:, order].contiguous()
    if kind == "vjp":
        acc, bar = _pair_sums(case, pos, x["acc_bar"][:, order])
        return {"pos": None, "acc": acc, "pos_bar": bar}
    mom = x["mom"][:, order].to(torch.float64)
    if kind == "reorder":
        acc = x["acc"][:, order].to(torch.float64)
        q = x["dt"] ** 2 / (2.0 * ETA * _params(case)["eps"])
        s = q * q * (acc * acc).sum(0)
        rung = torch.zeros(case["n"], dtype=torch.int64, device=pos.device)
        for l in range(N_RUNG - 1):
            rung += (s > 16.0 ** l).to(torch.int64)
        mom = mom + acc * (x["dt"] / 2.0 ** rung.to(torch.float64))
        return {"pos": _wrapped(pos + mom * x["dt"]), "rung_new": None, "mom": mom, "acc": None, "rung": None,
                "ids": None}
    if kind == "step":
        acc = _pair_sums(case, pos)[0]
        mom = mom + acc * x["dt"]
        return {"pos": _wrapped(pos + mom * x["dt"]), "mom": mom, "acc": acc}
    rung = x["rung"][order]
    due = rung >= case["rung_min"]
    acc = torch.where(due, _pair_sums(case, pos, receivers=due)[0], 0.0)
    mom = torch.where(due, mom + acc * (x["dt"] / 2.0 ** rung.to(torch.float64)), mom)
    return {"pos": _wrapped(pos + mom * (x["dt"] / 2.0 ** (N_RUNG - 1))), "mom": mom, "rung": None, "acc": acc}
