"""The work that users of this framework have it do, as measured cases.

A case is a plain dict; its "kind" says which public entry points of
paper_2011_14984_gb300.frost one pass calls, the rest are sizes and options:

  step    set_state, step, state: one top-level step of the integrator from a given state
          (snapshot in, snapshot out), the call that a simulation spends its time in
  batch   the same on a context of independent clusters (one launch for all of them)
  accel   accel_gradient of a set due to itself: accelerations, a~ and the gradient, the
          force evaluation of an integrator of one's own
  kick    accel_gradient_pairwise of two disjoint lists: the kick between a slow and a fast set
  newton  accel_gradient with the accelerations alone, of an index list due to itself
  level   timesteps of an index list, then its partition by a pivot step: one hierarchy level
  energy  energy, momentum and angular momentum, the diagnostics between snapshots

Systems are the generators' Plummer spheres (equal masses, a Kroupa mass spectrum, or that with
5 % of the stars in hard binaries), sizes those of the benchmark configurations (1024, 65536,
262144, the batch of 256 clusters) and of the hierarchy levels inside a 65536-body step, with
odd sizes and unsorted index lists in between.
"""

import math

import numpy as np
import torch

from paper_2011_14984_gb300 import ics
from paper_2011_14984_gb300.frost import (FROST_FLYBY_EXACT, FROST_SYM_ARITHMETIC,
                                          FROST_SYM_HARMONIC, Frost)

ETA = 0.2
DT = 2.0 ** -7      # the benchmark's top-level step
EPS_GRAD = 2.0 ** -7
SYMS = {"harmonic": FROST_SYM_HARMONIC, "arithmetic": FROST_SYM_ARITHMETIC,
        "flyby": FROST_SYM_HARMONIC | FROST_FLYBY_EXACT}


def listed():
    return [
        # the smallest system: an open cluster's core, every step one launch of the solver
        {"name": "step_64", "kind": "step", "n": 64, "precision": "mixed", "masses": "kroupa"},
        # a small cluster: a few grid levels above the solver, all of them latency
        {"name": "step_1k", "kind": "step", "n": 1024, "precision": "mixed", "masses": "equal"},
        # the benchmark's headline step
        {"name": "step_64k", "kind": "step", "n": 65536, "precision": "mixed", "masses": "equal"},
        # the same small cluster in the reference precision
        {"name": "step_1k_fp64", "kind": "step", "n": 1024, "precision": "fp64", "masses": "equal"},
        # an ensemble of independent clusters of 64 to 4096 stars
        {"name": "batch_256", "kind": "batch", "clusters": 256, "n_max": 4096, "precision": "mixed"},
        # one full force evaluation at the benchmark's size
        {"name": "accel_64k", "kind": "accel", "n": 65536, "precision": "mixed", "masses": "equal", "eps": 0.0},
        # and of a large cluster with a mass spectrum and hard binaries
        {"name": "accel_256k_binaries", "kind": "accel", "n": 262144, "precision": "mixed",
         "masses": "binaries", "eps": 0.0},
        # the reference precision, of a set that fills no tile evenly, softened
        {"name": "accel_8k_fp64", "kind": "accel", "n": 8191, "precision": "fp64", "masses": "kroupa", "eps": 1e-3},
        # the kick between the slow and the fast set of a middle level of the headline step
        {"name": "kick_17k_6k", "kind": "kick", "n": 16717, "n_b": 6101, "precision": "mixed",
         "masses": "equal", "eps": 0.0},
        # a small list inside a larger system: launches and latency count
        {"name": "newton_3001", "kind": "newton", "n": 3001, "precision": "mixed", "masses": "kroupa", "eps": 0.0},
        # the time-steps and the partition of the headline step's second level
        {"name": "level_40k", "kind": "level", "n": 40603, "precision": "mixed", "masses": "equal",
         "sym": "harmonic"},
        # diagnostics of the headline system
        {"name": "energy_64k", "kind": "energy", "n": 65536, "precision": "mixed", "masses": "equal"},
    ]


def _log_size(rng, lo, hi):
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return min(max(n, lo), hi)


def draw(rng):
    kind = rng.choice(["step", "step", "batch", "accel", "accel", "kick", "newton", "level", "level", "energy"])
    precision = rng.choice(["mixed", "mixed", "mixed", "fp64"])
    top = 65536 if precision == "mixed" else 8192
    masses = rng.choice(["equal", "kroupa"])
    eps = rng.choice([0.0, 0.0, 1e-3])
    if kind == "step":
        return {"kind": kind, "n": _log_size(rng, 64, 65536 if precision == "mixed" else 2048),
                "precision": precision, "masses": masses}
    if kind == "batch":
        # an ensemble's sizes as listed; fewer clusters, and smaller ones in FP64
        return {"kind": kind, "clusters": _log_size(rng, 8, 256), "n_max": 4096 if precision == "mixed" else 512,
                "precision": precision}
    if kind == "accel":
        return {"kind": kind, "n": _log_size(rng, 300, 4 * top if precision == "mixed" else top),
                "precision": precision, "masses": rng.choice(["equal", "kroupa", "binaries"]), "eps": eps}
    if kind == "kick":
        return {"kind": kind, "n": _log_size(rng, 60, top), "n_b": _log_size(rng, 60, top // 2),
                "precision": precision, "masses": masses, "eps": eps}
    if kind == "newton":
        return {"kind": kind, "n": _log_size(rng, 300, top), "precision": precision, "masses": masses, "eps": eps}
    if kind == "level":
        return {"kind": kind, "n": _log_size(rng, 300, top), "precision": precision, "masses": masses,
                "sym": rng.choice(["harmonic", "harmonic", "arithmetic", "flyby"])}
    return {"kind": "energy", "n": _log_size(rng, 300, 65536), "precision": precision, "masses": masses}


def _stars(n, masses, seed):
    if masses == "binaries":
        return ics.plummer_kroupa_binaries(n, seed)
    return ics.plummer(n, seed, ics.kroupa_masses(n, seed) if masses == "kroupa" else None)


def _system(case, seed):
    """Masses, positions, velocities and the case's index lists (host arrays)."""
    kind = case["kind"]
    rng = np.random.default_rng(seed + 17)
    if kind == "kick":
        n, nb = case["n"], case["n_b"]
        m, x, v = _stars(n + nb, case["masses"], seed)
        # the fast set is the centre, as in the hierarchy: the nb innermost stars
        order = np.argsort((x * x).sum(axis=1), kind="stable")
        return m, x, v, (rng.permutation(order[nb:]).astype(np.int32), np.sort(order[:nb]).astype(np.int32))
    if kind in ("newton", "level"):
        # a list of n particles of a somewhat larger system, in no order
        n = case["n"]
        total = n + n // 4 + 1
        m, x, v = _stars(total, case["masses"], seed)
        return m, x, v, (rng.permutation(total)[:n].astype(np.int32),)
    m, x, v = _stars(case["n"], case["masses"], seed)
    if kind == "energy":
        # on its way through a galaxy: P and L are not sums that cancel to nothing
        x, v = x + np.array([1.0, 0.0, 0.5]), v + np.array([0.1, 0.2, 0.05])
    return m, x, v, ()


def prepare(case, seed):
    kind, precision = case["kind"], case["precision"]
    if kind == "batch":
        # the batch workload's log-uniform sizes; the stars of every cluster from the seed
        u = np.random.default_rng(1000).random(case["clusters"])
        sizes = np.floor(64.0 * (case["n_max"] / 64.0) ** u).astype(np.int64)
        offsets = np.concatenate([[0], np.cumsum(sizes)])
        parts = [ics.plummer(int(n), 1000 * seed + k) for k, n in enumerate(sizes)]
        m, x, v = (np.concatenate([p[c] for p in parts]) for c in range(3))
        f = Frost(m, x, v, eta=ETA, precision=precision, offsets=offsets)
        return {"case": case, "f": f, "x": x, "v": v}
    m, x, v, lists = _system(case, seed)
    f = Frost(m, x, v, eta=ETA, precision=precision, eps_soft=case.get("eps", 0.0),
              sym=SYMS[case.get("sym", "harmonic")])
    state = {"case": case, "f": f, "lists": [torch.from_numpy(k).cuda() for k in lists]}
    if kind == "step":
        # a program's host copy of the snapshot
        state["x"], state["v"] = x, v
    if kind == "level":
        # a pivot among the set's steps, as a level of the hierarchy has it: about two in
        # three particles are slow
        tau = f.timesteps(state["lists"][0])
        state["pivot"] = float(torch.quantile(tau[: 1 << 20], 0.35))
    return state


def _kept(case, out):
    # mixed mode gives forces to about 1e-7 of their size, and a program keeps them as what
    # they are, 32-bit values; in FP64 mode it keeps 64 bits
    return {k: t.float() if case["precision"] == "mixed" else t for k, t in out.items()}


def run(state):
    case, f = state["case"], state["f"]
    kind = case["kind"]
    if kind in ("step", "batch"):
        f.set_state(state["x"], state["v"], 0.0)
        f.step(DT, 1)
        x, v, t = f.state()
        return {"x": x, "v": v, "t": t}
    if kind == "accel":
        return _kept(case, f.accel_gradient(eps_grad=EPS_GRAD))
    if kind == "kick":
        a, b = state["lists"]
        return _kept(case, f.accel_gradient_pairwise(a, b, EPS_GRAD))
    if kind == "newton":
        k = state["lists"][0]
        return _kept(case, f.accel_gradient(k, k, want=("acc",)))
    if kind == "level":
        k = state["lists"][0]
        tau = f.timesteps(k)
        slow, fast = f.partition(k, tau, state["pivot"])
        # the set in its new order, the slow ones first
        return {"tau": tau, "order": torch.cat([slow, fast]), "n_slow": int(slow.numel())}
    return f.energy()


def work(case):
    """Algorithmic work of a pass: 20 flops a Newtonian, 38 a gradient and 45 a time-step
    interaction, and every particle's input and output once in the types of the interface."""
    kind = case["kind"]
    if kind == "batch":
        # the sizes are log-uniform in [64, n_max]: their second moment
        top = case["n_max"]
        pairs = case["clusters"] * (top ** 2 - 64 ** 2) / (2 * math.log(top / 64))
        mean = (top - 64) / math.log(top / 64)
        return {"bytes": 104.0 * case["clusters"] * mean, "flops": 143.0 * pairs}
    n = case["n"]
    pairs = float(n) * (n - 1)
    if kind == "step":
        # whatever the hierarchy, a pair takes part in at least one time-step criterion, three
        # Newtonian kicks and one gradient per top-level step
        return {"bytes": 104.0 * n, "flops": 143.0 * pairs}
    if kind == "accel":
        return {"bytes": (32.0 + 72.0) * n, "flops": 58.0 * pairs}
    if kind == "kick":
        return {"bytes": (32.0 + 72.0) * (n + case["n_b"]), "flops": 58.0 * 2.0 * n * case["n_b"]}
    if kind == "newton":
        return {"bytes": (36.0 + 24.0) * n, "flops": 20.0 * pairs}
    if kind == "level":
        # the criteria of a pair serve both of its particles
        more = 20.0 if case["sym"] == "flyby" else 0.0
        return {"bytes": (60.0 + 8.0 + 4.0) * n, "flops": (45.0 / 2 + more) * pairs}
    return {"bytes": 56.0 * n, "flops": 10.0 * pairs / 2}


# ---- the same results in 64 bits, by plain torch -------------------------------------------

_ROWS = 1 << 25  # pairs in flight


def _pairs(x, i0, i1, y, eps):
    """Separations y_j - x_i and r^2 of the rows i0 .. i1."""
    d = [y[None, :, c] - x[i0:i1, None, c] for c in range(3)]
    return d, d[0] * d[0] + d[1] * d[1] + d[2] * d[2] + eps * eps


def _no_self(r2, i0, same):
    if same:
        k = torch.arange(r2.shape[0], device=r2.device)
        r2[k, k + i0] = math.inf


def _acc(x, y, my, eps, same):
    out = torch.empty_like(x)
    step = max(1, _ROWS // y.shape[0])
    for i0 in range(0, x.shape[0], step):
        i1 = min(x.shape[0], i0 + step)
        d, r2 = _pairs(x, i0, i1, y, eps)
        _no_self(r2, i0, same)
        w = my[None, :] / (r2 * r2.sqrt())
        for c in range(3):
            out[i0:i1, c] = (w * d[c]).sum(dim=1)
    return out


def _grad(x, ax, y, my, ay, eps, same):
    out = torch.empty_like(x)
    step = max(1, _ROWS // y.shape[0])
    for i0 in range(0, x.shape[0], step):
        i1 = min(x.shape[0], i0 + step)
        d, r2 = _pairs(x, i0, i1, y, eps)
        _no_self(r2, i0, same)
        a = [ay[None, :, c] - ax[i0:i1, None, c] for c in range(3)]
        w = 2.0 * my[None, :] / (r2 * r2.sqrt())
        q = 3.0 * (d[0] * a[0] + d[1] * a[1] + d[2] * a[2]) / r2
        for c in range(3):
            out[i0:i1, c] = (w * (a[c] - q * d[c])).sum(dim=1)
    return out


def _factor(d, sym):
    if sym == "arithmetic":
        return torch.where(d < 2.0, 1.0 / (1.0 - 0.5 * d.clamp(max=1.999)), 2.0 / d.clamp(min=2.0))
    q = 1.0 + (1.0 + d * d).sqrt()
    return torch.where(d >= 0.0, (q + d) / q, 2.0 / (q - d))


def _tau(m, x, v, sym):
    n = x.shape[0]
    a = _acc(x, x, m, 0.0, True) if sym == "flyby" else None
    out = torch.empty_like(m)
    step = max(1, _ROWS // n)
    for i0 in range(0, n, step):
        i1 = min(n, i0 + step)
        d, r2 = _pairs(x, i0, i1, x, 0.0)
        _no_self(r2, i0, True)
        u, v2 = _pairs(v, i0, i1, v, 0.0)
        r = r2.sqrt()
        rv = (d[0] * u[0] + d[1] * u[1] + d[2] * u[2]) / r2
        gm = m[i0:i1, None] + m[None, :]
        tff = (r2 * r / gm).sqrt()
        tfb = r / v2.sqrt()
        if sym == "flyby":
            va = sum(u[c] * (a[None, :, c] - a[i0:i1, None, c]) for c in range(3))
            rate = rv - va / v2
        else:
            rate = rv * (1.0 + gm / (v2 * r))
        t = tff * _factor(ETA * 1.5 * rv * tff, sym)
        tb = tfb * _factor(ETA * rate * tfb, sym)
        t = torch.fmin(t, tb)
        _no_self(t, i0, True)
        out[i0:i1] = ETA * t.min(dim=1).values
    return out


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def exact(case, seed):
    kind = case["kind"]
    if kind in ("step", "batch"):
        return None  # a whole integration
    m, x, v, lists = _system(case, seed)
    eps = case.get("eps", 0.0)
    if kind == "kick":
        (xa, ma), (xb, mb) = [(_dev(x[k]), _dev(m[k])) for k in lists]
        a = _acc(xa, xb, mb, eps, False)
        b = _acc(xb, xa, ma, eps, False)
        ga = _grad(xa, a, xb, mb, b, eps, False)
        gb = _grad(xb, b, xa, ma, a, eps, False)
        c = EPS_GRAD ** 2 / 48.0
        return {"acc_a": a, "acc_b": b, "acc_tilde_a": a + c * ga, "acc_tilde_b": b + c * gb,
                "grad_a": ga, "grad_b": gb}
    if lists:
        m, x, v = m[lists[0]], x[lists[0]], v[lists[0]]
    m, x, v = _dev(m), _dev(x), _dev(v)
    if kind == "level":
        return {"tau": _tau(m, x, v, case["sym"]), "order": None, "n_slow": None}
    if kind == "energy":
        pot = 0.0
        step = max(1, _ROWS // x.shape[0])
        for i0 in range(0, x.shape[0], step):
            i1 = min(x.shape[0], i0 + step)
            _, r2 = _pairs(x, i0, i1, x, eps)
            _no_self(r2, i0, True)
            pot = pot + (m[i0:i1] * (m[None, :] / r2.sqrt()).sum(dim=1)).sum()
        kin = 0.5 * (m * (v * v).sum(dim=1)).sum()
        pot = -0.5 * pot
        return {"T": float(kin), "U": float(pot), "E": float(kin + pot), "P": (m[:, None] * v).sum(dim=0),
                "L": (m[:, None] * torch.linalg.cross(x, v)).sum(dim=0)}
    a = _acc(x, x, m, eps, True)
    if kind == "newton":
        return {"acc": a}
    g = _grad(x, a, x, m, a, eps, True)
    return {"acc": a, "acc_tilde": a + EPS_GRAD ** 2 / 48.0 * g, "grad": g}
