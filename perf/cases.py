"""Measured cases of the collision-constraint step, through the package's
public entry points.

A case is a dict of plain values; ``kind`` names the call:

  step    Context.step on one periodic suspension
  springs Context.step with bilateral crosslinker springs set on the context
  batch   Context.step_batch on an ensemble of independent systems
  run     Context.run, a short Brownian trajectory (walls optional)
  grad    autograd.constrained_step, forward and backward
  phases  build_neighbors, assemble_constraints and solve_lcp one by one

``run`` restarts every pass from the prepared positions, so that each pass
does the same work; the two device copies are part of it.
"""
from __future__ import annotations

import math
import time

import numpy as np
import torch

import paper_2109_08206_gb300 as A
from paper_2109_08206_gb300 import workloads as W
from paper_2109_08206_gb300.autograd import constrained_step

DIAMETER, LENGTH, VISCOSITY, DT = 1.0, 10.0, 1.0, 1e-3


def listed():
    return [
        # one small box at a tight tolerance: method development, calibration
        # runs, many short jobs; latency of the iteration and of the launches
        {"name": "step_1k_fp64", "kind": "step", "n": 1000, "phi": 0.1309, "nematic": 0.0, "forces": "unit",
         "crosslinks": 0, "precision": "fp64", "tol": 1e-8, "graph": False, "records": True},
        # one bundle-sized box; contacts, forces and velocities kept for the
        # stress and the contact network
        {"name": "step_20k_mixed", "kind": "step", "n": 20000, "phi": 0.15, "nematic": 0.0, "forces": "thermal",
         "crosslinks": 0, "precision": "mixed", "tol": 1e-5, "graph": False, "records": True},
        # the production step of a cytoskeletal network: explicit crosslinker
        # forces, the step recorded once and replayed
        {"name": "step_100k_mixed", "kind": "step", "n": 100000, "phi": 0.10, "nematic": 0.0, "forces": "thermal",
         "crosslinks": 50000, "precision": "mixed", "tol": 1e-5, "graph": True, "records": False},
        # the same network in plain float64 (validation runs)
        {"name": "step_100k_fp64", "kind": "step", "n": 100000, "phi": 0.10, "nematic": 0.0, "forces": "thermal",
         "crosslinks": 50000, "precision": "fp64", "tol": 1e-5, "graph": False, "records": False},
        # a dense nematic pack, the largest single system
        {"name": "step_400k_nematic_mixed", "kind": "step", "n": 400000, "phi": 0.25, "nematic": 0.1,
         "forces": "thermal", "crosslinks": 0, "precision": "mixed", "tol": 1e-5, "graph": False, "records": False},
        # crosslinkers as bilateral constraints of the same solve
        {"name": "springs_100k_mixed", "kind": "springs", "n": 100000, "phi": 0.10, "springs": 50000,
         "precision": "mixed", "tol": 1e-5},
        # a parameter sweep of uneven nematic domains in one call
        {"name": "batch_256_mixed", "kind": "batch", "count": 256, "scale": 1.0, "precision": "mixed", "tol": 1e-5,
         "graph": True},
        # a handful of small replicas (error bars of one state point)
        {"name": "batch_16_small_mixed", "kind": "batch", "count": 16, "scale": 0.25, "precision": "mixed",
         "tol": 1e-5, "graph": True},
        # a confined pile pushed onto a wall, warm-started step after step
        {"name": "run_1k_walls_mixed", "kind": "run", "n": 1000, "phi": 0.10, "steps": 20, "walls": True,
         "precision": "mixed", "tol": 1e-5},
        # ten Brownian steps of the network
        {"name": "run_100k_mixed", "kind": "run", "n": 100000, "phi": 0.10, "steps": 10, "walls": False,
         "precision": "mixed", "tol": 1e-5},
        # gradient of a loss of the post-step centres (fitting forces, drag)
        {"name": "grad_20k_mixed", "kind": "grad", "n": 20000, "phi": 0.15, "precision": "mixed", "tol": 1e-5},
        # the phases called one by one (own force laws between assembly and solve)
        {"name": "phases_20k_fp64", "kind": "phases", "n": 20000, "phi": 0.15, "precision": "fp64", "tol": 1e-6},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "springs", "batch", "run", "grad", "phases"])
    fp64 = rng.random() < 0.3
    c = {"kind": kind, "precision": "fp64" if fp64 else "mixed"}
    if kind == "step":
        nematic = rng.random() < 0.4
        c["n"] = _log_int(rng, 500, 50_000 if fp64 else 400_000 if nematic else 150_000)
        c["phi"] = round(rng.uniform(0.10, 0.25) if nematic else rng.uniform(0.03, 0.12), 4)
        c["nematic"] = 0.1 if nematic else 0.0
        c["forces"] = "thermal"
        c["crosslinks"] = 0 if nematic or rng.random() < 0.5 else c["n"] // 2
        c["tol"] = rng.choice([1e-5, 1e-6, 1e-8]) if fp64 else 1e-5
        c["graph"] = rng.random() < 0.5
        c["records"] = rng.random() < 0.5
    elif kind == "springs":
        c["precision"] = "mixed"
        c.update(n=_log_int(rng, 1000, 100_000), phi=round(rng.uniform(0.05, 0.12), 4), tol=1e-5)
        c["springs"] = c["n"] // 2
    elif kind == "batch":
        c["precision"] = "mixed"
        c.update(count=_log_int(rng, 2, 256), scale=round(math.exp(rng.uniform(math.log(0.1), 0.0)), 3), tol=1e-5,
                 graph=rng.random() < 0.7)
    elif kind == "run":
        c["precision"] = "mixed"
        c.update(n=_log_int(rng, 500, 100_000), phi=round(rng.uniform(0.05, 0.10), 4), steps=rng.randint(4, 10),
                 walls=rng.random() < 0.4, tol=1e-5)
    elif kind == "grad":
        c.update(n=_log_int(rng, 500, 20_000), phi=round(rng.uniform(0.08, 0.15), 4), tol=1e-6 if fp64 else 1e-5)
    else:
        c.update(n=_log_int(rng, 500, 50_000), phi=round(rng.uniform(0.05, 0.15), 4), tol=1e-6 if fp64 else 1e-5)
    return c


# ------------------------------------------------------------------ inputs

def _suspension(case, seed, forces="thermal", crosslinks=0, nematic=0.0):
    box = W.box_for_fraction(case["n"], DIAMETER, LENGTH, case["phi"])
    return W.random_system(seed, case["n"], box, length=LENGTH, diameter=DIAMETER, viscosity=VISCOSITY, dt=DT,
                           nematic_spread=nematic if nematic > 0 else None, forces=forces, n_springs=crosslinks,
                           tol=case["tol"])


def _inputs(case, seed):
    """The host inputs of a case: a RodSystem (a list of them for a batch) and extras."""
    kind = case["kind"]
    if kind == "step":
        return _suspension(case, seed, case["forces"], case["crosslinks"], case["nematic"]), None
    if kind == "batch":
        # the sweep's state points are the case's, their configurations the seed's
        got = []
        for k, (n, length, phi, _, director) in enumerate(W.ensemble_specs(count=case["count"])):
            n = max(2, int(round(n * case["scale"])))
            box = max(W.box_for_fraction(n, DIAMETER, length, phi), length + 2 * DIAMETER + 1e-6)
            got.append(W.random_system(seed + k, n, box, length=length, nematic_spread=W.ENSEMBLE_SPREAD,
                                       director=director, forces="thermal", viscosity=VISCOSITY, dt=DT,
                                       tol=case["tol"]))
        return got, None
    if kind == "springs":
        s = _suspension(case, seed)
        return s, W.spring_set(s, case["springs"], seed=seed + 1)
    if kind == "run" and case["walls"]:
        # everything starts between the walls; a steady load pushes it onto the lower one
        s = _suspension(case, seed, forces="none")
        lo, hi = 2.0, s.box[2] - (LENGTH + 2.0 * DIAMETER) - 2.0
        s.x[:, 2] = lo + 6.0 + s.x[:, 2] / s.box[2] * (hi - lo - 12.0)
        s.f_nc[:, 2] = -2000.0
        return s, (2, lo, hi)
    if kind == "run":
        return _suspension(case, seed, forces="none", crosslinks=case["n"] // 2), None
    s = _suspension(case, seed)
    return s, W.loss_targets(s, seed=seed + 1) if kind == "grad" else None


def _dev(a, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dtype, device="cuda")


def prepare(case, seed):
    s, extra = _inputs(case, seed)
    kind = case["kind"]
    st = {"kind": kind}
    precision = A.FP64 if case["precision"] == "fp64" else A.MIXED
    if kind == "batch":
        off, x, quat, f, systems = W.batch_arrays(s)
        p = A.params_of(s[0], precision=precision, tol=case["tol"])
        st["tables"] = A.BatchSpec(systems, off)
    else:
        x, quat, f = s.x, s.quat, s.f_nc
        p = A.params_of(s, precision=precision, tol=case["tol"])
    n = x.shape[0]
    st["x0"], st["q0"], st["f"] = _dev(x), _dev(quat), _dev(f)
    rows = 12 * n + (len(extra["kappa"]) if kind == "springs" else 0)
    ctx = st["ctx"] = A.Context(p, n, rows)
    if kind in ("step", "springs", "batch", "run"):
        st["x"], st["q"] = torch.empty_like(st["x0"]), torch.empty_like(st["q0"])
    if kind == "step":
        if case["graph"]:
            ctx.set_step_graph(True)
        if case["records"]:
            st["pairs"] = torch.zeros((rows, 3), dtype=torch.int32, device="cuda")
            st["gamma"] = torch.zeros(rows, dtype=torch.float64, device="cuda")
            st["vel"] = torch.empty((n, 6), dtype=torch.float64, device="cuda")
    elif kind == "springs":
        ctx.set_springs(_dev(extra["ends"], torch.int32), _dev(extra["arms"]), _dev(extra["kappa"]),
                        _dev(extra["rest"]))
    elif kind == "batch":
        ctx.set_batch_graph(case["graph"])
    elif kind == "run":
        st["steps"], st["seed"] = case["steps"], seed % 1_000_003
        if extra is not None:
            ctx.set_walls(*extra)
    elif kind == "grad":
        st["target"] = _dev(extra)
        st["eta"] = torch.tensor(VISCOSITY, dtype=torch.float64, device="cuda")
        st["leaves"] = [t.requires_grad_(True) for t in (st["x0"], st["q0"], st["f"], st["eta"])]
    else:
        st["pairs"] = torch.zeros((rows, 3), dtype=torch.int32, device="cuda")
        for name, tail in (("phi", ()), ("dgeom", (9,)), ("lcp_q", ()), ("gamma", ())):
            st[name] = torch.zeros((rows, *tail), dtype=torch.float64, device="cuda")
    return st


# -------------------------------------------------------------------- pass

def run(st):
    kind, ctx = st["kind"], st["ctx"]
    if kind == "grad":
        xn, qn = constrained_step(ctx, *st["leaves"])
        loss = ((xn - st["target"]) ** 2).sum()
        gx, gq, gf, ge = torch.autograd.grad(loss, st["leaves"])
        return {"x": xn.detach(), "quat": qn.detach(), "loss": loss.detach(), "dx": gx, "dquat": gq, "df": gf,
                "deta": ge}
    if kind == "phases":
        pairs = ctx.build_neighbors(st["x0"], st["q0"], st["pairs"])
        phi, dgeom, q = ctx.assemble_constraints(st["x0"], st["q0"], st["f"], pairs)
        gamma, _ = ctx.solve_lcp(st["q0"], pairs, dgeom, q)
        m = pairs.shape[0]   # the program's own arrays, sized for the most constraints it expects
        out = {"phi": phi, "dgeom": dgeom, "lcp_q": q, "gamma": gamma}
        for name, t in out.items():
            st[name][:m] = t
        return {"pairs": st["pairs"], **{name: st[name] for name in out}}
    x, q = st["x"], st["q"]
    x.copy_(st["x0"])
    q.copy_(st["q0"])
    if kind == "batch":
        info = ctx.step_batch(st["tables"], None, x, q, st["f"])
        return {"x": x, "quat": q, "n_pairs": int(info.n_pairs)}
    if kind == "run":
        _, stats = ctx.run(x, q, st["steps"], kT=1.0, seed=st["seed"], first_step=0, f_ext=st["f"], warm_start=True)
        return {"x": x, "quat": q, "n_pairs": [int(d["n_pairs"]) for d in stats]}
    if "vel" in st:
        ctx.step(x, q, st["f"], pairs_out=st["pairs"], gamma_out=st["gamma"], vel_out=st["vel"])
        return {"x": x, "quat": q, "pairs": st["pairs"], "gamma": st["gamma"], "vel": st["vel"]}
    info = ctx.step(x, q, st["f"])
    return {"x": x, "quat": q, "n_pairs": int(info.n_pairs)}


def _rods(case):
    if case["kind"] != "batch":
        return case["n"]
    return case["count"] * 5300 * case["scale"]   # mean of a log-uniform draw in [500, 20000]


def work(case):
    """Rod state in (104 bytes a rod) and out (56), 84 bytes per constraint
    where the constraints are outputs; per rod about four constraints, whose
    geometry, columns and one sparse product with the mobility no method can
    leave out (about 200 and 50 operations)."""
    n, kind = _rods(case), case["kind"]
    m = 4 * n + case.get("springs", 0)
    steps = case.get("steps", 1)
    b = steps * n * (24 + 32 + 48 + 24 + 32)
    if case.get("records"):
        b += m * (12 + 8) + n * 48
    if kind == "springs":
        b += case["springs"] * (8 + 16 + 8 + 8)
    if kind == "phases":
        b = n * 104 + m * (12 + 8 + 72 + 8 + 8)
    if kind == "grad":
        b += n * (24 + 24 + 32 + 48)
    return {"bytes": float(b), "flops": float(steps * (250 * m + 300 * n) * (2 if kind == "grad" else 1))}


# ------------------------------------------------------- 64-bit plain torch

def _axis(q):
    s, a, b, c = q.unbind(1)
    return torch.stack([2 * (a * c + s * b), 2 * (b * c - s * a), s * s - a * a - b * b + c * c], 1)


def _dot(a, b):
    return (a * b).sum(1)


def _closest(dx, p, q, hl):
    """Arclengths of the closest points of two segments (clamped projections)."""
    a, b, c, d, e = _dot(p, p), _dot(p, q), _dot(q, q), _dot(p, dx), _dot(q, dx)
    s = torch.minimum(torch.maximum((b * e - c * d) / (a * c - b * b).clamp_min(1e-300), -hl), hl)
    t = (b * s + e) / c
    tc = torch.minimum(torch.maximum(t, -hl), hl)
    back = torch.minimum(torch.maximum((b * tc - d) / a, -hl), hl)
    return torch.where(t == tc, s, back), tc


def _shift(code, box):
    return torch.stack([code % 3 - 1, code // 3 % 3 - 1, code // 9 - 1], 1).to(box.dtype) * box


def _find(xw, p, box, length, system, first_of):
    """(i, j, image code) of every pair with a surface gap below D, sorted:
    cell lists with cells of at least L + 2 D, each of the 27 neighbours in turn."""
    rcut = length + 2 * DIAMETER
    nc = torch.clamp((box / rcut[:, None]).floor().long(), min=1, max=400)
    cell = torch.minimum((xw / box * nc).floor().long(), nc - 1)
    per = nc.prod(1)
    base = torch.cumsum(per[first_of], 0) - per[first_of]
    key = base[system] + (cell[:, 0] * nc[:, 1] + cell[:, 1]) * nc[:, 2] + cell[:, 2]
    keys, order = torch.sort(key)
    got = []
    for o in range(27):
        step = torch.tensor([o % 3 - 1, o // 3 % 3 - 1, o // 9 - 1], device=xw.device)
        at = cell + step
        k = torch.div(at, nc, rounding_mode="floor")
        at = at - k * nc
        want = base[system] + (at[:, 0] * nc[:, 1] + at[:, 1]) * nc[:, 2] + at[:, 2]
        lo, hi = torch.searchsorted(keys, want), torch.searchsorted(keys, want, right=True)
        cnt = hi - lo
        i = torch.repeat_interleave(torch.arange(len(xw), device=xw.device), cnt)
        j = order[torch.arange(len(i), device=xw.device) - (torch.cumsum(cnt, 0) - cnt)[i] + lo[i]]
        keep = j > i
        i, j = i[keep], j[keep]
        dx = xw[i] - xw[j] - k[i].double() * box[i]
        keep = _dot(dx, dx) < rcut[i] ** 2
        i, j, dx = i[keep], j[keep], dx[keep]
        s, t = _closest(dx, p[i], p[j], length[i] / 2)
        r = dx + s[:, None] * p[i] - t[:, None] * p[j]
        keep = r.norm(dim=1) - DIAMETER < DIAMETER
        i, j = i[keep], j[keep]
        kk = k[i]
        got.append(torch.stack([i, j, (kk[:, 0] + 1) + 3 * (kk[:, 1] + 1) + 9 * (kk[:, 2] + 1)], 1))
    got = torch.cat(got)
    return got[torch.argsort((got[:, 0] * len(xw) + got[:, 1]) * 27 + got[:, 2])]


def _move(p, length, eta, F):
    """Rod velocities U = M F [n, 6]."""
    perp = 4 * math.pi * eta * length / torch.log(2 * length / DIAMETER)
    rot, spin = perp * length ** 2 / 12, math.pi * eta * DIAMETER ** 2 * length
    pf, pt = _dot(p, F[:, :3])[:, None] * p, _dot(p, F[:, 3:])[:, None] * p
    return torch.cat([F[:, :3] / perp[:, None] + pf / perp[:, None],
                      F[:, 3:] / rot[:, None] + pt * (1 / spin - 1 / rot)[:, None]], 1)


def _columns(x, p, box, length, pairs):
    """Gap and the column's parts (normal, y_P x e, y_Q x e) of every pair."""
    i, j = pairs[:, 0], pairs[:, 1]
    dx = x[i] - x[j] - _shift(pairs[:, 2], box[i])
    s, t = _closest(dx, p[i], p[j], length[i] / 2)
    yp, yq = s[:, None] * p[i], t[:, None] * p[j]
    r = dx + yp - yq
    dist = r.norm(dim=1)
    e = r / dist[:, None]
    return dist - DIAMETER, e, torch.linalg.cross(yp, e), torch.linalg.cross(yq, e)


def _force(n, ij, col, g):
    e, ap, aq = col
    F = torch.zeros((n, 6), dtype=torch.float64, device=g.device)
    F = F.index_add(0, ij[0], torch.cat([e, ap], 1) * g[:, None])
    return F.index_add(0, ij[1], torch.cat([-e, -aq], 1) * g[:, None])


def _gaps(ij, col, U):
    e, ap, aq = col
    u, v = U[ij[0]], U[ij[1]]
    return _dot(e, u[:, :3] - v[:, :3]) + _dot(ap, u[:, 3:]) - _dot(aq, v[:, 3:])


def _contact_forces(n, p, length, ij, col, q, comp, seconds=12.0, want=2e-12):
    """min 1/2 g^T A g + q^T g with A = D^T M D + comp, g >= 0 where comp < 0:
    projected Barzilai-Borwein steps on the diagonally scaled problem, to the
    largest projected gradient (times h / D) below ``want``.  None if the
    time runs out."""
    hard = comp < 0
    soft = comp.clamp_min(0.0)
    apply = lambda g: _gaps(ij, col, _move(p, length, VISCOSITY, _force(n, ij, col, g))) + soft * g
    e, ap, aq = col
    w = 0.0
    for side, arm in ((0, ap), (1, aq)):
        F = torch.cat([e, arm], 1)
        w = w + (F * _move(p[ij[side]], length[ij[side]], VISCOSITY, F)).sum(1)
    sc = (w + soft) ** -0.5
    g, grad = torch.zeros_like(q), q * sc            # scaled force g / sc and scaled gradient
    project = lambda v: torch.where(hard, v.clamp_min(0.0), v)
    step, began, best = None, time.monotonic(), (math.inf, None)
    for k in range(200_000):
        pg = torch.where(hard & (g <= 0), grad.clamp_max(0.0), grad)
        if k % 10 == 0:
            r = float((pg / sc).abs().max()) * DT / DIAMETER if len(q) else 0.0
            if r < best[0]:
                best = (r, g.clone())
            if r <= want or (r < 1e-10 and time.monotonic() - began > seconds / 2):
                break
            if time.monotonic() - began > seconds:
                return None
        if step is None:
            step = (pg * pg).sum() / (pg * sc * apply(sc * pg)).sum()
        new = project(g - step * grad)
        gnew = sc * (apply(sc * new) + q)
        s, y = new - g, gnew - grad
        sy = (s * y).sum()
        step = torch.where(sy > 0, (s * s).sum() / sy if k % 2 else sy / (y * y).sum(), step)
        g, grad = new, gnew
    return best[1] * sc


def _rows(t, rows):
    """t with zero rows after it, as the program's arrays are."""
    return torch.cat([t, torch.zeros((rows - t.shape[0], *t.shape[1:]), dtype=t.dtype, device=t.device)])


def exact(case, seed):
    kind = case["kind"]
    if kind == "run":
        return None   # the steps' differences add up over the trajectory
    s, extra = _inputs(case, seed)
    if kind == "batch":
        off, x, quat, f, systems = W.batch_arrays(s)
        cnt = _dev(np.diff(off), torch.int64)
        system = torch.repeat_interleave(torch.arange(len(systems), device="cuda"), cnt)
        first = _dev(off[:-1], torch.int64)
        box = _dev([list(b) for b, _ in systems])[system]
        length = _dev([v for _, v in systems])[system]
    else:
        x, quat, f = s.x, s.quat, s.f_nc
        system = torch.zeros(len(x), dtype=torch.int64, device="cuda")
        first = torch.zeros(1, dtype=torch.int64, device="cuda")
        box, length = _dev([list(s.box)]).expand(len(x), 3), torch.full((len(x),), LENGTH, dtype=torch.float64,
                                                                      device="cuda")
    x, quat, f = _dev(x), _dev(quat), _dev(f)
    n = len(x)
    p = _axis(quat)
    xw = torch.remainder(x, box)
    pairs = _find(xw, p, box, length, system, first)
    phi, *col = _columns(xw, p, box, length, pairs)
    ij = (pairs[:, 0], pairs[:, 1])
    if kind == "springs":
        ends, arms = _dev(extra["ends"], torch.int64), _dev(extra["arms"])
        yp, yq = arms[:, :1] * p[ends[:, 0]], arms[:, 1:] * p[ends[:, 1]]
        r = xw[ends[:, 0]] + yp - xw[ends[:, 1]] - yq
        r = r - box[0] * torch.round(r / box[0])
        dist = r.norm(dim=1)
        e = r / dist[:, None]
        more = (e, torch.linalg.cross(yp, e), torch.linalg.cross(yq, e))
        col = [torch.cat([a, b]) for a, b in zip(col, more)]
        ij = tuple(torch.cat([ij[k], ends[:, k]]) for k in (0, 1))
        gap = torch.cat([phi, dist - _dev(extra["rest"])])
        comp = torch.cat([torch.full_like(phi, -1.0), 1 / (DT * _dev(extra["kappa"]))])
    else:
        gap, comp = phi, torch.full_like(phi, -1.0)
    q = gap / DT + _gaps(ij, col, _move(p, length, VISCOSITY, f))
    g = _contact_forces(n, p, length, ij, col, q, comp)
    if g is None:
        return None
    if kind == "phases":
        return {"pairs": None, **{name: _rows(t, 12 * n) for name, t in (
            ("phi", phi), ("dgeom", torch.cat(col, 1)), ("lcp_q", q), ("gamma", g))}}
    U = _move(p, length, VISCOSITY, f + _force(n, ij, col, g))
    w = U[:, 3:]
    v = quat[:, 1:]
    turn = torch.cat([-_dot(w, v)[:, None], quat[:, :1] * w + torch.linalg.cross(w, v)], 1)
    qn = quat + 0.5 * DT * turn
    qn = qn / qn.norm(dim=1, keepdim=True)
    if kind == "grad":
        return dict(_gradient(x, quat, f, box, length, pairs, g, _dev(extra)), quat=qn)
    xn = torch.remainder(xw + DT * U[:, :3], box)
    if case.get("records"):
        # a dense pack's contact forces are not unique, its velocities are
        return {"x": xn, "quat": qn, "pairs": None, "gamma": _rows(g, 12 * n) if case["nematic"] == 0 else None,
                "vel": U}
    return {"x": xn, "quat": qn, "n_pairs": None}


def _gradient(x, quat, f, box, length, pairs, g, target):
    """Loss and its gradient on the pair list and the active set {g > 0}: with
    A_AA lam = (D^T M u)_A, dL = d[loss - lam . (gaps + D^T U)_A] at fixed g, lam."""
    n = len(x)
    pairs, g = pairs[g > 0], g[g > 0]
    ij = (pairs[:, 0], pairs[:, 1])
    eta = torch.tensor(VISCOSITY, dtype=torch.float64, device=x.device)
    var = [t.clone().requires_grad_(True) for t in (x, quat, f, eta)]

    def forward(x, quat, f, eta):
        p = _axis(quat)
        phi, *col = _columns(x + (torch.remainder(x, box) - x).detach(), p, box, length, pairs)
        U = _move(p, length, eta, f + _force(n, ij, col, g))
        xn = x + DT * U[:, :3]
        return xn, ((xn - target) ** 2).sum(), phi / DT + _gaps(ij, col, U), p, col

    xn, loss, gaps, p, col = forward(*var)
    with torch.no_grad():
        apply = lambda v: _gaps(ij, col, _move(p, length, VISCOSITY, _force(n, ij, col, v)))
        u = torch.cat([2 * DT * (xn - target), torch.zeros_like(xn)], 1)
        r = _gaps(ij, col, _move(p, length, VISCOSITY, u))
        lam, d, rr = torch.zeros_like(r), r.clone(), (r * r).sum()
        stop = 1e-26 * float(rr)
        for k in range(4000):
            Ad = apply(d)
            a = rr / (d * Ad).sum()
            lam, r = lam + a * d, r - a * Ad
            new = (r * r).sum()
            if k % 20 == 0 and float(new) <= stop:
                break
            d, rr = r + new / rr * d, new
    gx, gq, gf, ge = torch.autograd.grad(loss - (lam * gaps).sum(), var)
    gq = gq - quat * _dot(quat, gq)[:, None]
    return {"x": xn.detach(), "loss": loss.detach(), "dx": gx, "dquat": gq, "df": gf, "deta": ge}
