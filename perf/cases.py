"""The work this library is measured on: builds of interval-MDP abstractions in
both precisions, batches of builds, a served burst, controller synthesis,
region vectors and sampled-noise builds, each through its public entry point.

A case names a system of ``workloads`` (or a seeded linear one), its grid as
"NxNx...", a precision, a cutoff and the entry point. The seed moves what a
user would change between two runs of the same model: offsets, noise scales,
input points, boxes, draws. Pairs come back in buffers of a size the case
fixes (about a fifth more than they need, the rest zero), so that every seed's
outputs have one layout.
"""

from __future__ import annotations

import math
from dataclasses import replace

import numpy as np
import torch

from paper_2401_03555_gb300 import impact
from paper_2401_03555_gb300 import workloads as W


def listed():
    return [
        # the smallest call: one 2-D grid of about 1e3 cells rebuilt into kept
        # buffers inside a user's outer loop; launches and host work count
        dict(name="linear2d-small-fp32", entry="builder", system="linear", cells="33x31", inputs=4,
             precision="fp32", cutoff=1e-8),
        # the 2-D robot, dense, plain FP64: a first run of the tool, one call
        # from a problem to its IMDP
        dict(name="robot2d-dense-fp64", entry="build", system="robot", cells="21x21",
             precision="fp64", cutoff=0.0),
        # the 3-D vehicle in FP64 on an uneven grid (trigonometric images)
        dict(name="unicycle-fp64", entry="builder", system="unicycle", cells="21x19x13",
             precision="fp64", cutoff=1e-8),
        # the 5-D rooms in FP64 on an uneven grid (affine images, five factors)
        dict(name="room5d-fp64", entry="builder", system="room", cells="5x6x5x6x5",
             precision="fp64", cutoff=1e-8),
        # the full vehicle, FP32-sound, into kept buffers
        dict(name="unicycle-fp32", entry="builder", system="unicycle", cells="51x51x25",
             precision="fp32", cutoff=1e-8),
        # the headline build: 11^5 rooms, FP32-sound, into kept buffers
        dict(name="room5d-fp32", entry="builder", system="room", cells="11x11x11x11x11",
             precision="fp32", cutoff=1e-8),
        # the 7-D building: deep prefix trees of narrow windows
        dict(name="building7d-fp32", entry="builder", system="building", cells="6x6x6x6x6x6x6",
             precision="fp32", cutoff=1e-8),
        # many uneven builds in one captured graph (a design-space sweep)
        dict(name="batch24-fp32", entry="graph", system="batch", systems=24, min_cells=1000,
             max_cells=20000, precision="fp32", cutoff=1e-8),
        # a burst at the request server: submit, wait, take the results out of
        # the server's memory and give it back
        dict(name="serve8-fp32", entry="serve", system="batch", systems=8, min_cells=1000,
             max_cells=20000, building="5x5x5x5x5x5x5", precision="fp32", cutoff=1e-8),
        # controller synthesis on the dense robot: interval iteration until
        # the bounds meet
        dict(name="synth-robot-fp64", entry="synth", system="robot", cells="21x21",
             precision="fp64", cutoff=0.0, spec="reach", optimistic=False, horizon=0,
             with_regions=False),
        # the paper's target and avoid vectors over the full room grid
        dict(name="regions-room5d-fp64", entry="regions", system="room", cells="11x11x11x11x11",
             precision="fp64", cutoff=1e-8, mode="cells"),
        # correlated noise given by draws
        dict(name="mc-room5d-fp32", entry="mc", system="room", cells="7x7x7x7x7",
             precision="fp32", cutoff=2e-3, draws=1024),
    ]


# --------------------------------------------------------------------------
# more cases of the same ranges
# --------------------------------------------------------------------------

def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _cells(rng, n, lo, hi, most):
    while True:
        c = [rng.randint(lo, hi) for _ in range(n)]
        if math.prod(c) <= most:
            return "x".join(map(str, c))


def draw(rng):
    entry = rng.choice(["builder"] * 6 + ["graph", "serve", "synth", "synth", "regions", "regions",
                                          "mc"])
    prec = rng.choice(["fp32", "fp64"])
    if entry == "builder":
        system = rng.choice(["robot", "unicycle", "room", "building", "linear", "linear", "images"])
        if system == "robot":   # dense: one call from a problem to its IMDP
            cutoff = rng.choice([0.0, 1e-8])
            return dict(entry="builder" if cutoff else "build", system=system,
                        cells=_cells(rng, 2, 5, 41, 1600), precision=prec, cutoff=cutoff)
        if system == "unicycle":
            a, b = (_log(rng, 7, 48 if prec == "fp32" else 19) for _ in range(2))
            c = rng.randint(5, 25 if prec == "fp32" else 13)
            return dict(entry=entry, system=system, cells=f"{a}x{b}x{c}", precision=prec,
                        cutoff=rng.choice([1e-8, 1e-6]))
        if system == "room":
            big = 10 if prec == "fp32" else 6
            return dict(entry=entry, system=system,
                        cells=_cells(rng, 5, 3, big, 100000 if prec == "fp32" else 3600),
                        precision=prec, cutoff=rng.choice([1e-8, 1e-6]))
        if system == "building":
            return dict(entry=entry, system=system, cells=_cells(rng, 7, 3, 6, 150000),
                        precision="fp32", cutoff=1e-8)
        n = rng.choice([2, 3, 4, 5])
        total = _log(rng, 1e3, 5e4 if prec == "fp32" and system == "linear" else 2e3)
        side = max(3, round(total ** (1.0 / n)))
        cells = "x".join(str(max(2, side + rng.choice([-1, 0, 0, 1]))) for _ in range(n))
        return dict(entry=entry, system=system, cells=cells,
                    inputs=rng.choice([4, 8, 9, 27] if prec == "fp32" else [4, 8, 9]),
                    precision=prec, cutoff=rng.choice([1e-8, 1e-8, 1e-6]))
    if entry == "graph":
        return dict(entry=rng.choice(["graph", "into"]), system="batch", systems=rng.randint(3, 24),
                    min_cells=1000, max_cells=_log(rng, 2000, 20000), precision="fp32", cutoff=1e-8)
    if entry == "serve":
        return dict(entry=entry, system="batch", systems=rng.randint(2, 8), min_cells=1000,
                    max_cells=_log(rng, 2000, 20000), building=_cells(rng, 7, 3, 5, 40000),
                    precision="fp32", cutoff=1e-8)
    if entry == "synth":
        if rng.random() < 0.6:
            system, cells = "robot", _cells(rng, 2, 7, 25, 500)
            cutoff = rng.choice([0.0, 1e-8])
        else:
            system, cells, cutoff = "unicycle", _cells(rng, 3, 5, 13, 1200), 1e-8
        return dict(entry=entry, system=system, cells=cells, precision=prec, cutoff=cutoff,
                    spec=rng.choice(["reach", "safety"]), optimistic=rng.random() < 0.3,
                    horizon=rng.choice([0, 10, 40]) if system == "robot" else rng.randint(5, 40),
                    with_regions=rng.random() < 0.3)
    if entry == "regions":
        system = rng.choice(["robot", "unicycle", "room", "building"])
        cells = {"robot": lambda: _cells(rng, 2, 9, 90, 8100),
                 "unicycle": lambda: _cells(rng, 3, 9, 41, 30000),
                 "room": lambda: _cells(rng, 5, 4, 11, 120000),
                 "building": lambda: _cells(rng, 7, 3, 6, 150000)}[system]()
        return dict(entry=entry, system=system, cells=cells, precision=prec, cutoff=1e-8,
                    mode=rng.choice(["box", "cells"]))
    system = rng.choice(["robot", "unicycle", "room"])
    cells = {"robot": lambda: _cells(rng, 2, 7, 41, 1200),
             "unicycle": lambda: _cells(rng, 3, 7, 19, 3000),
             "room": lambda: _cells(rng, 5, 4, 8, 14000)}[system]()
    return dict(entry="mc", system=system, cells=cells, precision=prec,
                cutoff=rng.choice([1e-3, 4e-3]), draws=_log(rng, 256, 2048))


# --------------------------------------------------------------------------
# problems
# --------------------------------------------------------------------------

def _ints(text):
    return [int(v) for v in text.split("x")]


def _linear(cells, n_inputs, cutoff, model, rng):
    """A linear system of the batched family with its sizes given: `model`
    seeds A, B and the noise scales, `rng` moves the offsets and the noise."""
    n = len(cells)
    move, rng = rng, np.random.default_rng(model)
    m = {4: 2, 9: 2, 8: 3, 27: 3}[n_inputs]
    pts = {4: 2, 9: 3, 8: 2, 27: 3}[n_inputs]
    q, r = np.linalg.qr(rng.standard_normal((n, n)))
    q = q * np.sign(np.diag(r))[None, :]
    width = 2.0 / np.asarray(cells, np.float64)
    spread = np.exp(np.linspace(math.log(0.1), 0.0, n + 2)[1:-1])
    mesh = np.meshgrid(*([np.linspace(-1.0, 1.0, pts)] * m), indexing="ij")
    return W.Problem(
        name="linear", kind=W.AFFINE, lo=np.full(n, -1.0), hi=np.full(n, 1.0),
        cells=np.asarray(cells, np.int32),
        inputs=np.stack([g.reshape(-1) for g in mesh], axis=1),
        sigma=width * rng.permutation(spread) * move.uniform(0.99, 1.01, n), cutoff=cutoff,
        A=0.9 * (q * rng.uniform(0.5, 1.0, n)[None, :]) @ q.T,
        B=rng.normal(0.0, 0.3, (n, m)), c=width * move.uniform(-0.02, 0.02, n))


def _problem(case, seed):
    rng = np.random.default_rng(1000003 * (seed + 1))
    cells, cutoff = _ints(case["cells"]), float(case["cutoff"])
    system = case["system"]
    if system in ("linear", "images"):
        p = _linear(cells, case["inputs"], cutoff, 17, rng)
        if system == "images":
            lo, hi = _images(p)
            grow = torch.as_tensor(rng.uniform(0.0, 0.2, tuple(lo.shape))).to(lo) * (hi - lo)
            p = W.with_images(p, torch.stack([lo, hi + grow], dim=2).cpu().numpy())
        return p
    if system == "robot":
        p = W.robot_2d()
        p = replace(p, c=rng.uniform(-0.1, 0.1, 2))
    elif system == "unicycle":
        p = W.unicycle_3d()
        p = replace(p, inputs=p.inputs * rng.uniform(0.98, 1.02, (1, 2)))
    elif system == "room":
        p = W.room_5d()
        p = replace(p, c=p.c + rng.uniform(-0.02, 0.02, 5))
    else:
        p = W.building_7d()
        p = replace(p, c=rng.uniform(-0.01, 0.01, 7))
    return replace(W.with_cells(p, cells), cutoff=cutoff,
                   sigma=p.sigma * rng.uniform(0.99, 1.01, len(p.sigma)))


def _batch(case, seed):
    """Uneven systems: dimensions 2..5 in turn, cells log-spaced, 4..27 inputs."""
    rng = np.random.default_rng(1000003 * (seed + 1))
    k = int(case["systems"])
    totals = np.exp(np.linspace(math.log(case["min_cells"]), math.log(case["max_cells"]), k))
    inputs = [4, 9, 8, 27]
    probs = []
    for i in range(k):
        n = 2 + i % 4
        side = max(2, round(totals[(5 * i + 2) % k] ** (1.0 / n)))
        probs.append(_linear([side] * n, inputs[(i // 4 + i) % 4], float(case["cutoff"]),
                             100 + i, rng))
    if case.get("building"):
        probs[k // 2] = _problem(dict(case, system="building", cells=case["building"]), seed)
    return probs


def _boxes(p, seed):
    """A target box and an avoid box in seeded places, as (lo, hi) lists."""
    rng = np.random.default_rng(7 * seed + 5)
    w = p.hi - p.lo
    t0 = p.lo + w * rng.uniform(0.55, 0.65, p.n)
    a0 = p.lo + w * rng.uniform(0.1, 0.2, p.n)
    return [(t0, t0 + 0.3 * w)], [(a0, a0 + 0.25 * w)]


def _draws(p, case, seed):
    rng = np.random.default_rng(13 * seed + 3)
    cov = np.outer(p.sigma, p.sigma) * (0.7 * np.eye(p.n) + 0.3)
    return rng.standard_normal((int(case["draws"]), p.n)) @ np.linalg.cholesky(cov).T


_SPEC = {"reach": impact.REACH_AVOID, "safety": impact.SAFETY}


def prepare(case, seed):
    entry, prec = case["entry"], case["precision"]
    s = {"entry": entry, "precision": prec, "case": case}
    if entry in ("graph", "into"):
        b = impact.Batch(_batch(case, seed), prec)
        rows = impact.alloc_rows(b.rows)
        ws = b.alloc_workspace()
        room = sum(_room(q) for q in _batch(case, 0))
        pairs = _pairs(room, prec)
        s.update(batch=b, rows=rows, ws=ws, room=room, pairs=pairs)
        if entry == "graph":
            s["graph"] = b.graph(rows, pairs, room, ws)
        return s
    if entry == "serve":
        s["server"] = impact.Server(prec, memory_budget=24 << 30)
        s["probs"] = _batch(case, seed)
        s["pairs"] = [_pairs(_room(q), prec) for q in _batch(case, 0)]
        return s
    p = _problem(case, seed)
    s["prob"] = p
    if entry == "builder":
        dev = None if p.images is None else torch.as_tensor(p.images).cuda().contiguous()
        room = _room(_problem(case, 0))
        b = s["builder"] = impact.Builder(p, prec, capacity=room, images=dev)
        for v in b.pairs_buf.values():
            v.zero_()
    elif entry == "synth":
        t, a = _boxes(p, seed)
        s["csr"] = impact.build(p, prec)
        s["labels"] = impact.label_cells(p, t, a)
        s["regions"] = (impact.region_vectors(p, t, a, "cells", prec) if case["with_regions"]
                        else None)
    elif entry == "regions":
        s["boxes"] = _boxes(p, seed)
    elif entry == "mc":
        s["draws"] = _draws(p, case, seed)
        s["pairs"] = _pairs(_mc_room(case), prec)
    return s


def _pairs(room, precision):
    return {k: v.zero_() for k, v in impact.alloc_pairs(room, precision).items()}


def _taken(c, pairs):
    """A result taken out into the caller's own buffers (row arrays copied)."""
    for k, v in pairs.items():
        v[:c.nnz].copy_(getattr(c, k))
    return {**{k: v.clone() for k, v in _csr(c).items() if k not in pairs}, **pairs}


def _csr(c):
    return {"row_ptr": c.row_ptr, "col": c.col, "lo": c.lo, "up": c.up, "sink_lo": c.sink_lo,
            "sink_up": c.sink_up, "trunc": c.trunc, "row_flags": c.row_flags}


def run(s):
    entry = s["entry"]
    if entry == "builder":
        b = s["builder"]
        b.run()
        return {**b.rows_buf, **b.pairs_buf}
    if entry == "build":
        return _csr(impact.build(s["prob"], s["precision"]))
    if entry in ("graph", "into"):
        if entry == "graph":
            s["graph"].launch()
        else:
            s["batch"].build_into(s["rows"], s["pairs"], s["room"], s["ws"])
        return {**s["rows"], **s["pairs"]}
    if entry == "serve":
        srv = s["server"]
        tickets = [srv.submit(p) for p in s["probs"]]
        for t in tickets:
            srv.poll(t, wait=True)
        # results are views of the server's memory until their release: the
        # copies have to be done before it
        out = [_taken(srv.result(t), q) for t, q in zip(tickets, s["pairs"])]
        torch.cuda.current_stream().synchronize()
        for t in tickets:
            srv.release(t)
        return out
    if entry == "synth":
        c = s["case"]
        r = impact.synthesize(s["csr"], s["prob"], s["labels"], spec=_SPEC[c["spec"]], eps=1e-6,
                              optimistic=c["optimistic"], horizon=c["horizon"],
                              regions=s["regions"])
        return {"p_min": r.p_min, "p_max": r.p_max, "policy": r.policy,
                "iterations": list(r.iterations)}
    if entry == "regions":
        v = impact.region_vectors(s["prob"], *s["boxes"], s["case"]["mode"], s["precision"])
        return {"r_lo": v.r_lo, "r_up": v.r_up, "a_lo": v.a_lo, "a_up": v.a_up}
    return _taken(impact.build_mc(s["prob"], s["draws"], s["precision"]), s["pairs"])


# --------------------------------------------------------------------------
# the work of one pass
# --------------------------------------------------------------------------

def _kept_per_row(p, samples=1024):
    """Mean kept pairs of a row (sampled rows, 64-bit factors)."""
    if p.cutoff <= 0:
        return p.total_cells
    rows = torch.as_tensor(np.random.default_rng(0).integers(0, p.rows, samples)).cuda()
    mlo, mhi = (x[rows] for x in _images(p)) if p.kind == W.IMAGES else _images(p, rows)
    step = max(1, int(4e7) // p.total_cells)
    total = 0
    for r in range(0, samples, step):
        up = torch.ones((mlo[r:r + step].shape[0], 1), dtype=torch.float64, device="cuda")
        for d in range(p.n):
            u = _factors(p, d, mlo[r:r + step, d], mhi[r:r + step, d])[0]
            up = (up[:, :, None] * u[:, None, :]).reshape(up.shape[0], -1)
        total += int((up >= p.cutoff).sum())
    return total / samples


def _room(p):
    """Pairs the buffers of a problem's results hold (from its seed-0 model)."""
    if p.cutoff <= 0:
        return p.rows * p.total_cells
    return 1024 * math.ceil(1.2 * _kept_per_row(p) * p.rows / 1024 + 1)


def _mc_kept(case, samples=64):
    p = _problem(case, 0)
    rows = torch.as_tensor(np.random.default_rng(0).integers(0, p.rows, samples)).cuda()
    return _mc_rows(p, case, _draws(p, case, 0), *_images(p, rows))["up"].numel() / samples


def _mc_room(case):
    return 1024 * math.ceil(1.4 * _mc_kept(case) * _problem(case, 0).rows / 1024 + 1)


def work(case):
    entry = case["entry"]
    pair = 12 if case["precision"] == "fp32" else 20
    per_row = 8 + 3 * 8 + 4
    if entry in ("graph", "into", "serve"):
        probs = _batch(case, 0)
    else:
        probs = [_problem(case, 0)]
    p = probs[0]
    if entry == "regions":
        return {"bytes": 32.0 * p.rows, "flops": 4.0 * p.rows * p.n * 3}
    if entry == "mc":
        # each draw's cell in each dimension at both image ends; pairs kept
        # are the cells met by at least cutoff of the draws
        return {"bytes": p.rows * (_mc_kept(case) * pair + per_row) + 8.0 * p.n * case["draws"],
                "flops": 2.0 * p.rows * p.n * case["draws"]}
    if entry == "synth":
        nnz = p.rows * _kept_per_row(p)
        sweeps = case["horizon"] or 100
        return {"bytes": nnz * pair + p.rows * per_row + p.total_cells * 21.0,
                "flops": 2.0 * 4.0 * nnz * sweeps}
    by = fl = 0.0
    for q in probs:
        nnz = q.rows * _kept_per_row(q)
        by += nnz * pair + q.rows * per_row
        if q.kind == W.IMAGES:
            by += 16.0 * q.rows * q.n
        fl += 2.0 * nnz
    return {"bytes": by, "flops": fl}


# --------------------------------------------------------------------------
# the definitions in 64 bits
# --------------------------------------------------------------------------

def _edges(p, d):
    n = int(p.cells[d])
    h = (float(p.hi[d]) - float(p.lo[d])) / n
    e = float(p.lo[d]) + torch.arange(n + 1, dtype=torch.float64, device="cuda") * h
    e[n] = float(p.hi[d])
    return e


def _images(p, rows=None):
    """[m_lo, m_hi] of every row (or of `rows`) and dimension."""
    if p.kind == W.IMAGES:
        im = torch.as_tensor(p.images).cuda()
        return im[:, :, 0].contiguous(), im[:, :, 1].contiguous()
    if rows is None:
        rows = torch.arange(p.rows, device="cuda")
    u = torch.as_tensor(np.asarray(p.inputs, np.float64)).cuda()[rows % p.n_inputs]
    cell, idx = rows // p.n_inputs, [None] * p.n
    for d in range(p.n - 1, -1, -1):
        idx[d] = cell % int(p.cells[d])
        cell = cell // int(p.cells[d])
    e = [_edges(p, d) for d in range(p.n)]
    x0 = [e[d][idx[d]] for d in range(p.n)]
    x1 = [e[d][idx[d] + 1] for d in range(p.n)]
    lo, hi = [], []
    if p.kind == W.UNICYCLE:
        v, om = u[:, 0], u[:, 1]
        for d, f, peak in ((0, torch.cos, 0.0), (1, torch.sin, math.pi / 2)):
            a, b = f(x0[2]), f(x1[2])
            top, low = torch.maximum(a, b), torch.minimum(a, b)
            for k in range(-4, 5):   # extrema of the heading's cosine or sine
                t = peak + k * math.pi
                inside = (x0[2] <= t) & (t <= x1[2])
                if k % 2 == 0:
                    top = torch.where(inside, 1.0, top)
                else:
                    low = torch.where(inside, -1.0, low)
            lo.append(x0[d] + torch.minimum(v * low, v * top))
            hi.append(x1[d] + torch.maximum(v * low, v * top))
        lo.append(x0[2] + om)
        hi.append(x1[2] + om)
    else:
        for d in range(p.n):
            a = b = torch.zeros_like(x0[0])
            for k in range(p.n):
                s, t = float(p.A[d, k]) * x0[k], float(p.A[d, k]) * x1[k]
                a, b = a + torch.minimum(s, t), b + torch.maximum(s, t)
            off = torch.full_like(a, float(p.c[d]))
            for k in range(u.shape[1]):
                off = off + float(p.B[d, k]) * u[:, k]
            lo.append(a + off)
            hi.append(b + off)
    return torch.stack(lo, 1), torch.stack(hi, 1)


def _mass(c, e, m, sigma):
    """Mass of [c, e] around the mean m, in the form whose terms are small tails."""
    a, b = (c - m) / (sigma * math.sqrt(2.0)), (e - m) / (sigma * math.sqrt(2.0))
    f = torch.special.erfc
    right, left = 0.5 * (f(a) - f(b)), 0.5 * (f(-b) - f(-a))
    return torch.where(a >= 0, right, torch.where(b <= 0, left, 1.0 - 0.5 * f(-a) - 0.5 * f(b)))


def _bounds(c, e, mlo, mhi, sigma):
    mid = torch.minimum(torch.maximum(0.5 * (c + e), mlo), mhi)
    return (_mass(c, e, mid, sigma),
            torch.minimum(_mass(c, e, mlo, sigma), _mass(c, e, mhi, sigma)))


def _factors(p, d, mlo, mhi):
    """Upper and lower factor of every cell of dimension d, per row."""
    e = _edges(p, d)
    return _bounds(e[None, :-1], e[None, 1:], mlo[:, None], mhi[:, None], float(p.sigma[d]))


def _sinks(p, mlo, mhi):
    up = low = 1.0
    for d in range(p.n):
        c, e = (torch.tensor(float(v), dtype=torch.float64, device="cuda") for v in
                (p.lo[d], p.hi[d]))
        u, v = _bounds(c, e, mlo[:, d], mhi[:, d], float(p.sigma[d]))
        up, low = up * u, low * v
    return 1.0 - up, 1.0 - low


def _dense_rows(p, mlo, mhi):
    up = low = torch.ones((mlo.shape[0], 1), dtype=torch.float64, device="cuda")
    for d in range(p.n):
        u, v = _factors(p, d, mlo[:, d], mhi[:, d])
        up = (up[:, :, None] * u[:, None, :]).reshape(mlo.shape[0], -1)
        low = (low[:, :, None] * v[:, None, :]).reshape(mlo.shape[0], -1)
    return up, low


def _padded(parts, room):
    v = torch.cat(parts)
    return torch.cat([v, v.new_zeros(max(0, room - v.numel()))])


def _exact_build(p, precision, room, only_sinks=False):
    mlo, mhi = _images(p)
    sl, su = _sinks(p, mlo, mhi)
    out = {"row_ptr": None, "col": None, "lo": None, "up": None, "sink_lo": sl, "sink_up": su,
           "trunc": None, "row_flags": None}
    if precision == "fp32" and float(sl.max()) < 1e-3:
        # FP32-sound sink bounds are good to about 2e-6 absolute: of a sink
        # that is never reached in earnest the lower one says nothing
        out["sink_lo"] = None
    if only_sinks or p.rows * p.total_cells > 2e9:
        return out
    # the kept set of FP32-sound builds is that of its own upper bounds: the
    # pairs have no 64-bit value of the same layout unless every cell is kept
    pairs = precision == "fp64" or p.cutoff <= 0
    step = max(1, int(4e7) // p.total_cells)
    los, ups, trunc = [], [], []
    for r in range(0, p.rows, step):
        up, low = _dense_rows(p, mlo[r:r + step], mhi[r:r + step])
        keep = up >= p.cutoff
        trunc.append(torch.where(keep, 0.0, up).sum(1))
        if pairs:
            los.append(low[keep])
            ups.append(up[keep])
    out["trunc"] = torch.cat(trunc)
    if pairs:
        out["lo"], out["up"] = _padded(los, room), _padded(ups, room)
    return out


def _exact_regions(p, case, boxes):
    mlo, mhi = _images(p)
    sl, su = _sinks(p, mlo, mhi)
    sums = []
    for (b,) in boxes:
        up = low = 1.0
        for d in range(p.n):
            e = _edges(p, d)
            mid = 0.5 * (e[:-1] + e[1:])
            inside = torch.nonzero((mid >= float(b[0][d])) & (mid <= float(b[1][d]))).reshape(-1)
            if inside.numel() == 0:
                u = v = torch.zeros(p.rows, dtype=torch.float64, device="cuda")
            elif case["mode"] == "box":
                u, v = _bounds(e[inside[0]], e[inside[-1] + 1], mlo[:, d], mhi[:, d],
                               float(p.sigma[d]))
            else:
                u = v = 0.0
                for i in inside.tolist():
                    x, y = _bounds(e[i], e[i + 1], mlo[:, d], mhi[:, d], float(p.sigma[d]))
                    u, v = u + x, v + y
            up, low = up * u, low * v
        sums.append((low, up))
    return {"r_lo": sums[0][0], "r_up": sums[0][1], "a_lo": sl + sums[1][0],
            "a_up": su + sums[1][1]}


def _mc_rows(p, case, draws, mlo, mhi):
    """Kept shares and row terms of rows with the images given, by counting."""
    S, n = draws.shape
    cells = [int(c) for c in p.cells]
    w = torch.as_tensor(draws).cuda()
    k0 = n // 2
    step = max(1, int(3e8) // (S * max(math.prod(cells[:k0]), math.prod(cells[k0:]))))
    parts = {k: [] for k in ("lo", "up", "sink_lo", "sink_up", "trunc")}

    def cell_of(d, y):
        e = _edges(p, d)
        c = torch.searchsorted(e, y.contiguous(), right=True) - 1
        return torch.where(y == e[-1], cells[d] - 1, c)

    def counts(marks):
        halves = []
        for part in (marks[:k0], marks[k0:]):
            x = part[0]
            for m in part[1:]:
                x = (x[:, :, :, None] * m[:, :, None, :]).reshape(x.shape[0], S, -1)
            halves.append(x)
        return torch.bmm(halves[0].transpose(1, 2), halves[1]).reshape(halves[0].shape[0], -1)

    for r in range(0, mlo.shape[0], step):
        met, held, inside, outside = [], [], True, False
        for d in range(n):
            a = cell_of(d, w[None, :, d] + mlo[r:r + step, d, None])
            b = cell_of(d, w[None, :, d] + mhi[r:r + step, d, None])
            inside = inside & (a >= 0) & (b <= cells[d] - 1)
            outside = outside | (b < 0) | (a > cells[d] - 1)
            t = torch.arange(cells[d], device="cuda")
            met.append(((a[:, :, None] <= t) & (t <= b[:, :, None])).float())
            held.append(((a[:, :, None] == t) & (t == b[:, :, None])).float())
        up, low = counts(met).double(), counts(held).double()
        keep = up / S >= float(case["cutoff"])
        parts["up"].append(up[keep] / S)
        parts["lo"].append(low[keep] / S)
        parts["trunc"].append(torch.where(keep, 0.0, up).sum(1) / S)
        parts["sink_up"].append((~inside).double().mean(1))
        parts["sink_lo"].append(outside.double().mean(1))
    return {k: torch.cat(v) for k, v in parts.items()}


def _exact_mc(p, case, draws):
    if float(p.rows) * draws.shape[0] * p.total_cells > 6e12:
        return None
    out = dict.fromkeys(["row_ptr", "col", "lo", "up", "sink_lo", "sink_up", "trunc", "row_flags"])
    out.update(_mc_rows(p, case, draws, *_images(p)))
    room = _mc_room(case)
    out["lo"], out["up"] = _padded([out["lo"]], room), _padded([out["up"]], room)
    return out


def _exact_synth(p, case, labels):
    """Interval iteration with the sorting method, dense in 64 bits."""
    T, J = p.total_cells, p.n_inputs
    mlo, mhi = _images(p)
    up, low = _dense_rows(p, mlo, mhi)
    drop = up < p.cutoff
    sl, su = _sinks(p, mlo, mhi)
    zero = torch.zeros_like(sl)
    # successors: the cells, the sink, the truncated mass
    w_lo = torch.cat([torch.where(drop, 0.0, low), sl[:, None], zero[:, None]], 1)
    w_up = torch.cat([torch.where(drop, 0.0, up), su[:, None],
                      torch.where(drop, up, 0.0).sum(1)[:, None]], 1)
    width, rest = w_up - w_lo, (1.0 - w_lo.sum(1)).clamp_min(0.0)
    reach = case["spec"] == "reach"
    free = labels == 0
    hold = (labels == (1 if reach else 2)).double()

    def lp(v, maximize):
        v = torch.cat([v, v.new_tensor([0.0 if reach else 1.0, 1.0 if maximize else 0.0])])
        order = torch.argsort(v, descending=maximize)
        ws = width[:, order]
        before = torch.cumsum(ws, 1) - ws
        fill = torch.minimum(ws, (rest[:, None] - before).clamp_min(0.0))
        return w_lo @ v + fill @ v[order]

    lower_max = not reach
    first = not lower_max if case["optimistic"] else lower_max
    policy, ends = None, {}
    for phase, maximize in enumerate((first, not first)):
        v0 = torch.where(free, 0.0, hold)
        v1 = v0.clone() if case["horizon"] else torch.where(free, 1.0, hold)
        for _ in range(case["horizon"] or 10000):
            q = [lp(v, maximize).reshape(T, J) for v in (v0, v1)]
            if phase == 0:
                best = [x.max(1) if reach else x.min(1) for x in q]
                policy = best[1 if first else 0].indices
                new = [x.values for x in best]
            else:
                new = [x.gather(1, policy[:, None])[:, 0] for x in q]
            v0, v1 = (torch.where(free, x.clamp(0.0, 1.0), hold) for x in new)
            if not case["horizon"] and float((v1 - v0).abs().max()) <= 1e-6:
                break
        if reach:
            ends["p_max" if maximize else "p_min"] = v1 if maximize else v0
        else:
            ends["p_min" if maximize else "p_max"] = 1.0 - (v1 if maximize else v0)
    return {**ends, "policy": None, "iterations": None}


def exact(case, seed):
    entry, prec = case["entry"], case["precision"]
    if entry == "serve":
        return [_exact_build(p, prec, 0, only_sinks=True) for p in _batch(case, seed)]
    if entry in ("graph", "into"):
        parts = [_exact_build(p, prec, 0, only_sinks=True) for p in _batch(case, seed)]
        return {k: None if parts[0][k] is None else torch.cat([q[k] for q in parts])
                for k in parts[0]}
    p = _problem(case, seed)
    if entry == "regions":
        return _exact_regions(p, case, _boxes(p, seed))
    if entry == "mc":
        return _exact_mc(p, case, _draws(p, case, seed))
    if entry == "synth":
        # FP32 bounds are another IMDP; region vectors add successors
        if prec != "fp64" or case["with_regions"] or p.rows * p.total_cells > 4e6:
            return None
        t, a = _boxes(p, seed)
        return _exact_synth(p, case, torch.as_tensor(W.region_labels(p, t, a)).cuda())
    return _exact_build(p, prec, _room(_problem(case, 0)))
