"""The work that is timed: what a program that uses this library calls, over the sizes it calls it with.

A case names a kind of call and its sizes:

  step        one outer step of the integrator on a state the program holds on the GPU: set_state, evolve,
              get_state (a coupled code hands its bodies over, steps them and takes them back)
  dkd         a program's own splitting level from the unit calls: components, drift, kick, drift
  graph       the time-step graph of a state as an edge list
  components  the component labels of a caller-held state, with no allocation by the library
  energy      the conserved quantities, which every run checks as it goes
"""
import math

import numpy as np
import torch

from paper_1407_7105_gb300 import cc, ics

ETA = 0.03


def listed():
    return [
        # the smallest cluster that is run by itself: one step is mostly latency and launches
        {"name": "step_fp64_plummer256", "kind": "step", "ics": "plummer", "n": 256, "form": "fp64", "dt": 1 / 64},
        # an ordinary open-cluster model: a softened sphere of about a thousand bodies
        {"name": "step_mixed_soft1024", "kind": "step", "ics": "plummer", "n": 1024, "form": "mixed", "dt": 1 / 64,
         "eps": 1 / 256},
        # the production run: a rich cluster in the mixed form
        {"name": "step_mixed_plummer16384", "kind": "step", "ics": "plummer", "n": 16384, "form": "mixed",
         "dt": 1 / 256},
        # the same cluster in the reference form, which a result is checked with
        {"name": "step_fp64_plummer16384", "kind": "step", "ics": "plummer", "n": 16384, "form": "fp64",
         "dt": 1 / 256},
        # a young clumpy cluster with a mass spectrum: the largest single system, hard binaries among its clumps
        {"name": "step_mixed_fractal65536", "kind": "step", "ics": "fractal", "n": 65536, "form": "mixed",
         "dt": 1 / 256},
        # a cluster whose primordial binaries go to the Kepler solver
        {"name": "step_kepler_binaries32768", "kind": "step", "ics": "binaries", "n": 32768, "form": "mixed",
         "dt": 1 / 256, "kepler": 1},
        # a survey of small systems, triples and clumps, stepped together
        {"name": "step_mixed_systems4096", "kind": "step", "ics": "systems", "nsys": 4096, "form": "mixed",
         "dt": 1 / 64},
        # the split of interactions instead of particles, at a ragged size
        {"name": "step_ok_fp64_plummer5003", "kind": "step", "ics": "plummer", "n": 5003, "form": "fp64",
         "dt": 1 / 256, "split": "ok"},
        # an own integrator built from the unit calls
        {"name": "dkd_mixed_plummer40009", "kind": "dkd", "ics": "plummer", "n": 40009, "form": "mixed",
         "dt": 1 / 256},
        # who is close to whom: the graph of a snapshot, for an analysis
        {"name": "graph_plummer10007", "kind": "graph", "ics": "plummer", "n": 10007, "dt": 1 / 256},
        # the components of another code's bodies, inside that code's own memory budget
        {"name": "components_plummer30011", "kind": "components", "ics": "plummer", "n": 30011, "dt": 1 / 256},
        # the diagnostics of the largest system
        {"name": "energy_plummer65536", "kind": "energy", "ics": "plummer", "n": 65536, "dt": 1 / 256},
    ]


def _size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["mixed", "mixed", "fp64", "fractal", "binaries", "systems", "other", "dkd", "graph",
                       "components", "energy"])
    if what in ("mixed", "fp64"):
        n = _size(rng, 64, 16384)
        return {"kind": "step", "ics": "plummer", "n": n, "form": what, "dt": 1 / 64 if n < 2048 else 1 / 256,
                "eps": rng.choice([0.0, 1 / 256])}
    if what == "fractal":
        return {"kind": "step", "ics": "fractal", "n": _size(rng, 4096, 65536), "form": "mixed", "dt": 1 / 256}
    if what == "binaries":
        # (h_fp64: forces in 64 bits inside the close components, as a careful run asks for)
        return {"kind": "step", "ics": "binaries", "n": _size(rng, 2048, 32768), "form": "mixed", "dt": 1 / 256,
                "kepler": 1, "h_fp64": rng.choice([0.0, 1 / 256 / 64])}
    if what == "systems":
        return {"kind": "step", "ics": "systems", "nsys": _size(rng, 16, 4096), "form": "mixed", "dt": 1 / 64}
    if what == "other":
        return {"kind": "step", "ics": "plummer", "n": _size(rng, 256, 8192), "dt": 1 / 256,
                **rng.choice([{"split": "ok", "form": "fp64"}, {"split": "hold", "form": "mixed"}])}
    if what == "dkd":
        return {"kind": "dkd", "ics": "plummer", "n": _size(rng, 256, 40009),
                "form": rng.choice(["mixed", "mixed", "fp64"]), "dt": 1 / 256}
    if what == "graph":
        return {"kind": "graph", "ics": "plummer", "n": _size(rng, 64, 16384), "dt": 1 / 256}
    if what == "components":
        return {"kind": "components", "ics": "plummer", "n": _size(rng, 64, 32768), "dt": 1 / 256}
    return {"kind": "energy", "ics": rng.choice(["plummer", "binaries"]), "n": _size(rng, 256, 65536), "dt": 1 / 256}


# ------------------------------------------------------------------ inputs
def _plummer(n, seed):
    """An equal-mass sphere in N-body units: E = -1/4 with its own potential energy, in virial equilibrium."""
    m, x, v = ics.plummer(n, seed=seed, exact_scale=False)
    return m, *ics.scale_to_nbody_units(m, x, v, Q=0.5, exact=False, W=_potential(m, x, 0.0))


def _fractal(n, seed):
    """The clumpy cluster with a mass spectrum, in N-body units."""
    x, v = ics.box_fractal_raw(n, seed=seed)
    m = ics.salpeter_masses(n, seed, 9100)
    x, v = ics._com_frame(m, x, v)
    return m, *ics.scale_to_nbody_units(m, x, v, Q=0.3, exact=False, W=_potential(m, x, 0.0))


def _systems(nsys, seed):
    """Triples and clumps of log-uniform 3..512 bodies, each in its own units; the survey's sizes stay, its states
    are the seed's."""
    coin, size = ics.uniform(1, 31, nsys), ics.uniform(1, 32, nsys)
    parts = []
    for k in range(nsys):
        if coin[k] < 0.5:
            parts.append(ics.hierarchical_triple(seed, 100000 + 37 * k))
        else:
            n = int(round(3 * math.exp(math.log(512 / 3) * size[k])))
            parts.append(ics.plummer(n, seed=seed * 4099 + k, exact_scale=True))
    off = np.concatenate([[0], np.cumsum([p[0].shape[0] for p in parts])])
    return tuple(np.concatenate([p[q] for p in parts], axis=-1) for q in range(3)) + (off,)


def _state(case, seed):
    seed = 1 + seed % 1000003
    off = None
    if case["ics"] == "plummer":
        m, x, v = _plummer(case["n"], seed)
    elif case["ics"] == "fractal":
        m, x, v = _fractal(case["n"], seed)
    elif case["ics"] == "binaries":
        m, x, v = ics.plummer_with_binaries(case["n"], seed=seed)
    else:
        m, x, v, off = _systems(case["nsys"], seed)
    if case["kind"] == "energy":
        # a cluster on its way through a galaxy: momentum and angular momentum are not zero
        x = x + np.array([[3.0], [-2.0], [0.5]])
        v = v + np.array([[0.2], [0.7], [-0.4]])
    return m, np.ascontiguousarray(x), np.ascontiguousarray(v), off


def _params(case):
    split = {"cc": cc.SPLIT_CC, "hold": cc.SPLIT_HOLD, "ok": cc.SPLIT_OK}[case.get("split", "cc")]
    return cc.default_params(dt=case["dt"], eta=ETA, eps=case.get("eps", 0.0), kepler=case.get("kepler", 0),
                             h_fp64=case.get("h_fp64", 0.0), split=split,
                             precision=cc.PREC_MIXED if case.get("form") == "mixed" else cc.PREC_FP64)


def prepare(case, seed):
    m, x, v, off = _state(case, seed)
    s = {"case": case, "m": torch.tensor(m, device="cuda"), "x": torch.tensor(x, device="cuda"),
         "v": torch.tensor(v, device="cuda"), "params": _params(case)}
    n = m.shape[0]
    if case["kind"] == "components":
        s["labels"] = torch.zeros(n, dtype=torch.int32, device="cuda")
        s["ncomp"] = torch.zeros(1, dtype=torch.int64, device="cuda")
        return s
    s["ctx"] = cc.Context(s["m"], s["x"], s["v"], params=s["params"])
    if case["kind"] == "graph":
        s["edges"] = np.empty((64 * n, 2), dtype=np.int32)  # the analysis' own edge buffer
    if off is not None:
        s["ctx"].set_systems(off)
    if case["kind"] in ("step", "dkd"):
        s["x1"], s["v1"] = torch.empty_like(s["x"]), torch.empty_like(s["v"])
        s["labels"] = torch.zeros(n, dtype=torch.int32, device="cuda")
    return s


def run(s):
    case, ctx, h = s["case"], s.get("ctx"), s["case"]["dt"]
    if case["kind"] == "step":
        ctx.set_state(0.0, s["m"], s["x"], s["v"])
        ctx.evolve(h)
        ctx.get_state(x3=s["x1"], v3=s["v1"], alloc=False)
        return {"x": s["x1"], "v": s["v1"]}
    if case["kind"] == "dkd":
        ctx.set_state(0.0, None, s["x"], s["v"])
        labels, ncomp = ctx.components(h, labels_out=s["labels"])
        ctx.drift(labels, 0.5 * h)
        ctx.kick(labels, h)
        ctx.drift(labels, 0.5 * h)
        ctx.get_state(x3=s["x1"], v3=s["v1"], alloc=False)
        return {"x": s["x1"], "v": s["v1"], "labels": labels, "ncomp": ncomp}
    if case["kind"] == "graph":
        edges, count, near = ctx.timestep_graph(h, cap=s["edges"].shape[0])
        s["edges"][:count] = edges
        s["edges"][count:] = -1
        return {"edges": s["edges"], "count": count, "near": near}
    if case["kind"] == "components":
        cc.components_noalloc(s["m"], s["x"], s["v"], h, s["labels"], s["ncomp"], params=s["params"])
        return {"labels": s["labels"], "ncomp": s["ncomp"]}
    e, p, ang = ctx.energy()
    return {"energy": e, "momentum": p, "angular_momentum": ang}


# ------------------------------------------------------------------ work
TAU_FLOPS, KICK_FLOPS, POT_FLOPS = 47, 25, 13  # a pair's time step, its kick on both bodies, its potential


def work(case):
    """The outermost level's pairs, which no step goes without (what its components need below it depends on the
    state), and the state in and out once."""
    if case["ics"] == "systems":
        # half of the systems triples, half clumps of log-uniform 3..512 bodies
        n, pairs = case["nsys"] * 52, case["nsys"] * 7000
    else:
        n, pairs = case["n"], case["n"] * (case["n"] - 1) / 2
    if case["kind"] == "energy":
        return {"bytes": 56 * n + 56, "flops": POT_FLOPS * pairs}
    if case["kind"] in ("graph", "components"):
        return {"bytes": 56 * n + 4 * n, "flops": TAU_FLOPS * pairs}
    return {"bytes": 104 * n, "flops": (TAU_FLOPS + KICK_FLOPS) * pairs}


# ------------------------------------------------------------------ the same in plain 64 bits
# The definitions, set by set: sets of at most SMALL bodies in numpy, larger ones in torch, row block by row block.
SMALL = 96


def _tau(xp, dx, dv, mu, eps2):
    r2 = (dx * dx).sum(0) + eps2
    v2 = (dv * dv).sum(0)
    rv = (dx * dv).sum(0)
    r = xp.sqrt(r2)
    tff = ETA * xp.sqrt(r2 * r / mu)
    tff = tff / (1 - 0.5 * (1.5 * tff * rv / r2).clip(max=1.0))
    tfb = ETA * r / xp.sqrt(v2)
    tfb = tfb / (1 - 0.5 * (tfb * rv / r2 * (1 + mu / (r * v2))).clip(max=1.0))
    return xp.minimum(tff, tfb)


def _rows(n):
    step = max(1, (1 << 25) // n)
    return [(a, min(n, a + step)) for a in range(0, n, step)]


def _cuda(*arrays):
    return [torch.tensor(a, device="cuda") for a in arrays]


def _edges(m, x, v, h, eps2):
    n = m.shape[0]
    if n <= SMALL:
        i, j = np.triu_indices(n, 1)
        on = _tau(np, x[:, i] - x[:, j], v[:, i] - v[:, j], m[i] + m[j], eps2) < h
        return i[on], j[on]
    tm, tx, tv = _cuda(m, x, v)
    found = []
    for a, b in _rows(n):
        t = _tau(torch, tx[:, a:b, None] - tx[:, None, :], tv[:, a:b, None] - tv[:, None, :],
                 tm[a:b, None] + tm[None, :], eps2)
        e = torch.nonzero(t < h)
        e[:, 0] += a
        found.append(e[e[:, 0] < e[:, 1]])
    e = torch.cat(found).cpu().numpy()
    return e[:, 0], e[:, 1]


def _labels(n, i, j):
    lab = np.arange(n)
    while True:
        new = lab.copy()
        low = np.minimum(lab[i], lab[j])
        np.minimum.at(new, i, low)
        np.minimum.at(new, j, low)
        np.minimum.at(new, lab[i], low)
        np.minimum.at(new, lab[j], low)
        new = new[new]
        if np.array_equal(new, lab):
            return lab
        lab = new


def _potential(m, x, eps2):
    tm, tx = _cuda(m, x)
    pot = torch.zeros((), dtype=torch.float64, device="cuda")
    for a, b in _rows(m.shape[0]):
        r2 = ((tx[:, None, :] - tx[:, a:b, None]) ** 2).sum(0) + eps2
        r2[torch.arange(b - a), torch.arange(a, b)] = math.inf
        pot -= 0.5 * (tm[a:b, None] * tm[None, :] / r2.sqrt()).sum()
    return pot.item()


def _kick(m, x, v, lab, h, eps2):
    n = m.shape[0]
    if n <= SMALL:
        dx = x[:, None, :] - x[:, :, None]
        r2 = (dx * dx).sum(0) + eps2
        other = lab[:, None] != lab[None, :]
        w = np.where(other, m[None, :] / np.where(other, r2 * np.sqrt(r2), 1.0), 0.0)
        return v + h * (w[None] * dx).sum(2)
    tm, tx, tl = _cuda(m, x, lab)
    a3 = []
    for a, b in _rows(n):
        dx = tx[:, None, :] - tx[:, a:b, None]
        r2 = (dx * dx).sum(0) + eps2
        w = torch.where(tl[a:b, None] != tl[None, :], tm[None, :] / (r2 * r2.sqrt()), torch.zeros_like(r2))
        a3.append((w[None] * dx).sum(2))
    return v + h * torch.cat(a3, 1).cpu().numpy()


def _pair(m, x, v, h, eps2):
    """A two-body set: its own recursion in plain numbers."""
    ma, mb = float(m[0]), float(m[1])
    r0, r1, r2 = (float(x[k, 0] - x[k, 1]) for k in range(3))
    u0, u1, u2 = (float(v[k, 0] - v[k, 1]) for k in range(3))
    mu, todo = ma + mb, [h]
    while todo:
        g = todo.pop()
        q = r0 * r0 + r1 * r1 + r2 * r2 + eps2
        w = u0 * u0 + u1 * u1 + u2 * u2
        rv = r0 * u0 + r1 * u1 + r2 * u2
        r = math.sqrt(q)
        tau = ETA * math.sqrt(q * r / mu)
        tau = tau / (1 - 0.5 * min(1.5 * tau * rv / q, 1.0))
        if w > 0.0:
            fb = ETA * r / math.sqrt(w)
            tau = min(tau, fb / (1 - 0.5 * min(fb * rv / q * (1 + mu / (r * w)), 1.0)))
        if tau < g:
            todo += [0.5 * g, 0.5 * g]
            continue
        r0, r1, r2 = r0 + 0.5 * g * u0, r1 + 0.5 * g * u1, r2 + 0.5 * g * u2
        q = r0 * r0 + r1 * r1 + r2 * r2 + eps2
        f = -g * mu / (q * math.sqrt(q))
        u0, u1, u2 = u0 + f * r0, u1 + f * r1, u2 + f * r2
        r0, r1, r2 = r0 + 0.5 * g * u0, r1 + 0.5 * g * u1, r2 + 0.5 * g * u2
    c, cv = (x @ m) / mu + h * (v @ m) / mu, (v @ m) / mu
    d, dv = np.array([r0, r1, r2]), np.array([u0, u1, u2])
    x[:, 0], x[:, 1] = c + mb / mu * d, c - ma / mu * d
    v[:, 0], v[:, 1] = cv + mb / mu * dv, cv - ma / mu * dv


def _step_cc(m, x, v, h, eps2, hold):
    if m.shape[0] == 2:
        return _pair(m, x, v, h, eps2)
    i, j = _edges(m, x, v, h, eps2)
    lab = _labels(m.shape[0], i, j)
    size = np.bincount(lab, minlength=lab.shape[0])[lab]
    if hold and i.size:
        lab = np.where(size > 1, lab[size > 1].min(), lab)
    parts = [np.flatnonzero(lab == c) for c in np.unique(lab[size > 1])]
    rest = size == 1
    for half in range(2):
        for p in parts:
            px, pv = x[:, p], v[:, p]
            _step_cc(m[p], px, pv, 0.5 * h, eps2, hold)
            x[:, p], v[:, p] = px, pv
        if half == 0 and len(parts[0] if parts else ()) < m.shape[0]:
            x[:, rest] += 0.5 * h * v[:, rest]
            v[:] = _kick(m, x, v, lab, h, eps2)
            x[:, rest] += 0.5 * h * v[:, rest]


def _step_ok(m, x, v, i, j, mine, h, eps2):
    """The interactions (i, j) among the bodies `mine`; i is None for all pairs, at the outer step."""
    if i is None:
        a, b = _edges(m, x, v, h, eps2)
    else:
        fast = _tau(np, x[:, i] - x[:, j], v[:, i] - v[:, j], m[i] + m[j], eps2) < h
        a, b = i[fast], j[fast]
    sub = np.unique(np.concatenate([a, b]))
    rest = np.setdiff1d(mine, sub, assume_unique=True)
    for half in range(2):
        if a.size:
            _step_ok(m, x, v, a, b, sub, 0.5 * h, eps2)
        if half == 0:
            x[:, rest] += 0.5 * h * v[:, rest]
            if i is None:  # every pair, less the fast ones
                v[:] = _kick(m, x, v, np.arange(m.shape[0]), h, eps2)
                si, sj, sign = a, b, -1.0
            else:
                si, sj, sign = i[~fast], j[~fast], 1.0
            dx = x[:, sj] - x[:, si]
            r2 = (dx * dx).sum(0) + eps2
            f = sign * h * dx / (r2 * np.sqrt(r2))
            for k in range(3):
                v[k] += np.bincount(si, f[k] * m[sj], m.shape[0]) - np.bincount(sj, f[k] * m[si], m.shape[0])
            x[:, rest] += 0.5 * h * v[:, rest]


def exact(case, seed):
    if case["kind"] in ("graph", "components"):
        return None  # whole numbers
    if case.get("kepler") or case["ics"] in ("fractal", "systems"):
        if case["kind"] != "energy":
            return None  # too many small sets for a plain program
    m, x, v, _ = _state(case, seed)
    h, eps2 = case["dt"], case.get("eps", 0.0) ** 2
    if case["kind"] == "energy":
        return {"energy": float(0.5 * (m * (v * v).sum(0)).sum()) + _potential(m, x, eps2), "momentum": v @ m,
                "angular_momentum": np.cross(x.T, v.T).T @ m}
    if case["kind"] == "dkd":
        i, j = _edges(m, x, v, h, eps2)
        lab = _labels(m.shape[0], i, j)
        rest = np.bincount(lab, minlength=lab.shape[0])[lab] == 1
        x[:, rest] += 0.5 * h * v[:, rest]
        v = _kick(m, x, v, lab, h, eps2)
        x[:, rest] += 0.5 * h * v[:, rest]
        return {"x": x, "v": v, "labels": None, "ncomp": None}
    if case.get("split") == "ok":
        _step_ok(m, x, v, None, None, np.arange(m.shape[0]), h, eps2)
    else:
        _step_cc(m, x, v, h, eps2, case.get("split") == "hold")
    return {"x": x, "v": v}
