"""Workloads the library's speed is measured on, each through its public entry points.

A case is a dict of plain values; ``listed()`` gives the fixed ones and ``draw(rng)`` more of
the same ranges. ``prepare(case, seed)`` builds what a program holds before the call (the
particles, the handle, device buffers), ``run(state)`` is one pass, ``work(case)`` the bytes and
floating-point operations a pass cannot do without, and ``exact(case, seed)`` the results in
64-bit arithmetic from plain torch.

Kinds of work:

- ``force``: acceleration, jerk and potential of the whole system (``ni`` = 0; prediction
  included, as in every step) or of ``ni`` members (a due set) from all ``n`` particles, into
  device buffers;
- ``snap``: the 6th-order scheme's evaluation (with the snap) of the whole system, host arrays;
- ``ext``: the field of ``n`` particles at ``ni`` outside positions, host arrays in and out (what a
  tree code or a bridge asks of the direct solver);
- ``shared``: Hermite steps of one common size;
- ``block``: block time steps over ``span`` from a checkpoint;
- ``batch``: shared steps of many clusters of uneven size in one graph replay;
- ``serve``: a burst of force and integration requests of uneven size through the request loop.

FP32 pair arithmetic (plain or double-single) gives results of FP32 accuracy, so these cases hand
their outputs on in single precision; FP64 pairs hand on binary64.
"""
import math

import numpy as np
import torch

from paper_1409_5474_gb300 import nbody

SHARED_DT = 1.0 / 256
BATCH_DT = 1.0 / 512
ETA = 0.01
DT_MAX = 1.0 / 16
FLOPS_PAIR = 60   # acc + jerk + pot of one pair, the metric's count
FLOPS_SNAP = 97   # acc + jerk + snap + pot


def listed():
    return [
        # the tail of a block step: three particles due among 65536
        {"name": "force_tiny", "kind": "force", "n": 65536, "ni": 3, "variant": "f32ds"},
        # an ordinary due set, a ragged count
        {"name": "force_due", "kind": "force", "n": 65536, "ni": 1531, "variant": "f32ds"},
        # a full evaluation of a large cluster with a mass spectrum
        {"name": "force_whole", "kind": "force", "n": 262144, "ni": 0, "variant": "f32ds"},
        # the plain FP32 kind, an odd size
        {"name": "force_f32", "kind": "force", "n": 40961, "ni": 0, "variant": "f32"},
        # the native FP64 kind (extreme mass ratios, reference runs), an odd size
        {"name": "force_f64", "kind": "force", "n": 6007, "ni": 0, "variant": "f64"},
        # the 6th-order scheme's evaluation
        {"name": "snap", "kind": "snap", "n": 20011, "variant": "f32ds"},
        # outside positions in a cluster's field
        {"name": "ext", "kind": "ext", "n": 50000, "ni": 10007, "variant": "f32ds"},
        # the small plain method: 1024 particles, FP64, one shared step
        {"name": "shared_f64", "kind": "shared", "n": 1024, "steps": 16, "variant": "f64"},
        # block steps of a small cluster, where every step is latency
        {"name": "block_small", "kind": "block", "n": 2500, "span": 0.0625, "variant": "f32ds"},
        # block steps at the size of a production run: due sets from 1 to all particles
        {"name": "block_large", "kind": "block", "n": 65536, "span": 0.0625, "variant": "f32ds"},
        # many independent clusters, sizes log-uniform
        {"name": "batch", "kind": "batch", "systems": 512, "n_lo": 16, "n_hi": 4096, "steps": 8,
         "variant": "f32ds"},
        # a burst of requests from a hybrid code, half forces, half integrations
        {"name": "serve", "kind": "serve", "requests": 16, "n_lo": 256, "n_hi": 16384,
         "span": 0.0625, "variant": "f32ds"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("force", "force", "due", "due", "f64", "snap", "ext", "shared", "block",
                       "batch", "serve"))
    if kind == "force":
        return {"kind": "force", "n": _log_int(rng, 300, 200000), "ni": 0,
                "variant": rng.choice(("f32ds", "f32ds", "f32"))}
    if kind == "due":
        n = _log_int(rng, 4000, 200000)
        return {"kind": "force", "n": n, "ni": _log_int(rng, 1, n // 3),
                "variant": rng.choice(("f32ds", "f32ds", "f32ds", "f64")) if n < 20000 else "f32ds"}
    if kind == "f64":
        return {"kind": "force", "n": _log_int(rng, 300, 12000), "ni": 0, "variant": "f64"}
    if kind == "snap":
        return {"kind": "snap", "n": _log_int(rng, 500, 60000), "variant": "f32ds"}
    if kind == "ext":
        return {"kind": "ext", "n": _log_int(rng, 500, 100000), "ni": _log_int(rng, 5, 60000),
                "variant": "f32ds"}
    if kind == "shared":
        f64 = rng.random() < 0.5
        return {"kind": "shared", "n": _log_int(rng, 256, 3000 if f64 else 20000),
                "steps": rng.choice((1, 4, 16)), "variant": "f64" if f64 else "f32ds"}
    if kind == "block":
        return {"kind": "block", "n": _log_int(rng, 500, 20000), "span": 0.0625,
                "variant": rng.choice(("f32ds", "f32ds", "f32ds", "f32"))}
    if kind == "batch":
        return {"kind": "batch", "systems": _log_int(rng, 40, 500), "n_lo": 16,
                "n_hi": _log_int(rng, 512, 4096), "steps": rng.choice((1, 4, 8)),
                "variant": "f32ds"}
    return {"kind": "serve", "requests": rng.choice((4, 8, 12, 16)), "n_lo": 256,
            "n_hi": _log_int(rng, 1024, 16384), "span": 0.0625, "variant": "f32ds"}


# ---- inputs ---------------------------------------------------------------------


def _plummer(n, rng, spectrum=False):
    """Plummer sphere in N-body units: m (n,), pos (n, 3), vel (n, 3). Speeds by inverting the
    cumulative distribution of q = v / v_esc, g(q) = q^2 (1 - q^2)^(7/2), on a fine grid."""
    def directions():
        c = rng.uniform(-1.0, 1.0, n)
        phi = rng.uniform(0.0, 2.0 * math.pi, n)
        s = np.sqrt(1.0 - c * c)
        return np.stack([s * np.cos(phi), s * np.sin(phi), c], axis=1)

    x = rng.uniform(1e-9, 0.997, n)   # enclosed mass fraction, to about 22 scale lengths
    r = 1.0 / np.sqrt(x ** (-2.0 / 3.0) - 1.0)
    grid = np.linspace(0.0, 1.0, 8193)
    cum = np.concatenate([[0.0], np.cumsum((lambda q: q * q * (1.0 - q * q) ** 3.5)(
        0.5 * (grid[1:] + grid[:-1])))])
    q = np.interp(rng.uniform(0.0, 1.0, n) * cum[-1], cum, grid)
    vesc = math.sqrt(2.0) * (1.0 + r * r) ** -0.25
    m = np.exp(0.5 * rng.standard_normal(n)) if spectrum else np.ones(n)
    m /= m.sum()
    scale = 3.0 * math.pi / 16.0
    pos = scale * r[:, None] * directions()
    vel = (q * vesc)[:, None] * directions() / math.sqrt(scale)
    pos -= (m[:, None] * pos).sum(axis=0)
    vel -= (m[:, None] * vel).sum(axis=0)
    return m, pos, vel


def _galaxy(n, rng):
    """Plummer sphere with a central point mass of 1% of its mass."""
    m, pos, vel = _plummer(n - 1, rng)
    return (np.concatenate([[0.01], 0.99 * m]), np.concatenate([np.zeros((1, 3)), pos]),
            np.concatenate([np.zeros((1, 3)), vel]))


def _sizes(count, lo, hi):
    """count sizes spread evenly over the logarithm of [lo, hi]."""
    u = (np.arange(count) + 0.5) / count
    return np.rint(np.exp(math.log(lo) + u * (math.log(hi) - math.log(lo)))).astype(np.int64)


def _eps(case):
    return {"force": 1e-4, "snap": 1e-3, "ext": 1e-3, "shared": 1.0 / 64, "block": 1e-3}[case["kind"]]


def _inputs(case, seed):
    """Particles (and whatever else the case draws), as host arrays, from the seed alone."""
    rng = np.random.default_rng(int(seed))
    kind = case["kind"]
    if kind == "batch":
        sizes = _sizes(case["systems"], case["n_lo"], case["n_hi"])
        rng.shuffle(sizes)
        return {"systems": [_plummer(int(n), rng) for n in sizes], "eps": 0.25 / np.cbrt(sizes)}
    if kind == "serve":
        sizes = _sizes(case["requests"], case["n_lo"], case["n_hi"])
        order = np.random.default_rng(5).permutation(case["requests"])  # arrival order
        return {"requests": [_galaxy(int(sizes[k]), rng) for k in order]}
    n = case["n"]
    d = {"p": _plummer(n, rng, spectrum=kind in ("force", "ext", "snap"))}
    if kind == "force" and case["ni"]:
        d["idx"] = np.sort(rng.permutation(n)[: case["ni"]]).astype(np.int32)
    if kind == "ext":
        _, d["pos"], d["vel"] = _plummer(case["ni"], rng)
    return d


def _evolves(k):
    """Every second request is an integration."""
    return k % 2 == 1


def _request_eps(n):
    return 0.25 / n ** (1.0 / 3.0)


# ---- the passes -----------------------------------------------------------------


class _Records:
    """Systems given as (m, pos, vel) in the form nbody.Batch takes."""

    def __init__(self, m, pos, vel):
        self.m, self.pos, self.vel = m, pos, vel


def prepare(case, seed):
    d = _inputs(case, seed)
    kind, variant = case["kind"], case["variant"]
    s = {"case": dict(case)}
    if kind == "batch":
        s["batch"] = nbody.Batch([_Records(*p) for p in d["systems"]], d["eps"], BATCH_DT,
                                 variant=variant)
        s["batch"].step(0)  # the initial evaluation
        return s
    if kind == "serve":
        s["server"] = nbody.Server(variant=nbody.VARIANTS[variant], eta=ETA, dt_max=DT_MAX)
        s["requests"] = [(m, np.ascontiguousarray(pos.T), np.ascontiguousarray(vel.T),
                          _request_eps(len(m))) for m, pos, vel in d["requests"]]
        return s
    more = {"shared_dt": SHARED_DT} if kind == "shared" else {}
    if kind == "snap":
        more["order"] = 6
    s["sys"] = sy = nbody.System(*d["p"], variant=variant, eps=_eps(case), eta=ETA, dt_max=DT_MAX,
                                 **more)
    if kind == "force":
        ni = case["ni"] or case["n"]
        nbody.nb_set_stream(sy.h, torch.cuda.current_stream().cuda_stream)
        sy.predict(0.0)
        s["idx"] = torch.from_numpy(d["idx"]).cuda() if case["ni"] else None
        s["out"] = torch.empty((7, ni), dtype=torch.float64, device="cuda")
    elif kind == "snap":
        nbody.nb_init(sy.h)
    elif kind == "ext":
        sy.predict(0.0)
        s["pos"], s["vel"] = (np.ascontiguousarray(d[k].T) for k in ("pos", "vel"))
    elif kind == "shared":
        nbody.nb_init(sy.h)
        s["t"] = 0.0
    elif kind == "block":
        nbody.nb_init(sy.h)
        s["checkpoint"] = sy.state()
    return s


def _as(variant, *arrays):
    """Outputs at the accuracy of the pair arithmetic."""
    return tuple(a if variant == "f64" else a.astype(np.float32) for a in arrays)


def run(s):
    case = s["case"]
    kind, variant = case["kind"], case["variant"]
    if kind == "force":
        h, out = s["sys"].h, s["out"]
        if s["idx"] is None:
            nbody.nb_predict(h, 0.0)
        p, row = out.data_ptr(), out.stride(0) * 8
        nbody.nb_force_dev(h, s["idx"].data_ptr() if s["idx"] is not None else 0, out.shape[1],
                           p, p + 3 * row, p + 6 * row)
        out = out.clone() if variant == "f64" else out.to(torch.float32)
        return out[:3], out[3:6], out[6]
    if kind == "snap":
        s["sys"].predict(0.0)
        return _as(variant, *s["sys"].force_snap())
    if kind == "ext":
        return _as(variant, *s["sys"].force_ext(s["pos"], s["vel"]))
    if kind == "shared":
        s["t"] += case["steps"] * SHARED_DT
        s["sys"].step(s["t"])
        return _as(variant, *nbody.nb_get_particles(s["sys"].h)[1:])
    if kind == "block":
        s["sys"].set_state(s["checkpoint"])
        s["sys"].step(case["span"])
        return _as(variant, *nbody.nb_get_particles(s["sys"].h)[1:])
    if kind == "batch":
        s["batch"].step(case["steps"])
        return _as(variant, *s["batch"].get()[:2])
    srv = s["server"]
    tickets = [srv.evolve(*r, case["span"]) if _evolves(k) else srv.force(*r)
               for k, r in enumerate(s["requests"])]
    got = [srv.wait(t) for t in tickets]
    return [_as(variant, *((g["pos"], g["vel"]) if _evolves(k) else (g["acc"], g["jerk"], g["pot"])))
            for k, g in enumerate(got)]


# ---- the work a pass cannot do without --------------------------------------------


def _block_steps_per_particle(n, span):
    """Mean count of steps a particle takes over span at eta = 0.01: a fit to 14.1, 18.6, 24.0 and
    33.9 steps in 1/16 time unit, counted on Plummer spheres of 500, 2500, 10000 and 65536."""
    return 73.8 * n ** 0.18 * span


def work(case):
    kind, n = case["kind"], case.get("n", 0)
    state = 56.0  # m, pos, vel of a particle in binary64
    if kind in ("force", "snap", "ext"):
        ni = case.get("ni") or n
        rows = 10 if kind == "snap" else 7
        flops = float(ni) * n * (FLOPS_SNAP if kind == "snap" else FLOPS_PAIR)
        given = 48.0 * ni if kind == "ext" else 4.0 * ni if case.get("ni") else 0.0
        return {"bytes": state * n + given + rows * 8.0 * ni, "flops": flops}
    if kind == "shared":
        return {"bytes": 2 * 13 * 8.0 * n, "flops": FLOPS_PAIR * float(n) * n * case["steps"]}
    if kind == "block":
        pairs = _block_steps_per_particle(n, case["span"]) * float(n) * n
        return {"bytes": 2 * 15 * 8.0 * n, "flops": FLOPS_PAIR * pairs}
    if kind == "batch":
        sizes = _sizes(case["systems"], case["n_lo"], case["n_hi"]).astype(float)
        return {"bytes": 2 * 13 * 8.0 * float(sizes.sum()),
                "flops": FLOPS_PAIR * float((sizes ** 2).sum()) * case["steps"]}
    sizes = _sizes(case["requests"], case["n_lo"], case["n_hi"]).astype(float)
    order = np.random.default_rng(5).permutation(case["requests"])
    pairs, size = 0.0, 0.0
    for k, which in enumerate(order):
        q = sizes[which]
        pairs += q * q * ((1.0 + _block_steps_per_particle(q, case["span"])) if _evolves(k) else 1.0)
        size += q * (state + (48.0 if _evolves(k) else 56.0))
    return {"bytes": float(size), "flops": FLOPS_PAIR * float(pairs)}


# ---- the same results in 64 bits ----------------------------------------------------

_CHUNK = 1 << 25  # pairs held at once


def _force64(xi, vi, x, v, m, eps, own=None, ai=None, a=None):
    """acc, jerk (ni, 3) and pot (ni,) of positions xi from the particles x; own: their indices
    among x (the self pair leaves the potential; its other terms are 0). With the accelerations
    ai, a also the snap, before pot."""
    ni, n = xi.shape[0], x.shape[0]
    names = 2 if a is None else 3
    vec = [torch.empty((ni, 3), dtype=torch.float64, device=xi.device) for _ in range(names)]
    pot = torch.empty(ni, dtype=torch.float64, device=xi.device)
    for k in range(0, ni, max(1, _CHUNK // n)):
        b = slice(k, min(ni, k + max(1, _CHUNK // n)))
        d = [x[None, :, c] - xi[b, None, c] for c in range(3)]
        w = [v[None, :, c] - vi[b, None, c] for c in range(3)]
        r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2] + eps * eps
        rinv2 = 1.0 / r2
        mr = m[None, :] * torch.sqrt(rinv2)
        pot[b] = -mr.sum(dim=1)
        mr3 = mr * rinv2
        rv = (d[0] * w[0] + d[1] * w[1] + d[2] * w[2]) * rinv2
        for c in range(3):
            vec[0][b, c] = (mr3 * d[c]).sum(dim=1)
            vec[1][b, c] = (mr3 * (w[c] - 3.0 * rv * d[c])).sum(dim=1)
        if a is not None:
            g = [a[None, :, c] - ai[b, None, c] for c in range(3)]
            beta = (w[0] * w[0] + w[1] * w[1] + w[2] * w[2] + d[0] * g[0] + d[1] * g[1]
                    + d[2] * g[2]) * rinv2 + rv * rv
            for c in range(3):
                vec[2][b, c] = (mr3 * (g[c] - 6.0 * rv * (w[c] - 3.0 * rv * d[c])
                                       - 3.0 * beta * d[c])).sum(dim=1)
    if own is not None:
        pot += m[own] / eps
    return (*vec, pot)


def _cuda(*arrays):
    return tuple(torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in arrays)


def _rows(*tensors):
    return tuple((t.T if t.dim() == 2 else t).contiguous().cpu().numpy() for t in tensors)


def _correct64(x, v, a, j, h, a1, j1):
    """Hermite corrector over h (n, 1): new x, v, and a2, a3 at the end of the step."""
    xp, vp = _predict64(x, v, a, j, h)
    a2 = (-6.0 * (a - a1) - h * (4.0 * j + 2.0 * j1)) / h ** 2
    a3 = (12.0 * (a - a1) + 6.0 * h * (j + j1)) / h ** 3
    return (xp + h ** 4 / 24.0 * a2 + h ** 5 / 120.0 * a3, vp + h ** 3 / 6.0 * a2
            + h ** 4 / 24.0 * a3, a2 + h * a3, a3)


def _predict64(x, v, a, j, h):
    return x + h * v + h ** 2 / 2.0 * a + h ** 3 / 6.0 * j, v + h * a + h ** 2 / 2.0 * j


def _shared64(p, eps, dt, steps):
    m, x, v = _cuda(*p)
    own = torch.arange(len(m), device="cuda")
    h = torch.full((len(m), 1), dt, dtype=torch.float64, device="cuda")
    a, j, _ = _force64(x, v, x, v, m, eps, own)
    for _ in range(steps):
        xp, vp = _predict64(x, v, a, j, h)
        a1, j1, _ = _force64(xp, vp, xp, vp, m, eps, own)
        x, v, _, _ = _correct64(x, v, a, j, h, a1, j1)
        a, j = a1, j1
    return x, v


def _quantized64(raw, t):
    """The largest power of two <= raw, at most DT_MAX, that divides t."""
    d = torch.exp2(torch.floor(torch.log2(raw))).clamp(2.0 ** -30, DT_MAX)
    while True:
        bad = torch.floor(t / d) * d != t
        if not bool(bad.any()):
            return d
        d = torch.where(bad, 0.5 * d, d)


def _block64(p, eps, span):
    m, x, v = _cuda(*p)
    own = torch.arange(len(m), device="cuda")
    a, j, _ = _force64(x, v, x, v, m, eps, own)
    t = torch.zeros(len(m), dtype=torch.float64, device="cuda")
    dt = _quantized64(ETA * a.norm(dim=1) / j.norm(dim=1), 0.0 * t)
    while True:
        now = (t + dt).min()
        if float(now) > span:
            return x, v
        due = torch.nonzero(t + dt == now)[:, 0]
        xp, vp = _predict64(x, v, a, j, (now - t)[:, None])
        a1, j1, _ = _force64(xp[due], vp[due], xp, vp, m, eps, due)
        h = dt[due, None]
        x1, v1, a2, a3 = _correct64(x[due], v[due], a[due], j[due], h, a1, j1)
        x[due], v[due], a[due], j[due], t[due] = x1, v1, a1, j1, now
        na, nj, n2, n3 = (u.norm(dim=1) for u in (a1, j1, a2, a3))
        raw = torch.sqrt(ETA * (na * n2 + nj ** 2) / (nj * n3 + n2 ** 2))
        dt[due] = _quantized64(torch.minimum(raw, 2.0 * dt[due]), t[due])


def exact(case, seed):
    d = _inputs(case, seed)
    kind = case["kind"]
    if kind == "force":
        m, x, v = _cuda(*d["p"])
        own = torch.from_numpy(d["idx"]).cuda().long() if case["ni"] else torch.arange(
            len(m), device="cuda")
        return _rows(*_force64(x[own], v[own], x, v, m, _eps(case), own))
    if kind == "snap":
        m, x, v = _cuda(*d["p"])
        own = torch.arange(len(m), device="cuda")
        a0, _, _ = _force64(x, v, x, v, m, _eps(case), own)
        return _rows(*_force64(x, v, x, v, m, _eps(case), own, a0, a0))
    if kind == "ext":
        m, x, v = _cuda(*d["p"])
        return _rows(*_force64(*_cuda(d["pos"], d["vel"]), x, v, m, _eps(case)))
    if kind == "shared":
        return _rows(*_shared64(d["p"], _eps(case), SHARED_DT, case["steps"]))
    if kind == "block":
        # larger systems take minutes
        return _rows(*_block64(d["p"], _eps(case), case["span"])) if case["n"] <= 4096 else None
    if kind == "batch":
        got = [_shared64(p, e, BATCH_DT, case["steps"]) for p, e in zip(d["systems"], d["eps"])]
        return _rows(*(torch.cat([g[c] for g in got]) for c in range(2)))
    # the integrations of the larger requests take minutes
    out = []
    for k, p in enumerate(d["requests"]):
        eps = _request_eps(len(p[0]))
        if _evolves(k):
            out.append(_rows(*_block64(p, eps, case["span"])) if len(p[0]) <= 1024 else (None, None))
        else:
            m, x, v = _cuda(*p)
            out.append(_rows(*_force64(x, v, x, v, m, eps, torch.arange(len(m), device="cuda"))))
    return out
