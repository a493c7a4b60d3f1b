"""What users of the solver have it do, as cases that can be timed and checked.

A case is a dict of plain values.  ``listed()`` gives the standing cases,
``draw(rng)`` more of the same ranges, ``prepare(case, seed)`` what a program
holds before the call (inputs, and the solver, batch or server it keeps),
``run(state)`` one pass through the public entry points, ``work(case)`` the
bytes and operations the path cannot do without, ``exact(case, seed)`` the
result of a plain 64-bit evaluation of the method written here with torch.

Four kinds of case:

* ``event``  -- one event on a solver that is kept: set the state, advance it,
                read the result (``shasta.Solver``).  ``every`` > 0 reads the
                five totals after that many steps each, as a program that
                watches conservation does.
* ``batch``  -- many uneven events added to one pool, advanced together, read
                and removed (``shasta.Batch``).
* ``serve``  -- host arrays submitted to the serving loop and drained
                (``shasta.Server``).
* ``totals`` -- the five sums of caller-owned fields (``totals_noalloc``).
"""
import math
import random

import numpy as np
import torch

from paper_1206_0919_gb300 import shasta

LAM = 0.4
BAG_B, BAG_EC = 0.1, 0.5
TABLE_N, TABLE_DE = 20001, 0.005
FP32_FIELD, FP64_FIELD = 4, 8
# arithmetic of the method per cell and sweep: nine field passes of about 15
# operations, two recoveries of about 30, two sets of transport factors
FLOPS = 220


# ------------------------------------------------------------------ cases --

def _event(name, nx, ny, nz, precision, data, steps, bc="reflect", eos="ideal",
           fields="primitives", every=0):
    c = dict(kind="event", nx=nx, ny=ny, nz=nz, precision=precision, data=data, steps=steps, bc=bc,
             eos=eos, fields=fields, every=every)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the five sums of resident fields, called between other work: the
        # smallest call there is, latency and launches
        dict(name="totals_100", kind="totals", nx=100, ny=100, nz=100),
        # a small event of a scan over many: launch and chain latency
        _event("event_48_fp32", 48, 48, 48, "fp32", "hot", 30),
        # a program that advances step by step and watches the totals; the
        # conserved state in and out, as at a checkpoint
        _event("monitor_64_fp32", 64, 64, 64, "fp32", "flow", 12, bc="periodic",
               fields="conserved", every=1),
        # the planar shock tube in double, the accuracy reference
        _event("tube_64_fp64", 64, 64, 64, "fp64", "tube", 40),
        # a tabulated equation of state
        _event("table_96_fp32", 96, 96, 96, "fp32", "hot", 24, eos="table"),
        # odd extents, frozen ghosts, the bag model, compensated recovery
        _event("bag_ragged_mixed", 131, 97, 110, "mixed", "flow", 24, bc="frozen", eos="bag"),
        # the recovery in double on a single-precision state
        _event("recovery64_128", 128, 128, 128, "mixed_fp64", "hot", 12),
        # double precision on a ragged mid-size grid
        _event("bag_ragged_fp64", 143, 129, 151, "fp64", "flow", 6, bc="periodic", eos="bag"),
        # the standard event: 200^3 hot spots in single precision
        _event("hot_200_fp32", 200, 200, 200, "fp32", "hot", 75),
        # the large grid, from checkpoint to checkpoint
        _event("blast_512_fp32", 512, 512, 512, "fp32", "blast", 6, fields="conserved"),
        # uneven events advanced as one batch
        dict(name="batch_mixed", kind="batch", events=10, sizes_seed=3, precision="mixed",
             steps=48),
        # a burst of requests through the serving loop, host memory to host
        # memory, half on the bag model
        dict(name="serve_burst", kind="serve", events=8, sizes_seed=4, steps=150),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["event", "batch", "serve", "totals"], [15, 2, 1, 2])[0]
    if kind == "totals":
        return dict(kind=kind, nx=_log_int(rng, 20, 300), ny=_log_int(rng, 20, 300),
                    nz=_log_int(rng, 20, 300))
    if kind == "batch":
        return dict(kind=kind, events=rng.randint(3, 10), sizes_seed=rng.randrange(1 << 20),
                    precision=rng.choice(["fp32", "mixed"]), steps=_log_int(rng, 6, 48))
    if kind == "serve":
        return dict(kind=kind, events=rng.randint(2, 8), sizes_seed=rng.randrange(1 << 20),
                    steps=rng.randint(20, 150))
    precision = rng.choice(["fp32", "fp32", "mixed", "fp64", "mixed_fp64"])
    eos = rng.choice(["ideal", "ideal", "bag", "table"])
    if eos == "table" and precision not in ("fp32", "fp64"):
        eos = "bag"
    hi = 340 if precision in ("fp32", "mixed") and eos != "table" else 150
    n = _log_int(rng, 40, hi)
    dims = [max(17, int(n * rng.uniform(0.7, 1.35))) for _ in range(3)]
    if rng.random() < 0.3:
        dims = [n, n, n]
    cells = dims[0] * dims[1] * dims[2]
    per_step = cells / (2e8 if precision == "fp64" else 1e9 if hi == 150 else 2e10)
    steps = max(1, min(rng.choice([1, 6, 12, 30, 60]), int(0.1 / per_step)))
    every = rng.choice([0, 0, 0, 1, 2])
    return _event(None, dims[0], dims[1], dims[2], precision,
                  rng.choice(["hot", "flow", "blast", "tube"]), steps,
                  bc=rng.choice(["reflect", "periodic", "frozen"]), eos=eos,
                  fields=rng.choice(["primitives", "conserved"]), every=every)


def _batch_events(case):
    """Grid size, hot spots and equation of state of each event of a batch or
    serving case (the request mix: part of the case, not of its inputs)."""
    r = random.Random(case["sizes_seed"])
    if case["kind"] == "batch":
        return [dict(N=r.choice([48, 64, 96, 128, 160]), spots=r.randint(5, 40), eos="ideal",
                     flow=0.1) for _ in range(case["events"])]
    return [dict(N=r.choices([64, 96, 128, 192], [.4, .3, .2, .1])[0], spots=r.randint(5, 40),
                 eos="ideal" if i % 2 == 0 else "bag", flow=0.0) for i in range(case["events"])]


# ----------------------------------------------------------------- inputs --

def _coords(nx, ny, nz):
    c = [torch.arange(n, dtype=torch.float64, device="cuda") + 0.5 for n in (nx, ny, nz)]
    return c[0][None, None, :], c[1][None, :, None], c[2][:, None, None]


def _hot(nx, ny, nz, rng, spots, flow):
    """Gaussian hot spots on a background of 1e-6, n = e^(3/4), optionally with
    a radial flow."""
    x, y, z = _coords(nx, ny, nz)
    e = torch.full((nz, ny, nx), 1e-6, dtype=torch.float64, device="cuda")
    for _ in range(spots):
        c = [rng.uniform(n / 4, 3 * n / 4) for n in (nx, ny, nz)]
        s = rng.uniform(3.0, 8.0)
        a = 10.0 ** rng.uniform(-1.0, 1.0)
        g = [torch.exp(-((q - m) ** 2) / (2 * s * s)) for q, m in zip((x, y, z), c)]
        e += (a * g[2]) * (g[1] * g[0])
    rb = min(nx, ny, nz) / 2.0
    v = [(flow * (q - n / 2.0) / rb).expand(nz, ny, nx).contiguous()
         for q, n in zip((x, y, z), (nx, ny, nz))]
    return [e, v[0], v[1], v[2], e ** 0.75]


def _blast(nx, ny, nz, rng):
    """A steep spherical blast near the centre."""
    x, y, z = _coords(nx, ny, nz)
    rad = min(nx, ny, nz) * 0.08 * rng.uniform(0.9, 1.1)
    c = [n / 2.0 + rng.uniform(-2, 2) for n in (nx, ny, nz)]
    r2 = (x - c[0]) ** 2 + (y - c[1]) ** 2 + (z - c[2]) ** 2
    inside = r2 < rad * rad
    e = torch.where(inside, 1e3 * rng.uniform(0.8, 1.2), 0.1).to(torch.float64)
    zero = torch.zeros_like(e)
    return [e, zero, zero.clone(), zero.clone(), e ** 0.75]


def _tube(nx, ny, nz, rng):
    """A planar shock tube along x."""
    e_l, e_r = rng.uniform(0.9, 1.1), rng.uniform(0.009, 0.011)
    left = (torch.arange(nx, device="cuda") < nx // 2).expand(nz, ny, nx)
    e = torch.where(left, e_l, e_r).to(torch.float64).contiguous()
    n = torch.where(left, 1.0, 0.01).to(torch.float64).contiguous()
    zero = torch.zeros_like(e)
    return [e, zero, zero.clone(), zero.clone(), n]


def _prims(case, seed):
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    rng = random.Random(seed)
    if case["data"] == "tube":
        return _tube(nx, ny, nz, rng)
    if case["data"] == "blast":
        return _blast(nx, ny, nz, rng)
    return _hot(nx, ny, nz, rng, 30, 0.0 if case["data"] == "hot" else 0.3)


def _table():
    """p(e) = e/3 softened around e = 1, as a crossover: slope between 0.20 and 0.37."""
    e = np.arange(TABLE_N) * TABLE_DE
    return e / 3.0 - 0.08 * e * np.exp(-((np.log(np.maximum(e, 1e-12))) ** 2))


def _conserved(prims, eos):
    e, vx, vy, vz, n = prims
    g2 = 1.0 / (1.0 - ((vx * vx + vy * vy) + vz * vz))
    p = _eos_p(e, eos)
    w = (e + p) * g2
    return [w - p, w * vx, w * vy, w * vz, n * torch.sqrt(g2)]


def _inputs(case, seed):
    """The five input arrays of an event, float64 on the GPU."""
    f = _prims(case, seed)
    return _conserved(f, case["eos"]) if case["fields"] == "conserved" else f


def _event_inputs(case, seed):
    """The five primitive arrays of each event of a batch or serving case."""
    rng = random.Random(seed)
    return [_hot(e["N"], e["N"], e["N"], rng, e["spots"], e["flow"]) for e in _batch_events(case)]


def _totals_inputs(case, seed):
    # fields of an event in flight: the conserved state of flowing hot spots
    f = _hot(case["nx"], case["ny"], case["nz"], random.Random(seed), 12, 0.3)
    return _conserved(f, "ideal")


# ---------------------------------------------------------------- prepare --

def _empties(shape, k):
    return [torch.empty(shape, dtype=torch.float64, device="cuda") for _ in range(k)]


def prepare(case, seed):
    st = dict(case=case)
    if case["kind"] == "totals":
        st["fields"] = _totals_inputs(case, seed)
        st["out"] = torch.empty(5, dtype=torch.float64, device="cuda")
        return st
    if case["kind"] == "batch":
        st["inputs"] = _event_inputs(case, seed)
        st["events"] = _batch_events(case)
        cells = sum(e["N"] ** 3 + 32 for e in st["events"])
        st["batch"] = shasta.Batch(cells, precision=case["precision"], max_events=64)
        st["out"] = [_empties(i[0].shape, 6) for i in st["inputs"]]
        return st
    if case["kind"] == "serve":
        st["inputs"] = [[a.cpu().numpy() for a in i] for i in _event_inputs(case, seed)]
        st["events"] = _batch_events(case)
        st["server"] = shasta.Server(8 << 30, precision="fp32")
        return st
    table = dict(table=_table(), table_de=TABLE_DE) if case["eos"] == "table" else {}
    st["inputs"] = _inputs(case, seed)
    st["solver"] = shasta.Solver((case["nx"], case["ny"], case["nz"]), lam=LAM,
                                 precision=case["precision"], bc=case["bc"], eos=case["eos"],
                                 bag_B=BAG_B, bag_ec=BAG_EC, **table)
    st["out"] = _empties(st["inputs"][0].shape, 5 if case["fields"] == "conserved" else 6)
    return st


# -------------------------------------------------------------------- run --

def run(st):
    case = st["case"]
    if case["kind"] == "totals":
        shasta.totals_noalloc(*st["fields"], st["out"])
        return st["out"]
    if case["kind"] == "batch":
        b = st["batch"]
        ids = [b.add_primitives((e["N"],) * 3, f, lam=LAM, eos=e["eos"])
               for e, f in zip(st["events"], st["inputs"])]
        b.step(case["steps"])
        for i, out in zip(ids, st["out"]):
            b.get_primitives(i, out)
        for i in ids:
            b.remove(i)
        return st["out"]
    if case["kind"] == "serve":
        srv = st["server"]
        tickets = [srv.submit((e["N"],) * 3, f, case["steps"], lam=LAM, eos=e["eos"], bag_B=BAG_B,
                              bag_ec=BAG_EC) for e, f in zip(st["events"], st["inputs"])]
        srv.drain(60.0)
        res = [srv.poll(t)["prims"] for t in tickets]
        return [[r[k] for k in ("e", "vx", "vy", "vz", "n", "p")] for r in res]
    s = st["solver"]
    if case["fields"] == "conserved":
        s.set_conserved(st["inputs"])
    else:
        s.set_primitives(*st["inputs"])
    sums = []
    if case["every"]:
        left = case["steps"]
        while left > 0:
            k = min(left, case["every"])
            s.step(k)
            sums.append(s.totals())
            left -= k
    else:
        s.step(case["steps"])
    out = s.get_conserved(st["out"]) if case["fields"] == "conserved" else \
        list(s.get_primitives(st["out"]).values())
    return [out, np.stack(sums)] if sums else [out]


# ------------------------------------------------------------------- work --

def work(case):
    if case["kind"] == "totals":
        n = case["nx"] * case["ny"] * case["nz"]
        return dict(bytes=5 * 8 * n, flops=5 * n)
    if case["kind"] in ("batch", "serve"):
        n = sum(e["N"] ** 3 for e in _batch_events(case))
        word, ends, every = FP32_FIELD, 5 * 8 + 6 * 8, 0
    else:
        n = case["nx"] * case["ny"] * case["nz"]
        word = FP64_FIELD if case["precision"] == "fp64" else FP32_FIELD
        ends = 5 * 8 + (5 if case["fields"] == "conserved" else 6) * 8
        every = -(-case["steps"] // case["every"]) if case["every"] else 0
    # one read and one write of the five fields per sweep, the inputs and the
    # results in double, one read of the state per set of totals
    return dict(bytes=n * (case["steps"] * 3 * 2 * 5 * word + ends + every * 5 * word),
                flops=n * (case["steps"] * 3 * FLOPS + 60))


# ------------------------------------------------- the method in 64 bits --
#
# Dimensionally split relativistic SHASTA (arXiv:1206.0919, Sec. 2-3), each
# operation on whole arrays: a sweep recovers velocity and pressure, takes the
# half step with lambda/2, recovers again and takes the full step from the old
# state.  The axis of the sweep is the last one of every array.

AXES = (0, 1, 2, 0, 2, 1, 2, 0, 1, 2, 1, 0, 1, 2, 0, 1, 0, 2)


def _table_p(e, tab):
    x = e / TABLE_DE
    k = torch.floor(x).clamp(0, TABLE_N - 2)
    i = k.long()
    return tab[i] + (x - k) * (tab[i + 1] - tab[i])


_tab = {}


def _tab64():
    if "t" not in _tab:
        _tab["t"] = torch.from_numpy(_table()).cuda()
    return _tab["t"]


def _eos_p(e, eos):
    if eos == "table":
        return _table_p(e, _tab64())
    if eos == "bag":
        return torch.where(e > BAG_EC, (e - 4.0 * BAG_B) / 3.0, e / 3.0)
    return e / 3.0


def _solve(E, M, eos):
    """Rest-frame energy density and pressure from E and |M|."""
    if eos == "table":
        tab = _tab64()
        safe = torch.where(E > 0, E, 1.0)
        v = M / (safe + _table_p(safe, tab))
        for _ in range(200):
            new = M / (safe + _table_p(safe - M * v, tab))
            d = (new - v).abs().max()
            v = new
            if float(d) <= 1e-14:
                break
        e = safe - M * v
        return e, _table_p(e, tab)
    p = (E - M) * (E + M) / (torch.sqrt(4 * E * E - 3 * M * M) + E)
    e = 3 * p
    if eos == "bag":
        B, ec = BAG_B, BAG_EC
        r = 4 * (E - B) ** 2 - 3 * M * M
        eb = (3 * ((E - M) * (E + M)) - 4 * B * E) / (torch.sqrt(r.clamp(min=0)) + (E - 2 * B))
        high = e > ec
        root = high & (E > ec) & (r >= 0) & (eb > ec)
        gap = high & ~root
        e = torch.where(root, eb, torch.where(gap, torch.full_like(e, ec), e))
        p = torch.where(root, (eb - 4 * B) / 3, torch.where(gap, M * M / (E - ec) - E, p))
    return e, p


def _recover(U, eos, delta):
    """e, the momenta clamped to |M| <= (1 - delta) E, E + p, p; vacuum where E <= 0."""
    E = U[0]
    M = torch.sqrt((U[1] * U[1] + U[2] * U[2]) + U[3] * U[3])
    lim = (1.0 - delta) * E
    over = M > lim
    scale = torch.where(over, lim / torch.where(over, M, 1.0), 1.0)
    e, p = _solve(E, torch.where(over, lim, M), eos)
    return e, scale, E + p, p, E > 0


def _w_p(U, par, eos, delta):
    _, scale, h, p, ok = _recover(U, eos, delta)
    w = U[1 + par] * scale / h
    return torch.where(ok, w, 0.0), torch.where(ok, p, 0.0)


def _pad(a, lo, hi):
    return torch.cat([lo, a, hi], dim=-1)


def _ghosts(U, par, bc, frozen):
    """The five fields with three ghost cells at each end of the last axis."""
    n = U[0].shape[-1]
    if bc == "frozen":
        return [_pad(a, lo.expand(*lo.shape[:-1], 3), hi.expand(*hi.shape[:-1], 3))
                for a, (lo, hi) in zip(U, frozen)]
    q = torch.cat([torch.arange(-3, 0), torch.arange(n, n + 3)])
    if bc == "periodic":
        src, neg = q % n, torch.zeros_like(q, dtype=torch.bool)
    else:
        m = q % (2 * n)
        src, neg = torch.where(m < n, m, 2 * n - 1 - m), m >= n
    src = src.to(U[0].device)
    sign = torch.where(neg, -1.0, 1.0).to(torch.float64).to(U[0].device)
    out = []
    for k, a in enumerate(U):
        g = a[..., src]
        if k == 1 + par:
            g = g * sign
        out.append(_pad(a, g[..., :3], g[..., 3:]))
    return out


def _shasta_pass(U, w, p, par, tau):
    """One SHASTA pass of the five padded fields: the interior cells' new values."""
    eps = tau * w
    den = 1.0 + (eps[..., 1:] - eps[..., :-1])
    qp = (0.5 - eps[..., 1:-1]) / den[..., 1:]
    qm = (0.5 + eps[..., 1:-1]) / den[..., :-1]
    a, b, c = 0.5 * qp * qp, 0.5 * qm * qm, qp + qm
    pw = p * w
    out = []
    for k, u in enumerate(U):
        d = u[..., 1:] - u[..., :-1]
        uh = (a * d[..., 1:] - b * d[..., :-1]) + c * u[..., 1:-1]
        if k in (0, 1 + par):
            f = pw if k == 0 else p
            uh = uh + (0.5 * tau) * (f[..., :-2] - f[..., 2:])
        dh = uh[..., 1:] - uh[..., :-1]
        m = dh[..., 1:-1] - 0.125 * ((d[..., 3:-1] + d[..., 1:-3]) - 2 * d[..., 2:-2])
        aph = 0.125 * m
        s = torch.sign(aph)
        A = s * torch.clamp(torch.minimum(torch.minimum(s * dh[..., 2:], aph.abs()),
                                          s * dh[..., :-2]), min=0.0)
        out.append(uh[..., 2:-2] - (A[..., 1:] - A[..., :-1]))
    return out


def _sweep(U, axis, bc, eos, delta, frozen):
    dim = 2 - axis
    lines = [a.transpose(dim, 2) for a in U]
    fz = None if frozen is None else [(lo.transpose(dim, 2), hi.transpose(dim, 2))
                                      for lo, hi in frozen[axis]]
    out = [torch.empty_like(a) for a in U]
    olines = [a.transpose(dim, 2) for a in out]
    total = lines[0].numel()
    chunk = max(1, lines[0].shape[0] * (1 << 25) // max(total, 1))  # bounds the temporaries
    for lo in range(0, lines[0].shape[0], chunk):
        sl = slice(lo, lo + chunk)
        old = [a[sl].contiguous() for a in lines]
        f = None if fz is None else [(x[sl], y[sl]) for x, y in fz]
        g = _ghosts(old, axis, bc, f)
        w, p = _w_p(g, axis, eos, delta)
        half = _ghosts(_shasta_pass(g, w, p, axis, 0.5 * LAM), axis, bc, f)
        w, p = _w_p(half, axis, eos, delta)
        for o, v in zip(olines, _shasta_pass(g, w, p, axis, LAM)):
            o[sl] = v
    return out


def _advance(U, step0, steps, bc, eos, delta, frozen):
    for s in range(step0, step0 + steps):
        for k in range(3):
            U = _sweep(U, AXES[3 * (s % 6) + k], bc, eos, delta, frozen)
    return U


def _prims_of(U, eos, delta):
    e, scale, h, p, ok = _recover(U, eos, delta)
    v = [torch.where(ok, U[1 + a] * scale / h, 0.0) for a in range(3)]
    n = U[4] * torch.sqrt(((e + p) / h).clamp(min=0))
    return [torch.where(ok, e, 0.0), *v, torch.where(ok, n, 0.0), torch.where(ok, p, 0.0)]


def _exact_event(prims_or_cons, conserved, precision, bc, eos, steps, every):
    delta = 1e-10 if precision == "fp64" else 1e-6
    U = prims_or_cons if conserved else _conserved(prims_or_cons, eos)
    if precision != "fp64":
        U = [a.to(torch.float32).to(torch.float64) for a in U]
    frozen = None
    if bc == "frozen":
        frozen = [[(a.narrow(2 - ax, 0, 1).clone(),
                    a.narrow(2 - ax, a.shape[2 - ax] - 1, 1).clone()) for a in U]
                  for ax in range(3)]
    sums, done = [], 0
    while done < steps:
        k = min(every or steps, steps - done)
        U = _advance(U, done, k, bc, eos, delta, frozen)
        done += k
        if every:
            sums.append([float(a.sum()) for a in U])
    out = U if conserved else _prims_of(U, eos, delta)
    return out, np.array(sums)


def exact(case, seed):
    if case["kind"] == "totals":
        return torch.stack([a.sum() for a in _totals_inputs(case, seed)])
    if case["kind"] in ("batch", "serve"):
        res = []
        for e, f in zip(_batch_events(case), _event_inputs(case, seed)):
            out, _ = _exact_event(f, False, "fp32", "reflect", e["eos"], case["steps"], 0)
            res.append(out if case["kind"] == "batch" else [a.cpu().numpy() for a in out])
        return res
    out, sums = _exact_event(_inputs(case, seed), case["fields"] == "conserved",
                             case["precision"], case["bc"], case["eos"], case["steps"],
                             case["every"])
    return [out, sums] if case["every"] else [out]
