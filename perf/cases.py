"""What a user of this framework has it do, as cases that can be timed and compared.

A case is one Chord Length Sampling problem (or a batch of them) and a number of
histories.  A pass walks the next histories of the handle's numbering and reads
the tallies: the loop of a program that adds histories until its standard errors
are small enough.  Sizes are the repository's workloads (workloads.py, the tests
and bench.py).

`exact` walks the same histories in plain torch, in 64 bits, draw for draw: the
random numbers of a history are defined by (seed, history, case) alone.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1708_00765_gb300 as cls
from paper_1708_00765_gb300 import _native, workloads

NBATCH = 64  # statistics batches of a run (the library's default)
COUNTS = ("n_histories", "nR", "nT", "nA", "n_coll", "n_interface", "n_reflect", "n_events", "max_events", "n_capped")
MEANS = ("R", "T", "A", "total_flux", "sigma_R", "sigma_T", "sigma_A", "sigma_total_flux", "track0", "track1")
ROD, EXTRUDED, BOX, SLAB, BOX_X = 1, 2, 3, 11, 13


def _one(name, n, precision, *, workload="", suite="", d=0, L=0.0, nbins=0, source="incident", schedule="history",
         outcomes=False):
    return {"name": name, "kind": "single", "workload": workload, "suite": suite, "d": d, "L": L, "nbins": nbins,
            "cases": 1, "n": n, "precision": precision, "source": source, "schedule": schedule, "outcomes": outcomes}


def _many(name, kind, cases, n, precision, nbins):
    return {"name": name, "kind": kind, "workload": "sweep", "suite": "", "d": 0, "L": 0.0, "nbins": nbins,
            "cases": cases, "n": n, "precision": precision, "source": "incident", "schedule": "history",
            "outcomes": False}


def listed():
    return [
        # a first look at a problem, and the inner call of a parameter search: latency and launches
        _one("rod_1e3_fp64", 1_000, "fp64", workload="rod"),
        # the rod workload at its own size
        _one("rod_1e5_fp64", 100_000, "fp64", workload="rod"),
        # one configuration of benchmark suite II (volume source), the paper's d = 1 slab; ragged history count
        _one("slab_volume_1e6_fp64", 1_000_003, "fp64", suite="2c", d=SLAB, L=10.0, nbins=100, source="volume"),
        # one configuration of benchmark suite I in the extruded geometry, odd mesh
        _one("extruded_3e5_fp64", 300_001, "fp64", suite="1c", d=EXTRUDED, L=10.0, nbins=33),
        # the 3D box workload in the default precision
        _one("box_1e7_fp64", 10_000_000, "fp64", workload="box"),
        # the same box at its full size in FP32 tracking: the longest single call
        _one("box_1e8_fp32", 100_000_000, "fp32", workload="box"),
        # the box walked by its x-marginal, every history's outcome recorded
        _one("box_x_outcomes_4e6_fp32", 4_000_000, "fp32", workload="box_x", outcomes=True),
        # long histories on a fine mesh (diffusive box): history-based and event-based tracking
        _one("diffusive_1e6_fp32", 1_000_000, "fp32", workload="diffusive"),
        _one("diffusive_event_1e6_fp32", 1_000_000, "fp32", workload="diffusive", schedule="event"),
        # the 256-case sweep, FP32 tracking, one graph replay
        _many("sweep_256x1e6_fp32", "batch", 256, 1_000_000, "fp32", 100),
        # a study of fewer cases and few histories each, default precision
        _many("sweep_48x2e4_fp64", "batch", 48, 20_000, "fp64", 100),
        # the allocation-free entry point with its largest number of cases
        _many("noalloc_64x2e4_fp64", "noalloc", 64, 20_000, "fp64", 50),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("single", "single", "single", "suite", "suite", "batch", "noalloc"))
    precision = rng.choice(("fp64", "fp32"))
    nbins = _log_int(rng, 1, 1000)
    if kind == "batch":
        cases = _log_int(rng, 2, 256)
        c = _many("", kind, cases, _log_int(rng, 500, 3e7 / cases), precision, nbins)
    elif kind == "noalloc":
        cases = _log_int(rng, 1, 64)
        c = _many("", kind, cases, _log_int(rng, 500, 3e6 / cases), "fp64", nbins)
    elif kind == "suite":
        d = rng.choice((ROD, EXTRUDED, BOX, SLAB, BOX_X))
        c = _one("", _log_int(rng, 500, 3e6), precision, suite=rng.choice("123") + rng.choice("abc"), d=d,
                 L=rng.choice((1.0, 5.0, 10.0)), nbins=nbins, source=rng.choice(("incident", "volume")))
    else:
        w = rng.choice(("rod", "box", "box", "box_x", "diffusive"))
        top = 1e6 if w == "diffusive" else 1e7
        c = _one("", _log_int(rng, 500, top), precision, workload=w, outcomes=rng.random() < 0.15,
                 schedule="event" if rng.random() < 0.15 else "history")
    del c["name"]
    return c


def _params(case):
    """The case's problems, rows of (sigma0, sigma1, lambda0, lambda1, c0, c1, L, d, nbins)."""
    if case["workload"] == "sweep":
        return workloads.batch_sweep(case["cases"], seed=7, nbins=case["nbins"])
    if case["suite"]:
        p = workloads.suite_case(case["suite"], d=case["d"], L=case["L"], nbins=case["nbins"])
    else:
        p = {"rod": workloads.ROD_L10, "box": workloads.BOX_L10, "box_x": workloads.BOX_L10_X,
             "diffusive": workloads.BOX_DIFFUSIVE}[case["workload"]]
    return np.asarray([p], dtype=np.float64)


def _key(seed):
    """The Philox key of a seed: 64 bits, both words in use."""
    return (int(seed) * 0x9E3779B97F4A7C15 + 0x1F123BB5) & ((1 << 62) - 1)


def prepare(case, seed):
    params = _params(case)
    nc, n = params.shape[0], case["n"]
    s = {"kind": case["kind"], "n": n, "seed": _key(seed), "cases": nc, "outcomes": None}
    if case["kind"] == "noalloc":
        nb = int(params[0, 8])
        s.update(params=params, first=0, stride=nb,
                 flux=torch.zeros((nc, NBATCH, nb), dtype=torch.float64, device="cuda"),
                 stats=torch.zeros((nc, 4), dtype=torch.float64, device="cuda"),
                 counters=torch.zeros((nc, 9), dtype=torch.int64, device="cuda"))
        return s
    prob = cls.Problem(params if case["kind"] == "batch" else params[0], batch=case["kind"] == "batch")
    prob.set_option("precision", case["precision"])
    prob.set_option("schedule", case["schedule"])
    prob.set_option("source", case["source"])
    if case["outcomes"]:
        s["outcomes"] = torch.empty(nc * n, dtype=torch.uint8, device="cuda")
        prob.record_outcomes(s["outcomes"].data_ptr(), s["outcomes"].numel())
    s["prob"] = prob
    return s


def run(s):
    stream = torch.cuda.current_stream()
    if s["kind"] == "noalloc":
        rc = _native.run_noalloc(s["params"], s["first"], s["n"], s["seed"], NBATCH, s["stride"], s["flux"].data_ptr(),
                                 s["stats"].data_ptr(), s["counters"].data_ptr(), stream=stream)
        if rc != cls.CLS_OK:
            raise cls.ClsError(rc, "cls_run_noalloc")
        s["first"] += s["n"]
        return {"flux": s["flux"], "stats": s["stats"], "counters": s["counters"]}
    prob = s["prob"]
    prob.run(s["n"], s["seed"], stream=stream)
    tallies = [prob.tallies(k) for k in range(s["cases"])]
    out = {k: np.array([t[k] for t in tallies], dtype=np.int64) for k in COUNTS}
    out.update({k: np.array([t[k] for t in tallies]) for k in MEANS})
    out["flux"] = np.stack([t["flux"] for t in tallies])
    out["flux_sigma"] = np.stack([t["flux_sigma"] for t in tallies])
    if s["outcomes"] is not None:
        out["outcomes"] = s["outcomes"]
    return out


# ------------------------------------------------- the same walk in plain torch
M32 = 0xFFFFFFFF


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 of 32-bit words held in int64 tensors."""
    k0, k1 = seed & M32, (seed >> 32) & M32
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = ((p1 >> 32) & M32) ^ c1 ^ k0, p1 & M32, ((p0 >> 32) & M32) ^ c3 ^ k1, p0 & M32
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return c0, c1, c2, c3


def _draws(block0, h, ci, seed):
    """The six draws of Philox blocks block0, block0 + 1, block0 + 2 of each history: uniforms
    in [0, 1) with 53 bits."""
    b = torch.stack([block0, block0 + 1, block0 + 2])
    w = _philox(b, (h & M32).expand_as(b), (h >> 32).expand_as(b), ci.expand_as(b), seed)
    even, odd = ((w[0] << 21) | (w[1] >> 11)), ((w[2] << 21) | (w[3] >> 11))
    return torch.stack([even, odd], 1).reshape(6, -1).double() * 2.0**-53


def _walk(params, n, seed, source, max_steps=None, device="cuda"):
    """Walk histories [0, n) of every problem; raw tallies per problem (counts, sums, flux
    per statistics batch) and each history's outcome."""
    P = torch.tensor(np.asarray(params), dtype=torch.float64, device=device)
    nc, nb = P.shape[0], P[:, 8].long()
    nbmax = int(nb.max())
    blen = 1024 * max(1, -(-n // (1024 * NBATCH)))
    ends = torch.zeros(nc * NBATCH * (nbmax + 1), dtype=torch.float64, device=device)    # end bins of the flights
    inner = torch.zeros_like(ends)                                                       # differences of their interior bins
    cnt = torch.zeros((nc, 10), dtype=torch.int64, device=device)
    sums = torch.zeros((nc, 4), dtype=torch.float64, device=device)
    outcome = torch.zeros(nc * n, dtype=torch.uint8, device=device)
    ci = torch.arange(nc, device=device).repeat_interleave(n)
    h = torch.arange(n, device=device).repeat(nc)
    d, L = P[ci, 7].long(), P[ci, 6]
    p0 = P[ci, 2] / (P[ci, 2] + P[ci, 3])
    u = _draws(torch.zeros_like(h), h, ci, seed)
    vol = 1 if source == "volume" else 0
    zero = torch.zeros_like(L)
    rod, thin, box = d == ROD, (d == SLAB) | (d == BOX_X), d == BOX
    x = L * u[0] if vol else zero
    mu_at = torch.where(box, 2, torch.where(d == EXTRUDED, 1, 0)) + vol   # draw that gives mu (3D, extruded, slab)
    umu, uphi = u.gather(0, mu_at[None])[0], u.gather(0, (mu_at + 1)[None])[0]
    mu = 2 * umu - 1 if vol else umu.sqrt()
    st = (1 - mu * mu).clamp_min(0).sqrt() if not vol else (4 * umu * (1 - umu)).sqrt()
    st = (1 - umu).sqrt() if not vol else st
    a, b = st * torch.cos(2 * math.pi * uphi), st * torch.sin(2 * math.pi * uphi)
    wx, wy, wz = (a, b, mu) if vol else (mu, a, b)
    w1 = torch.where(u[1] < 0.5, 1.0, -1.0).double() if vol else zero + 1
    wx = torch.where(rod, w1, torch.where(thin, mu, wx))
    flat = rod | thin
    wy, wz = torch.where(flat, zero, wy), torch.where(flat, zero, wz)
    y = torch.where(flat, zero, L * u[vol])
    z = torch.where(box, L * u[vol + 1], zero)
    j = torch.where(rod, 1 + 2 * vol, torch.where(thin, 2 + vol, torch.where(box, 5, 4) + vol))
    m = (u.gather(0, (j - 1)[None])[0] >= p0).long()
    t0, t1 = zero.clone(), zero.clone()
    ev = torch.zeros_like(h)
    s = dict(ci=ci, h=h, d=d, L=L, x=x, y=y, z=z, wx=wx, wy=wy, wz=wz, j=j, m=m, t0=t0, t1=t1, ev=ev)
    del u, a, b, st, mu, umu, uphi, mu_at, w1, p0, zero, rod, thin, box, flat
    steps = 0
    while s["ci"].numel() and (max_steps is None or steps < max_steps):
        steps += 1
        if device != "cpu" and s["ci"].numel() < 4096:   # the last histories: small operations are quicker on the host
            device = "cpu"
            s = {k: v.cpu() for k, v in s.items()}
            P, nb, ends, inner, cnt, sums, outcome = (v.cpu() for v in (P, nb, ends, inner, cnt, sums, outcome))
        ci, h, d, L, j, m = s["ci"], s["h"], s["d"], s["L"], s["j"], s["m"]
        x, y, z, wx, wy, wz = s["x"], s["y"], s["z"], s["wx"], s["wy"], s["wz"]
        u = _draws(j >> 1, h, ci, seed)
        odd = (j & 1).bool()
        u = [torch.where(odd, u[k + 1], u[k]) for k in range(5)]
        sig, lam, c = P[ci, m], P[ci, 2 + m], P[ci, 4 + m]
        l_c = torch.where(sig > 0, -torch.log1p(-u[0]) / sig, math.inf)
        l_i = -lam * torch.log1p(-u[1])
        l_i = torch.where(d == SLAB, l_i / wx.abs(), torch.where(d == EXTRUDED, l_i / (1 - wz * wz).sqrt(), l_i))

        def face(r, w):
            e = ((torch.where(w > 0, L, 0.0) - r) / w).clamp_min(0)
            return torch.where(w == 0, math.inf, e)

        box, wide = d == BOX, (d == BOX) | (d == EXTRUDED)
        l_x = face(x, wx)
        l_y = torch.where(wide, face(y, wy), math.inf)
        l_z = torch.where(box, face(z, wz), math.inf)
        l_b = torch.minimum(l_x, torch.minimum(l_y, l_z))
        lat = l_b < l_x
        bnd = (l_b <= l_c) & (l_b <= l_i)
        coll = ~bnd & (l_c <= l_i)
        leak = bnd & ~lat
        l = torch.where(bnd, l_b, torch.where(coll, l_c, l_i))
        x1 = torch.where(leak, torch.where(wx > 0, L, 0.0), x + l * wx)
        # score the flight
        s["t0"] = s["t0"] + torch.where(m == 0, l, 0.0)
        s["t1"] = s["t1"] + torch.where(m == 1, l, 0.0)
        nbi = nb[ci]
        idx = nbi / L
        lo, hi = torch.minimum(x, x1).clamp_min(0) * idx, torch.minimum(torch.maximum(x, x1), L) * idx
        k0 = torch.minimum(lo.long(), nbi - 1)
        k1 = torch.where(wx == 0, k0, torch.minimum(hi.long(), nbi - 1))
        per = 1 / (idx * wx.abs())                         # track length in a whole bin
        same = k0 == k1
        e0 = torch.where(same, l, (1 - (lo - k0)) * per)
        e1 = torch.where(same, 0.0, (hi - k1) * per)
        row = (ci * NBATCH + h // blen) * (nbmax + 1)
        ends.index_add_(0, row + k0, e0)
        ends.index_add_(0, row + k1, e1)
        mid = torch.where(k1 > k0 + 1, per, 0.0)
        inner.index_add_(0, row + torch.minimum(k0 + 1, nbi), mid)
        inner.index_add_(0, row + k1, -mid)
        # move
        on_y, on_z = bnd & lat & (l_y == l_b), bnd & lat & (l_z == l_b)
        s["x"] = x1
        s["y"] = torch.where(on_y, torch.where(wy > 0, L, 0.0), y + l * wy)
        s["z"] = torch.where(on_z, torch.where(wz > 0, L, 0.0), z + l * wz)
        wy, wz = torch.where(on_y, -wy, wy), torch.where(on_z, -wz, wz)
        # collision: scatter or absorb
        scat = coll & (u[2] < c)
        absorb = coll & ~scat
        mu = 2 * u[3] - 1
        st = (4 * u[3] * (1 - u[3])).sqrt()
        rod, thin = d == ROD, (d == SLAB) | (d == BOX_X)
        new = torch.where(rod, torch.where(u[3] < 0.5, 1.0, -1.0).double(),
                          torch.where(thin, mu, st * torch.cos(2 * math.pi * u[4])))
        s["wx"] = torch.where(scat, new, wx)
        s["wy"] = torch.where(scat & wide, st * torch.sin(2 * math.pi * u[4]), wy)
        s["wz"] = torch.where(scat & wide, mu, wz)
        cross = ~bnd & ~coll
        s["m"] = torch.where(cross, 1 - m, m)
        s["j"] = j + 2 + coll.long() + torch.where(scat, torch.where(wide, 2, 1), 0)
        s["ev"] = s["ev"] + 1
        out0, outl = leak & (wx <= 0), leak & (wx > 0)
        for col, mask in ((1, out0), (2, outl), (3, absorb), (4, coll), (5, cross), (6, bnd & lat), (7, None)):
            cnt[:, col] += torch.bincount(ci if mask is None else ci[mask], minlength=nc)
        dead = leak | absorb
        if bool(dead.any()):
            dc, t0, t1 = ci[dead], s["t0"][dead], s["t1"][dead]
            t = t0 + t1
            for q, v in enumerate((t, t * t, t0, t1)):
                sums[:, q].index_add_(0, dc, v)
            cnt[:, 8].scatter_reduce_(0, dc, s["ev"][dead], "amax")
            outcome[dc * n + h[dead]] = torch.where(out0, 0, torch.where(outl, 1, 2))[dead].to(torch.uint8)
            s = {k: v[~dead] for k, v in s.items()}
    cnt[:, 0] = n
    shape = (nc, NBATCH, nbmax + 1)
    flux = (ends.view(shape) + inner.view(shape).cumsum(-1))[:, :, :nbmax]
    sizes = np.array([max(0, min(blen, n - b * blen)) for b in range(NBATCH)], dtype=np.float64)
    return cnt.cpu().numpy(), sums.cpu().numpy(), flux.cpu().numpy(), sizes, outcome.cpu().numpy()


def _results(case, params, cnt, sums, flux, sizes, outcome):
    """What `run` returns, from raw tallies; counts are whole numbers that FP32 tracking takes from
    its own flights, so they have a 64-bit value in FP64 only."""
    if case["kind"] == "noalloc":
        order = [1, 2, 3, 4, 5, 6, 7, 9, 8]
        return {"flux": flux, "stats": sums, "counters": cnt[:, order]}
    n = float(case["n"])
    exact_counts = case["precision"] == "fp64"
    out = {k: cnt[:, i] if exact_counts else None for i, k in enumerate(COUNTS)}
    for i, k in ((1, "R"), (2, "T"), (3, "A")):
        out[k] = cnt[:, i] / n
        out["sigma_" + k] = np.sqrt(out[k] * (1 - out[k]) / (n - 1))
    out["total_flux"] = sums[:, 0] / n
    out["sigma_total_flux"] = np.sqrt(np.maximum(sums[:, 1] / n - out["total_flux"] ** 2, 0) / (n - 1))
    out["track0"], out["track1"] = sums[:, 2] / n, sums[:, 3] / n
    dx = (params[:, 6] / params[:, 8])[:, None]
    out["flux"] = flux.sum(1) / (n * dx)
    used = sizes > 0
    B = int(used.sum())
    if B < 2:
        out["flux_sigma"] = None
    else:
        xb = flux[:, used] / (sizes[used][None, :, None] * dx[:, None])
        var = ((sizes[used] / n) ** 2)[None, :, None] * (xb - out["flux"][:, None]) ** 2
        out["flux_sigma"] = np.sqrt(var.sum(1) * B / (B - 1))
    if case["outcomes"]:
        out["outcomes"] = outcome if exact_counts else None
    return out


def exact(case, seed):
    histories = case["n"] * case["cases"]
    if case["workload"] == "diffusive" or histories > 30_000_000:
        return None  # histories of 10^4 events, or too many of them: minutes of plain torch
    params = _params(case)
    return _results(case, params, *_walk(params, case["n"], _key(seed), case["source"]))


_PER_HISTORY = {}


def work(case):
    """Operations of the algorithm: per history from a pilot walk of a few hundred histories -- half
    a Philox block (40) and 2 to form the number per draw; per event two logarithms and scalings
    (6), 3 for each tracked axis' boundary distance, the choice (5), the move (1 per axis), bin
    coordinates, end partials and bookkeeping (8) and one add per bin touched; per 3D scatter 11,
    per history 20.  Bytes: the case table in, the tallies (and outcomes) out."""
    params = _params(case)
    key = (case["workload"], case["suite"], case["d"], case["L"], case["nbins"], case["cases"], case["source"])
    if key not in _PER_HISTORY:
        pilot = max(8, 512 // len(params))
        cnt, sums, _, _, _ = _walk(params, pilot, _key(1), case["source"], max_steps=1500, device="cpu")
        ops = 0.0
        for p, c, t in zip(params, cnt.astype(float), sums[:, 0]):
            axes = {ROD: 1, SLAB: 1, BOX_X: 1, EXTRUDED: 2, BOX: 3}[int(p[7])]
            scatters = c[4] - c[3]
            draws = (3 + axes) * pilot + 2 * c[7] + c[4] + (2 if axes > 1 else 1) * scatters
            bins = c[7] + (1.0 if p[7] == ROD else 0.5) * t * p[8] / p[6]
            ops += 42 * draws + (19 + 4 * axes) * c[7] + bins + (11 if axes > 1 else 2) * scatters + 20 * pilot
        _PER_HISTORY[key] = float(ops) / (pilot * len(params))
    histories = case["n"] * len(params)
    nb = int(params[0, 8])
    flux = NBATCH * nb * 8 if case["kind"] == "noalloc" else 2 * nb * 8
    return {"bytes": len(params) * (72 + flux + 20 * 8) + (histories if case["outcomes"] else 0),
            "flops": _PER_HISTORY[key] * histories}
