"""Timed cases of the powder-pattern engine, through its public entry points.

A case is a plain dict. Three kinds of pass:

* ``pattern`` -- the merged peak lists of a batch of structures: Handle.pattern_batch
  ("eager") or a replay of Handle.graph ("graph") on buffers the caller keeps.
* ``grad``    -- one refinement step: autograd.broadened_pattern, a mean-square loss
  against a target pattern, and its gradients.
* ``augment`` -- training patterns: Handle.pattern_augmented with a pseudo-Voigt
  profile, preferred orientation and noise per structure.

The batches are the seeded generators of paper_2602_11709_gb300.synth, which stand in
for the MC3D and COD sets of the paper (Sec. 4) at their sizes.
"""
import math

import numpy as np
import torch

from paper_2602_11709_gb300 import adapter, autograd, synth, xrd

CU, MO = synth.CU_KA, synth.MO_KA


def _pattern(name, batch, n, precision="fp32_phasefix", wavelength=CU, tt_min=0.0, tt_max=90.0, cutoff=1e-3,
             scaled=True, refl=False, call="eager", runs=False, point_group=""):
    return {"name": name, "kind": "pattern", "batch": batch, "n": n, "precision": precision,
            "wavelength": wavelength, "tt_min": tt_min, "tt_max": tt_max, "cutoff": cutoff, "scaled": scaled,
            "refl": refl, "call": call, "runs": runs, "point_group": point_group}


def listed():
    return [
        # one small cell at a time, in FP64: an interactive calculator call
        _pattern("one cell, fp64", "nacl", 1, precision="fp64"),
        # a handful of cells per call, as a screening loop makes them
        _pattern("a few cells", "mixed", 24),
        # a generation step of an ML workflow: a thousand small cells
        _pattern("small cells", "small", 1024),
        # the same with the phase reduced in FP64, replayed as a graph
        _pattern("small cells, fp64 phase", "small", 1024, precision="fp32_phase64", call="graph"),
        # reference-quality patterns of a thousand cells
        _pattern("small cells, fp64", "small", 1024, precision="fp64", call="graph"),
        # symmetric and disordered cells: merged peaks, families of a point group, every peak kept
        _pattern("hexagonal cells", "hexdis", 256, tt_min=5.0, tt_max=110.0, cutoff=0.0, point_group="6/mmm"),
        # a database pass: 100 000 cells of mixed size, default options, the launch shape that tuning picks
        _pattern("database", "mixed", 100_000, call="graph", runs=True),
        # the paper's own setting (Mo K-alpha, 2-60 degrees, every peak, unscaled), with the reflection list
        _pattern("database, Mo, all peaks", "mixed", 20_000, wavelength=MO, tt_min=2.0, tt_max=60.0, cutoff=0.0,
                 scaled=False, refl=True),
        # large cells, 200 to 2000 atoms, with the launch shape that tuning picks
        _pattern("large cells", "large", 256, tt_min=5.0, tt_max=120.0, call="graph", runs=True),
        # the largest single structure of the paper's Sec. 4.2: 940 atoms, 6e5 reflections
        _pattern("largest cell", "stress", 1, wavelength=MO, tt_min=2.0, tt_max=60.0),
        # one refinement step of 512 structures, forward and backward
        {"name": "refinement step", "kind": "grad", "n": 512, "n_pts": 4096, "fwhm": 0.1},
        # training patterns of a thousand structures
        {"name": "training patterns", "kind": "augment", "n": 1024, "n_pts": 4096},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["pattern"] * 8 + ["grad"] * 2 + ["augment"] * 2)
    if kind == "grad":
        return {"kind": "grad", "n": _log_int(rng, 4, 512), "n_pts": _log_int(rng, 500, 5000),
                "fwhm": round(rng.uniform(0.06, 0.3), 3)}
    if kind == "augment":
        return {"kind": "augment", "n": _log_int(rng, 4, 800), "n_pts": _log_int(rng, 500, 5000)}
    batch = rng.choice(["small", "small", "mixed", "mixed", "mixed", "hexdis", "large", "stress"])
    # a batch of large cells or of the wide range stays with the fast path: it is the one that scales to it
    precision = "fp32_phasefix" if batch in ("large", "stress") else rng.choice(["fp32_phasefix"] * 3 + ["fp64", "fp32_phase64"])
    most = {"fp32_phasefix": {"small": 8192, "mixed": 30_000, "hexdis": 700, "large": 128, "stress": 1},
            "fp32_phase64": {"small": 3000, "mixed": 5000, "hexdis": 700},
            "fp64": {"small": 600, "mixed": 600, "hexdis": 500}}[precision][batch]
    n = _log_int(rng, 1, most)
    if batch == "stress":  # one cell, its size set by the angle range
        c = _pattern("", batch, 1, wavelength=MO, tt_min=2.0, tt_max=round(rng.uniform(20.0, 60.0), 2))
    elif batch == "large":
        c = _pattern("", batch, n, tt_min=5.0, tt_max=round(rng.uniform(60.0, 120.0), 2), runs=rng.random() < 0.5)
    else:
        c = _pattern("", batch, n, precision=precision, tt_min=rng.choice([0.0, 2.0, 5.0]),
                     tt_max=round(rng.uniform(40.0, 110.0), 2), runs=precision == "fp32_phasefix" and rng.random() < 0.2)
    # all peaks kept is the choice of callers who filter later; large batches with the cutoff are the default call
    c["cutoff"], c["scaled"] = (1e-3, True) if rng.random() < 0.6 else (0.0, rng.random() < 0.5)
    c["refl"] = batch != "stress" and rng.random() < 0.15
    c["point_group"] = rng.choice(["", "6/mmm"]) if batch == "hexdis" else ""
    c["call"] = rng.choice(["eager", "graph"])
    del c["name"]
    return c


def _redraw(b, rng, bmax, sites=False):
    """The batch with other contents: the cells keep their shapes (their axes in another order), so the number of
    reflections and atoms is the case's, and everything else is drawn. sites: records of one site stay together."""
    n = b.n_atoms
    if sites:
        lattice, (_, site) = b.lattice, np.unique(b.frac, axis=0, return_inverse=True)
        frac = rng.random((int(site.max()) + 1, 3))[site.reshape(-1)]
    else:
        axes = rng.permuted(np.tile(np.arange(3), (b.n_struct, 1)), axis=1)
        lattice = np.hstack([np.take_along_axis(b.lattice[:, :3], axes, 1), np.take_along_axis(b.lattice[:, 3:], axes, 1)])
        frac = rng.random((n, 3))
    return synth.Batch(lattice, b.atom_off, frac, rng.integers(1, synth.ZMAX + 1, n).astype(np.int16),
                       b.occ if sites else rng.permutation(b.occ), rng.uniform(0.0, bmax, n), synth.coef_table(rng))


def _host(case, seed):
    """(batch, options, ...) of a case, as host arrays."""
    rng = np.random.default_rng(seed)
    if case["kind"] == "grad":
        b, _, opts, grid = synth.grad(n=case["n"])
        grid.n_pts, grid.dt, grid.fwhm = case["n_pts"], 85.0 / (case["n_pts"] - 1), case["fwhm"]
        b = _redraw(b, rng, 2.0)
        n = b.n_struct
        lattice = np.hstack([b.lattice[:, :3] * (1.0 + rng.uniform(-0.005, 0.005, (n, 3))),
                             b.lattice[:, 3:] + rng.uniform(-0.2, 0.2, (n, 3))])
        target = synth.Batch(lattice, b.atom_off, (b.frac + rng.normal(0.0, 0.01, b.frac.shape)) % 1.0, b.Z, b.occ,
                             np.clip(b.B + rng.uniform(-0.1, 0.1, b.n_atoms), 0.0, None), b.coef)
        return b, opts, grid, target
    if case["kind"] == "augment":
        b, opts = synth.small(n=case["n"])
        opts.tt_min, opts.tt_max = 5.0, 90.0
        grid = synth.Grid(n_pts=case["n_pts"], dt=85.0 / (case["n_pts"] - 1))
        return _redraw(b, rng, 2.0), opts, grid, synth.augment(case["n"], case["n_pts"], seed=seed)
    if case["batch"] == "nacl":
        b, _ = synth.nacl(seed=seed)
        b.B = np.full(8, rng.uniform(0.3, 0.8))
    else:
        b, _ = getattr(synth, case["batch"])(n=case["n"])
        b = _redraw(b, rng, {"hexdis": 1.5, "large": 3.0, "stress": 3.0}.get(case["batch"], 2.0), case["batch"] == "hexdis")
    opts = synth.Opts(case["wavelength"], case["tt_min"], case["tt_max"], 1e-5, case["cutoff"], int(case["scaled"]))
    return b, opts


def prepare(case, seed):
    if case["kind"] == "grad":
        base, opts, grid, target = _host(case, seed)
        h = xrd.Handle(0)
        cuda = lambda a: torch.from_numpy(a).cuda()  # noqa: E731
        fixed = autograd.FixedBatch.from_host(base)
        with torch.no_grad():
            y0 = autograd.broadened_pattern(cuda(target.frac), cuda(target.B), cuda(target.lattice), fixed, opts, grid, h)
        p = [cuda(a).requires_grad_(True) for a in (base.frac, base.B, base.lattice)]
        return {"kind": "grad", "h": h, "params": p, "fixed": fixed, "opts": opts, "grid": grid, "target": y0}
    if case["kind"] == "augment":
        b, opts, grid, aug = _host(case, seed)
        h = xrd.Handle(0)
        db, o, g = xrd.DeviceBatch.from_host(b), xrd.make_opts(opts), xrd.make_grid(grid)
        t = {k: torch.from_numpy(getattr(aug, k)).cuda() for k in ("fwhm", "eta", "po_dir", "po_r", "noise_sigma", "z")}
        n = db.n_struct
        return {"kind": "augment", "h": h, "db": db, "o": o, "g": g, "aug": t,
                "ws": xrd.workspace(h.query_sizes(db, o).ws_grad_bytes),
                "y": torch.empty(n, case["n_pts"], dtype=torch.float32, device="cuda"),
                "status": torch.zeros(n, dtype=torch.int32, device="cuda"),
                "totals": torch.zeros(4, dtype=torch.int64, device="cuda")}
    b, opts = _host(case, seed)
    h = xrd.Handle(0)
    if case["runs"]:
        h.set_sf_shape(128, 2, 1)
    if case["point_group"]:
        h.set_point_group(adapter.laue_group_ops(case["point_group"]))
    db, o = xrd.DeviceBatch.from_host(b), xrd.make_opts(opts, case["precision"])
    sz = h.query_sizes(db, o)
    out = xrd.PatternBuffers(db.n_struct, sz.n_refl, refl=case["refl"])
    s = {"kind": "pattern", "h": h, "db": db, "o": o, "out": out, "ws": xrd.workspace(sz.ws_bytes), "graph": None}
    if case["call"] == "graph":
        s["graph"] = h.graph(db, o, out, s["ws"])
    return s


_FIELDS = ("peak_off", "two_theta", "intensity", "d_hkl", "fam_off", "hkl", "mult", "status", "totals", "flags")
_REFL = ("refl_off", "refl_hkl", "refl_tt", "refl_I")


def run(s):
    if s["kind"] == "grad":
        y = autograd.broadened_pattern(*s["params"], s["fixed"], s["opts"], s["grid"], s["h"])
        loss = torch.nn.functional.mse_loss(y, s["target"])
        d_frac, d_B, d_lat = torch.autograd.grad(loss, s["params"])
        return {"y": y.detach(), "loss": loss.detach(), "d_frac": d_frac, "d_B": d_B, "d_lat": d_lat}
    if s["kind"] == "augment":
        a = s["aug"]
        s["h"].pattern_augmented(s["db"], s["o"], s["g"], a["fwhm"], a["eta"], s["y"], s["status"], s["totals"], s["ws"],
                                 po_dir=a["po_dir"], po_r=a["po_r"], noise_z=a["z"], noise_sigma=a["noise_sigma"])
        return {"y": s["y"], "status": s["status"], "totals": s["totals"]}
    if s["graph"] is not None:
        s["graph"].launch()
    else:
        s["h"].pattern_batch(s["db"], s["o"], s["out"], s["ws"])
    return {k: getattr(s["out"], k) for k in _FIELDS + (_REFL if s["out"].refl else ())}


def _volumes(lattice):
    c = np.cos(np.radians(lattice[:, 3:]))
    return lattice[:, :3].prod(axis=1) * np.sqrt(1.0 - (c ** 2).sum(axis=1) + 2.0 * c.prod(axis=1))


def work(case):
    """Friedel-unique reflections from the volume of the sphere; a term is the phase (5 operations), its sine and
    cosine (2), the displacement factor (2), the weight (1) and the two sums (4); FP32 or FP64 outputs."""
    b, o = _host(case, 1)[:2]
    r = [2.0 * math.sin(math.radians(t) / 2.0) / o.wavelength for t in (o.tt_min, o.tt_max)]
    refl = 2.0 / 3.0 * math.pi * (r[1] ** 3 - r[0] ** 3) * _volumes(b.lattice)
    atoms = np.diff(b.atom_off)
    terms, R = float((refl * atoms).sum()), float(refl.sum())
    n_in = 48.0 * b.n_struct + 8.0 * (b.n_struct + 1) + 42.0 * b.n_atoms + b.coef.size * 8.0
    if case["kind"] == "grad":  # a second pass over the terms, and one Gaussian value per reflection and window point
        window = 2.0 * 6.0 * case["fwhm"] / 2.355 / (85.0 / (case["n_pts"] - 1))
        return {"bytes": n_in + 2.0 * 4.0 * b.n_struct * case["n_pts"] + 16.0 * b.n_atoms + 24.0 * b.n_struct,
                "flops": 14.0 * terms + 22.0 * terms + 2.0 * 6.0 * R * window}
    if case["kind"] == "augment":  # Lorentzian at every grid point
        return {"bytes": n_in + 8.0 * b.n_struct * case["n_pts"], "flops": 14.0 * terms + 5.0 * R * case["n_pts"]}
    kept = 1.0 if case["cutoff"] == 0.0 else 0.8
    out = R * kept * (24.0 + 8.0 + 16.0) + (R * 28.0 if case["refl"] else 0.0) + 20.0 * b.n_struct
    return {"bytes": n_in + out, "flops": 14.0 * terms}


# ---- 64-bit values of the outputs ----

def _cell(lat):
    """Reciprocal metric of one cell (torch float64 [6])."""
    a, b, c = lat[0], lat[1], lat[2]
    ca, cb, cg = (torch.cos(torch.deg2rad(lat[i])) for i in (3, 4, 5))
    row = lambda *v: torch.stack(v)  # noqa: E731
    return torch.linalg.inv(torch.stack([row(a * a, a * b * cg, a * c * cb), row(a * b * cg, b * b, b * c * ca),
                                         row(a * c * cb, b * c * ca, c * c)]))


def _half_sphere(lat, o):
    """(h, k, l) [R][3] of the reflections in range, one per Friedel pair (first nonzero index positive)."""
    r0, r1 = (2.0 * math.sin(math.radians(t) / 2.0) / o.wavelength for t in (o.tt_min, o.tt_max))
    H, K, L = (int(r1 * float(v)) + 1 for v in lat[:3])
    ax = lambda lo, hi: torch.arange(lo, hi + 1, device=lat.device, dtype=torch.float64)  # noqa: E731
    out, G = [], _cell(lat)
    for h0 in range(0, H + 1, 8):  # slabs of h bound the memory
        h, k, l = (t.reshape(-1) for t in torch.meshgrid(ax(h0, min(h0 + 7, H)), ax(-K, K), ax(-L, L), indexing="ij"))
        q = G[0, 0] * h * h + G[1, 1] * k * k + G[2, 2] * l * l + 2.0 * (G[0, 1] * h * k + G[0, 2] * h * l + G[1, 2] * k * l)
        first = (h > 0) | ((h == 0) & ((k > 0) | ((k == 0) & (l > 0))))
        m = first & (q <= r1 * r1) & (q >= r0 * r0)
        out.append(torch.stack([h[m], k[m], l[m]], dim=1))
    return torch.cat(out)


def _intensities(hkl, lat, frac, Z, occ, B, coef, o):
    """(q, I) of every reflection: |F|^2 and the Lorentz-polarisation factor in 64 bits."""
    q = torch.einsum("ri,ij,rj->r", hkl, _cell(lat), hkl)
    zs, inv = torch.unique(Z, return_inverse=True)
    parts = []
    for hk, qq in zip(hkl.split(16384), q.split(16384)):
        s2 = (0.25 * qq)[:, None]
        fz = zs.double()[None, :].expand(len(qq), -1)
        for i in range(4):
            fz = fz - 41.78214 * s2 * coef[zs, i, 0][None, :] * torch.exp(-coef[zs, i, 1][None, :] * s2)
        phi = 2.0 * math.pi * torch.remainder(hk @ frac.T, 1.0)
        w = occ[None, :] * fz[:, inv] * torch.exp(-B[None, :] * s2)
        parts.append((w * torch.cos(phi)).sum(1) ** 2 + (w * torch.sin(phi)).sum(1) ** 2)
    X = q * (o.wavelength ** 2 / 4.0)
    return q, torch.cat(parts) * (1.0 + (1.0 - 2.0 * X) ** 2) / (X * torch.sqrt(1.0 - X))


def _two_theta(q, o):
    return torch.rad2deg(2.0 * torch.asin((0.5 * o.wavelength * torch.sqrt(q)).clamp(max=1.0)))


def _peaks(q, I, o):
    """Merged peaks of sorted reflections: (2theta, intensity, d); a peak holds what lies within tt_tol of its first."""
    tt = _two_theta(q, o)
    start = torch.ones_like(tt, dtype=torch.bool)
    start[1:] = tt[1:] - tt[:-1] >= o.tt_tol
    idx = torch.arange(len(tt), device=tt.device)
    while True:
        anchor = torch.cummax(torch.where(start, idx, torch.zeros_like(idx)), 0).values
        late = tt - tt[anchor] >= o.tt_tol
        first = late & ~torch.cat([late.new_zeros(1), late[:-1] & (anchor[1:] == anchor[:-1])])
        if not bool(late.any()):
            break
        start = start | first
    s = torch.nonzero(start).reshape(-1)
    sums = torch.zeros(len(s), dtype=torch.float64, device=tt.device).index_add_(0, torch.cumsum(start, 0) - 1, 2.0 * I)
    top = sums.max()
    keep = sums > o.rel_cutoff * top if o.rel_cutoff > 0 else torch.ones_like(sums, dtype=torch.bool)
    y = 100.0 * (sums / top) if o.scaled and float(top) > 0 else sums
    return tt[s][keep], y[keep], 1.0 / torch.sqrt(q[s][keep])


def _atoms(b, s, dev):
    sl = b.atoms_of(s)
    return [torch.from_numpy(np.ascontiguousarray(a[sl])).to(dev) for a in (b.frac, b.Z.astype(np.int64), b.occ, b.B)]


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    host = _host(case, seed)
    b, o = host[:2]
    if case["kind"] == "pattern" and (case["batch"] == "large" or case["n"] > 1500):
        return None  # tens of seconds to minutes of 64-bit sums
    coef = torch.from_numpy(b.coef).to(dev)
    lat = torch.from_numpy(b.lattice).to(dev)
    if case["kind"] == "pattern":
        got, lists, total = [], [], 0
        for s in range(b.n_struct):
            hkl = _half_sphere(lat[s], o)
            total += len(hkl)
            if not len(hkl):
                continue
            q, I = _intensities(hkl, lat[s], *_atoms(b, s, dev), coef, o)
            q, order = torch.sort(q)
            got.append(_peaks(q, I[order], o))
            lists.append((_two_theta(q, o), I[order]))
        pad = lambda parts: torch.cat(parts + [torch.zeros(max(total, 1) - sum(map(len, parts)), dtype=torch.float64, device=dev)])  # noqa: E731
        r = dict.fromkeys(_FIELDS)
        r.update({k: pad([g[i] for g in got]) for i, k in enumerate(("two_theta", "intensity", "d_hkl"))})
        if case["refl"]:
            r.update(dict.fromkeys(_REFL))
            r["refl_tt"] = pad([v[0] for v in lists])
            if case["batch"] in ("small", "mixed"):  # equal |g| in symmetric cells: their order is by index there
                r["refl_I"] = pad([v[1] for v in lists])
        return r
    grid = host[2]
    t = grid.t0 + grid.dt * torch.arange(grid.n_pts, dtype=torch.float64, device=dev)
    if case["kind"] == "augment":
        aug, rows = host[3], []
        for s in range(b.n_struct):
            hkl = _half_sphere(lat[s], o)
            q, I = _intensities(hkl, lat[s], *_atoms(b, s, dev), coef, o)
            G, n = _cell(lat[s]), torch.from_numpy(aug.po_dir[s]).to(dev)
            c2 = (hkl @ G @ n) ** 2 / (q * (n @ G @ n))
            pr = float(aug.po_r[s])
            amp = 2.0 * I * (pr * pr * c2 + (1.0 - c2).clamp(min=0.0) / pr) ** -1.5
            w, eta, y = float(aug.fwhm[s]), float(aug.eta[s]), torch.zeros_like(t)
            for tt, a in zip(_two_theta(q, o).split(2048), amp.split(2048)):
                x2 = (2.0 * (t[None, :] - tt[:, None]) / w) ** 2
                pv = eta * 2.0 / (math.pi * w) / (1.0 + x2) + (1.0 - eta) * (2.0 / w) * math.sqrt(math.log(2.0) / math.pi) * torch.exp2(-x2)
                y = y + a @ pv
            z = torch.from_numpy(aug.z[s]).to(dev).double()
            rows.append(y + float(aug.noise_sigma[s]) * torch.sqrt(y.clamp(min=0.0)) * z)
        return {"y": torch.stack(rows), "status": None, "totals": None}

    sigma = grid.fwhm / (2.0 * math.sqrt(2.0 * math.log(2.0)))
    W = math.ceil(6.0 * sigma / grid.dt)

    def broadened(batch, s, frac, Z, occ, B, la):
        q, I = _intensities(_half_sphere(la.detach(), o), la, frac, Z, occ, B, coef, o)
        y = torch.zeros(grid.n_pts, dtype=torch.float64, device=dev)
        tt = _two_theta(q, o)
        cell = torch.floor((tt.detach() - grid.t0) / grid.dt).long()
        at = cell[:, None] + torch.arange(-W, W + 2, device=dev)[None, :]
        inside = (at >= 0) & (at < grid.n_pts)
        at = at.clamp(0, grid.n_pts - 1)
        v = 2.0 * I[:, None] * torch.exp(-(t[at] - tt[:, None]) ** 2 / (2.0 * sigma * sigma)) * inside
        return y.index_add(0, at.reshape(-1), v.reshape(-1))

    target, tlat = host[3], torch.from_numpy(host[3].lattice).to(dev)
    ys, loss, grads = [], 0.0, ([], [], [])
    for s in range(b.n_struct):
        frac, Z, occ, B = _atoms(b, s, dev)
        with torch.no_grad():
            y0 = broadened(target, s, *_atoms(target, s, dev), tlat[s])
        p = [frac.requires_grad_(True), B.requires_grad_(True), lat[s].clone().requires_grad_(True)]
        y = broadened(b, s, p[0], Z, occ, p[1], p[2])
        e = ((y - y0) ** 2).sum() / (b.n_struct * grid.n_pts)
        for into, g in zip(grads, torch.autograd.grad(e, p)):
            into.append(g)
        ys.append(y.detach())
        loss += float(e.detach())
    return {"y": torch.stack(ys), "loss": torch.tensor(loss, dtype=torch.float64), "d_frac": torch.cat(grads[0]),
            "d_B": torch.cat(grads[1]), "d_lat": torch.stack(grads[2])}
