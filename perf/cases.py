"""Timed cases: the work that users of this framework have it do, through its
public entry points (``capi`` and ``autograd``), with a plain 64-bit torch
statement of the same results.

Kinds of cases:

- ``step``: ``lp_step`` calls on a cube, a column, a batch of columns or a
  periodic layer, from a smooth flow on a jittered lattice (what a collapsing
  column looks like between calls). Every pass starts from the same state, by
  one device copy, as the explicit step blows up over long runs.
- ``sweep``: truncated stencils of per-particle radius (``lp_build_neighbors``)
  and the derivatives of several fields on them (``lp_fit_derivatives``).
- ``stress``: the stress of a given flow: stencils, velocity derivatives,
  ``lp_mui_stress``.
- ``adjoint``: a differentiable run, forward and backward (``lp_step_diff``).

Material values, lattice spacings, radii and time steps are those of
``paper_2206_14061_gb300.workloads`` and of the tests.
"""
import math

import numpy as np
import torch

from paper_2206_14061_gb300 import autograd, capi

MUI = dict(mu_s=0.38, mu_2=0.64, I0=0.28, d=5e-4, rho_s=2500.0)
EOS = dict(phi_c=0.60, phi_min=0.35, phi_max=0.59, beta=400.0, alpha=-400.0 * 0.59)
PREC = dict(fp64=capi.LP_FP64, mixed_ff=capi.LP_MIXED_FF)
LAUNCH = dict(kernels=capi.LP_LAUNCH_KERNELS, graph=capi.LP_LAUNCH_GRAPH)
KEEP = dict(nearest=capi.LP_KEEP_NEAREST, octants=capi.LP_KEEP_OCTANTS)
FIELDS = ("x", "y", "z", "u", "v", "w", "V")
DT = 1e-5


def _step(name, geom, size, prec, steps, **kw):
    c = dict(name=name, kind="step", geom=geom, size=size, prec=prec, steps=steps, calls=1,
             launch="kernels", skin=0.0, ghosts=False, heun=False, host=False, flow=0.5, phi=0.585)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: an 8^3 cube for four steps, float-float fits, graph replay
        _step("cube512_ff", "cube", 8, "mixed_ff", 4, launch="graph", skin=0.1, flow=0.1),
        # the 8,000-particle cube of the tests for its 50 steps, every option at its default (FP64)
        _step("cube8k_fp64", "cube", 20, "fp64", 50, flow=0.05, phi=0.5),
        # the benchmark's column (786,000 particles), its default configuration, collapsing
        _step("column786k_ff", "column", 50, "mixed_ff", 10, launch="graph", skin=0.1),
        # the same column in FP64, for users who want no float-float
        _step("column786k_fp64", "column", 50, "fp64", 4, launch="graph", skin=0.1),
        # the benchmark's end-to-end loop: one step a call on pinned host arrays, lists kept
        _step("column786k_host_ff", "column", 50, "mixed_ff", 1, calls=4, skin=0.1, host=True),
        # the parameter study: 256 independent columns with free-surface ghosts in one call
        # (4.8 M particles, the largest case)
        _step("batch256_ghosts_ff", "batch", 256, "mixed_ff", 5, launch="graph", skin=0.1,
              ghosts=True, phi=0.5),
        # the paper's compacting layer: periodic sides, ghosts at the top (ragged: 97 cells wide)
        _step("layer282k_ghosts_ff", "layer", 97, "mixed_ff", 6, launch="graph", skin=0.1,
              ghosts=True, phi=0.5),
        # Heun's method on a mid-size column, ghosts, FP64
        _step("column49k_heun_fp64", "column", 20, "fp64", 6, launch="graph", skin=0.1,
              ghosts=True, heun=True, phi=0.5),
        # the derivative-operator sweep at its stated size: 48 nearest, four fields
        dict(name="sweep2m_ff", kind="sweep", side=126, prec="mixed_ff", keep="nearest", cap=48,
             nf=4),
        # one field on a small lattice in FP64 with octant-balanced stencils
        dict(name="sweep59k_octants_fp64", kind="sweep", side=39, prec="fp64", keep="octants",
             cap=32, nf=1),
        # strain rate and stress of a given flow, FP64 (the diagnostics of a run)
        dict(name="stress170k_fp64", kind="stress", size=30, prec="fp64"),
        # gradients of a run with ghosts, forward and backward
        dict(name="adjoint25k", kind="adjoint", size=16, steps=12, every=6, flow=0.5),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(("step", "step", "step", "step", "sweep", "stress", "adjoint"))
    if kind == "step":
        geom = rng.choice(("cube", "column", "column", "batch", "layer"))
        n = log_int(600, 2400000)  # particles, and what each shape makes of them
        size = {"cube": lambda: max(8, round(min(n, 400000) ** (1 / 3))),
                "column": lambda: max(6, round((n / (2 * math.pi)) ** (1 / 3))),
                "batch": lambda: max(2, min(128, round(n / 18700))),
                "layer": lambda: max(7, round(math.sqrt(n / 30)))}[geom]()
        prec = rng.choice(("mixed_ff", "mixed_ff", "mixed_ff", "fp64"))
        ghosts = rng.random() < 0.4
        host = rng.random() < 0.15
        c = dict(kind="step", geom=geom, size=size, prec=prec,
                 steps=1 if host else rng.randint(1, 3) if n > 300000 else rng.randint(1, 12),
                 calls=rng.randint(2, 4) if host else 1,
                 launch=rng.choice(("graph", "kernels")), skin=0.1 if host else rng.choice((0.0, 0.1, 0.1, 0.2)),
                 ghosts=ghosts, heun=rng.random() < 0.15, host=host,
                 flow=round(rng.uniform(0.05, 0.5), 3), phi=rng.choice((0.5, 0.585)))
        return c
    if kind == "sweep":
        side = log_int(12, 110)
        return dict(kind="sweep", side=side, prec=rng.choice(("mixed_ff", "mixed_ff", "fp64")),
                    keep=rng.choice(("nearest", "nearest", "octants")), cap=rng.choice((32, 48, 64)),
                    nf=rng.randint(1, 5))
    if kind == "stress":
        return dict(kind="stress", size=log_int(7, 45), prec=rng.choice(("mixed_ff", "fp64")))
    return dict(kind="adjoint", size=log_int(6, 16), steps=rng.randint(2, 12),
                every=rng.randint(1, 6), flow=round(rng.uniform(0.2, 0.5), 3))


# ------------------------------------------------------------------ inputs


def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _cylinder(R, H, h, g):
    nr = int(math.ceil(R / h))
    c = (np.arange(-nr, nr) + 0.5) * h
    X, Y = np.meshgrid(c, c, indexing="xy")
    keep = X * X + Y * Y <= R * R
    X, Y = X[keep], Y[keep]
    Z = (np.arange(int(round(H / h))) + 0.5) * h
    p = np.stack([np.tile(X, Z.size), np.tile(Y, Z.size), np.repeat(Z, X.size)])
    return p + g.uniform(-0.05 * h, 0.05 * h, size=p.shape)


def _box(nx, ny, nz, h, jitter, g):
    z, y, x = np.meshgrid((np.arange(nz) + 0.5) * h, (np.arange(ny) + 0.5) * h,
                          (np.arange(nx) + 0.5) * h, indexing="ij")
    p = np.stack([x.ravel(), y.ravel(), z.ravel()])
    return p + g.uniform(-jitter * h, jitter * h, size=p.shape)


def _flow(p, R, H, U, phi, radial):
    """State rows x, y, z, u, v, w, V: a spreading (radial) or shearing flow
    that vanishes at the floor, solid fraction falling slightly with height."""
    x, y, z = p
    s = U * z / H
    u, v = (s * x / R, s * y / R) if radial else (s, 0.2 * s * np.cos(2 * math.pi * x / R))
    w = -0.05 * s * (z / H)
    return np.stack([x, y, z, u, v, w, 1.0 / (phi - 0.02 * z / H)])


def _step_inputs(c, seed):
    """(state rows [7, n], column offsets or None, mu_s per column, parameters)."""
    g = np.random.default_rng([int(seed), 77])
    U = c.get("flow", 0.5) * g.uniform(0.9, 1.1)
    phi, geom, size = c.get("phi", 0.5), c.get("geom", "column"), c["size"]
    h, offs, mus, L = 1e-3, None, [MUI["mu_s"]], 0.0
    if geom == "cube":
        st = _flow(_box(size, size, size, h, 0.05, g), size * h, size * h, U, phi, False)
    elif geom == "column":
        R = 0.02
        h = R / size
        st = _flow(_cylinder(R, 2 * R, h, g), R, 2 * R, U, phi, True)
    elif geom == "layer":
        L = size * h
        st = _flow(_box(size, size, 30, h, 0.05, g), L, 30 * h, U, phi, False)
        st[:2] = np.mod(st[:2], L)
    else:
        cols = np.random.default_rng([size, 76])  # sizes of the case, whatever the seed
        N = np.round(np.exp(cols.uniform(math.log(2000), math.log(64000), size=size)))
        a, mus = cols.uniform(0.5, 6.0, size=size), list(g.uniform(0.30, 0.45, size=size))
        parts = []
        for n, k in zip(N, a):
            R = h * (n / (math.pi * k)) ** (1.0 / 3.0)
            parts.append(_flow(_cylinder(R, k * R, h, g), R, k * R, 0.2 * U, phi, True))
        offs = np.concatenate([[0], np.cumsum([q.shape[1] for q in parts])]).astype(np.int32)
        st = np.concatenate(parts, axis=1)
    prm = dict(h=h, radius=2.2 * h, gx=0.0, gy=0.0, gz=-9.81, floor_z=0.0, mirror_mode=1,
               precision=PREC[c.get("prec", "fp64")], rebuild_every=1,
               launch_mode=LAUNCH[c.get("launch", "kernels")], skin=c.get("skin", 0.0) * h,
               free_surface=int(c.get("ghosts", False)), time_scheme=int(c.get("heun", False)),
               period_x=L, period_y=L, keep_lists=int(c.get("host", False)))
    return torch.from_numpy(st).to(_dev()), offs, mus, prm


def _sweep_inputs(c, seed):
    g = np.random.default_rng([int(seed), 78])
    h, side = 1e-3, c["side"]
    dev = _dev()
    p = torch.from_numpy(_box(side, side, side, h, 0.2, g)).to(dev)
    radius = torch.from_numpy(g.uniform(1.8 * h, 2.6 * h, size=side ** 3)).to(dev)
    fields = []
    for _ in range(c["nf"]):  # a sum of plane waves of 1 to 8 periods per edge
        s = torch.zeros_like(p[0])
        for k in range(1, 9):
            e = g.standard_normal(3)
            e *= 2 * math.pi * k / (side * h) / np.linalg.norm(e)
            s += g.standard_normal() * torch.sin(e[0] * p[0] + e[1] * p[1] + e[2] * p[2]
                                                 + g.uniform(0, 2 * math.pi))
        fields.append(s)
    return p, radius, fields, h


# ------------------------------------------------------------ prepare, run


def prepare(case, seed):
    kind = case["kind"]
    if kind == "sweep":
        p, radius, fields, h = _sweep_inputs(case, seed)
        n = p.shape[1]
        return dict(case=case, x=p[0], y=p[1], z=p[2], radius=radius, fields=fields, h=h,
                    ctx=capi.Context(n, cap=64))
    if kind == "stress":
        init, _, _, prm = _step_inputs(dict(case, phi=0.5), seed)
        return dict(case=case, f=dict(zip(FIELDS, init)), prm=prm,
                    ctx=capi.Context(init.shape[1], cap=64))
    if kind == "adjoint":
        init, _, _, prm = _step_inputs(dict(case, ghosts=True), seed)
        g = np.random.default_rng([int(seed), 79])
        lam = torch.from_numpy(g.standard_normal(tuple(init.shape))).to(init.device)
        theta = torch.tensor([MUI["mu_s"], MUI["mu_2"], MUI["I0"]], dtype=torch.float64,
                             device=init.device)
        return dict(case=case, init=init, seed=lam, theta=theta, prm=prm,
                    ctx=capi.Context(init.shape[1], cap=64))
    init, offs, mus, prm = _step_inputs(case, seed)
    n = init.shape[1]
    buf = torch.empty((7, n), dtype=torch.float64, pin_memory=True) if case["host"] else torch.empty_like(init)
    return dict(case=case, init=init, buf=buf, f=dict(zip(FIELDS, buf)), offs=offs, prm=prm,
                mui=[dict(MUI, mu_s=float(m)) for m in mus],
                ctx=capi.Context(n, max_columns=len(mus), cap=64), stream=torch.cuda.Stream())


def run(s):
    c = s["case"]
    if c["kind"] == "step":
        with torch.cuda.stream(s["stream"]):
            s["buf"].copy_(s["init"], non_blocking=True)
            for _ in range(c["calls"]):
                capi.lp_step(s["ctx"], s["f"], s["mui"], EOS, s["prm"], DT, c["steps"],
                             column_offsets=s["offs"], stream=s["stream"])
        return s["f"]
    if c["kind"] == "sweep":
        nb = capi.lp_build_neighbors(s["ctx"], s["x"], s["y"], s["z"], radius=s["radius"],
                                     mirror_mode=0, cap=c["cap"], keep_nearest=KEEP[c["keep"]])
        return capi.lp_fit_derivatives(s["ctx"], s["x"], s["y"], s["z"], nb, s["fields"],
                                       [1.0] * c["nf"], s["h"], precision=PREC[c["prec"]])
    if c["kind"] == "stress":
        f, q = s["f"], s["prm"]
        nb = capi.lp_build_neighbors(s["ctx"], f["x"], f["y"], f["z"], r_const=q["radius"])
        d = capi.lp_fit_derivatives(s["ctx"], f["x"], f["y"], f["z"], nb, [f["u"], f["v"], f["w"]],
                                    [-1.0] * 3, q["h"], precision=q["precision"])
        o = capi.lp_mui_stress(s["ctx"], MUI, EOS, f["V"], d[:, :, :3].reshape(-1, 9))
        return dict(o, d=d)
    theta = s["theta"].detach().requires_grad_(True)
    st = {k: r.detach().requires_grad_(True) for k, r in zip(FIELDS, s["init"])}
    out = autograd.lp_step_diff(s["ctx"], theta, st, MUI, EOS, s["prm"], DT, c["steps"], c["every"])
    g = torch.autograd.grad([out[k] for k in FIELDS], [theta] + [st[k] for k in FIELDS],
                            list(s["seed"]))
    return dict(out={k: out[k].detach() for k in FIELDS}, dtheta=g[0],
                dstate=dict(zip(FIELDS, g[1:])))


def work(case):
    """Inputs read once and outputs written once; the method's own flops: per
    step and particle about 36 stencil rows, the 9 x 9 factor and the solves
    (pass 1: 176 a row and 1000; pass 2: 50 a row and 400)."""
    kind = case["kind"]
    if kind == "sweep":
        n, m = case["side"] ** 3, case["cap"]
        return dict(bytes=n * 8.0 * (4 + 10 * case["nf"]),
                    flops=n * (m * (80.0 + 19.0 * case["nf"]) + 400 + 170 * case["nf"]))
    size = case["size"]
    per = {"cube": size ** 3, "column": 2 * math.pi * size ** 3, "batch": 18700.0 * size,
           "layer": 30.0 * size ** 2}
    n = per[case.get("geom", "column")]
    if kind == "stress":
        return dict(bytes=n * 8.0 * (7 + 27 + 9), flops=n * (36 * 176.0 + 1100))
    one = 36 * 226.0 + 1400
    if kind == "adjoint":
        return dict(bytes=n * 8.0 * 7 * 4, flops=3 * n * one * case["steps"])
    stages = 2 if case["heun"] else 1
    return dict(bytes=n * 8.0 * 14 * case["calls"],
                flops=n * one * case["steps"] * case["calls"] * stages)


# --------------------------------------------------- the results in 64 bits

CHUNK = 1 << 17


def _cells(p, col, r, periods):
    """Cell table of edge >= r: sorted keys, their order, dimensions and origin."""
    lo = [0.0 if periods[a] else float(p[a].min()) for a in range(3)]
    hi = [periods[a] or float(p[a].max()) for a in range(3)]
    w = r * (1 + 1e-9)
    dim = [max(1, int((hi[a] - lo[a]) / w)) if periods[a] else int((hi[a] - lo[a]) / w) + 1
           for a in range(3)]
    edge = [periods[a] / dim[a] if periods[a] else w for a in range(3)]
    c = [((p[a] - lo[a]) / edge[a]).floor().long() for a in range(3)]
    c = [c[a] % dim[a] if periods[a] else c[a].clamp(0, dim[a] - 1) for a in range(3)]
    key = ((col * dim[2] + c[2]) * dim[1] + c[1]) * dim[0] + c[0]
    order = torch.argsort(key, stable=True)
    return key[order].contiguous(), order, dim, lo, edge


def _near(d, L):
    if not L:
        return d
    return torch.where(d > 0.5 * L, d - L, torch.where(d < -0.5 * L, d + L, d))


def _candidates(p, col, cells, periods, rows, mirrored):
    """Particles (or their floor mirrors) in the 27 cells around `rows`: ids, mask."""
    ks, order, dim, lo, edge = cells
    q = [p[0][rows], p[1][rows], -p[2][rows] if mirrored else p[2][rows]]
    c = [((q[a] - lo[a]) / edge[a]).floor().long() for a in range(3)]
    at, end = [], []
    for oz in (-1, 0, 1):
        for oy in (-1, 0, 1):
            for ox in (-1, 0, 1):
                k = [c[0] + ox, c[1] + oy, c[2] + oz]
                ok = torch.ones_like(c[0], dtype=torch.bool)
                for a in range(3):
                    if periods[a]:
                        k[a] = k[a] % dim[a]
                    else:
                        ok &= (k[a] >= 0) & (k[a] < dim[a])
                key = ((col[rows] * dim[2] + k[2]) * dim[1] + k[1]) * dim[0] + k[0]
                key = torch.where(ok, key, torch.full_like(key, -1))
                at.append(torch.searchsorted(ks, key))
                end.append(torch.searchsorted(ks, key, right=True))
    at, end = torch.stack(at, 1), torch.stack(end, 1)
    most = max(1, int((end - at).max()))
    slot = at[:, :, None] + torch.arange(most, device=at.device)
    ok = slot < end[:, :, None]
    ids = order[slot.clamp(max=order.numel() - 1)]
    return ids.flatten(1), ok.flatten(1)


def _pair_d2(p, rows, ids, mir, periods):
    """Squared distances of `rows` to ids, the mirrored ones at -z, as printed in FP64."""
    dx = _near(p[0][ids] - p[0][rows][:, None], periods[0])
    dy = _near(p[1][ids] - p[1][rows][:, None], periods[1])
    zj = p[2][ids]
    dz = torch.where(mir, -zj, zj) - p[2][rows][:, None]
    return (dx * dx + dy * dy) + dz * dz, (dx, dy, dz)


def _stencils(p, col, r, mirrors, periods, cap, keep=None):
    """Stencils (ids, mirror flag, mask), each [n, cap]: every neighbour within
    r (a number or one a particle), or the first `cap` by `keep`."""
    n = p.shape[1]
    per = torch.is_tensor(r)
    rmax = float(r.max()) if per else r
    cells = _cells(p, col, rmax, periods)
    out = []
    for b in range(0, n, CHUNK // 2):
        rows = torch.arange(b, min(n, b + CHUNK // 2), device=p.device)
        ids, ok = _candidates(p, col, cells, periods, rows, False)
        ok &= ids != rows[:, None]
        mir = torch.zeros_like(ok)
        if mirrors and bool((p[2][rows] < rmax).any()):
            im, om = _candidates(p, col, cells, periods, rows, True)
            ids, ok = torch.cat([ids, im], 1), torch.cat([ok, om], 1)
            mir = torch.cat([mir, torch.ones_like(om)], 1)
        d2, off = _pair_d2(p, rows, ids, mir, periods)
        rr = (r[rows] * r[rows])[:, None] if per else r * r
        ok &= d2 <= rr
        if keep is None:
            at = ok.long().cumsum(1) - 1
            if int(at.max()) >= cap:
                raise RuntimeError("a stencil is larger than its capacity")
        else:
            o = torch.argsort(torch.where(ok, d2, torch.full_like(d2, math.inf)), dim=1, stable=True)
            o = o[:, :160]
            ids, ok, mir = ids.gather(1, o), ok.gather(1, o), mir.gather(1, o)
            rank = torch.arange(o.shape[1], device=o.device).expand_as(o)
            if keep == "octants":  # by rank within the octant, then by distance
                q = sum((f.gather(1, o) >= 0).long() << k for k, f in enumerate(off))
                rnd = torch.zeros_like(q)
                for k in range(8):
                    m = (q == k) & ok
                    rnd = torch.where(m, m.long().cumsum(1) - 1, rnd)
                key = torch.where(ok, rnd * 1024 + rank, torch.full_like(rnd, 1 << 40))
                o = torch.argsort(key, dim=1)
                ids, ok, mir = ids.gather(1, o), ok.gather(1, o), mir.gather(1, o)
                rank = torch.arange(o.shape[1], device=o.device).expand_as(o)
            ok &= rank < cap
            at = rank
        at = torch.where(ok, at, torch.full_like(at, cap))
        one = []
        for v in (ids, mir, ok):
            t = torch.zeros((rows.numel(), cap + 1), dtype=v.dtype, device=v.device)
            one.append(t.scatter_(1, at, v)[:, :cap])
        one[2] = torch.arange(cap, device=p.device) < ok.sum(1, keepdim=True)
        out.append(one)
    return [torch.cat([o[k] for o in out]) for k in range(3)]


def _ghost_flags(p, col, sten, prm, periods):
    """Entries whose point reflection through the particle is a ghost: the
    one-sided test and the placement on the fixed-point grid."""
    ids, mir, ok = sten
    K = 1.0
    while K * prm["radius"] > 8192.0:
        K *= 0.5
    while 2 * K * prm["radius"] <= 8192.0:
        K *= 2.0
    R2 = round((K * prm["radius"]) ** 2)
    hk = prm["h"] * K
    clear2 = round((0.5 * hk) * (0.5 * hk))
    X = [torch.round(p[a] * K).long() for a in range(3)]
    Zm = torch.round(-p[2] * K).long()
    flag = torch.zeros_like(ok)
    for b in range(0, ok.shape[0], CHUNK):
        e = min(ok.shape[0], b + CHUNK)
        i, m, k = ids[b:e], mir[b:e], ok[b:e]
        o = []
        for a in range(3):
            d = (torch.where(m, Zm[i], X[2][i]) if a == 2 else X[a][i]) - X[a][b:e, None]
            if periods[a]:
                P = round(K * periods[a])
                d = torch.where(2 * d > P, d - P, torch.where(2 * d < -P, d + P, d))
            o.append(d)
        w = (R2 - (o[0] * o[0] + o[1] * o[1] + o[2] * o[2])).clamp(min=0) * k
        S = [(w * d).sum(1) for d in o]
        s2 = (S[0].double() ** 2 + S[1].double() ** 2) + S[2].double() ** 2
        lim = (0.22 * hk) * w.sum(1).double()
        hit = torch.nonzero(s2 > lim * lim).flatten()
        for c in range(0, hit.numel(), 1 << 14):
            t = hit[c:c + (1 << 14)]
            q = [d[t] for d in o]
            ds = sum(q[a] * S[a][t][:, None] for a in range(3)).double()
            dep = 0.5 * hk
            f = k[t] & (ds > 0) & (ds * ds >= (dep * dep * s2[t])[:, None])
            zi = p[2][b + t][:, None]
            zk = torch.where(m[t], -p[2][i[t]], p[2][i[t]])
            f &= (zi + zi) - zk >= 0.0
            for j in range(ok.shape[1]):  # no entry within h/2 of the reflection
                r2 = sum((q[a] + q[a][:, j:j + 1]) ** 2 for a in range(3))
                f[:, j] &= ~((r2 < clear2) & k[t]).any(1)
            flag[b + t] = f
    return flag


def _basic(A, B):
    """Least squares by column-pivoted Householder QR, basic solution: columns
    past the rank (|R_kk| > 1e-8 |R_00|) get 0. A [t, m, 9], B [t, m, f]."""
    t = torch.arange(A.shape[0], device=A.device)
    perm = torch.arange(9, device=A.device).repeat(A.shape[0], 1)
    for k in range(9):
        best = (A[:, k:, k:] ** 2).sum(1).argmax(1) + k
        for v in (A.transpose(1, 2), perm):  # swap columns k and best
            a, b = v[:, k].clone(), v[t, best].clone()
            v[:, k], v[t, best] = b, a
        v = A[:, k:, k].clone()
        v[:, 0] += torch.where(v[:, 0] >= 0, 1.0, -1.0) * v.norm(dim=1)
        f = (v * v).sum(1)
        f = torch.where(f > 0, 2.0 / f, f)[:, None]
        A[:, k:] -= v[:, :, None] * (f * (v[:, :, None] * A[:, k:]).sum(1))[:, None]
        B[:, k:] -= v[:, :, None] * (f * (v[:, :, None] * B[:, k:]).sum(1))[:, None]
    r = torch.stack([A[:, k, k] for k in range(9)], 1)
    full = ((r.abs() > 1e-8 * r[:, :1].abs()).long().cumprod(1) > 0)[:, :, None]
    y = torch.zeros((A.shape[0], 9, B.shape[2]), dtype=A.dtype, device=A.device)
    for k in range(8, -1, -1):
        q = B[:, k] - (A[:, k, k + 1:, None] * y[:, k + 1:]).sum(1)
        y[:, k] = torch.where(full[:, k], q / r[:, k, None], torch.zeros_like(q))
    return torch.zeros_like(y).scatter_(1, perm[:, :, None].expand_as(y), y)


def _lsq(d, w, bs):
    """Least squares of every field of `bs` on the Taylor rows of the offsets d
    (rows with w = 0 left out): the normal equations with one refinement, and
    pivoted QR for stencils too poor for them."""
    a = [d[0], d[1], d[2], 0.5 * d[0] * d[0], 0.5 * d[1] * d[1], 0.5 * d[2] * d[2],
         d[0] * d[1], d[0] * d[2], d[1] * d[2]]
    a = [v * w for v in a]
    L, poor = {}, w.sum(1) < 9
    for j in range(9):
        s = s0 = (a[j] * a[j]).sum(1)
        for k in range(j):
            s = s - L[j, k] * L[j, k]
        poor = poor | ~(s > 1e-5 * s0)
        L[j, j] = torch.sqrt(s)
        for i in range(j + 1, 9):
            s = (a[i] * a[j]).sum(1)
            for k in range(j):
                s = s - L[i, k] * L[j, k]
            L[i, j] = s / L[j, j]

    def solve(r):
        y = []
        for i in range(9):
            s = r[i]
            for k in range(i):
                s = s - L[i, k] * y[k]
            y.append(s / L[i, i])
        c = [None] * 9
        for i in range(8, -1, -1):
            s = y[i]
            for k in range(i + 1, 9):
                s = s - L[k, i] * c[k]
            c[i] = s / L[i, i]
        return c

    out = []
    for b in bs:
        c = solve([(v * b).sum(1) for v in a])
        r = b * w
        for v, q in zip(a, c):
            r = r - v * q[:, None]
        out.append([q + e for q, e in zip(c, solve([(v * r).sum(1) for v in a]))])
    at = torch.nonzero(poor).flatten()
    if at.numel() and not bs[0].requires_grad:
        pad = max(0, 9 - w.shape[1])
        A = torch.nn.functional.pad(torch.stack([v[at] for v in a], 2), (0, 0, 0, pad))
        B = torch.nn.functional.pad(torch.stack([(b * w)[at] for b in bs], 2), (0, 0, 0, pad))
        y = _basic(A, B)
        for f, c in enumerate(out):
            for k in range(9):
                c[k][at] = y[:, k, f]
    return out


def _rows(s, sten, ghost, b, e, prm, periods):
    """Scaled offsets and weights of the rows of particles b..e, ghost rows after them."""
    ids, mir, ok = (v[b:e] for v in sten)
    _, d = _pair_d2(s[:3], torch.arange(b, e, device=s[0].device), ids, mir, periods)
    d = [v / prm["h"] for v in d]
    w = ok.to(d[0].dtype)
    if ghost is not None:
        d = [torch.cat([v, -v], 1) for v in d]
        w = torch.cat([w, ghost[b:e].to(w.dtype)], 1)
    return ids, mir, d, w


class _S(list):
    """Seven rows that index like a [7, n] tensor."""

    @property
    def shape(self):
        return (len(self), self[0].shape[0])


def _derivs(s, th, sten, ghost, prm, periods, mus, heun):
    """du/dt, V^{n+1} and V_t of the semi-discrete system (one stage)."""
    n, h = s[0].shape[0], prm["h"]
    g2 = []
    for b in range(0, n, CHUNK):
        e = min(n, b + CHUNK)
        ids, mir, d, w = _rows(s, sten, ghost, b, e, prm, periods)
        bs = []
        for k in (3, 4, 5):  # no-slip floor: mirrors carry -u; ghosts the particle's own u
            v = torch.where(mir, -s[k][ids], s[k][ids]) - s[k][b:e, None]
            bs.append(torch.cat([v, torch.zeros_like(v)], 1) if ghost is not None else v)
        c = _lsq(d, w, bs)
        G = [[c[i][j] / h for j in range(3)] for i in range(3)]
        div = G[0][0] + G[1][1] + G[2][2]
        t = div / 3.0
        gd = [G[0][0] - t, G[1][1] - t, G[2][2] - t, 0.5 * (G[0][1] + G[1][0]),
              0.5 * (G[0][2] + G[2][0]), 0.5 * (G[1][2] + G[2][1])]
        ss = 0.5 * (gd[0] ** 2 + gd[1] ** 2 + gd[2] ** 2) + gd[3] ** 2 + gd[4] ** 2 + gd[5] ** 2
        gn = torch.where(ss > 0, torch.sqrt(torch.where(ss > 0, ss, torch.ones_like(ss))), 0.0 * ss)
        dd = [c[0][3] + c[1][6] + c[2][7], c[0][6] + c[1][4] + c[2][8], c[0][7] + c[1][8] + c[2][5]]
        ld = [(0.5 * (c[i][3] + c[i][4] + c[i][5]) + dd[i] / 6.0) / (h * h) for i in range(3)]
        g2.append(gd + [gn] + ld + [div])
    q = [torch.cat([v[k] for v in g2]) for k in range(11)]
    gd, gn, ld, div = q[:6], q[6], q[7:10], q[10]
    Vn = s[6] + DT * (s[6] * div)
    Vf = s[6] if heun else Vn  # the V of pass 2
    phi = 1.0 / Vf
    inertial = (phi > EOS["phi_min"]) & (phi <= EOS["phi_max"])
    acc = [[], [], []]
    for b in range(0, n, CHUNK):
        e = min(n, b + CHUNK)
        ids, mir, d, w = _rows(s, sten, ghost, b, e, prm, periods)
        bg = torch.where(mir, torch.zeros_like(gn[ids]), gn[ids]) - gn[b:e, None]
        bv = Vf[ids] - Vf[b:e, None]
        if ghost is not None:
            pg = EOS["phi_min"] * (1 - 1e-3)
            den = torch.where(inertial, EOS["phi_c"] - phi, torch.ones_like(phi))[b:e]
            gg = torch.where(inertial[b:e], gn[b:e] * ((EOS["phi_c"] - pg) / den), gn[b:e])
            bg = torch.cat([bg, (gg - gn[b:e])[:, None].expand_as(bg)], 1)
            bv = torch.cat([bv, (1.0 / pg - Vf[b:e])[:, None].expand_as(bv)], 1)
        c = _lsq(d, w, [bg, bv])
        cg, cV = [c[0][j] / h for j in range(3)], [c[1][j] / h for j in range(3)]
        a = EOS["phi_c"] - EOS["phi_min"]
        om = torch.where(inertial, EOS["phi_c"] - phi, torch.ones_like(phi))[b:e]
        mu_s = th[0][b:e] if mus is None else mus[b:e]
        k = 4.0 * a * a * MUI["d"] * MUI["d"]
        M, den = -k / (om * om), a * th[2] + om
        mu = (a * mu_s * th[2] + th[1] * om) / den
        N, S = -M * mu, -2.0 * k / (om * om * om)
        R = -S * mu + M * (a * th[2] * (th[1] - mu_s)) / (den * den)
        V, G = Vf[b:e], gn[b:e]
        T = [v[b:e] for v in gd]
        T = [[T[0], T[3], T[4]], [T[3], T[1], T[5]], [T[4], T[5], T[2]]]
        for i in range(3):
            tV = sum(T[i][j] * cV[j] for j in range(3))
            tG = sum(T[i][j] * cg[j] for j in range(3))
            f = V * (-(G / (V * V)) * (S * G * cV[i] + R * tV) + 2.0 * M * G * cg[i] + N * tG
                     + N * G * ld[i][b:e])
            solid = EOS["beta"] * cV[i] / V
            gas = phi[b:e] <= EOS["phi_min"]
            f = torch.where(inertial[b:e], f, torch.where(gas, torch.zeros_like(f), solid))
            acc[i].append(f + (prm["gx"], prm["gy"], prm["gz"])[i])
    return [torch.cat(v) for v in acc], Vn


def _wrap(x, L):
    return x if not L else torch.where(x >= L, x - L, torch.where(x < 0, x + L, x))


def _advance(s, th, sten, ghost, prm, periods, mus, heun):
    a, Vn = _derivs(s, th, sten, ghost, prm, periods, mus, heun)
    u = [s[3 + i] + DT * a[i] for i in range(3)]
    x = [s[i] + (DT * s[3 + i] if heun else 0.5 * DT * (s[3 + i] + u[i])) for i in range(3)]
    return _S([_wrap(x[i], periods[i]) for i in range(3)] + u + [Vn])


def _one_step(s, th, sten, ghost, prm, periods, mus):
    heun = bool(prm["time_scheme"])
    y = _advance(s, th, sten, ghost, prm, periods, mus, heun)
    if heun:
        y = _advance(y, th, sten, ghost, prm, periods, mus, True)
        y = _S([_wrap(s[i] + 0.5 * _near(y[i] - s[i], periods[i]), periods[i]) if i < 3
                else 0.5 * (s[i] + y[i]) for i in range(7)])
    return y


def _topology(s, col, prm, periods):
    p = torch.stack([v.detach() for v in s[:3]])
    sten = _stencils(p, col, prm["radius"], True, periods, 64)
    ghost = _ghost_flags(p, col, sten, prm, periods) if prm["free_surface"] else None
    most = int(sten[2].sum(1).max())
    sten = [v[:, :most] for v in sten]
    return sten, None if ghost is None else ghost[:, :most]


def _exact_step(c, seed):
    init, offs, mus, prm = _step_inputs(c, seed)
    n, dev = init.shape[1], init.device
    col = torch.zeros(n, dtype=torch.long, device=dev)
    mu = torch.full((n,), MUI["mu_s"], dtype=torch.float64, device=dev)
    if offs is not None:
        size = torch.tensor(np.diff(offs), device=dev)
        col = torch.repeat_interleave(torch.arange(len(mus), device=dev), size)
        mu = torch.tensor(mus, dtype=torch.float64, device=dev)[col]
    periods = (prm["period_x"], prm["period_y"], 0.0)
    s = _S(init)
    for _ in range(c["steps"] * c["calls"]):
        sten, ghost = _topology(s, col, prm, periods)
        s = _one_step(s, (None, MUI["mu_2"], MUI["I0"]), sten, ghost, prm, periods, mu)
    return {k: v.cpu() for k, v in zip(FIELDS, s)} if c["host"] else dict(zip(FIELDS, s))


def _exact_fit(s, sten, fields, signs, h):
    n, out = s[0].shape[0], []
    scale = torch.tensor([1 / h] * 3 + [1 / (h * h)] * 6, dtype=torch.float64, device=s[0].device)
    for b in range(0, n, CHUNK):
        e = min(n, b + CHUNK)
        ids, mir, d, w = _rows(s, sten, None, b, e, dict(h=h), (0, 0, 0))
        bs = [torch.where(mir, q * f[ids], f[ids]) - f[b:e, None] for f, q in zip(fields, signs)]
        c = _lsq(d, w, bs)
        out.append(torch.stack([torch.stack(v, 1) for v in c], 1) * scale)
    return torch.cat(out)


def _exact_stress(case, seed):
    init, _, _, prm = _step_inputs(dict(case, phi=0.5), seed)
    col = torch.zeros(init.shape[1], dtype=torch.long, device=init.device)
    sten, _ = _topology(_S(init), col, prm, (0.0, 0.0, 0.0))
    d = _exact_fit(_S(init), sten, list(init[3:6]), [-1.0] * 3, prm["h"])
    G = d[:, :, :3]
    t = (G[:, 0, 0] + G[:, 1, 1] + G[:, 2, 2]) / 3.0
    g = torch.stack([G[:, 0, 0] - t, G[:, 1, 1] - t, G[:, 2, 2] - t,
                     0.5 * (G[:, 0, 1] + G[:, 1, 0]), 0.5 * (G[:, 0, 2] + G[:, 2, 0]),
                     0.5 * (G[:, 1, 2] + G[:, 2, 1])], 1)
    gn = torch.sqrt(0.5 * (g[:, :3] ** 2).sum(1) + (g[:, 3:] ** 2).sum(1))
    phi = 1.0 / init[6]
    gas, solid = phi <= EOS["phi_min"], phi > EOS["phi_max"]
    a, om = EOS["phi_c"] - EOS["phi_min"], EOS["phi_c"] - phi
    P = MUI["rho_s"] * (2 * a * MUI["d"] * gn / om) ** 2
    mu = (a * MUI["mu_s"] * MUI["I0"] + MUI["mu_2"] * om) / (a * MUI["I0"] + om)
    eta = MUI["rho_s"] * 4 * a * a * MUI["d"] ** 2 / (om * om) * mu * gn
    zero = torch.zeros_like(P)
    P = torch.where(solid, MUI["rho_s"] * (EOS["alpha"] + EOS["beta"] * phi), torch.where(gas, zero, P))
    eta = torch.where(gas | solid, zero, eta)
    regime = torch.where(gas, 0, torch.where(solid, 2, 1)).to(torch.int8)
    return dict(gdot=g, gdot_norm=gn, P=P, eta=eta, regime=regime, d=d)


def _exact_adjoint(c, seed):
    from torch.utils.checkpoint import checkpoint
    st = _step_inputs(dict(c, ghosts=True), seed)
    init, prm = st[0], st[3]
    n, dev = init.shape[1], init.device
    lam = torch.from_numpy(np.random.default_rng([int(seed), 79])
                           .standard_normal(tuple(init.shape))).to(dev)
    theta = torch.tensor([MUI["mu_s"], MUI["mu_2"], MUI["I0"]], dtype=torch.float64, device=dev,
                         requires_grad=True)
    first = [v.clone().requires_grad_(True) for v in init]
    col = torch.zeros(n, dtype=torch.long, device=dev)
    s, periods = _S(first), (0.0, 0.0, 0.0)
    for k in range(c["steps"]):
        if k % c["every"] == 0:
            sten, ghost = _topology(s, col, prm, periods)
            if int(sten[2].sum(1).min()) < 9:
                return None  # the gradient of such a stencil is left out by definition

        def step(t, *v, sten=sten, ghost=ghost):
            return tuple(_one_step(_S(v), (t[0].expand(n), t[1], t[2]), sten, ghost, prm, periods,
                                   None))

        s = _S(checkpoint(step, theta, *s, use_reentrant=False))
    g = torch.autograd.grad(list(s), [theta] + first, list(lam))
    return dict(out={k: v.detach() for k, v in zip(FIELDS, s)}, dtheta=g[0],
                dstate=dict(zip(FIELDS, g[1:])))


def exact(case, seed):
    if case["kind"] == "step":
        return _exact_step(case, seed)
    if case["kind"] == "stress":
        return _exact_stress(case, seed)
    if case["kind"] == "adjoint":
        return _exact_adjoint(case, seed)
    p, radius, fields, h = _sweep_inputs(case, seed)
    col = torch.zeros(p.shape[1], dtype=torch.long, device=p.device)
    sten = _stencils(p, col, radius, False, (0.0, 0.0, 0.0), case["cap"], case["keep"])
    return _exact_fit(_S(p), sten, fields, [1.0] * case["nf"], h)
