"""LP_FP64 on stencils that one fixed-point scale cannot hold.

The rows of LP_FP64 are summed in fixed point laid out for the stencil radius.
A particle whose stencil is thin along an axis, or small against the radius, or
has entries far outside it, takes plain FP64 rows, and its results are as good
as any other's. The reference solves the least-squares problem itself in
extended precision, or is the oracle's step.

Errors are measured in each coefficient's own units: a derivative along an axis
on which the stencil extends over `a` lattice spacings counts times `a`.
"""
import numpy as np
import pytest

from paper_2206_14061_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

TOL = 1e-11  # of the largest coefficient: what LP_FP64 derivatives are held to


@pytest.fixture(scope="module")
def capi():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_14061_gb300 import build
    build.build()
    from paper_2206_14061_gb300 import capi as C
    C.lib()
    return C


def T(a):
    return torch.tensor(np.ascontiguousarray(a, dtype=np.float64), device="cuda:0")


def _lattice(k, jitter, seed=7):
    i = np.arange(k)
    X = np.stack(np.meshgrid(i, i, i, indexing="ij")).reshape(3, -1) - 0.5 * (k - 1)
    return X + np.random.default_rng(seed).uniform(-jitter, jitter, X.shape)


def _lists(X, r):
    """Caller's stencils: entries within r (rows [n, cap], counts)."""
    d = np.linalg.norm(X[:, :, None] - X[:, None, :], axis=0)
    np.fill_diagonal(d, np.inf)
    rows = [np.nonzero(d[i] <= r)[0] for i in range(X.shape[1])]
    cnt = np.array([len(q) for q in rows], dtype=np.int32)
    nbr = np.zeros((X.shape[1], 64), dtype=np.int32)
    for i, q in enumerate(rows):
        nbr[i, :len(q)] = q
    return nbr, cnt


def _own(capi, ctx, nbr, cnt):
    t = torch.tensor(np.ascontiguousarray(nbr.T).ravel(), dtype=torch.int32, device="cuda:0")
    c = torch.tensor(cnt, dtype=torch.int32, device="cuda:0")
    nb = capi.Neighbors(ctx, capi.LpNeighbors(t.data_ptr(), c.data_ptr(), len(cnt),
                                              nbr.shape[1], 0))
    nb.keep = (t, c)
    return nb


def _columns(d):
    x, y, z = d
    return np.stack([x, y, z, x * x / 2, y * y / 2, z * z / 2, x * y, x * z, y * z], -1)


def _reference(X, nbr, cnt, F, pick=None):
    """Coefficients [n, nf, 9] of the stored positions in units of X, by normal
    equations in extended precision (columns scaled; 64 bits or more)."""
    pick = np.arange(X.shape[1]) if pick is None else pick
    L = np.longdouble
    live = np.arange(nbr.shape[1]) < cnt[pick, None]
    j = np.where(live, nbr[pick], pick[:, None])  # (a row of zeros)
    A = _columns(X.astype(L)[:, j] - X.astype(L)[:, pick, None])
    b = F.astype(L)[:, j] - F.astype(L)[:, pick, None]
    s = np.sqrt((A * A).sum(1))
    s[s == 0] = 1
    A = A / s[:, None]
    G = (A[:, :, :, None] * A[:, :, None, :]).sum(1) + np.eye(9) * (cnt[pick] < 9)[:, None, None]
    R = (A[None, :, :, :] * b[:, :, :, None]).sum(2)
    for k in range(9):  # Cholesky, the factor in the lower triangle
        G[:, k, k] = np.sqrt(G[:, k, k])
        G[:, k + 1:, k] /= G[:, k, k, None]
        for m in range(k + 1, 9):
            G[:, m:, m] -= G[:, m:, k] * G[:, m, k, None]
    for k in range(9):
        R[..., k] = (R[..., k] - (G[:, k, :k] * R[..., :k]).sum(-1)) / G[:, k, k]
    for k in reversed(range(9)):
        R[..., k] = (R[..., k] - (G[:, k + 1:, k] * R[..., k + 1:]).sum(-1)) / G[:, k, k]
    return np.moveaxis(R / s, 0, 1).astype(np.float64)


def _error(got, ref, scale, fit):
    """Largest error over the particles `fit`, in units of the stencil's own
    extents (scale: their length per axis), of each field's largest one."""
    a, b, c = scale
    u = np.array([a, b, c, a * a, b * b, c * c, a * b, a * c, b * c])
    e = np.abs((got - ref) * u)[fit].max(axis=(0, 2))
    return float((e / np.abs(ref * u)[fit].max(axis=(0, 2))).max())


def _fields(X):
    return np.stack([np.sin(0.4 * X[0] + 0.3 * X[1] - 0.2 * X[2]) + 2.0,
                     X[0] * X[2] - 0.5 * X[1] ** 2 + X[1] + 0.3 * X[2]])


@pytest.mark.parametrize("built", [False, True])
@pytest.mark.parametrize("axis", [0, 2])
@pytest.mark.parametrize("aspect", [1.0, 0.3, 0.1, 0.03, 0.01, 1e-3, 1e-4])
def test_fit_of_a_stencil_thin_along_an_axis(capi, aspect, axis, built):
    """A lattice compressed along one axis. Caller's stencils, or those the
    context built before the compression (the range is then their radius)."""
    h, X = 1e-3, _lattice(7, 0.1)
    F = _fields(X)
    ctx = capi.Context(X.shape[1], cap=64)
    if built:
        nb = capi.lp_build_neighbors(ctx, *[T(c) for c in X * h], r_const=1.9 * h, mirror_mode=0)
        nbr, cnt = nb.export()
    else:
        nbr, cnt = _lists(X, 1.9)
        nb = _own(capi, ctx, nbr, cnt)
    s = np.ones(3)
    s[axis] = aspect
    P = X * s[:, None] * h
    got = capi.lp_fit_derivatives(ctx, *[T(c) for c in P], nb, [T(f) for f in F], [1.0, 1.0],
                                  h).cpu().numpy()
    assert ctx.sync()["flags"] == 0
    ref = _reference(P, nbr, cnt, F)
    fit = cnt >= 17  # (with fewer entries FP64 itself is worse)
    assert fit.sum() > 200
    err = _error(got, ref, s * h, fit)
    print(f"aspect {aspect:g} axis {axis} built {built}: {err:.2e}")
    assert err <= TOL
    ctx.close()


def _params(pd, **kw):
    prm = {k: pd[k] for k in ("h", "radius", "gx", "gy", "gz", "floor_z", "mirror_mode")}
    prm.update(precision=0, rebuild_every=1, launch_mode=0, skin=0.0, free_surface=0)
    prm.update(kw)
    return prm


def _step_both(capi, orc, P, vel, radius, dt, mode=0):
    """One LP_FP64 step on the device and by the oracle: the changes of u, v, w."""
    wl = W.cube(6)
    pd = dict(W.param_dict(wl), h=1e-3, radius=radius, mirror_mode=0, dt=dt, gz=0.0)
    n = P.shape[1]
    st = dict(zip(capi.FIELDS, [*P, *vel, np.full(n, 1.0 / 0.5)]))
    ref, _ = orc.step(st, orc.params(**pd), 1, brute=n < 4000)
    ctx = capi.Context(n, cap=64)
    dev = {k: T(v) for k, v in st.items()}
    mui = {k: pd[k] for k in ("mu_s", "mu_2", "I0", "d", "rho_s")}
    eos = {k: pd[k] for k in ("phi_c", "phi_min", "phi_max", "alpha", "beta")}
    capi.lp_step(ctx, dev, mui, eos, _params(pd, launch_mode=mode), dt, 1)
    d = ctx.sync()
    ctx.close()
    assert d["flags"] == 0
    du = np.stack([dev[k].cpu().numpy() - st[k] for k in "uvw"])
    dr = np.stack([ref[k] - st[k] for k in "uvw"])
    return du, dr


@pytest.mark.parametrize("mode", [0, 2])
@pytest.mark.parametrize("side", [20, 80, 170])
@pytest.mark.parametrize("aspect", [0.5, 0.3, 0.1, 0.03, 0.01])
def test_step_of_a_sheet(capi, orc, aspect, side, mode):
    """Three lattice layers `aspect` h apart (at the four-lane, two-lane and
    one-thread launch shapes, and in the persistent launch): the velocity
    change against the oracle's. The flow varies by the same amount over h in
    every direction of the sheet, so the largest terms are those across it."""
    h = 1e-3
    i, k = np.arange(side), np.arange(3)
    X = np.stack(np.meshgrid(i, i, k, indexing="ij")).reshape(3, -1).astype(float)
    X += np.random.default_rng(3).uniform(-0.05, 0.05, X.shape)
    vel = 1e-2 * np.stack([np.sin(0.5 * X[0] + 0.7 * X[2]), np.cos(0.4 * X[1] - 0.5 * X[2]),
                           np.sin(0.3 * X[0] - 0.4 * X[1] + 0.6 * X[2])])
    P = (X + 2.0) * h * np.array([1.0, 1.0, aspect])[:, None]
    # |d_z u| = 1e-2 / (h aspect); V changes by less than 1 %
    dt = 1e-3 * aspect
    du, dr = _step_both(capi, orc, P, vel, 1.5 * h, dt, mode)
    inner = ((X[:2] > 1.5) & (X[:2] < side - 2.5)).all(0)
    # u + du is rounded to 2^-53 u
    floor = 2.0 ** -52 * np.abs(vel).max()
    err, big = np.abs(du - dr)[:, inner].max() - floor, np.abs(dr)[:, inner].max()
    print(f"aspect {aspect:g} n {P.shape[1]} mode {mode}: {err / big:.2e}")
    assert err <= TOL * big


@pytest.mark.parametrize("size", [1.0, 0.3, 0.1, 0.02])
def test_step_of_small_clusters(capi, orc, size):
    """Clusters of 3^3 particles `size` h apart, far from one another: offsets
    far below the radius, the same along all axes."""
    h = 1e-3
    X = _lattice(3, 0.1)
    g = np.random.default_rng(4)
    parts, vels = [], []
    for c in range(40):
        Y = X + g.uniform(-0.02, 0.02, X.shape)
        at = 8.0 * np.array([c % 4, (c // 4) % 4, c // 16])[:, None] + 3.0
        parts.append((Y * size + at) * h)
        vels.append(1e-2 * np.stack([np.sin(0.5 * Y[0] + 0.7 * Y[2]),
                                     np.cos(0.4 * Y[1] - 0.5 * Y[2]),
                                     np.sin(0.3 * Y[0] - 0.4 * Y[1] + 0.6 * Y[2])]))
    P, vel = np.concatenate(parts, 1), np.concatenate(vels, 1)
    # the largest offset in a cluster of spacing h is below the radius
    du, dr = _step_both(capi, orc, P, vel, 4.0 * h, 1e-3 * size)
    floor = 2.0 ** -52 * np.abs(vel).max()
    err = np.abs(du - dr).max() - floor
    print(f"size {size:g}: {err / np.abs(dr).max():.2e}")
    assert err <= TOL * np.abs(dr).max()


def _turn(r, bits):
    """Length after which fixed-point positions repeat, laid out for radius r."""
    return bits * 2.0 ** np.frexp(r)[1]


@pytest.mark.parametrize("lists", ["own", "built", "mirrors"])
@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("turns", [0.3, 1, 3, 1000, 3e6])
def test_fit_of_entries_far_along_an_axis(capi, turns, axis, lists):
    """A lattice whose layers are whole turns of the fixed-point positions apart
    along one axis: the entries look near. Caller's stencils, those the context
    built before the layers moved, and caller's with every entry of a higher
    layer given as the floor mirror of a particle below the floor."""
    h, X = 1e-3, _lattice(7, 0.05)
    base = np.round(X)
    ctx = capi.Context(2 * X.shape[1], cap=64)
    P = X * h
    nbr, cnt = _lists(X, 1.9)
    nb = None
    if lists == "built":
        nb = capi.lp_build_neighbors(ctx, *[T(c) for c in P], r_const=1.9 * h, mirror_mode=0)
        nbr, cnt = nb.export()
    apart = turns * _turn(1.9 * h if lists == "built" else 4 * h, 64.0)
    P[axis] = base[axis] * apart + (X - base)[axis] * h
    F, floor, sign = _fields(X), 0.0, [1.0, 1.0]
    if lists == "mirrors":
        n = X.shape[1]
        up = (np.arange(64) < cnt[:, None]) & (base[2][nbr] > base[2][:, None])
        floor = -4.0 * (apart if axis == 2 else h)
        P = np.concatenate([P, np.stack([P[0], P[1], 2.0 * floor - P[2]])], 1)
        at = P.copy()
        at[2, n:] = 2.0 * floor - P[2, n:]  # as the stored positions have them
        ref_nbr = np.concatenate([np.where(up, nbr + n, nbr), np.zeros_like(nbr)])
        nbr = np.concatenate([np.where(up, (nbr + n) | np.int32(-2 ** 31), nbr),
                              np.zeros_like(nbr)])
        cnt = np.concatenate([cnt, np.zeros_like(cnt)])
        F = np.concatenate([F, -F], 1)  # (odd fields: the mirrors have F again)
        sign = [-1.0, -1.0]
        ref_F = np.concatenate([F[:, :n], F[:, :n]], 1)
    else:
        at, ref_nbr, ref_F = P, nbr, F
    if nb is None:
        nb = _own(capi, ctx, nbr, cnt)
    got = capi.lp_fit_derivatives(ctx, *[T(c) for c in P], nb, [T(f) for f in F], sign, h,
                                  floor_z=floor).cpu().numpy()
    assert ctx.sync()["flags"] == 0
    fit = cnt >= 26
    assert fit.sum() >= 100
    ref = np.zeros_like(got)
    ref[fit] = _reference(at, ref_nbr, cnt, ref_F, np.nonzero(fit)[0])
    s = np.full(3, h)
    s[axis] = apart
    err = _error(got, ref, s, fit)
    print(f"turns {turns:g} axis {axis} {lists}: {err:.2e}")
    assert err <= TOL
    ctx.close()


@pytest.mark.parametrize("mode", [0, 2])
@pytest.mark.parametrize("side", [7, 26, 31])
@pytest.mark.parametrize("axis", [0, 2])
def test_step_on_held_stencils_that_spread(capi, orc, axis, side, mode):
    """A dilute gas (no stress) whose layers move a turn of the fixed-point
    positions apart in the first step; the second takes the same stencils."""
    h, dt, radius = 1e-3, 1e-3, 1.9e-3
    X = _lattice(side, 0.05)
    base = np.round(X - X.min(1)[:, None])
    vel = np.zeros_like(X)
    vel[axis] = base[axis] * _turn(radius, 16.0) / dt
    wl = W.cube(6)
    pd = dict(W.param_dict(wl), h=h, radius=radius, mirror_mode=0, dt=dt, gz=0.0)
    n = X.shape[1]
    st = dict(zip(capi.FIELDS, [*(X * h), *vel, np.full(n, 1.0 / 0.2)]))
    ref, _ = orc.step(st, orc.params(**pd), 2, rebuild_every=2, brute=n < 4000)
    ctx = capi.Context(n, cap=64)
    dev = {k: T(v) for k, v in st.items()}
    mui = {k: pd[k] for k in ("mu_s", "mu_2", "I0", "d", "rho_s")}
    eos = {k: pd[k] for k in ("phi_c", "phi_min", "phi_max", "alpha", "beta")}
    capi.lp_step(ctx, dev, mui, eos, _params(pd, launch_mode=mode, rebuild_every=2), dt, 2)
    assert ctx.sync()["flags"] == 0
    ctx.close()
    # (two layers from the surface: V of the outermost is an extrapolation, may
    # leave the gas regime, and then changes velocities that the next one sees)
    inner = ((base > 1.5) & (base < side - 2.5)).all(0)
    err = np.abs(dev["V"].cpu().numpy() - ref["V"])[inner].max() / ref["V"][inner].max()
    print(f"n {n} mode {mode}: {err:.2e}")
    assert err <= TOL
    for k in "xyzuvw":
        assert np.allclose(dev[k].cpu().numpy()[inner], ref[k][inner], rtol=1e-12, atol=0), k


@pytest.mark.parametrize("h", [1e60, 1e69, 1e70, 1e72, 1e75, 1e77])
def test_fit_with_h_far_above_the_spacing(capi, h):
    """h is only the unit of the offsets: fourth powers of 1 / h near the
    smallest normal number."""
    X = _lattice(7, 0.1)
    nbr, cnt = _lists(X, 1.9)
    F = _fields(X)
    for built in (False, True):
        ctx = capi.Context(X.shape[1], cap=64)
        nb = (capi.lp_build_neighbors(ctx, *[T(c) for c in X], r_const=1.9, mirror_mode=0)
              if built else _own(capi, ctx, nbr, cnt))
        got = capi.lp_fit_derivatives(ctx, *[T(c) for c in X], nb, [T(f) for f in F], [1.0, 1.0],
                                      h).cpu().numpy()
        assert ctx.sync()["flags"] == 0
        fit = cnt >= 17
        err = _error(got, _reference(X, nbr, cnt, F), np.ones(3), fit)
        print(f"h {h:g} built {built}: {err:.2e}")
        assert err <= TOL
        ctx.close()


@pytest.mark.parametrize("ratio", [1, 20, 60, 500, 1000, 2000, 4000, 10000])
def test_fit_of_small_stencils_near_the_origin(capi, ratio):
    """Radii 1 : ratio in one call, the small ones where coordinates have more
    bits than the layout for the largest keeps: 64 roundings of FP64."""
    big = 2.2e-3
    X = _lattice(7, 0.1)
    d = big / ratio / 1.9
    P = np.concatenate([X * d, np.full((3, 1), 1.0)], 1)
    rad = np.append(np.full(X.shape[1], 1.9 * d), big)
    ctx = capi.Context(P.shape[1], cap=64)
    nb = capi.lp_build_neighbors(ctx, *[T(c) for c in P], radius=T(rad), mirror_mode=0)
    nbr, cnt = nb.export()
    F = np.concatenate([_fields(X), np.zeros((2, 1))], 1)
    got = capi.lp_fit_derivatives(ctx, *[T(c) for c in P], nb, [T(f) for f in F], [1.0, 1.0],
                                  d).cpu().numpy()
    assert ctx.sync()["flags"] == 0
    ctx.close()
    fit = cnt >= 26
    assert fit.sum() >= 100
    ref = np.zeros_like(got)
    ref[fit] = _reference(P, nbr, cnt, F, np.nonzero(fit)[0])
    err = _error(got, ref, np.full(3, d), fit)
    print(f"ratio {ratio}: {err:.2e}")
    assert err <= 64 * 2.0 ** -53
