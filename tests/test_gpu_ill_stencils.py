"""lp_fit_derivatives on lattices with little jitter and few entries a stencil,
a third of which are poorly conditioned (small pivots of the normal equations):
few of them take the pivoted QR fit, many the normal equations as all others,
and no number of them overflows a queue.
"""
import numpy as np
import pytest

from test_gpu_fixed_range import T, _columns, _lattice, _reference

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def capi():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2206_14061_gb300 import build
    build.build()
    from paper_2206_14061_gb300 import capi as C
    C.lib()
    return C


def _pivots(X, nbr, cnt, pick):
    """Smallest pivot of the normal equations relative to its diagonal."""
    live = np.arange(nbr.shape[1]) < cnt[pick, None]
    j = np.where(live, nbr[pick], pick[:, None])
    A = _columns(X[:, j] - X[:, pick, None])
    G = (A[:, :, :, None] * A[:, :, None, :]).sum(1)
    d = np.einsum("naa->na", G).copy()
    p = np.full(len(pick), np.inf)
    for k in range(9):
        p = np.minimum(p, G[:, k, k] / d[:, k])
        G[:, k + 1:, k + 1:] -= (G[:, k + 1:, k, None] * G[:, k, None, k + 1:]
                                 / G[:, k, k, None, None])
    return p


@pytest.mark.parametrize("prec,eps", [(0, 2.0 ** -53), (2, 2.0 ** -44)])
# few (13 of 1728 below 2^-7) and many (380, 2200; 310 and 1700 below 2^-10)
@pytest.mark.parametrize("side,jitter,cap", [(12, 0.2, 48), (9, 0.03, 12), (20, 0.03, 12)])
def test_poorly_conditioned_stencils(capi, side, jitter, cap, prec, eps):
    """Errors against extended precision. The sums have 12 rows of up to 2^3 (entries
    up to 2, fields up to 1, spacings up to 2), the solve 9 steps: 2^10 units in
    the last place (2^12 with 48 rows), amplified by at most 1 / pivot^2."""
    h, X = 1e-3, _lattice(side, jitter)
    P = X * h
    ctx = capi.Context(X.shape[1], cap=64)
    nb = capi.lp_build_neighbors(ctx, *[T(c) for c in P], r_const=2.2 * h, mirror_mode=0, cap=cap,
                                 keep_nearest=1)
    nbr, cnt = nb.export()
    F = np.stack([np.sin(0.4 * X[0] + 0.3 * X[1] - 0.2 * X[2]), np.cos(0.3 * X[0] - 0.5 * X[2])])
    got = [capi.lp_fit_derivatives(ctx, *[T(c) for c in P], nb, [T(f) for f in F], [1.0, 1.0],
                                   h, precision=prec).cpu().numpy() for _ in range(2)]
    d = ctx.sync()
    ctx.close()
    assert d["flags"] == 0
    assert np.array_equal(got[0], got[1])
    pick = np.arange(X.shape[1])
    p = _pivots(X, nbr, cnt, pick)
    pick, p = pick[p > 2e-4], p[p > 2e-4]  # (below, LP_MIXED_FF refuses)
    assert (p < 2.0 ** -7).sum() > (64 if cap == 12 else 0)
    ref = _reference(P, nbr, cnt, F, pick)
    u = np.array([h] * 3 + [h * h] * 6)
    err = np.abs((got[0][pick] - ref) * u).max((1, 2))
    print(f"n {X.shape[1]} prec {prec}: below 2^-7 {(p < 2.0 ** -7).sum()}, 2^-10 "
          f"{(p < 2.0 ** -10).sum()}, largest error {err.max():.1e}, in bounds "
          f"{(err * p * p).max() / eps:.2f}")
    assert (err * p * p <= 2 ** (10 if cap == 12 else 12) * eps).all()


@pytest.mark.parametrize("prec", [0, 2])
def test_more_poorly_conditioned_stencils_than_the_queue_holds(capi, prec):
    """A sheet of two layers, over 2^20 of them: every stencil is fitted
    (coefficients start as NaN) and quadratic fields come back."""
    h, k = 1e-3, 800
    i = np.arange(k)
    X = np.stack(np.meshgrid(i, i, np.arange(2), indexing="ij")).reshape(3, -1).astype(float)
    X += np.random.default_rng(7).uniform(-0.03, 0.03, X.shape)
    n = X.shape[1]
    ctx = capi.Context(n, cap=32)
    P = [T(c * h) for c in X]
    nb = capi.lp_build_neighbors(ctx, *P, r_const=2.2 * h, mirror_mode=0, cap=17, keep_nearest=1)
    Xg = [p / h for p in P]
    F = [Xg[0] * Xg[1] / k + 0.5 * Xg[2] ** 2 - Xg[0]]
    out = torch.full((n, 1, 9), float("nan"), dtype=torch.float64, device="cuda:0")
    capi.lp_fit_derivatives(ctx, *P, nb, F, [1.0], h, precision=prec, out=out)
    d = ctx.sync()
    ctx.close()
    assert d["flags"] == 0
    assert d["n_fallback"] < n // 10
    assert bool(torch.isfinite(out).all())
    err = (out[:, 0, 0] * h - (Xg[1] / k - 1.0)).abs()
    assert float(err.max()) < 1e-3
    assert float((err < (1e-10 if prec == 0 else 1e-6)).double().mean()) > 0.99


@pytest.mark.parametrize("prec,unit,aspect", [(0, 3e-10, 1.0), (0, 1e-3, 1.0), (0, 1.0, 1e-5),
                                              (2, 1e-3, 1.0), (2, 1.0, 1e-4)])
def test_poorly_conditioned_stencils_whose_columns_differ_in_size(capi, prec, unit, aspect):
    """The spacing `unit` h, compressed along z to `aspect`: pivots relative to
    the columns are those of the lattice, but the QR fit's rank, relative to
    the largest column, would leave out the smallest."""
    h, X = 1.0, _lattice(5, 0.06, seed=11)
    P = X * unit
    ctx = capi.Context(X.shape[1], cap=64)
    nb = capi.lp_build_neighbors(ctx, *[T(c) for c in P], r_const=2.2 * unit, mirror_mode=0,
                                 cap=12, keep_nearest=1)
    nbr, cnt = nb.export()
    P[2] *= aspect
    F = np.stack([np.sin(0.4 * X[0] + 0.3 * X[1] - 0.2 * X[2]), np.cos(0.3 * X[0] - 0.5 * X[2])])
    got = capi.lp_fit_derivatives(ctx, *[T(c) for c in P], nb, [T(f) for f in F], [1.0, 1.0], h,
                                  precision=prec).cpu().numpy()
    assert ctx.sync()["flags"] == 0
    ctx.close()
    pick = np.arange(X.shape[1])
    p = _pivots(X, nbr, cnt, pick)
    pick, p = pick[p > 2e-4], p[p > 2e-4]
    ill = (p < (2.0 ** -7 if prec == 0 else 2.0 ** -10)).sum()
    ref = _reference(P, nbr, cnt, F, pick)
    u, v = unit, unit * aspect
    err = np.abs((got[pick] - ref) * np.array([u, u, v, u * u, u * u, v * v, u * u, u * v, u * v]))
    err = err.max((1, 2))
    eps = 2.0 ** -53 if prec == 0 else 2.0 ** -44
    print(f"prec {prec} unit {unit:g} aspect {aspect:g}: {ill} ill, largest error "
          f"{err.max():.1e}, in bounds {(err * p * p).max() / eps:.2f}")
    assert 0 < ill and (err * p * p <= 2 ** 10 * eps).all()
