"""The pivoted QR fits of lp_fit_derivatives (stencils that the normal equations
refuse) against the oracle's, which are the same algorithm: rank and basic
solution.
"""
import numpy as np
import pytest

from test_gpu_fixed_range import T, _fields, _lattice, _lists, _own

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


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("axes,value", [("xyz", np.nan), ("z", np.nan), ("x", np.inf),
                                        ("y", -np.inf)])
def test_stencils_with_an_entry_that_is_not_finite(capi, orc, axes, value, prec):
    """Particle 171 is in its neighbours' lists: columns without its offset are
    fitted, all others are beyond the rank."""
    h, X = 1e-3, _lattice(7, 0.1)
    nbr, cnt = _lists(X, 1.9)
    P, F = X * h, _fields(X)
    for a in axes:
        P["xyz".index(a), 171] = value
    ctx = capi.Context(X.shape[1], cap=64)
    got = capi.lp_fit_derivatives(ctx, *[T(c) for c in P], _own(capi, ctx, nbr, cnt),
                                  [T(f) for f in F], [1.0, 1.0], h, precision=prec).cpu().numpy()
    ctx.close()
    ref, rank = orc.fit(*P, nbr, cnt, F, [1.0, 1.0], h)
    sees = np.array([171 in nbr[i, :cnt[i]] for i in range(len(cnt))])
    sees[171] = True
    assert sees.sum() > 20 and (rank[sees] < 9).all()
    assert np.array_equal(np.isnan(got[sees]), np.isnan(ref[sees]))
    u = np.array([h] * 3 + [h * h] * 6)
    err = np.abs((got - ref) * u)[sees]
    print(f"{axes} {value} prec {prec}: ranks {set(rank[sees])}, {np.nanmax(err):.1e}")
    assert np.nanmax(err) <= 1e-11 * np.abs(F).max()


@pytest.mark.parametrize("prec", [0, 2])
@pytest.mark.parametrize("nf", [1, 4, 6])
@pytest.mark.parametrize("side,r", [(5, 1.2), (10, 1.2), (11, 1.2), (17, 1.2)])
def test_refused_stencils_few_and_many(capi, orc, side, r, nf, prec):
    """Six entries at most, so every particle takes the QR fit: up to 1216 of
    them a warp each, above that a thread each."""
    h, X = 1e-3, _lattice(side, 0.05)
    P = X * h
    ctx = capi.Context(X.shape[1], cap=64)
    nb = capi.lp_build_neighbors(ctx, *[T(c) for c in P], r_const=r * h, mirror_mode=0)
    nbr, cnt = nb.export()
    F = np.stack([np.sin((0.4 + 0.1 * f) * X[0] + 0.3 * X[1] - 0.2 * X[2]) for f in range(nf)])
    got = capi.lp_fit_derivatives(ctx, *[T(c) for c in P], nb, [T(f) for f in F], [1.0] * nf, h,
                                  precision=prec).cpu().numpy()
    d = ctx.sync()
    ctx.close()
    assert d["flags"] == 0 and d["n_fallback"] == X.shape[1]
    ref, rank = orc.fit(*P, nbr, cnt, F, [1.0] * nf, h)
    u = np.array([h] * 3 + [h * h] * 6)
    # (a near tie of two norms may pivot otherwise; pivots that small amplify)
    err = (np.abs(got - ref) * u).max((1, 2))
    print(f"n {X.shape[1]} nf {nf}: {err.max():.1e}, ranks {set(rank)}")
    assert np.quantile(err, 0.999) <= 1e-11


@pytest.mark.parametrize("nf", [1, 3, 5])
@pytest.mark.parametrize("rows", [9, 20, 33, 48, 64])
def test_rank_deficient_stencils_of_any_size(capi, orc, rows, nf):
    """Entries in one plane: rank 5 (columns without z), one and two rows a lane."""
    g = np.random.default_rng(rows)
    h, n = 1e-3, 40
    X = np.concatenate([g.uniform(-1, 1, (2, n * (rows + 1))), np.zeros((1, n * (rows + 1)))])
    X[0] += np.repeat(10.0 * np.arange(n), rows + 1)
    P, m = X * h, X.shape[1]
    own = np.arange(n) * (rows + 1)
    nbr, cnt = np.zeros((m, 64), dtype=np.int32), np.zeros(m, dtype=np.int32)
    nbr[own, :rows] = own[:, None] + 1 + np.arange(rows)
    cnt[own] = rows
    F = np.stack([np.sin(0.4 * X[0] + (0.3 + 0.1 * f) * X[1]) for f in range(nf)])
    ctx = capi.Context(m, cap=64)
    got = capi.lp_fit_derivatives(ctx, *[T(c) for c in P], _own(capi, ctx, nbr, cnt),
                                  [T(f) for f in F], [1.0] * nf, h).cpu().numpy()
    ctx.close()
    ref, rank = orc.fit(*P, nbr, cnt, F, [1.0] * nf, h)
    assert (rank[own] == 5).all()
    err = np.abs((got - ref) * np.array([h] * 3 + [h * h] * 6))[own].max()
    print(f"rows {rows} nf {nf}: {err:.1e}")
    assert err <= 1e-11
