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
