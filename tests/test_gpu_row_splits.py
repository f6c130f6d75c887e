"""The fixed-point rows of LP_FP64, the ghost lanes and the truncated stencils
at the edges of their launch shapes.

Whole-number sums do not depend on who adds them: the per-phase kernels (four or
two lanes, three or four blocks per SM by particle count) give the bits of the
persistent launch, which takes one thread per particle throughout.
"""
import numpy as np
import pytest

from paper_2206_14061_gb300 import workloads as W

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


def T(a):
    return torch.tensor(np.ascontiguousarray(a, dtype=np.float64), device="cuda:0")


@pytest.mark.parametrize("ghosts", [0, 1])
@pytest.mark.parametrize("n", [1, 31, 33, 129, 14592, 14593, 29184, 29185, 58368, 58369])
def test_step_bits_do_not_depend_on_the_row_split(capi, n, ghosts):
    wl = W.cube(next(s for s in (6, 25, 39) if s ** 3 >= n))
    pd = W.param_dict(wl)
    mui = {k: pd[k] for k in ("mu_s", "mu_2", "I0", "d", "rho_s")}
    eos = {k: pd[k] for k in ("phi_c", "phi_min", "phi_max", "alpha", "beta")}
    runs = []
    for mode in (0, 2):
        prm = {k: pd[k] for k in ("h", "radius", "gx", "gy", "gz", "floor_z", "mirror_mode")}
        prm.update(precision=0, rebuild_every=1, launch_mode=mode, skin=0.0, free_surface=ghosts)
        ctx = capi.Context(n, cap=64)
        st = {k: T(wl.state[k][:n]) for k in capi.FIELDS}
        capi.lp_step(ctx, st, mui, eos, prm, pd["dt"], 2)
        d = ctx.sync()
        runs.append((st, d["n_ghosts"], d["n_fallback"]))
        ctx.close()
    assert runs[0][1:] == runs[1][1:]
    assert n < 1000 or not ghosts or runs[0][1] > 0
    for k in capi.FIELDS:
        assert torch.equal(runs[0][0][k], runs[1][0][k]), k


@pytest.mark.parametrize("nf", [1, 2, 3, 4, 5, 7])
@pytest.mark.parametrize("h,offset", [(1e-3, 0.0), (1e-3, 1e3), (7e5, 0.0)])
def test_fit_fp64_recovers_quadratics_of_any_scale(capi, nf, h, offset):
    """Quadratic fields of very different magnitudes, some outside the fixed
    point range (the plain FP64 rows then take the particle), and a field with
    one infinite value. Tolerance, in lattice units: differences up to 30 over
    at most 48 rows, 2^-53 each, amplified by at most 2^14 (smallest pivot
    2^-7, squared; smaller ones go to the QR fit), and the positions' rounding
    at the offset."""
    rng = np.random.default_rng(5)
    i = np.arange(9)
    X = np.stack(np.meshgrid(i, i, i, indexing="ij")).reshape(3, -1) - 4.0
    X = X + rng.uniform(-0.15, 0.15, X.shape)
    P = [T((c + offset) * h) for c in X]
    q = [p / h - offset for p in P]  # as the stored positions have them
    base = q[0] * q[1] + 0.5 * q[2] ** 2 - q[0] + 0.25
    scale = [1.0, 1e-200, 1e30, 0.0, 1e6, 1e200, 1.0]
    fields = [base * s for s in scale]
    fields[6] = torch.where(torch.arange(base.numel(), device=base.device) == 5, torch.inf, base)
    ctx = capi.Context(base.numel(), cap=64)
    nb = capi.lp_build_neighbors(ctx, *P, r_const=2.6 * h, mirror_mode=0, cap=48, keep_nearest=1)
    nbr, cnt = nb.export()
    out = capi.lp_fit_derivatives(ctx, *P, nb, fields[:nf], [1.0] * nf, h)
    ref = torch.zeros(base.numel(), 9, dtype=torch.float64, device=base.device)
    ref[:, 0], ref[:, 1], ref[:, 2] = q[1] - 1.0, q[0], q[2]
    ref[:, 5], ref[:, 6] = 1.0, 1.0
    unit = torch.tensor([h] * 3 + [h * h] * 6, dtype=torch.float64, device=base.device)
    tol = 30 * 48 * 2.0 ** -53 * 2 ** 14 * (1.0 + 8 * offset)
    for f in range(nf):
        got, keep = out[:, f] * unit, torch.ones(base.numel(), dtype=torch.bool, device=base.device)
        if f == 6:
            sees = np.zeros(base.numel(), bool)
            sees[5] = True
            for s in range(base.numel()):
                sees[s] |= 5 in nbr[s, :cnt[s]]
            keep = T(sees) == 0.0
            assert not bool(torch.isfinite(got[~keep]).all(1).any())
        s = scale[f]
        assert float((got[keep] - s * ref[keep]).abs().max()) <= tol * max(s, 0.0), (f, s)
    ctx.close()


@pytest.mark.parametrize("keep", [1, 2])
@pytest.mark.parametrize("cap", [1, 16, 32, 33, 48, 64])
@pytest.mark.parametrize("jitter,stretch", [(0.0, 1.0), (0.2, 1.0), (0.2, 9.0)])
def test_truncated_stencils_match_the_oracle(capi, orc, keep, cap, jitter, stretch):
    """Distance ties (a lattice), full and partial stencils, and a sparse
    domain with many empty cells; entries in the oracle's order."""
    rng = np.random.default_rng(3)
    i = np.arange(11)
    X = np.stack(np.meshgrid(i, i, i, indexing="ij")).reshape(3, -1) + 0.5
    p = (X * stretch + rng.uniform(-jitter, jitter, X.shape)) * 1e-3
    rad = rng.uniform(1.8e-3, 2.6e-3, p.shape[1])
    ctx = capi.Context(p.shape[1], cap=64)
    nb = capi.lp_build_neighbors(ctx, T(p[0]), T(p[1]), T(p[2]), radius=T(rad), mirror_mode=1,
                                 cap=cap, keep_nearest=keep)
    got, cnt = nb.export()
    ref, rcnt, _ = orc.neighbors(*p, radius=rad, mirror_mode=1, cap=cap, keep_nearest=keep,
                                 brute=False)
    rcnt = np.minimum(rcnt, cap)
    mask = np.arange(cap) < rcnt[:, None]
    assert np.array_equal(cnt, rcnt)
    assert np.array_equal(np.where(mask, got, 0), np.where(mask, ref, 0))
    ctx.close()
