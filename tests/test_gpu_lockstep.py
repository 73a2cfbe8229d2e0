"""Lockstep Krylov loops: sizes at which their sums take another path, smoother
counts, members that stop early, and setups whose null vectors form several groups."""
import numpy as np
import pytest

import sw_inputs as si
from oracle import operators

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sw():
    import paper_1801_07823_gb300 as m
    return m


# 16 x 16: a sum in one CTA (two elements per thread on the coarse levels); 1024 x 640:
# more elements than threads in a capped grid
@pytest.mark.parametrize("L0,L1,smooth,precision", [
    (16, 16, 0, "FP64"), (16, 16, 1, "FP64"), (16, 16, 3, "MIXED"), (48, 16, 0, "MIXED"),
    (48, 16, 1, "MIXED"), (1024, 640, 2, "MIXED")])
def test_solve_residuals(sw, L0, L1, smooth, precision):
    m, tol = 0.1, 1e-9
    th = si.heatbath_u1(L0, L1, 6.0, 5, seed=L0, device="cuda")
    ctx = sw.sw_context_create(0)
    g = sw.sw_gauge_load(ctx, th)
    p = sw.sw_mg_params_default()
    p.precision = getattr(sw, "SW_MG_" + precision)
    p.smoother_iters = smooth
    p.setup_maxiter = 20
    full = smooth > 0  # a coarse correction alone cannot reach every error: one step of it
    if not full:
        p.outer_maxiter = 1
    h = sw.sw_mg_setup(g, m, 2, [(4, 4)], [8], params=p, seed=3)
    D = operators.dirac(th, m)
    B = np.stack([si.gaussian_complex(7 + k, L0 * L1) for k in range(5)])
    B[2] = 0.0
    B[3] *= 1e-12
    many = precision == "MIXED" and L0 < 1024
    for k in (0, 2, 3):
        x = np.zeros_like(B[k])
        st = sw.sw_mg_solve(h, B[k], x, tol, allow_noconv=not full)
        r = np.linalg.norm(B[k] - D @ x) / max(np.linalg.norm(B[k]), 1e-300)
        # rounding of the two residuals: some 1e-15 |D| |x| / |b|, |D|/m = 30
        assert abs(r - st["true_resid"]) <= 1e-12, (k, r, st)
        assert not full or (st["converged"] and r <= tol + 1e-12), (k, r, st)
    if many:
        X = np.zeros_like(B)
        sts = sw.sw_mg_solve_batch(h, B, X, tol, allow_noconv=not full)
        for k in range(5):
            r = np.linalg.norm(B[k] - D @ X[k]) / max(np.linalg.norm(B[k]), 1e-300)
            assert abs(r - sts[k]["true_resid"]) <= 1e-12
            assert not full or (sts[k]["converged"] and r <= tol + 1e-12)
        X0 = np.zeros_like(B[:2])
        sts = sw.sw_mg_solve_batch(h, np.zeros_like(X0), X0, tol)  # nothing to do
        assert all(s["converged"] for s in sts) and not X0.any()
    h.free()
    g.free()
    ctx.free()


def test_setup_groups(sw):
    """1024^2: two null vectors to a group.  P P^dag does not depend on their order."""
    L, nv = 1024, 3
    th = si.heatbath_u1(L, L, 6.0, 2, seed=1, device="cuda")
    ctx = sw.sw_context_create(0)
    g = sw.sw_gauge_load(ctx, th)
    psi = np.stack([si.gaussian_complex(20 + i, L * L) for i in range(nv)])
    v = si.gaussian_complex(11, L * L)
    got = []
    for order in ([0, 1, 2], [2, 0, 1]):
        p = sw.sw_mg_params_default()
        p.setup_maxiter = 6
        p.setup_passes = 2
        h = sw.sw_mg_setup(g, 0.1, 2, [(8, 8)], [nv], params=p, psi0=[psi[order]])
        nc = (L // 16) ** 2 * 2 * nv
        c, e = np.zeros(nc, complex), np.zeros_like(v)
        sw.sw_mg_transfer(h, 1, 0, v, c)
        sw.sw_mg_transfer(h, 1, 1, c, e)
        got.append(e)
        h.free()
    # orthonormalisation of 3 well-conditioned vectors of 64 elements: some 100 roundings
    assert np.linalg.norm(got[1] - got[0]) <= 1e-12 * np.linalg.norm(got[0])
    assert np.linalg.norm(got[0]) > 0
    g.free()
    ctx.free()
