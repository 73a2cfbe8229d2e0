"""The coarsest solver in one cluster (small coarsest levels, all SMs) against
its form with a grid barrier, which a context that holds half of the SMs runs."""
import numpy as np
import pytest

import sw_inputs as si

pytestmark = pytest.mark.gpu


# eight-row items of the coarsest level: 1 (one CTA), 27 (uneven shares), 96 (the most), 100 (none)
@pytest.mark.parametrize("L0,L1,nvec", [(16, 16, [3, 2]), (48, 48, [8, 12]), (64, 96, [8, 16]),
                                        (80, 80, [8, 16])])
def test_cluster_form(L0, L1, nvec):
    """The products are the same integers and only the norms are added in another order, so the
    solves agree to the solve tolerance over the smallest eigenvalue."""
    import paper_1801_07823_gb300 as sw
    m = 0.1
    th = si.heatbath_u1(L0, L1, 6.0, 20, seed=L0 + L1, device="cuda")
    b = si.gaussian_complex(7, L0 * L1)
    res = []
    for den in (1, 2):
        ctx = sw.sw_context_create(0)
        sw.sw_context_set_sm_share(ctx, 1, den)
        g = sw.sw_gauge_load(ctx, th)
        h = sw.sw_mg_setup(g, m, 3, [(4, 4), (2, 2)], nvec, seed=2)
        x = np.zeros_like(b)
        s = sw.sw_mg_solve(h, b, x, 1e-10)
        assert s["converged"] and s["true_resid"] <= 1e-10
        zero = np.ones_like(b)
        assert sw.sw_mg_solve(h, np.zeros_like(b), zero, 1e-10)["converged"] and not zero.any()
        res.append((s["coarsest_iters"] / s["coarsest_solves"], x))
        h.free()
        g.free()
        ctx.free()
    (i1, x1), (i2, x2) = res
    assert abs(i1 - i2) <= max(1.0, 0.05 * i1)
    # |x1 - x2| <= 2 tol |b| / m, the smallest singular value of D being at least m
    assert np.linalg.norm(x1 - x2) <= 2e-10 / m * np.linalg.norm(b)
