"""A negative coarsest_tol is a tolerance that no residual meets: every coarsest solve runs
coarsest_maxiter iterations."""
import numpy as np
import pytest

import sw_inputs as si

pytestmark = pytest.mark.gpu


# the coarsest kernel in a cluster and in a grid, the queued loop, the batched kernel
@pytest.mark.parametrize("form", ["cluster", "grid", "loop", "batch64", "batch32"])
def test_fixed_number_of_coarsest_iterations(monkeypatch, form):
    import paper_1801_07823_gb300 as sw
    L, m, cap = 64, 0.05, 5
    th = si.heatbath_u1(L, L, 6.0, 20, seed=6, device="cuda")
    b = si.gaussian_complex(11, L * L)
    ctx = sw.sw_context_create(0)
    if form == "grid":
        sw.sw_context_set_sm_share(ctx, 1, 2)
    if form == "loop":
        monkeypatch.setenv("SW_CGNE_LOOP", "1")
    p = sw.sw_mg_params_default()
    p.coarsest_tol, p.coarsest_maxiter = -2.0, cap
    if form.startswith("batch"):
        p.precision = sw.SW_MG_MIXED
        p.batch_iterates = sw.SW_PREC_FP32 if form == "batch32" else sw.SW_PREC_FP64
    g = sw.sw_gauge_load(ctx, th)
    h = sw.sw_mg_setup(g, m, 3, [(4, 4), (2, 2)], [8, 12], params=p, seed=2)
    if form.startswith("batch"):
        B = np.stack([b, 2j * b[::-1]])
        stats = sw.sw_mg_solve_batch(h, B, np.zeros_like(B), 1e-8)
    else:
        stats = [sw.sw_mg_solve(h, b, np.zeros_like(b), 1e-8)]
    for st in stats:
        assert st["converged"] and st["coarsest_solves"] > 0
        assert st["coarsest_iters"] == cap * st["coarsest_solves"]
    h.free()
    g.free()
    ctx.free()
