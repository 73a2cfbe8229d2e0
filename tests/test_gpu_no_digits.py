"""Hierarchies without digit entries (too large for them, or no memory left): the FP64-pipe
stencils and the queued coarsest solver do their work."""
import numpy as np
import pytest

import sw_inputs as si
from tests.gpu_helpers import assemble_stencil, relerr

pytestmark = pytest.mark.gpu


# compiled block sizes (16, 24) and others (6, 10), and a limit that only the larger level exceeds
@pytest.mark.parametrize("nvec,limit", [([8, 12], 0), ([3, 5], 0), ([8, 12], 10000)])
@pytest.mark.parametrize("mixed", [False, True])
def test_without_digit_entries(monkeypatch, nvec, limit, mixed):
    """Stencils against the exported Y (1e-13: rounding of sums of at most 120 terms); solves with
    and without to the tolerance and, since only roundings differ, in the same outer iterations to
    one."""
    import paper_1801_07823_gb300 as sw
    from oracle import operators
    L0, L1, m = 48, 32, 0.05
    th = si.heatbath_u1(L0, L1, 6.0, 20, seed=4, device="cuda")
    b = si.gaussian_complex(9, L0 * L1)
    D = operators.dirac(th, m)
    p = sw.sw_mg_params_default()
    if mixed:
        p.precision = sw.SW_MG_MIXED
    its = []
    for lim in (None, limit):
        if lim is not None:
            monkeypatch.setenv("SW_DIGIT_ENTRIES", str(lim))
        ctx = sw.sw_context_create(0)
        g = sw.sw_gauge_load(ctx, th)
        h = sw.sw_mg_setup(g, m, 3, [(4, 4), (2, 2)], nvec, params=p, seed=2)
        for level in (2, 3):
            e0, e1, nc = sw.sw_mg_level_info(h, level)
            A = assemble_stencil(sw.sw_mg_export_Y(h, level), e0, e1)
            v = si.gaussian_complex(level, e0 * e1 * nc)
            out = np.zeros_like(v)
            for dagger in (0, 1):
                sw.sw_mg_apply_level(h, level, sw.SW_PREC_FP64, dagger, v, out)
                assert relerr(out, (A.conj().T if dagger else A) @ v) <= 1e-13
        x = np.zeros_like(b)
        st = sw.sw_mg_solve(h, b, x, 1e-10)
        assert st["converged"] and np.linalg.norm(b - D @ x) <= 1e-10 * np.linalg.norm(b)
        its.append(st["outer_iters"])
        h.free()
        g.free()
        ctx.free()
    assert abs(its[0] - its[1]) <= 1
