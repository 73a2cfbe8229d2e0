"""FP64 stencil products by digit arithmetic on the tensor cores, against long
double on the library's own exported stencil, and the coarsest solver on them."""
import numpy as np
import pytest

import sw_inputs as si

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sw():
    import paper_1801_07823_gb300 as m
    return m


def neighbours(e0, e1):
    X = np.arange(e0 * e1)
    X0, X1 = X % e0, X // e0
    return [X, (X0 + 1) % e0 + e0 * X1, (X0 - 1) % e0 + e0 * X1, X0 + e0 * ((X1 + 1) % e1),
            X0 + e0 * ((X1 - 1) % e1)]


def blocks(Y, e0, e1, dagger):
    """[sites, 5, nc, nc]: block d multiplies the vector of neighbour d."""
    if not dagger:
        return Y
    nb = neighbours(e0, e1)
    return np.stack([Y[nb[d], o].conj().transpose(0, 2, 1) for d, o in enumerate((0, 2, 1, 4, 3))],
                    axis=1)


def reference(B, v, e0, e1):
    """(product, bound on the digit product's error), both [sites, nc].

    A product is rounded once to FP64 (2^-53 of it).  Before that every term
    loses at most 2^-58 of the largest entry times the largest vector component
    it meets: digit products of level 8 and above (7 of at most 2^-62 in that
    unit, and less beyond) and the roundings of the entry (2^-64) and of the
    vector (2^-62); scales are powers of two, a factor of two on either side.
    Largest entry: of the whole level for the adjoint, whose rows are scaled as
    columns.  10 nc real terms in a component."""
    ns, _, nc, _ = B.shape
    w = v.reshape(ns, nc)
    nb = neighbours(e0, e1)
    out = np.zeros((ns, nc), np.clongdouble)
    for d in range(5):
        out += np.einsum("xij,xj->xi", B[:, d].astype(np.clongdouble), w[nb[d]].astype(np.clongdouble))
    vmax = np.max([np.abs(w[n]).max(axis=1) for n in nb], axis=0)
    amax = np.abs(B).max()
    return out, 2.0 ** -53 * np.abs(out) + 10 * nc * 2.0 ** -56 * amax * vmax[:, None]


# extents 1, 2, 3 and more; row groups and k-steps with and without padding; one to four
# rows groups per k-step; sites that fill the GPU and sites whose rows are split over CTAs
CASES = [(16, 16, (4, 4), 1), (8, 8, (4, 4), 5), (24, 16, (4, 4), 3), (32, 32, (4, 4), 8),
         (64, 32, (4, 4), 12), (48, 48, (2, 2), 20), (16, 32, (4, 4), 32), (16, 16, (4, 4), 33),
         (8, 16, (4, 4), 64), (128, 128, (2, 2), 4)]


@pytest.mark.parametrize("L0,L1,block,nv", CASES)
def test_level_product_against_long_double(sw, L0, L1, block, nv):
    th = si.heatbath_u1(L0, L1, 6.0, 5, seed=L0 + nv, device="cuda")
    ctx = sw.sw_context_create(0)
    g = sw.sw_gauge_load(ctx, th)
    p = sw.sw_mg_params_default()
    p.setup_maxiter = 4
    h = sw.sw_mg_setup(g, 0.05, 2, [block], [nv], params=p, seed=3)
    e0, e1, nc = sw.sw_mg_level_info(h, 2)
    Y = sw.sw_mg_export_Y(h, 2)
    n = e0 * e1 * nc
    gauss = si.gaussian_complex(11, n)
    wide = gauss * 2.0 ** (40 * np.sin(np.arange(n)))  # neighbours of very different size
    point = np.zeros(n, complex)
    point[n // 2] = 1 - 2j
    for dagger in (0, 1):
        B = blocks(Y, e0, e1, dagger)
        for v in (gauss, wide, point, gauss * 1e-290, gauss * 1e290, np.zeros(n, complex)):
            out = np.full(n, 7.0 + 0j)
            sw.sw_mg_apply_level(h, 2, sw.SW_PREC_FP64, dagger, np.ascontiguousarray(v), out)
            ref, bound = reference(B, v, e0, e1)
            err = np.abs(out.reshape(ref.shape) - ref)
            assert np.all(err <= np.maximum(bound, 5e-324)), (dagger, float((err / bound).max()))
        for bad in (np.inf, np.nan):  # only the sites around it, and there nothing finite is made up
            v = gauss.copy()
            v[n // 3] = bad
            out = np.empty(n, complex)
            sw.sw_mg_apply_level(h, 2, sw.SW_PREC_FP64, dagger, v, out)
            hit = np.any([np.asarray(nb) == (n // 3) // nc for nb in neighbours(e0, e1)], axis=0)
            o = out.reshape(-1, nc)
            assert np.all(np.isfinite(o[~hit])) and not np.any(np.isfinite(o[hit].real))
    h.free()
    g.free()
    ctx.free()


def test_coarsest_solver_on_few_sms(sw):
    """With all SMs a CTA's rows fit one chunk of shared memory; on one or two
    of the SMs the kernel walks several chunks per phase.  The products are the
    same integers, only the norms are added in another order, so the solves
    agree to the solve tolerance."""
    L, nvec = 64, [16, 32]
    th = si.heatbath_u1(L, L, 6.0, 20, seed=5, device="cuda")
    b = si.gaussian_complex(7, L * L)
    res = {}
    for den in (1, 76, 152):
        ctx = sw.sw_context_create(0)
        sw.sw_context_set_sm_share(ctx, 1, den)
        g = sw.sw_gauge_load(ctx, th)
        h = sw.sw_mg_setup(g, 0.1, 3, [(4, 4), (2, 2)], nvec, seed=2)
        x = np.zeros_like(b)
        res[den] = (sw.sw_mg_solve(h, b, x, 1e-10), x)
        h.free()
        g.free()
        ctx.free()
    s1, x1 = res[1]
    for den in (76, 152):
        s, x = res[den]
        assert s["true_resid"] <= 1e-10
        assert abs(s["coarsest_iters"] - s1["coarsest_iters"]) <= 0.05 * s1["coarsest_iters"]
        assert np.linalg.norm(x - x1) <= 1e-8 * np.linalg.norm(x1)
