"""Range of the digit products: rows of very different entries on vectors of very different
elements.  The bound is per row and neighbourhood, as the header states it."""
import numpy as np
import pytest

import sw_inputs as si
from tests.test_gpu_digits import blocks, neighbours

pytestmark = pytest.mark.gpu


def reference(Y, v, e0, e1, dagger):
    """(product, bound), both [sites, nc]: 2^-53 of the component, and 2^-58 of the largest product
    of the scales for each of its 10 nc real terms.  Forward: a row's largest component and the
    largest vector component of the five sites, either rounded up to a power of two.  Adjoint: the
    rows' scales multiply the vector's elements."""
    ns, _, nc, _ = Y.shape
    B, w, nb = blocks(Y, e0, e1, dagger), v.reshape(ns, nc), neighbours(e0, e1)
    out = np.zeros((ns, nc), np.clongdouble)
    for d in range(5):
        out += np.einsum("xij,xj->xi", B[:, d].astype(np.clongdouble), w[nb[d]].astype(np.clongdouble))
    comp = lambda z: np.maximum(np.abs(z.real), np.abs(z.imag))
    up = lambda z: 2.0 ** np.ceil(np.log2(np.maximum(z, 1e-300)) + 1e-9)
    row = up(comp(Y).max(axis=(1, 3)))  # [sites, nc], of the forward operator
    if dagger:
        scale = np.max([(up(comp(w)) * row)[n].max(axis=1) for n in nb], axis=0)[:, None]
    else:
        scale = row * np.max([up(comp(w))[n].max(axis=1) for n in nb], axis=0)[:, None]
    return out, 2.0 ** -53 * np.abs(out) + 10 * nc * 2.0 ** -58 * scale


@pytest.mark.parametrize("mass", [0.5, 1e-4])
def test_graded_rows_and_vectors(mass):
    """A block plaquette close to pi at small mass: rows of A between 1 and 1/m.  Vectors graded
    over 2^-20 .. 2^20 within a site, along rows, and from site to site."""
    import paper_1801_07823_gb300 as sw
    L0, L1, nv = 48, 32, 12
    th = si.heatbath_u1(L0, L1, 6.0, 10, seed=2, device="cuda")
    th = th.cpu().numpy() if hasattr(th, "cpu") else np.array(th)
    x, y = 8, 4
    th[0, y, x] += np.pi - 1e-4 - (th[0, y, x] + th[1, y, x + 1] - th[0, y + 1, x] - th[1, y, x])
    ctx = sw.sw_context_create(0)
    g = sw.sw_gauge_load(ctx, th)
    p = sw.sw_mg_params_default()
    p.setup_maxiter = 2
    h = sw.sw_mg_setup(g, mass, 2, [(4, 4)], [nv], params=p, seed=3)
    e0, e1, nc = sw.sw_mg_level_info(h, 2)
    Y, n = sw.sw_mg_export_Y(h, 2), e0 * e1 * nc
    gauss, k, rows = si.gaussian_complex(5, n), np.arange(n), np.abs(Y).max(axis=(1, 3)).reshape(-1)
    for dagger in (0, 1):
        for v in (gauss * 2.0 ** (20 * np.sin(k)), gauss / rows, gauss * 2.0 ** (k // nc % 41 - 20)):
            out = np.empty(n, complex)
            sw.sw_mg_apply_level(h, 2, sw.SW_PREC_FP64, dagger, np.ascontiguousarray(v), out)
            ref, bound = reference(Y, v, e0, e1, dagger)
            assert np.all(np.abs(out.reshape(ref.shape) - ref) <= bound)
    h.free()
    g.free()
    ctx.free()
