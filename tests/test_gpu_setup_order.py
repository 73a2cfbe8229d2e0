"""Setup on a field with a nearly singular KD block (a block plaquette close to pi), where the
relaxation of the null vectors multiplies every rounding difference about a thousandfold per
step: one configuration has one hierarchy."""
import os

import numpy as np
import pytest

from tests.gpu_helpers import assemble_stencil, relerr

pytestmark = pytest.mark.gpu
L0, L1, NVEC, BLOCKS = 32, 48, [4, 6], [(4, 4), (2, 2)]
GOLDEN = os.path.join(os.path.dirname(__file__), "golden", "setup_order.txt")


class Dyadic:
    """Multiples of 2^-20 in [-1, 1) from a 64-bit linear congruential generator (Knuth's
    constants): the same numbers on every machine."""

    def __init__(self, seed):
        self.s = seed

    def draw(self, *shape):
        out = np.empty(int(np.prod(shape)))
        for k in range(out.size):
            self.s = (self.s * 6364136223846793005 + 1442695040888963407) % 2**64
            out[k] = ((self.s >> 40) & 0x1fffff) / 2.0**20 - 1.0
        return out.reshape(shape)

    def complex(self, *shape):
        z = self.draw(*shape, 2)
        return z[..., 0] + 1j * z[..., 1]


@pytest.fixture(scope="module")
def hier():
    import paper_1801_07823_gb300 as sw
    d = Dyadic(11)
    th = d.draw(2, L1, L0)
    x, y = 4, 2  # the plaquette of KD block (2, 1)
    th[0, y, x] += np.pi - 0.02 - (th[0, y, x] + th[1, y, x + 1] - th[0, y + 1, x] - th[1, y, x])
    sizes = [L0 * L1, (L0 // 8) * (L1 // 8) * 2 * NVEC[0]]
    psi0 = [d.complex(nv, n) for nv, n in zip(NVEC, sizes)]
    p = sw.sw_mg_params_default()
    p.setup_maxiter = 8
    ctx = sw.sw_context_create(0)
    g = sw.sw_gauge_load(ctx, th)
    h = sw.sw_mg_setup(g, 0.01, 3, BLOCKS, NVEC, params=p, psi0=psi0)
    fields = []
    for level in (1, 2):
        e0, e1, nc = sw.sw_mg_level_info(h, level + 1)
        v = d.complex(sizes[level - 1])
        r = np.zeros(e0 * e1 * nc, dtype=complex)
        sw.sw_mg_transfer(h, level, 0, v, r)
        w = d.complex(r.size)
        a = np.zeros_like(r)
        sw.sw_mg_apply_level(h, level + 1, sw.SW_PREC_FP64, 0, w, a)
        fields.append((v, r, w, a))
    yield sw, h, fields
    h.free()
    g.free()
    ctx.free()


def outputs(fields):
    return np.concatenate([np.concatenate([r, a]) for _, r, _, a in fields])


def test_values(hier):
    """Restrictions and stencils of both levels against recorded values, which were computed when
    the library had plain FP64 products and tree sums only.  An application itself agrees to a few
    units of 1e-16; a relaxation with sums of another order moved these values by 1.3e-7."""
    ref = np.loadtxt(GOLDEN, dtype=float)
    got = outputs(hier[2])
    assert np.linalg.norm(got - (ref[:, 0] + 1j * ref[:, 1])) <= 1e-9 * np.linalg.norm(ref)


def test_own_operators(hier):
    """P^dag P = 1, and restriction and stencil against the exported P and Y (1e-13: rounding of
    sums of at most 160 terms)."""
    sw, h, fields = hier
    for level in (1, 2):
        v, r, w, a = fields[level - 1]
        nv = NVEC[level - 1]
        P = sw.sw_mg_export_P(h, level, nv)
        agg, chir = sw.sw_mg_level_maps(h, level)
        e0, e1, nc = sw.sw_mg_level_info(h, level + 1)
        D = np.zeros((P.shape[0], r.size), dtype=complex)
        col = agg * nc + np.where(chir > 0, 0, nv)
        D[np.arange(P.shape[0])[:, None], col[:, None] + np.arange(nv)] = P
        assert np.max(np.abs(D.conj().T @ D - np.eye(r.size))) <= 1e-12
        u = v.copy()
        if level == 1:  # the even KD blocks take part
            s = np.arange(v.size)
            u[((s % L0 // 2 + s // L0 // 2) & 1) == 1] = 0
        assert relerr(r, D.conj().T @ u) <= 1e-13
        assert relerr(a, assemble_stencil(sw.sw_mg_export_Y(h, level + 1), e0, e1) @ w) <= 1e-13
