"""The FP64 Dslash, half of whose products are formed in integers: fields whose
sites differ widely, vanish, underflow or are not finite."""
import numpy as np
import pytest

import sw_inputs as si

pytestmark = pytest.mark.gpu
EX, LD = np.clongdouble, np.longdouble


@pytest.fixture(scope="module")
def sw():
    import paper_1801_07823_gb300 as m
    return m


def field(kind, L0, L1):
    n = L0 * L1
    v = si.gaussian_complex(3, n).reshape(L1, L0)
    y, x = np.indices((L1, L0))
    if kind == "even":
        v[(x + y) % 2 == 1] = 0
    elif kind == "point":
        v[...] = 0
        v[1, L0 - 1] = 2.5 - 1j
    elif kind == "wide":  # neighbours up to 400 orders of magnitude apart
        v *= 10.0 ** np.random.default_rng(1).uniform(-200, 200, (L1, L0))
    elif kind == "large":
        v *= 1e300
    elif kind == "small":
        v *= 1e-300
    elif kind == "subnormal":
        v *= 2.0 ** -1060
    return np.ascontiguousarray(v)


def hops(th, v):
    """(sum of the hops, largest component among the neighbours) in extended precision."""
    eta = 1 - 2 * (np.arange(th.shape[2]) % 2)
    w = [EX(0.5) * np.exp(EX(1j) * th[0].astype(LD)), EX(0.5) * eta * np.exp(EX(1j) * th[1].astype(LD))]
    out = np.zeros(v.shape, dtype=EX)
    top = np.zeros(v.shape, dtype=LD)
    mag = np.maximum(np.abs(v.real), np.abs(v.imag)).astype(LD)
    u = v.astype(EX)
    for mu, ax in ((0, 1), (1, 0)):
        out += w[mu] * np.roll(u, -1, ax) - np.roll(w[mu].conj() * u, 1, ax)
        top = np.maximum(top, np.maximum(np.roll(mag, -1, ax), np.roll(mag, 1, ax)))
    return out, top


@pytest.mark.parametrize("kind", ["gauss", "even", "point", "wide", "large", "small", "subnormal"])
@pytest.mark.parametrize("L0,L1", [(4, 4), (260, 8)])
def test_dslash_bound(sw, kind, L0, L1):
    """Per component: nine roundings of a partial sum (mass term, eight products with a link
    component of at most 1/2), which bound the integer form too; 2^-50 of the largest neighbour
    for the links (good to 2 units in the last place); a few units of the subnormal range."""
    th = np.random.default_rng(L0).uniform(-np.pi, np.pi, (2, L1, L0))
    v = field(kind, L0, L1)
    ctx = sw.sw_context_create(0)
    g = sw.sw_gauge_load(ctx, th)
    h, top = hops(th, v)
    for op, sg in ((sw.SW_OP_D, 1), (sw.SW_OP_DDAG, -1)):
        out = np.full_like(v, np.nan).reshape(-1)
        sw.sw_dslash(g, 0.07, op, sw.SW_PREC_FP64, v.reshape(-1), out)
        out = out.reshape(L1, L0)
        ref = LD(0.07) * v.astype(EX) + sg * h
        for part in ("real", "imag"):
            got, want, x = (getattr(a, part) for a in (out, ref, v))
            part_sum = LD(0.07) * np.abs(x) + 4 * top
            tol = 9 * LD(2) ** -53 * part_sum + LD(2) ** -50 * top + LD(2) ** -1072
            assert np.all(np.abs(got - want) <= tol)
    g.free()
    ctx.free()


@pytest.mark.parametrize("bad", [np.nan, np.inf, complex(0.0, -np.inf)])
def test_not_finite_stays_local(sw, bad):
    L0, L1, m = 16, 12, 0.05
    th = np.random.default_rng(2).uniform(-np.pi, np.pi, (2, L1, L0))
    v = field("gauss", L0, L1)
    w = v.copy()
    w[5, 6] = bad
    ctx = sw.sw_context_create(0)
    g = sw.sw_gauge_load(ctx, th)
    a, b = np.zeros(v.size, complex), np.zeros(v.size, complex)
    sw.sw_dslash(g, m, sw.SW_OP_D, sw.SW_PREC_FP64, v.reshape(-1), a)
    sw.sw_dslash(g, m, sw.SW_OP_D, sw.SW_PREC_FP64, w.reshape(-1), b)
    off = ~np.isfinite(b.reshape(L1, L0))
    assert off[5, 6] and off[5, 5] and off[5, 7] and off[4, 6] and off[6, 6] and off.sum() == 5
    assert np.array_equal(a[~off.reshape(-1)], b[~off.reshape(-1)])
    g.free()
    ctx.free()
