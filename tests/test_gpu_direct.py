"""Calls that work on the caller's device fields without staging, against the
same calls on host fields, and where they must stage after all."""
import numpy as np
import pytest

import sw_inputs as si
from oracle import operators

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sw():
    import paper_1801_07823_gb300 as m
    return m


@pytest.fixture(scope="module")
def torch():
    import torch as t
    return t


def device_run(torch, f, v, nout, how):
    """f(in, out) on device fields: two buffers, one buffer, or overlapping pieces of one."""
    n = len(v)
    x = torch.from_numpy(v).cuda()
    if how == "apart":
        out = torch.empty(nout, dtype=torch.complex128, device="cuda")
        f(x, out)
    elif how == "same":
        out = x if nout <= n else torch.cat([x, torch.zeros(nout - n, dtype=x.dtype, device="cuda")])
        f(out[:n], out[:nout])
        out = out[:nout]
    else:
        buf = torch.zeros(n + nout + 8, dtype=torch.complex128, device="cuda")
        buf[4:4 + n] = x
        out = buf[7:7 + nout]
        f(buf[4:4 + n], out)
    return out.cpu().numpy()


@pytest.mark.parametrize("L0,L1", [(4, 4), (12, 8), (20, 36), (520, 12)])
@pytest.mark.parametrize("op", ["SW_OP_A", "SW_OP_ADAG", "SW_OP_S"])
def test_kd_operators_in_place(sw, torch, L0, L1, op):
    th = si.heatbath_u1(L0, L1, 6.0, 5, seed=L0, device="cuda")
    ctx = sw.sw_context_create(0)
    g = sw.sw_gauge_load(ctx, th)
    n = L0 * L1
    v = si.gaussian_complex(5, n)
    ref = np.full(n, 3.0 + 0j)
    sw.sw_dslash(g, 0.05, getattr(sw, op), sw.SW_PREC_FP64, v, ref)
    for how in ("apart", "same", "overlap"):
        got = device_run(torch, lambda a, b: sw.sw_dslash(g, 0.05, getattr(sw, op),
                                                          sw.SW_PREC_FP64, a, b), v, n, how)
        assert np.array_equal(got, ref), how
    if op == "SW_OP_S":
        out = torch.from_numpy(v).cuda()
        sw.sw_dslash_schur_noalloc(g, 0.05, out, out)
        assert np.array_equal(out.cpu().numpy(), ref)
    g.free()
    ctx.free()


# a group of one KD block, several groups, columns that do not fill the threads, all blocks (D)
@pytest.mark.parametrize("L0,L1,block,nvec,fine_d", [
    (16, 16, (2, 2), [3, 4], 0), (32, 16, (4, 4), [24, 5], 0), (32, 32, (4, 2), [64, 2], 0),
    (16, 32, (2, 4), [33, 2], 0), (32, 32, (4, 4), [8, 4], 1)])
def test_level_calls_on_device_fields(sw, torch, L0, L1, block, nvec, fine_d):
    th = si.heatbath_u1(L0, L1, 6.0, 5, seed=L1, device="cuda")
    ctx = sw.sw_context_create(0)
    g = sw.sw_gauge_load(ctx, th)
    p = sw.sw_mg_params_default()
    p.setup_maxiter = 3
    p.fine_operator = fine_d
    h = sw.sw_mg_setup(g, 0.05, 3, [block, (2, 2)], nvec, params=p, seed=3)
    n = [a * b * c for a, b, c in (sw.sw_mg_level_info(h, k) for k in (1, 2, 3))]
    P = sw.sw_mg_export_P(h, 1, nvec[0])
    agg, chir = sw.sw_mg_level_maps(h, 1)
    maps = sw.sw_debug_maps(g, *block)
    used = np.ones(n[0], bool) if fine_d else maps["kd_parity"] == 0
    col = agg * 2 * nvec[0] + np.where(chir > 0, 0, nvec[0])
    calls = [(lambda a, b, k=k, d=d: sw.sw_mg_transfer(h, k, d, a, b),
              n[k - 1] if d == 0 else n[k], n[k] if d == 0 else n[k - 1], (k, d))
             for k in (1, 2) for d in (0, 1)]
    calls += [(lambda a, b, k=k, d=d: sw.sw_mg_apply_level(h, k, sw.SW_PREC_FP64, d, a, b),
               n[k - 1], n[k - 1], ("apply", k, d)) for k, d in ((1, 0), (2, 0), (2, 1), (3, 1))]
    for f, nin, nout, what in calls:
        v = si.gaussian_complex(9, nin)
        ref = np.full(nout, 3.0 + 0j)
        f(v, ref)
        for how in ("apart", "same", "overlap"):
            assert np.array_equal(device_run(torch, f, v, nout, how), ref), (what, how)
        # at most 2 blocks * 2 sites * 16 terms a column, or nv terms a site: 64 roundings
        if what == (1, 0):
            full = np.zeros(nout, complex)
            for i in range(nvec[0]):
                np.add.at(full, (col + i)[used], (P[:, i].conj() * v)[used])
            assert np.abs(ref - full).max() <= 64 * 2.0 ** -52 * np.abs(v).max() * np.abs(P).max() * 8
        if what == (1, 1):
            e = sum(P[:, i] * v[col + i] for i in range(nvec[0])) * used
            assert np.abs(ref - e).max() <= 64 * 2.0 ** -52 * np.abs(v).max() * np.abs(P).max() * 8
    h.free()
    g.free()
    ctx.free()


# one CTA, part of a CTA's warps idle, ragged runs, several sites per thread; a few SMs only
@pytest.mark.parametrize("L0,L1,den", [(4, 4, 1), (4, 12, 1), (20, 12, 1), (64, 128, 1),
                                       (64, 64, 76), (32, 32, 152)])
def test_even_odd_cg_sizes(sw, L0, L1, den):
    m = 0.05
    th = si.heatbath_u1(L0, L1, 6.0, 10, seed=3, device="cuda")
    ctx = sw.sw_context_create(0)
    sw.sw_context_set_sm_share(ctx, 1, den)
    g = sw.sw_gauge_load(ctx, th)
    b = si.gaussian_complex(7, L0 * L1)
    D = operators.dirac(th, m)
    for cap in (1, 2, 100000):
        x = np.zeros_like(b)
        st = sw.sw_cg_eo_solve(g, m, b, x, 1e-10, cap, allow_noconv=True)
        r = np.linalg.norm(b - D @ x) / np.linalg.norm(b)
        assert st["outer_iters"] <= cap and abs(r - st["true_resid"]) <= 1e-12
    assert st["converged"] and r <= 1e-10
    b[3] = np.nan
    with pytest.raises(sw.SwError):
        sw.sw_cg_eo_solve(g, m, b, x, 1e-10)
    g.free()
    ctx.free()
