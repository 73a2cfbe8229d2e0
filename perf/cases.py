"""The calls of this library that a lattice program spends its time in, with their sizes.

Every case goes through the Python binding with device buffers, as a program
that keeps its fields on the GPU does.  Gauge fields are drawn from the
quenched compact U(1) ensemble of the Wilson plaquette action; sources and
operator inputs are complex Gaussian.

kinds
  dslash    one operator application (sw_dslash): D, D^dag, A, A^dag, S
  level     one application of the level-2 Galerkin stencil or its adjoint
  transfer  restriction or prolongation between two levels
  cg        CG on the even/odd system (sw_cg_eo_solve), the method one falls
            back on where no hierarchy is kept
  solve     one right-hand side on a hierarchy that is kept (sw_mg_solve)
  batch     several right-hand sides at once (sw_mg_solve_batch)
  config    a new gauge configuration: load, multigrid setup, one solve
"""
import math

import torch

import paper_1801_07823_gb300 as sw

OPS = {"D": sw.SW_OP_D, "Ddag": sw.SW_OP_DDAG, "A": sw.SW_OP_A, "Adag": sw.SW_OP_ADAG, "S": sw.SW_OP_S}
BLOCKS = [(4, 4), (2, 2), (2, 2)]  # KD blocks, then coarse sites per aggregate
TOL = 1e-10
CAP = 2048  # coarsest iteration cap of the Nv 24/32 hierarchies


def listed():
    return [
        # the smallest call: a test lattice, where the launch is all there is
        dict(name="dslash_32", kind="dslash", L0=32, L1=32, op="D", fp32=False, mass=0.05, beta=6.0),
        # a Krylov method on a large lattice, in both storage types
        dict(name="dslash_4096_f32", kind="dslash", L0=4096, L1=4096, op="D", fp32=True, mass=0.05, beta=6.0),
        dict(name="dslash_2048_f64", kind="dslash", L0=2044, L1=2052, op="Ddag", fp32=False, mass=0.05, beta=6.0),
        # a user's own Krylov solver on the preconditioned operators, ragged extents
        dict(name="schur_1024", kind="dslash", L0=1036, L1=1012, op="S", fp32=False, mass=0.01, beta=6.0),
        # coarse-operator studies and two-grid methods of a user's own: the
        # stencil of a large lattice (forward) and restriction into it
        dict(name="stencil_512", kind="level", L0=512, L1=512, nv=24, dagger=0, mass=0.01, beta=6.0),
        dict(name="restrict_512", kind="transfer", L0=512, L1=512, nv=24, level=1, direction=0, mass=0.01, beta=6.0),
        # the solver without a hierarchy
        dict(name="cg_256", kind="cg", L0=256, L1=256, mass=0.1, beta=6.0),
        # propagators on a configuration whose hierarchy is kept: the paper's
        # small lattice and null vectors, and the 256^2 hierarchy of the headline
        dict(name="solve_64", kind="solve", L0=64, L1=64, nv1=8, nv2=12, mixed=False, mass=0.01, beta=6.0),
        dict(name="solve_256", kind="solve", L0=256, L1=256, nv1=24, nv2=32, mixed=False, mass=0.01, beta=6.0),
        dict(name="solve_128_mixed", kind="solve", L0=128, L1=128, nv1=24, nv2=32, mixed=True, mass=0.01, beta=10.0),
        # many sources on one configuration
        dict(name="batch_128_16", kind="batch", L0=128, L1=128, nv1=24, nv2=32, nrhs=16, f32=True, mass=0.01, beta=6.0),
        # an ensemble run: every configuration is loaded, set up and solved once
        dict(name="config_64", kind="config", L0=64, L1=64, nv1=8, nv2=12, mass=0.05, beta=6.0),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _extent(rng, lo, hi, step):
    return max(lo, int(_log(rng, lo, hi)) // step * step)


def draw(rng):
    kind = rng.choice(["dslash", "dslash", "level", "transfer", "cg", "solve", "solve", "batch", "config"])
    beta = rng.choice([6.0, 10.0])
    c = dict(kind=kind)
    if kind == "dslash":
        c.update(L0=_extent(rng, 12, 4096, 4), L1=_extent(rng, 12, 4096, 4), op=rng.choice(list(OPS)), fp32=False)
        if c["op"] in ("D", "Ddag"):
            c["fp32"] = rng.random() < 0.5
        c["mass"] = round(_log(rng, 0.01, 0.1), 4)
    elif kind == "level":
        c.update(L0=_extent(rng, 64, 512, 8), L1=_extent(rng, 64, 512, 8), nv=rng.choice([6, 8, 12, 24, 32]),
                 dagger=rng.randrange(2), mass=round(_log(rng, 0.01, 0.1), 4))
    elif kind == "transfer":
        c.update(L0=_extent(rng, 64, 512, 16), L1=_extent(rng, 64, 512, 16), nv=rng.choice([6, 8, 12, 24, 32]),
                 level=rng.choice([1, 1, 2]), direction=rng.randrange(2), mass=round(_log(rng, 0.01, 0.1), 4))
    elif kind == "cg":
        c.update(L0=_extent(rng, 32, 256, 4), L1=_extent(rng, 32, 256, 4), mass=round(_log(rng, 0.05, 0.2), 4))
    else:
        nv1, nv2 = rng.choice([(6, 8), (8, 12), (12, 16), (24, 32)])
        top = 192 if kind == "solve" else 128 if kind == "batch" else 96
        c.update(L0=_extent(rng, 32, top, 16), L1=_extent(rng, 32, top, 16), nv1=nv1, nv2=nv2,
                 mass=round(_log(rng, 0.02, 0.1), 4))
        if kind == "solve":
            c["mixed"] = rng.random() < 0.5
        if kind == "batch":
            c.update(nrhs=rng.randint(2, 24), f32=rng.random() < 0.5)
    c["beta"] = beta
    return c


# ------------------------------------------------------------------ inputs


def _gauge(L0, L1, beta, gen):
    """theta[mu, x1, x0] of the compact U(1) Wilson action at coupling beta.

    In two dimensions the plaquette angles are independent with density
    proportional to exp(beta cos t); on the torus they also add up to a
    multiple of 2 pi.  They are drawn by inverting the tabulated distribution,
    the small excess of their sum is spread over the lattice, links with those
    plaquettes are summed up, and the two Polyakov phases and a gauge rotation
    are drawn uniformly.
    """
    dev, f8 = "cuda", torch.float64
    t = torch.linspace(-math.pi, math.pi, 8193, dtype=f8, device=dev)
    w = torch.exp(beta * (torch.cos(t) - 1.0))
    cdf = torch.cumulative_trapezoid(w, t)
    cdf = torch.cat([cdf.new_zeros(1), cdf / cdf[-1]])
    u = torch.rand((L1, L0), dtype=f8, device=dev, generator=gen)
    k = (torch.searchsorted(cdf, u) - 1).clamp(0, 8191)
    p = t[k] + (u - cdf[k]) / (cdf[k + 1] - cdf[k]).clamp_min(1e-300) * (t[1] - t[0])
    excess = p.sum() - 2 * math.pi * torch.round(p.sum() / (2 * math.pi))
    p -= excess / p.numel()
    th = torch.zeros((2, L1, L0), dtype=f8, device=dev)
    th[0, 1:] = -torch.cumsum(p, 0)[:-1]
    c = torch.cumsum(p.sum(0), 0)
    th[1, -1, 1:] = c[:-1]
    phases = 2 * math.pi * torch.rand(2, dtype=f8, device=dev, generator=gen)
    th[0, :, 0] += phases[0]
    th[1, 0, :] += phases[1]
    g = 2 * math.pi * torch.rand((L1, L0), dtype=f8, device=dev, generator=gen)
    th[0] += g - torch.roll(g, -1, 1)
    th[1] += g - torch.roll(g, -1, 0)
    return torch.remainder(th + math.pi, 2 * math.pi) - math.pi


def _gaussian(shape, gen, dtype=torch.complex128):
    x = torch.randn((*shape, 2), dtype=torch.float64, device="cuda", generator=gen)
    return torch.view_as_complex(x).to(dtype).contiguous()


def _nvec(case):
    if case["kind"] == "level":
        return [case["nv"]]
    if case["kind"] == "transfer":
        return [case["nv"]] if case["level"] == 1 else [case["nv"], 8]
    return [case["nv1"], case["nv2"]]


def _params(case):
    p = sw.sw_mg_params_default()
    p.coarsest_maxiter = CAP
    if case["kind"] in ("level", "transfer"):
        p.setup_maxiter = 8  # the shapes and sparsity are those of any setup
    if case.get("mixed") or case["kind"] == "batch":
        p.precision = sw.SW_MG_MIXED
    if case.get("f32"):
        p.batch_iterates = sw.SW_PREC_FP32
    return p


def _setup(case, g, seed):
    nv = _nvec(case)
    return sw.sw_mg_setup(g, case["mass"], len(nv) + 1, BLOCKS[:len(nv)], nv, params=_params(case), seed=seed)


class State:
    """A program's context, gauge field and hierarchy, and its buffers."""

    def __init__(self, case, seed):
        self.case, self.seed = case, seed
        self.handles = []
        gen = torch.Generator("cuda").manual_seed(seed)
        L0, L1, kind = case["L0"], case["L1"], case["kind"]
        self.theta = _gauge(L0, L1, case["beta"], gen)
        self.ctx = self.keep(sw.sw_context_create(0, torch.cuda.current_stream().cuda_stream))
        if kind != "config":
            self.gauge = self.keep(sw.sw_gauge_load(self.ctx, self.theta))
        if kind in ("level", "transfer", "solve", "batch"):
            self.mg = self.keep(_setup(case, self.gauge, seed))
        if kind in ("level", "transfer"):
            nin, nout = self.lengths()
            self.b = _gaussian((nin,), gen)
            self.x = torch.empty(nout, dtype=torch.complex128, device="cuda")
        else:
            shape = (case["nrhs"], L1, L0) if kind == "batch" else (L1, L0)
            self.b = _gaussian(shape, gen, torch.complex64 if case.get("fp32") else torch.complex128)
            self.x = torch.empty_like(self.b)

    def keep(self, h):
        self.handles.append(h)
        return h

    def lengths(self):
        case = self.case
        fine = case.get("level", 2)
        e0, e1, nc = sw.sw_mg_level_info(self.mg, fine)
        n = e0 * e1 * nc
        if case["kind"] == "level":
            return n, n
        e0, e1, nc = sw.sw_mg_level_info(self.mg, fine + 1)
        return (n, e0 * e1 * nc) if case["direction"] == 0 else (e0 * e1 * nc, n)

    def __del__(self):
        torch.cuda.synchronize()
        for h in reversed(self.handles):
            h.free()


def prepare(case, seed):
    return State(case, seed)


def run(state):
    c, kind = state.case, state.case["kind"]
    if kind == "dslash":
        prec = sw.SW_PREC_FP32 if c["fp32"] else sw.SW_PREC_FP64
        return sw.sw_dslash(state.gauge, c["mass"], OPS[c["op"]], prec, state.b, state.x)
    if kind == "level":
        return sw.sw_mg_apply_level(state.mg, 2, sw.SW_PREC_FP64, c["dagger"], state.b, state.x)
    if kind == "transfer":
        return sw.sw_mg_transfer(state.mg, c["level"], c["direction"], state.b, state.x)
    if kind == "cg":
        sw.sw_cg_eo_solve(state.gauge, c["mass"], state.b, state.x, TOL)
        return state.x
    if kind == "solve":
        sw.sw_mg_solve(state.mg, state.b, state.x, TOL)
        return state.x
    if kind == "batch":
        sw.sw_mg_solve_batch(state.mg, state.b, state.x, TOL)
        return state.x
    g = sw.sw_gauge_load(state.ctx, state.theta)
    mg = _setup(c, g, state.seed)
    sw.sw_mg_solve(mg, state.b, state.x, TOL)
    mg.free()
    g.free()
    return state.x


# ------------------------------------------------------------------ work


def _hierarchy(case):
    """(bytes of P and Y, [(sites, nc)] of the coarse levels), complex128."""
    e0, e1, dof, size, lev = case["L0"] // 2, case["L1"] // 2, case["L0"] * case["L1"], 0, []
    for nv, (b0, b1) in zip(_nvec(case), BLOCKS):
        size += 16 * dof * nv
        e0, e1 = e0 // b0, e1 // b1
        dof = e0 * e1 * 2 * nv
        size += 16 * e0 * e1 * 5 * (2 * nv) ** 2
        lev.append((e0 * e1, 2 * nv))
    return size, lev


def work(case):
    """Bytes: links (two complex numbers a site), vectors and, where the path
    reads one, the hierarchy, each once.  Flops of a solve: the operators at
    nominal iteration counts (10 outer; 3 intermediate each; 100 coarsest
    each; for CG 15 / mass), since the counts depend on the field."""
    N, kind = case["L0"] * case["L1"], case["kind"]
    el = 8 if case.get("fp32") else 16
    if kind == "dslash":
        if case["op"] == "S":  # even half in, whole field out
            return {"bytes": N * (2 * el + el // 2 + el), "flops": 98 * N // 2}
        return {"bytes": 4 * N * el, "flops": N * (38 if case["op"] in ("D", "Ddag") else 50)}
    if kind == "cg":
        return {"bytes": 4 * N * el, "flops": int(15 / case["mass"]) * N * 50}
    size, lev = _hierarchy(case)
    if kind == "level":
        sites, nc = lev[0]
        return {"bytes": 16 * (5 * nc * nc + 2 * nc) * sites, "flops": 40 * nc * nc * sites}
    if kind == "transfer":  # half of the fine sites take part on level 1
        nv = _nvec(case)[case["level"] - 1]
        fine = N // 2 if case["level"] == 1 else lev[0][0] * lev[0][1]
        coarse = lev[case["level"] - 1][0] * 2 * nv
        return {"bytes": 16 * (fine * (nv + 1) + coarse), "flops": 8 * fine * nv}
    n = case.get("nrhs", 1)
    (s2, c2), (s3, c3) = lev
    one = 10 * (6 * 49 * N + 3 * 6 * 40 * c2 * c2 * s2 + 3 * 100 * 80 * c3 * c3 * s3)
    return {"bytes": size + 32 * N + 32 * N * n, "flops": n * one}


# ------------------------------------------------------------------ 64-bit values


def _links(theta):
    L0 = theta.shape[2]
    u = torch.exp(1j * theta.to(torch.complex128))
    eta = 1.0 - 2.0 * (torch.arange(L0, device=theta.device) % 2).to(torch.float64)
    return 0.5 * u[0], 0.5 * eta * u[1]


def _hop(w, v):
    """sum_mu W_mu(s) v(s + mu) - W_mu(s - mu)^* v(s - mu) on [..., L1, L0]."""
    out = 0
    for wm, dim in ((w[0], -1), (w[1], -2)):
        out = out + wm * torch.roll(v, -1, dim) - torch.roll(wm.conj() * v, 1, dim)
    return out


def _blocks(v):
    """[..., L1, L0] -> [..., L1/2, L0/2, 4], site k of a block at (k & 1, k >> 1)."""
    L1, L0 = v.shape[-2:]
    v = v.reshape(*v.shape[:-2], L1 // 2, 2, L0 // 2, 2).transpose(-3, -2)
    return v.reshape(*v.shape[:-2], 4)


def _unblocks(v):
    B1, B0 = v.shape[-3:-1]
    v = v.reshape(*v.shape[:-1], 2, 2).transpose(-3, -2)
    return v.reshape(*v.shape[:-4], 2 * B1, 2 * B0)


def _block_matrix(w, mass):
    """The 2 x 2 blocks of D, mass included: [L1/2, L0/2, 4, 4]."""
    w0, w1 = _blocks(w[0]), _blocks(w[1])
    B = torch.zeros((*w0.shape, 4), dtype=torch.complex128, device=w0.device)
    for k in range(4):
        B[..., k, k] = mass
    for a, b, x in ((0, 1, w0), (2, 3, w0), (0, 2, w1), (1, 3, w1)):
        B[..., a, b] = x[..., a]
        B[..., b, a] = -x[..., a].conj()
    return B


def _operator(case, w, v):
    mass, op = case["mass"], case["op"]
    if op in ("D", "Ddag"):
        return mass * v + (_hop(w, v) if op == "D" else -_hop(w, v))
    Binv = torch.linalg.inv(_block_matrix(w, mass))

    def blk(M, z):
        return _unblocks((M @ _blocks(z).unsqueeze(-1)).squeeze(-1))

    def A(z):
        t = blk(Binv, z)
        return mass * t + _hop(w, t)

    if op == "A":
        return A(v)
    if op == "Adag":
        return blk(Binv.mH, mass * v - _hop(w, v))
    y, x = torch.meshgrid(torch.arange(v.shape[0], device=v.device), torch.arange(v.shape[1], device=v.device), indexing="ij")
    even = ((x // 2 + y // 2) % 2 == 0).to(torch.complex128)
    e = even * v
    odd = (1 - even) * A(e)
    return e - even * A(odd)


def _inverse(w, mass, b):
    """D^-1 b by CG on D^dag D with restarts from the true residual."""
    def D(v, s=1.0):
        return mass * v + s * _hop(w, v)

    def dot(a, c):
        return (a.conj() * c).real.sum((-1, -2), keepdim=True)

    x = torch.zeros_like(b)
    for _ in range(4):
        r = D(b - D(x), -1.0)
        d, p, rr = torch.zeros_like(b), r, dot(r, r)
        stop = 1e-14 * rr
        for k in range(20000):
            q = D(D(p), -1.0)
            a = rr / dot(p, q).clamp_min(1e-300)
            d, r = d + a * p, r - a * q
            new = dot(r, r)
            if k % 50 == 49 and bool((new <= stop).all()):
                break
            p, rr = r + new / rr.clamp_min(1e-300) * p, new
        x = x + d
    return x


def exact(case, seed):
    """The operators and D^-1 b in complex128; none for the coarse levels,
    whose null vectors are the library's own."""
    if case["kind"] in ("level", "transfer"):
        return None
    gen = torch.Generator("cuda").manual_seed(seed)
    L0, L1 = case["L0"], case["L1"]
    w = _links(_gauge(L0, L1, case["beta"], gen))
    shape = (case["nrhs"], L1, L0) if case["kind"] == "batch" else (L1, L0)
    b = _gaussian(shape, gen, torch.complex64 if case.get("fp32") else torch.complex128).to(torch.complex128)
    if case["kind"] == "dslash":
        return _operator(case, w, b)
    return _inverse(w, case["mass"], b)
