"""Workloads of the Wilson-clover multigrid library, through its ctypes binding.

Each case is one call sequence that a lattice-QCD program makes with device-resident
complex128 fields: the fine operator, the block projector pair, the coarse operator, the
smoother, the steps of a set-up (clover term, block orthonormalisation, Galerkin
coarsening), the learned network's forward and backward pass, and whole solves.  Results
of single-precision calls carry 24 bits, so the program keeps them as complex64 (half the
memory); FP64 calls and solves return complex128 as they come.

Conventions (the library's external layouts): site s = x + Lx (y + Ly (z + Lz t)), gauge
[4][V][3][3], spinors [nrhs][V][4][3], coarse fields [nrhs][Vc][nb], chiral basis
gamma_k = [[0, -i sigma_k], [i sigma_k, 0]], gamma_t = [[0, 1], [1, 0]].
"""
import math

import torch

from paper_1904_08678_gb300 import wcmg

DEV = "cuda:0"
C128 = torch.complex128
PREC = {"f64": wcmg.F64, "f32": wcmg.F32, "bf16": wcmg.BF16, "f16": wcmg.F16}


# ------------------------------------------------------------------ the cases
def _case(kind, dims, nrhs=1, prec="f32", block=(4, 4, 4, 4), nvec=24, levels=2, links="f32", eps=0.25, m0=-0.2):
    return dict(kind=kind, lx=dims[0], ly=dims[1], lz=dims[2], lt=dims[3], nrhs=nrhs, prec=prec, bx=block[0],
                by=block[1], bz=block[2], bt=block[3], nvec=nvec, levels=levels, links=links, eps=eps, m0=m0)


def listed():
    small, mid, big = (8, 8, 8, 16), (16, 16, 16, 32), (24, 24, 24, 48)
    full = (32, 32, 32, 64)
    named = {
        # the FP64 residual check of one vector on a test lattice: latency
        "apply_f64_x1_8c16": _case("apply", small, prec="f64", nvec=8, block=(2, 2, 2, 2)),
        # D on the twelve spin-colour sources of a propagator
        "apply_f32_x12_24c48": _case("apply", big, nrhs=12),
        # four minimal-residual steps on a batch of near-null candidates: a set-up sweep
        "smooth_f32_x24_16c32": _case("smooth", mid, nrhs=24),
        # block orthonormalisation of 24 candidates (double-float arithmetic)
        "nullvecs_df_16c32": _case("nullvecs", mid),
        # the Galerkin operator of the first coarse level
        "coarsen_f32_16c32": _case("coarsen", mid),
        # one coarse apply inside a solve on the largest lattice, BF16 links
        "coarse_bf16_x1_32c64": _case("coarse", full, links="bf16"),
        # the projector pair of one multigrid cycle, one residual
        "transfer_f32_x1_24c48": _case("transfer", big),
        # a new gauge configuration: clover term, then D in FP64 on one vector
        "gauge_f64_24c48": _case("gauge", big, prec="f64"),
        # one minibatch of the learned coarse correction's training, forward and backward
        "ptc_x4_16c32": _case("ptc", mid, nrhs=4),
        # a two-level solve for one source: launches and small grids count
        "solve_x1_16c32": _case("solve", mid),
        # a three-level solve for the twelve sources of a propagator
        "solve_x12_24c48": _case("solve", big, nrhs=12, levels=3, links="bf16"),
        # time to solution on a new configuration: gauge, set-up and solve, largest lattice
        "step_x1_32c64": _case("step", full, levels=3, links="bf16", eps=0.2, m0=-0.25),
    }
    return [dict(c, name=n) for n, c in named.items()]


def _draw_dims(rng, block, vmin, vmax, least=2):
    """Extents that are multiples of the block, ragged, volume log-uniform in [vmin, vmax]."""
    target = math.exp(rng.uniform(math.log(vmin), math.log(vmax)))
    n = [least] * 4
    while True:
        k = rng.choice((0, 1, 2, 3, 3))
        m = list(n)
        m[k] += 1
        if math.prod(a * b for a, b in zip(m, block)) > max(target, math.prod(a * b for a, b in zip(n, block)) + 1):
            return [a * b for a, b in zip(n, block)]
        n = m


def draw(rng):
    kind = rng.choice(("apply", "smooth", "nullvecs", "coarsen", "coarse", "transfer", "gauge", "ptc", "solve", "step"))
    block, nvec = rng.choice((((4, 4, 4, 4), 24), ((4, 4, 4, 4), 20), ((4, 4, 4, 4), 32), ((2, 2, 2, 2), 8),
                              ((3, 3, 3, 3), 20), ((4, 4, 4, 2), 16), ((4, 4, 4, 4), 24)))
    if kind == "apply":
        if rng.random() < 0.4:  # any extents: one-site aggregates
            block, nvec = (1, 1, 1, 1), 4
        dims = _draw_dims(rng, block, 4096, 500000, 5 if block[0] == 1 else 2)
        return _case(kind, dims, rng.choice((1, 1, 2, 3, 5, 12)), rng.choice(("f32", "f32", "f64")), block, nvec)
    if kind == "smooth":
        dims = _draw_dims(rng, block, 4096, 131072)
        return _case(kind, dims, rng.choice((1, 1, 4, 12, nvec)), "f32", block, nvec)
    if kind == "nullvecs":
        return _case(kind, _draw_dims(rng, block, 8192, 131072), 1, rng.choice(("f32", "f32", "f64")), block, nvec)
    if kind == "coarsen":
        return _case(kind, _draw_dims(rng, block, 8192, 131072), 1, "f32", block, nvec)
    if kind == "coarse":
        dims = _draw_dims(rng, block, 65536 if block[0] == 4 else 8192, 700000 if block[0] == 4 else 40000)
        return _case(kind, dims, rng.choice((1, 1, 12, 24)), "f32", block, nvec, 2, rng.choice(("f32", "bf16", "bf16")))
    if kind == "transfer":
        dims = _draw_dims(rng, block, 8192, 400000)
        return _case(kind, dims, rng.choice((1, 1, 2, 4, 12, 24)), rng.choice(("f32", "f32", "f32", "f64")), block, nvec)
    if kind == "gauge":
        return _case(kind, _draw_dims(rng, (1, 1, 1, 1), 8192, 663552, 5), 1, "f64", (1, 1, 1, 1), 4)
    if kind == "ptc":
        return _case(kind, _draw_dims(rng, (4, 4, 4, 4), 8192, 131072), rng.choice((1, 2, 4)))
    if kind == "solve" and rng.random() < 0.25:  # the library's default parameters: FP64 throughout
        return _case(kind, _draw_dims(rng, (2, 2, 2, 2), 1024, 8192), 1, "f64", (2, 2, 2, 2), 8, 2, "f32", 0.3, -0.1)
    levels = rng.choice((2, 3))
    nvec = rng.choice((20, 24, 24))
    unit = (4, 4, 4, 4) if levels == 2 else (8, 8, 8, 8)
    dims = _draw_dims(rng, unit, 16384, 400000, 2)
    nrhs = rng.choice((1, 1, 2, 4)) if kind == "solve" else 1
    return _case(kind, dims, nrhs, "f32", (4, 4, 4, 4), nvec, levels, "f32" if levels == 2 else rng.choice(("bf16", "f16")))


# ------------------------------------------------------------------ inputs
def _dims(c):
    return c["lx"], c["ly"], c["lz"], c["lt"]


def _block(c):
    return c["bx"], c["by"], c["bz"], c["bt"]


def _volume(c):
    return math.prod(_dims(c))


def _generator(seed, stream):
    g = torch.Generator(device=DEV)
    g.manual_seed((seed * 1000003 + stream) % 2**63)
    return g


def _gaussian(shape, seed, stream):
    """Independent N(0, 1) real and imaginary parts."""
    z = torch.randn(tuple(shape) + (2,), dtype=torch.float64, device=DEV, generator=_generator(seed, stream))
    return torch.view_as_complex(z)


def _gauge_field(c, seed):
    """SU(3) links exp(i eps X), X a unit Gaussian in the Gell-Mann basis."""
    n = 4 * _volume(c)
    out = torch.empty((n, 3, 3), dtype=C128, device=DEV)
    for s, lo in enumerate(range(0, n, 1 << 20)):
        m = min(1 << 20, n - lo)
        xi = c["eps"] * torch.randn((m, 8), dtype=torch.float64, device=DEV, generator=_generator(seed, 100 + s))
        x = torch.zeros((m, 3, 3), dtype=C128, device=DEV)
        r3 = 1 / math.sqrt(3.0)
        x[:, 0, 0], x[:, 1, 1], x[:, 2, 2] = (d.to(C128) for d in (xi[:, 2] + r3 * xi[:, 7], r3 * xi[:, 7] - xi[:, 2],
                                                                   -2 * r3 * xi[:, 7]))
        for (a, b), (k, l) in (((0, 1), (0, 1)), ((0, 2), (3, 4)), ((1, 2), (5, 6))):
            x[:, a, b] = torch.complex(xi[:, k], -xi[:, l])
            x[:, b, a] = torch.complex(xi[:, k], xi[:, l])
        u = torch.matrix_exp(1j * x)
        r0 = u[:, 0] / torch.linalg.vector_norm(u[:, 0], dim=-1, keepdim=True)
        r1 = u[:, 1] - (r0.conj() * u[:, 1]).sum(-1, keepdim=True) * r0
        r1 = r1 / torch.linalg.vector_norm(r1, dim=-1, keepdim=True)
        out[lo:lo + m] = torch.stack([r0, r1, torch.linalg.cross(r0, r1).conj()], 1)
    return out.reshape(4, _volume(c), 3, 3)


def _candidates(c, seed):
    """Near-null candidates: Gaussian fields mixed so that a panel's condition number is a few, up to about ten."""
    v = _gaussian((c["nvec"], _volume(c) * 12), seed, 2)
    m = 0.06 * _gaussian((c["nvec"], c["nvec"]), 12345, 3) + torch.eye(c["nvec"], device=DEV)
    return (m @ v).reshape(c["nvec"], _volume(c), 4, 3)


def _links(c, seed):
    """Coarse links of a hopping matrix: self block near 4, hops of order one half."""
    vc, nb = _volume(c) // math.prod(_block(c)), 2 * c["nvec"]
    a = (0.5 / math.sqrt(nb)) * _gaussian((9, vc, nb, nb), seed, 4)
    a[0] += 4.0 * torch.eye(nb, device=DEV)
    return a


def _context(c):
    f32 = c["prec"] == "f32"
    levels = c["levels"]
    big = _volume(c) >= 1 << 21
    nvec = [c["nvec"], 32 if big else 24][:levels - 1]
    p = wcmg.default_params(
        dims=_dims(c), n_levels=levels, blocks=[_block(c), (2, 2, 2, 2)][:levels - 1], nvec=nvec, m0=c["m0"], csw=1.0,
        setup_init_sweeps=3, setup_refine_sweeps=2 if f32 else 0, outer_maxiter=2000, outer_tol=1e-12,
        inner_prec=PREC[c["prec"]], coarse_link_prec=PREC[c["links"]], max_rhs=max(c["nrhs"], 1),
        use_graphs=1, autotune=1 if f32 else 0, ortho_df=1 if f32 else 0)
    return wcmg.Context(p)


def prepare(case, seed):
    c, k = case, case["kind"]
    s = {"case": c, "ctx": _context(c), "seed": seed}
    ctx, v, n = s["ctx"], _volume(c), c["nrhs"]
    if k != "coarse" and k != "transfer" and k != "nullvecs":
        s["U"] = _gauge_field(c, seed)
        if k != "gauge" and k != "step":
            ctx.set_gauge(s["U"])
    if k in ("apply", "smooth", "transfer", "gauge", "ptc", "solve", "step"):
        s["b"] = _gaussian((n, v, 4, 3), seed, 1)
        s["x"] = torch.zeros_like(s["b"])
    if k in ("coarsen", "transfer"):
        ctx.set_nullvecs(0, _candidates(c, seed))
    vc, nb = v // math.prod(_block(c)), 2 * c["nvec"]
    if k == "nullvecs":
        s["v"] = _candidates(c, seed)
        s["q"] = torch.empty_like(s["v"])
    elif k == "coarsen":
        s["A"] = torch.empty((9, vc, nb, nb), dtype=C128, device=DEV)
    elif k == "coarse":
        ctx.set_coarse_links(1, _links(c, seed))
        s["b"] = _gaussian((n, vc, nb), seed, 5)
        s["x"] = torch.empty_like(s["b"])
    elif k == "transfer":
        s["y"] = torch.empty((n, vc, nb), dtype=C128, device=DEV)
    elif k == "ptc":
        s["W"] = 0.05 * _gaussian((wcmg.PTC_NWEIGHTS,), seed, 6)
        ctx.ptc_set_weights(s["W"])
        s["g"] = _gaussian((n, v, 4, 3), seed, 7)
        s["gin"], s["gW"] = torch.empty_like(s["b"]), torch.empty_like(s["W"])
    elif k == "solve":
        ctx.setup_seeded(seed)
    torch.cuda.synchronize()
    return s


def run(state):
    s, c, ctx = state, state["case"], state["ctx"]
    k, n, prec = c["kind"], c["nrhs"], PREC[c["prec"]]
    keep = (lambda t: t.to(torch.complex64)) if c["prec"] == "f32" else (lambda t: t)
    if k == "apply":
        ctx.apply_D(s["b"], s["x"], n, prec)
        return keep(s["x"])
    if k == "smooth":
        ctx.krylov(0, 0, s["b"], s["x"], n, 4)
        return keep(s["x"])
    if k == "nullvecs":
        ctx.set_nullvecs(0, s["v"])
        ctx.get_nullvecs(0, s["q"])
        return s["q"]
    if k == "coarsen":
        ctx.coarsen(0)
        ctx.get_coarse_links(1, s["A"])
        return keep(s["A"])
    if k == "coarse":
        ctx.apply_coarse(1, s["b"], s["x"], n, prec)
        return keep(s["x"])
    if k == "transfer":
        ctx.restrict(0, s["b"], s["y"], n, prec)
        ctx.prolong(0, s["y"], s["x"], n, prec)
        return keep(s["y"]), keep(s["x"])
    if k == "gauge":
        ctx.set_gauge(s["U"])
        ctx.apply_D(s["b"], s["x"], n, prec)
        return s["x"]
    if k == "ptc":
        ctx.ptc_forward(s["b"], s["x"], n)
        ctx.ptc_backward(s["b"], s["g"], s["gin"], s["gW"], n)
        return keep(s["x"]), keep(s["gin"]), keep(s["gW"])
    if k == "step":
        ctx.set_gauge(s["U"])
        ctx.setup_seeded(s["seed"])
    ctx.solve(s["b"], s["x"], n)
    return s["x"]


def work(case):
    """Inputs read once, outputs written once, operands kept by the context at their precision."""
    c, k = case, case["kind"]
    v, n, nv = _volume(c), c["nrhs"], c["nvec"]
    r = 16 if c["prec"] == "f64" else 8          # the call's own precision, and what is kept of its result
    vc, nb = v // math.prod(_block(c)), 2 * nv
    op = 72 * v * r                              # links and clover term
    spinor = 12 * v * n
    if k == "apply":
        return {"bytes": spinor * (16 + r) + op, "flops": 1872 * v * n}
    if k == "smooth":
        return {"bytes": spinor * (16 + r) + op, "flops": 4 * (1872 + 12 * 24) * v * n}
    if k == "nullvecs":
        return {"bytes": 2 * nv * 12 * v * 16, "flops": 8 * 12 * v * nv * nv}
    if k == "coarsen":
        return {"bytes": op + nv * 12 * v * r + 9 * vc * nb * nb * r, "flops": v * nb * (1872 + 8 * 12 * nv)}
    if k == "coarse":
        link = 4 if c["links"] in ("bf16", "f16") else r
        return {"bytes": 9 * vc * nb * nb * link + vc * nb * n * (16 + r), "flops": 72 * vc * nb * nb * n}
    if k == "transfer":
        return {"bytes": 2 * nv * 12 * v * r + spinor * (16 + r) + 2 * vc * nb * n * r, "flops": 16 * 12 * v * nv * n}
    if k == "gauge":
        return {"bytes": 36 * v * 16 * 2 + spinor * 32, "flops": v * (36 * 216 + 1872)}
    if k == "ptc":
        fields = 12 * v * n
        return {"bytes": 36 * v * 8 + fields * (2 * 16 + 2 * r), "flops": 4 * 2 * v * n * 12 * 9 * (96 + 72)}
    # a solve: its operands once, and the cycles it takes are its own affair
    operands = op + nv * 12 * v * r + 9 * vc * nb * nb * (4 if c["links"] != "f32" else r)
    flops = 20 * v * n * (6 * 1872 + 16 * 12 * nv)
    if k == "step":
        return {"bytes": operands + 2 * 36 * v * 16 + spinor * 32, "flops": flops + v * nv * (14 * 1872 + 24 * 12 * nv)}
    return {"bytes": operands + spinor * 32, "flops": flops}


# ------------------------------------------------------------------ 64-bit references
_PAULI = torch.tensor([[[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]]], dtype=C128)


def _gammas():
    z = torch.zeros((2, 2), dtype=C128)
    g = [torch.cat([torch.cat([z, -1j * s], 1), torch.cat([1j * s, z], 1)], 0) for s in _PAULI]
    one = torch.eye(2, dtype=C128)
    g.append(torch.cat([torch.cat([z, one], 1), torch.cat([one, z], 1)], 0))
    return [m.to(DEV) for m in g]


class _Wilson:
    """D on [n, T, Z, Y, X, 4, 3] tensors, with plain torch."""

    def __init__(self, c, u, clover=True):
        lx, ly, lz, lt = _dims(c)
        self.shape = (lt, lz, ly, lx)
        self.u = [u[m].reshape(self.shape + (3, 3)) for m in range(4)]
        self.g = _gammas()
        self.one = torch.eye(4, dtype=C128, device=DEV)
        self.c = self._clover(c["m0"]) if clover else None

    def grid(self, f):
        return f.reshape(f.shape[:1] + self.shape + (4, 3))

    def _next(self, f, mu, sign, lead=0):
        """f(x + sign mu)."""
        return torch.roll(f, -sign, dims=lead + 3 - mu)

    def _clover(self, m0):
        c = torch.zeros(self.shape + (4, 3, 4, 3), dtype=C128, device=DEV)
        for m in range(4):
            for n in range(m + 1, 4):
                a, b, nx = self.u[m], self.u[n], self._next
                dag = lambda t: t.mH  # noqa: E731
                q = a @ nx(b, m, 1) @ dag(nx(a, n, 1)) @ dag(b)
                am, bn = nx(a, m, -1), nx(b, n, -1)
                q = q + b @ dag(nx(am, n, 1)) @ dag(nx(b, m, -1)) @ am
                q = q + dag(am) @ dag(nx(bn, m, -1)) @ nx(am, n, -1) @ bn
                q = q + dag(bn) @ nx(a, n, -1) @ nx(bn, m, 1) @ dag(a)
                f = 0.125j * (q - dag(q))
                sig = 0.5j * (self.g[m] @ self.g[n] - self.g[n] @ self.g[m])
                c += 0.5 * sig[:, None, :, None] * f[..., None, :, None, :]  # csw = 1
        c = c.reshape(self.shape + (12, 12))
        return c + (4.0 + m0) * torch.eye(12, dtype=C128, device=DEV)

    def hop(self, f, mu, sign):
        """The term of D that reads f(x + sign mu)."""
        p = self._next(f, mu, sign, 1)
        if sign > 0:
            t = p @ self.u[mu].transpose(-1, -2)
        else:
            t = p @ self._next(self.u[mu], mu, -1).conj()
        return -0.5 * torch.einsum("st,...tb->...sb", self.one - sign * self.g[mu], t)

    def site(self, f):
        return (f.reshape(f.shape[:-2] + (1, 12)) @ self.c.transpose(-1, -2)).reshape(f.shape)

    def __call__(self, f):
        out = torch.empty_like(f)
        for i in range(f.shape[0]):  # one field at a time: bounded temporaries
            o = self.site(f[i:i + 1])
            for mu in range(4):
                o += self.hop(f[i:i + 1], mu, 1)
                o += self.hop(f[i:i + 1], mu, -1)
            out[i] = o[0]
        return out


def _blocks(c, f):
    """[n, V, 12] -> [aggregate, chirality, n, sites in the aggregate * 6], aggregates in coarse order."""
    lx, ly, lz, lt = _dims(c)
    bx, by, bz, bt = _block(c)
    f = f.reshape(-1, lt // bt, bt, lz // bz, bz, ly // by, by, lx // bx, bx, 2, 6)
    f = f.permute(1, 3, 5, 7, 9, 0, 2, 4, 6, 8, 10)
    return f.reshape(_volume(c) // (bx * by * bz * bt), 2, f.shape[5], -1)


def _unblocks(c, a):
    """Inverse of _blocks."""
    lx, ly, lz, lt = _dims(c)
    bx, by, bz, bt = _block(c)
    n = a.shape[2]
    a = a.reshape(lt // bt, lz // bz, ly // by, lx // bx, 2, n, bt, bz, by, bx, 6)
    return a.permute(5, 0, 6, 1, 7, 2, 8, 3, 9, 4, 10).reshape(n, _volume(c), 12)


def _projector(c, seed):
    """Orthonormalised candidates as [aggregate, chirality, nvec, elements] (Cholesky QR, twice)."""
    a = _blocks(c, _candidates(c, seed).reshape(c["nvec"], _volume(c), 12)).transpose(-1, -2).contiguous()
    for _ in range(2):
        r = torch.linalg.cholesky(a.mH @ a).mH
        a = torch.linalg.solve_triangular(r, a, upper=True, left=False)
    return a.transpose(-1, -2)


def _exact_coarsen(c, seed):
    d = _Wilson(c, _gauge_field(c, seed))
    p = _projector(c, seed)
    na, nv = p.shape[0], c["nvec"]
    out = torch.zeros((9, na, 2 * nv, 2 * nv), dtype=C128, device=DEV)
    lx, ly, lz, lt = _dims(c)
    coord = torch.arange(_volume(c), device=DEV)
    xs = (coord % lx, coord // lx % ly, coord // (lx * ly) % lz, coord // (lx * ly * lz))
    cross = {}
    for mu in range(4):
        b, n = _block(c)[mu], _dims(c)[mu]
        for sign in (1, -1):
            cross[mu, sign] = (xs[mu] % b == (b - 1 if sign > 0 else 0)).reshape(-1, 1).to(torch.float64)
    for ch in range(2):
        for i in range(nv):
            half = torch.zeros((na, 2, 1, p.shape[3]), dtype=C128, device=DEV)
            half[:, ch, 0] = p[:, ch, i]
            f = d.grid(_unblocks(c, half).reshape(1, -1, 4, 3))
            own = d.site(f).reshape(1, -1, 12)
            pieces = []
            for mu in range(4):
                for sign in (1, -1):
                    h = d.hop(f, mu, sign).reshape(1, -1, 12)
                    pieces.append(h * cross[mu, sign])
                    own = own + h * (1 - cross[mu, sign])
            t = _blocks(c, torch.cat([own] + pieces))                       # [na, 2, 9, elements]
            out[:, :, :, ch * nv + i] = (p.conj() @ t.transpose(-1, -2)).permute(3, 0, 1, 2).reshape(9, na, 2 * nv)
    return out


def _exact_solve(c, d, b):
    """BiCGStab to 1e-13, all right-hand sides at once."""
    b = d.grid(b)
    dot = lambda p, q: (p.conj() * q).flatten(1).sum(1).reshape((-1,) + (1,) * 6)  # noqa: E731
    x, r = torch.zeros_like(b), b.clone()
    r0, p = r.clone(), r.clone()
    rho, bn = dot(r0, r), torch.linalg.vector_norm(b)
    for _ in range(600):
        v = d(p)
        al = rho / dot(r0, v)
        s = r - al * v
        t = d(s)
        om = dot(t, s) / dot(t, t)
        x += al * p + om * s
        r = s - om * t
        if torch.linalg.vector_norm(r) <= 1e-14 * bn:
            break
        new = dot(r0, r)
        p = r + (new / rho) * (al / om) * (p - om * v)
        rho = new
    true = torch.linalg.vector_norm(b - d(x)) / bn
    return x.reshape(x.shape[0], -1, 4, 3) if true < 3e-13 else None


def _exact_ptc(c, seed):
    d = _Wilson(c, _gauge_field(c, seed), clover=False)
    w = 0.05 * _gaussian((wcmg.PTC_NWEIGHTS,), seed, 6)
    b, g = (_gaussian((c["nrhs"], _volume(c), 4, 3), seed, k) for k in (1, 7))
    h = wcmg.PTC_HIDDEN

    def transport(f, k):
        mu, sign = (k - 1) // 2, 1 - 2 * ((k - 1) % 2)
        if k == 0:
            return f
        p = d._next(f, mu, sign, 1)
        return p @ (d.u[mu].transpose(-1, -2) if sign > 0 else d._next(d.u[mu], mu, -1).conj())

    back = lambda f, k: transport(f, k if k == 0 else k + 1 if k % 2 else k - 1)  # noqa: E731
    w1, w2 = w[:h * 144].reshape(h, 9, 4, 4), w[h * 144:].reshape(h, 9, 4, 4)
    outs, gins, gw = [], [], torch.zeros((2, h, 9, 4, 4), dtype=C128, device=DEV)
    for i in range(c["nrhs"]):
        f, go = d.grid(b[i:i + 1]), d.grid(g[i:i + 1])
        tf = [transport(f, k) for k in range(9)]
        tg = [back(go, k) for k in range(9)]  # T_k^dag gout
        out, gin = torch.zeros_like(f), torch.zeros_like(f)
        for j in range(h):
            hid = sum(torch.einsum("st,...tb->...sb", w1[j, k], tf[k]) for k in range(9))
            gh = sum(torch.einsum("ts,...tb->...sb", w2[j, k].conj(), tg[k]) for k in range(9))
            for k in range(9):
                th = transport(hid, k)
                out += torch.einsum("st,...tb->...sb", w2[j, k], th)
                gin += back(torch.einsum("ts,...tb->...sb", w1[j, k].conj(), gh), k)
                flat = lambda q: q.reshape(-1, 4, 3).transpose(0, 1).reshape(4, -1)  # noqa: E731
                gw[1, j, k] += flat(go) @ flat(th).mH
                gw[0, j, k] += flat(gh) @ flat(tf[k]).mH
        outs.append(out.reshape(-1, 4, 3))
        gins.append(gin.reshape(-1, 4, 3))
    return torch.stack(outs), torch.stack(gins), gw.reshape(-1)


def exact(case, seed):
    c, k, v, n = case, case["kind"], _volume(case), case["nrhs"]
    if k == "step" and v > 400000 or k == "solve" and v * n > 1200000:
        return None  # the plain solver would take too long
    if k == "nullvecs":
        return _unblocks(c, _projector(c, seed)).reshape(c["nvec"], v, 4, 3)
    if k == "coarse":
        nb = 2 * c["nvec"]
        lat = [a // b for a, b in zip(_dims(c), _block(c))][::-1]
        a, b = _links(c, seed), _gaussian((n, v // math.prod(_block(c)), nb), seed, 5)
        y = b.transpose(0, 1) @ a[0].transpose(-1, -2)
        for m in range(8):
            f = torch.roll(b.reshape([n] + lat + [nb]), -1 if m % 2 == 0 else 1, dims=4 - m // 2)
            y = y + f.reshape(n, -1, nb).transpose(0, 1) @ a[1 + m].transpose(-1, -2)
        return y.transpose(0, 1)
    if k == "coarsen":
        return _exact_coarsen(c, seed)
    if k == "ptc":
        return _exact_ptc(c, seed)
    b = _gaussian((n, v, 4, 3), seed, 1)
    if k == "transfer":
        p = _projector(c, seed)
        y = p.conj() @ _blocks(c, b.reshape(n, v, 12)).transpose(-1, -2)  # [na, 2, nvec, n]
        x = _unblocks(c, y.transpose(-1, -2) @ p)
        return y.reshape(p.shape[0], 2 * c["nvec"], n).permute(2, 0, 1), x.reshape(n, v, 4, 3)
    d = _Wilson(c, _gauge_field(c, seed))
    if k in ("apply", "gauge"):
        return d(d.grid(b)).reshape(n, v, 4, 3)
    if k == "smooth":
        r, x = d.grid(b), 0
        dot = lambda p, q: (p.conj() * q).flatten(1).sum(1).reshape((-1,) + (1,) * 6)  # noqa: E731
        for _ in range(4):
            p = d(r)
            al = dot(p, r) / dot(p, p)
            x = x + al * r
            r = r - al * p
        return x.reshape(n, v, 4, 3)
    return _exact_solve(c, d, b)
