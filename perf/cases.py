"""The work that a user of this framework has it do, as measurable cases.

A case is a dict of plain values.  ``prepare`` makes what the user's program
holds before the call (gauge field, sources, a ``Solver`` with its operator and,
where the call needs one, its multigrid setup), all on the GPU and from the seed
alone; ``run`` is one pass through the public entry points; ``exact`` gives the
same outputs in 64 bits from plain torch, with no code of the framework.

Kinds of cases:

* ``op``      -- a fine operator applied to one or several vectors (``Solver.apply``):
                 residual checks, eigenvalue and deflation codes, a user's own Krylov solver.
* ``force``   -- the gauge-link derivative (``Solver.force``): every step of a molecular-dynamics trajectory.
* ``solve``   -- ``Solver.solve`` by multigrid on a lattice whose setup exists: one source, or the twelve
                 spin-colour sources of a propagator.
* ``krylov``  -- ``Solver.solve`` by mixed-precision BiCGStab (no setup).
* ``grad``    -- a differentiated solve: forward and backward of ``dirac_solve``.
* ``remass``  -- ``Solver.update_mass``: the hierarchy rebuilt from kept null vectors for another mass,
                 returning the coarse operator it gives.
* ``fresh``   -- a new gauge configuration from the start: load, clover, setup and the solve of its sources.

Fields are the framework's synthetic ensemble, links exp(i eps H) smeared by
APE steps (alpha = 0.5): eps = 0.25 is the nearly free field of the benchmark
solve, eps = 1.0 the rough field of the comparison solvers, whose critical mass
lies below -0.65.  Results that are computed in single precision are kept by
the caller in single precision (complex64).
"""
import math

import torch

from paper_1011_2775_gb300 import binding as B
from paper_1011_2775_gb300.autograd import dirac_solve
from paper_1011_2775_gb300.solver import Solver

APE_STEPS = 5
CSW = 1.0
ANISO_W, ANISO_CSW_T = (0.3, 0.3, 0.3, 1.0), 1.4
TOL = 1e-10
# Multigrid parameters of the benchmark solve: coarse GCR(64) to a tenth.
MG = dict(tol_coarse=0.1, restart_coarse=64, maxit_fine=2000)
OPS = {"D": B.MG_OP_D, "DP": B.MG_OP_DP, "DR": B.MG_OP_DR, "BR": B.MG_OP_BR, "M": B.MG_OP_M, "MINV": B.MG_OP_MINV,
       "HOP": B.MG_OP_HOP}


# --------------------------------------------------------------------------- the cases
def _dims(c):
    return c["Lx"], c["Ly"], c["Lz"], c["Lt"]


def _volume(c):
    return c["Lx"] * c["Ly"] * c["Lz"] * c["Lt"]


def _lat(lx, ly, lz, lt):
    return dict(Lx=lx, Ly=ly, Lz=lz, Lt=lt)


def _mg(levels=2, b=(4, 4, 4, 4), nv=24, nv2=0, storage=B.MG_STORE_FP32):
    return dict(levels=levels, bx=b[0], by=b[1], bz=b[2], bt=b[3], nv=nv, nv2=nv2, storage=storage)


def listed():
    return [
        # The smallest call: one FP64 operator application on a few sites (a residual check inside somebody's
        # loop), half volume not a multiple of a thread block: launches, copies and allocations count.
        dict(name="op_d_fp64_6x4x8x10", kind="op", **_lat(6, 4, 8, 10), op="D", prec=B.MG_FP64, nrhs=1, eps=0.25,
             m0=-0.2, aniso=False),
        # The largest operator call: the single-precision even-odd operator on the twelve vectors of a
        # propagator of the largest lattice in use (bandwidth).
        dict(name="op_dr_fp32_12rhs_32x32x32x64", kind="op", **_lat(32, 32, 32, 64), op="DR", prec=B.MG_FP32, nrhs=12,
             eps=0.25, m0=-0.3, aniso=False),
        # The su(3) force of a molecular-dynamics step in FP64.
        dict(name="force_fp64_16x16x16x32", kind="force", **_lat(16, 16, 16, 32), prec=B.MG_FP64, su3=True, eps=1.0,
             m0=-0.5, aniso=False),
        # One source on a small lattice: the solve is a chain of short dependent launches.
        dict(name="solve_8x8x8x16", kind="solve", **_lat(8, 8, 8, 16), **_mg(), nrhs=1, eps=1.0, m0=-0.5),
        # The benchmark solve of the framework: one source, the lightest mass of its sweep.
        dict(name="solve_16x16x16x32", kind="solve", **_lat(16, 16, 16, 32), **_mg(), nrhs=1, eps=0.25, m0=-0.35),
        # The same system for the twelve sources of a propagator, 16-bit storage of the hierarchy.
        dict(name="solve_12rhs_fp16_16x16x16x32", kind="solve", **_lat(16, 16, 16, 32),
             **_mg(storage=B.MG_STORE_FP16), nrhs=12, eps=0.25, m0=-0.35),
        # A large lattice with BF16 storage, close to the critical mass of its field.
        dict(name="solve_bf16_24x24x24x48", kind="solve", **_lat(24, 24, 24, 48), **_mg(storage=B.MG_STORE_BF16),
             nrhs=1, eps=1.0, m0=-0.65),
        # Three levels (4^4, then 2^4 blocks): the intermediate level's GCR and cycles.
        dict(name="solve_3level_16x16x16x32", kind="solve", **_lat(16, 16, 16, 32), **_mg(levels=3, nv2=32), nrhs=1,
             eps=1.0, m0=-0.65),
        # The solver without a setup: mixed-precision BiCGStab, for one or two sources per configuration.
        dict(name="krylov_mp_16x16x16x32", kind="krylov", **_lat(16, 16, 16, 32), eps=1.0, m0=-0.5),
        # A training or fitting step that differentiates the solve, on a lattice whose coarse extents are odd.
        dict(name="grad_12x12x12x24", kind="grad", **_lat(12, 12, 12, 24), **_mg(), eps=1.0, m0=-0.5),
        # A mass sweep on one configuration: the hierarchy rebuilt from the null vectors in hand.
        dict(name="remass_16x16x16x32", kind="remass", **_lat(16, 16, 16, 32), **_mg(), eps=0.25, m0=-0.3),
        # A propagator on a configuration that has just arrived: load, clover, setup, twelve sources.
        dict(name="fresh_12rhs_16x16x16x32", kind="fresh", **_lat(16, 16, 16, 32), **_mg(), nrhs=12, eps=1.0, m0=-0.5),
    ]


def _even(rng, lo, hi):
    """An even extent, spread over the logarithm of the range."""
    return 2 * max(lo // 2, min(hi // 2, round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / 2)))


def _lattice(rng, most, lo=4, hi=32, hit=64):
    while True:
        c = _lat(_even(rng, lo, hi), _even(rng, lo, hi), _even(rng, lo, hi), _even(rng, lo, hit))
        if _volume(c) <= most:
            return c


def _blocked(rng, most, cmax=6):
    """A lattice of coarse extents 2 .. cmax (odd ones among them), blocks of 4 or 2 sites a side."""
    while True:
        b = tuple(rng.choice((4, 4, 4, 2)) for _ in range(4))
        if math.prod(b) < 64:
            continue
        n = [rng.randint(2, cmax) for _ in range(3)] + [rng.randint(2, 2 * cmax)]
        c = _lat(*(x * y for x, y in zip(b, n)))
        if _volume(c) <= most:
            return c, b


def draw(rng):
    kind = rng.choice(("op", "op", "op", "force", "solve", "solve", "solve", "krylov", "grad", "remass", "fresh"))
    mass = dict(eps=1.0, m0=round(rng.uniform(-0.5, -0.2), 3))
    store = rng.choice((B.MG_STORE_FP32, B.MG_STORE_FP16, B.MG_STORE_BF16))
    if kind == "op":
        n = rng.choice((1, 1, 2, 3, 4, 8, 12))
        lat = _lattice(rng, 32 * 32 * 32 * 64 * 12 // n // 2)
        aniso = rng.random() < 0.25
        return dict(kind=kind, **lat, op=rng.choice(sorted(OPS)), prec=rng.choice((B.MG_FP64, B.MG_FP32)), nrhs=n,
                    eps=rng.choice((0.25, 1.0)), m0=round(rng.uniform(-0.35, 0.2), 3), aniso=aniso)
    if kind == "force":
        return dict(kind=kind, **_lattice(rng, 16 * 16 * 16 * 32, hit=32), prec=rng.choice((B.MG_FP64, B.MG_FP32)),
                    su3=rng.random() < 0.5, eps=1.0, m0=-0.5, aniso=rng.random() < 0.25)
    if kind == "krylov":
        return dict(kind=kind, **_lattice(rng, 24 * 24 * 24 * 48, hit=48), **mass)
    if kind == "grad":
        lat, b = _blocked(rng, 16 * 16 * 16 * 32, 4)
        return dict(kind=kind, **lat, **_mg(b=b, nv=rng.choice((8, 16, 24))), **mass)
    if kind == "solve":
        n = rng.choice((1, 1, 1, 2, 5, 12))
        lat, b = _blocked(rng, 24 * 24 * 24 * 48 if n == 1 else 12 * 16 * 16 * 16 * 32 // n)
        return dict(kind=kind, **lat, **_mg(b=b, nv=rng.choice((8, 12, 16, 20, 24)), storage=store), nrhs=n, **mass)
    lat, b = _blocked(rng, 16 * 16 * 16 * 32, 4)
    more = dict(eps=rng.choice((0.25, 1.0)), m0=-0.3) if kind == "remass" else dict(nrhs=rng.choice((1, 4, 12)), **mass)
    return dict(kind=kind, **lat, **_mg(b=b, nv=rng.choice((8, 16, 24)), storage=store), **more)


def work(c):
    """One pass, counted per lattice site: links and clover held in the arithmetic's precision, caller's
    vectors and fields in complex128, each read or written once.  An iterative solve cannot do without
    one application of its operator; how many iterations it takes is the method's."""
    V, k = _volume(c), c["kind"]
    fields = 72 + 72                       # reals of the links and of the clover term
    hop, clover, mm = 1320, 504, 198       # flops of a hop (site), a clover term (site), a 3x3 complex product
    op = 2 * (hop + clover) / 2            # flops of D, or of D_r, for one site
    if k == "op":
        es = 8 if c["prec"] == B.MG_FP64 else 4
        return {"bytes": V * (fields * es + 384 * c["nrhs"]), "flops": V * op * c["nrhs"]}
    # hop: two outer products per link; clover: six planes of 22 products, the insertions
    dforce = 4 * 2 * 360 + 6 * (22 * mm + 288)
    if k == "force":
        es = 8 if c["prec"] == B.MG_FP64 else 4
        return {"bytes": V * (72 * es + 2 * 192 + 576), "flops": V * dforce}
    n = c.get("nrhs", 1)
    if k == "krylov":
        return {"bytes": V * (fields * 8 + 384), "flops": V * op}
    nv = c["nv"]
    sites = V // (c["bx"] * c["by"] * c["bz"] * c["bt"])
    coarse = sites * 9 * (2 * nv) ** 2     # complex numbers of the coarse operator
    pbytes = 8 if c["storage"] == B.MG_STORE_FP32 else 4
    solve = {"bytes": V * (fields * 8 + 12 * nv * pbytes + 384 * n) + coarse * pbytes, "flops": V * op * n}
    if k == "solve":
        return solve
    if k == "grad":
        return {"bytes": solve["bytes"] + V * (72 * 8 + 384 + 576), "flops": 2 * solve["flops"] + V * dforce}
    # block Gram-Schmidt of nv vectors; 2 nv columns hopped and projected on nv vectors (three slots a site)
    build = V * (12 * nv * nv * 8 + 2 * nv * (hop + clover) / 2 + 2 * nv * 6 * nv * 2 * 3 * 8)
    if k == "remass":
        return {"bytes": V * (fields * 8 + 12 * nv * (8 + pbytes)) + coarse * 8, "flops": build}
    return {"bytes": solve["bytes"] + V * (576 + 12 * nv * 8) + coarse * 8, "flops": solve["flops"] + build}


# --------------------------------------------------------------------------- inputs
def _dev():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _rng(seed, what):
    g = torch.Generator(device=_dev())
    g.manual_seed((int(seed) * 1009 + what) % (1 << 62))
    return g


def _mm(a, b):
    return sum(a[..., :, k, None] * b[..., None, k, :] for k in range(3))


def _dag(a):
    return a.transpose(-1, -2).conj()


def _su3(w):
    """Polar projection (Newton) and division by the cube root of the determinant."""
    for _ in range(14):
        r = w.unbind(-2)
        cof = [r[(i + 1) % 3][..., [1, 2, 0]] * r[(i + 2) % 3][..., [2, 0, 1]]
               - r[(i + 1) % 3][..., [2, 0, 1]] * r[(i + 2) % 3][..., [1, 2, 0]] for i in range(3)]
        det = (r[0] * cof[0]).sum(-1)
        w = 0.5 * (w + (torch.stack(cof, -2) / det[..., None, None]).conj())
    r = w.unbind(-2)
    det = (r[0] * (r[1][..., [1, 2, 0]] * r[2][..., [2, 0, 1]] - r[1][..., [2, 0, 1]] * r[2][..., [1, 2, 0]])).sum(-1)
    return w * torch.polar(torch.ones_like(det.real), -det.angle() / 3)[..., None, None]


def _gauge(dims, eps, seed):
    """Links [t][z][y][x][mu][3][3]: exp(i eps sum_a h_a lambda_a / 2), then the APE steps."""
    lx, ly, lz, lt = dims
    h = torch.randn((lt, lz, ly, lx, 4, 8), generator=_rng(seed, 1), dtype=torch.float64, device=_dev())
    m = torch.zeros(h.shape[:-1] + (3, 3), dtype=torch.complex128, device=h.device)
    for a, (i, j) in enumerate(((0, 1), (0, 2), (1, 2))):
        z = torch.complex(h[..., 2 * a], -h[..., 2 * a + 1])
        m[..., i, j], m[..., j, i] = z, z.conj()
    m[..., 0, 0], m[..., 1, 1] = h[..., 6] + h[..., 7] / 3 ** 0.5, h[..., 7] / 3 ** 0.5 - h[..., 6]
    m[..., 2, 2] = -2 * h[..., 7] / 3 ** 0.5
    m = m * (0.5j * eps / 16)
    u = one = torch.eye(3, dtype=torch.complex128, device=h.device)
    for k in range(10, 0, -1):   # Taylor series of the sixteenth, then four squarings
        u = one + _mm(m, u.expand_as(m)) / k
    for _ in range(4):
        u = _mm(u, u)
    del m, h
    u = list(u.unbind(4))
    for _ in range(APE_STEPS):
        new = []
        for mu in range(4):
            s = 0
            for nu in range(4):
                if nu != mu:
                    s = s + _mm(_mm(u[nu], u[mu].roll(-1, 3 - nu)), _dag(u[nu].roll(-1, 3 - mu)))
                    d = u[nu].roll(1, 3 - nu)
                    s = s + _mm(_mm(_dag(d), u[mu].roll(1, 3 - nu)), d.roll(-1, 3 - mu))
            new.append(_su3(0.5 * u[mu] + s / 12))
        u = new
    return torch.stack(u, 4).contiguous()


def _spinors(dims, n, seed, what):
    """n Gaussian vectors, Re and Im ~ N(0, 1/2), shape (n, t, z, y, x, 4, 3)."""
    lx, ly, lz, lt = dims
    return torch.randn((n, lt, lz, ly, lx, 4, 3), generator=_rng(seed, what), dtype=torch.complex128, device=_dev())


def _null_vectors(c, U, seed):
    """Smoothed random vectors, representable in FP32: Richardson steps on the operator."""
    W = Wilson(U, c["m0"] + 0.05, CSW)
    v = _spinors(_dims(c), c["nv"], seed, 7)
    for _ in range(3):
        v -= W.D(v) / 6.0
    return v.to(torch.complex64).to(torch.complex128).contiguous()


def _inputs(c, seed):
    """The tensors of a case, which prepare() and exact() share."""
    k, dims = c["kind"], _dims(c)
    st = {"U": _gauge(dims, c["eps"], seed)}
    if k == "force":
        st["lam"], st["psi"] = _spinors(dims, 2, seed, 3)
    elif k == "remass":
        st["V"] = _null_vectors(c, st["U"], seed)
    else:
        n = c.get("nrhs", 1)
        x = _spinors(dims, n, seed, 2)
        st["eta"] = x if n > 1 else x[0].contiguous()
    if k == "grad":
        st["chi"] = _spinors(dims, 1, seed, 4)[0].contiguous()
    return st


def _operator(S, c):
    if c.get("aniso"):
        S.set_clover_aniso(ANISO_W, CSW, ANISO_CSW_T, c["m0"])
    else:
        S.set_clover(CSW, c["m0"])


def prepare(c, seed):
    st = _inputs(c, seed)
    k = c["kind"]
    S = st["S"] = Solver(_dims(c))
    st["case"] = c
    if "levels" in c:
        blocks = [tuple(c[b] for b in ("bx", "by", "bz", "bt"))] + [(2, 2, 2, 2)] * (c["levels"] - 2)
        S.set_params(levels=c["levels"], blocks=blocks, nv=[c["nv"], c["nv2"]][:c["levels"] - 1], storage=c["storage"],
                     seed=1000 + seed % 1000, **MG)
    else:
        S.set_params(levels=1, maxit_fine=MG["maxit_fine"])
    if k == "fresh":
        return st
    S.load_gauge(st["U"])
    if k == "remass":
        S.set_clover(CSW, c["m0"] + 0.05)
        S.set_null_vectors(0, st.pop("V"))
        S.setup()
        (lx, ly, lz, lt), nc = S.level_info(1)
        st["Y"] = torch.empty((lt, lz, ly, lx, 8, nc, nc), dtype=torch.complex128, device=st["U"].device)
        st["X"] = torch.empty((lt, lz, ly, lx, nc, nc), dtype=torch.complex128, device=st["U"].device)
        return st
    _operator(S, c)
    if k in ("solve", "grad"):
        S.setup()
    if k == "grad":
        st["eta"].requires_grad_(True)
        st["U"].requires_grad_(True)
    return st


# --------------------------------------------------------------------------- one pass
def run(st):
    S, c = st["S"], st["case"]
    k = c["kind"]
    if k == "op":
        out = S.apply(OPS[c["op"]], st["eta"], prec=c["prec"], nrhs=c["nrhs"])
        return out if c["prec"] == B.MG_FP64 else out.to(torch.complex64)
    if k == "force":
        kind = (B.MG_FORCE_SU3 if c["su3"] else B.MG_FORCE_WIRTINGER)
        out = S.force(st["lam"], st["psi"], kind | (0 if c["prec"] == B.MG_FP64 else B.MG_FORCE_FP32))
        return out if c["prec"] == B.MG_FP64 else out.to(torch.complex64)
    if k == "solve":
        return S.solve(st["eta"], TOL)[0]
    if k == "krylov":
        return S.solve(st["eta"], TOL, B.MG_MODE_BICGSTAB_MP)[0]
    if k == "grad":
        psi = dirac_solve(S, st["eta"], st["U"], TOL)
        loss = (st["chi"].conj() * psi).real.sum()
        return (psi.detach(),) + torch.autograd.grad(loss, (st["eta"], st["U"]))
    if k == "remass":
        S.update_mass(c["m0"])
        B.mg_get_coarse_links(S.ctx, 1, st["Y"], st["X"])
        return st["Y"].to(torch.complex64), st["X"].to(torch.complex64)
    S.load_gauge(st["U"])
    _operator(S, c)
    S.setup()
    return S.solve(st["eta"], TOL)[0]


# --------------------------------------------------------------------------- the same in 64 bits
# gamma_mu psi: component s is phase[s] psi[perm[s]]
GAMMA = (((3, 2, 1, 0), (1j, 1j, -1j, -1j)), ((3, 2, 1, 0), (-1, 1, 1, -1)), ((2, 3, 0, 1), (1j, -1j, -1j, 1j)),
         ((2, 3, 0, 1), (1, 1, 1, 1)))
PLANES = tuple((m, n) for m in range(4) for n in range(m + 1, 4))


def _gamma(mu, psi):
    perm, phase = GAMMA[mu]
    ph = torch.tensor([complex(p) for p in phase], dtype=psi.dtype, device=psi.device)
    return psi[..., list(perm), :] * ph[:, None]


def _shift(psi, mu, d):
    """psi(x + d mu) for vectors (n, t, z, y, x, ...), antiperiodic in t."""
    r = psi.roll(-d, 4 - mu)
    if mu == 3:
        r = torch.cat((r[:, :-1], -r[:, -1:]) if d > 0 else (-r[:, :1], r[:, 1:]), 1)
    return r


def _colour(u, psi):
    """u psi for links (t, z, y, x, 3, 3) and vectors (n, t, z, y, x, 4, 3)."""
    return sum(u[..., None, :, b] * psi[..., :, b, None] for b in range(3))


class Wilson:
    """The Wilson-clover operator on whole vectors (n, t, z, y, x, 4, 3), complex128."""

    def __init__(self, U, m0, csw, weights=(1.0,) * 4, csw_t=None):
        self.U, self.w = U, weights
        u = U.unbind(4)
        eye = torch.eye(4, dtype=torch.complex128, device=U.device)[:, :, None]
        g = [_gamma(mu, eye)[..., 0] for mu in range(4)]   # row i: gamma_mu of the unit spinor i
        blocks = 0
        for mu, nu in PLANES:
            sig = 1j * (g[nu] @ g[mu]).T                    # i gamma_mu gamma_nu
            cf = 0.5j * (csw if nu != 3 or csw_t is None else csw_t)
            F = self._field(u, mu, nu)
            blocks = blocks + torch.stack([cf * torch.einsum("st,...ac->...satc", sig[2 * b:2 * b + 2, 2 * b:2 * b + 2], F)
                                           for b in range(2)], 4)
        A = blocks.reshape(U.shape[:4] + (2, 6, 6))
        self.A = A + (sum(weights) + m0) * torch.eye(6, dtype=torch.complex128, device=U.device)
        self.Ainv = None
        t, z, y, x = torch.meshgrid(*(torch.arange(n, device=U.device) for n in U.shape[:4]), indexing="ij")
        self.even = ((t + z + y + x) % 2 == 0).to(torch.complex128)[..., None, None]

    @staticmethod
    def _field(u, mu, nu):
        def at(m, *steps):
            v = u[m]
            for d, s in steps:
                v = v.roll(-s, 3 - d)
            return v

        q = _mm(_mm(u[mu], at(nu, (mu, 1))), _dag(_mm(u[nu], at(mu, (nu, 1)))))
        q = q + _mm(_mm(u[nu], _dag(_mm(at(nu, (mu, -1)), at(mu, (nu, 1), (mu, -1))))), at(mu, (mu, -1)))
        q = q + _mm(_dag(_mm(at(nu, (mu, -1), (nu, -1)), at(mu, (mu, -1)))), _mm(at(mu, (mu, -1), (nu, -1)), at(nu, (nu, -1))))
        q = q + _mm(_mm(_dag(at(nu, (nu, -1))), at(mu, (nu, -1))), _mm(at(nu, (nu, -1), (mu, 1)), _dag(u[mu])))
        f = (q - _dag(q)) / 8
        tr = f.diagonal(dim1=-2, dim2=-1).sum(-1) / 3
        return f - tr[..., None, None] * torch.eye(3, dtype=f.dtype, device=f.device)

    def inverse(self):
        if self.Ainv is None:
            f = self.A.reshape(-1, 6, 6)
            self.Ainv = torch.cat([torch.linalg.inv(x) for x in f.split(1 << 18)]).reshape(self.A.shape)
        return self.Ainv

    @staticmethod
    def _blocks(A, psi):
        v = psi.reshape(psi.shape[:-2] + (2, 6))
        return sum(A[..., :, j] * v[..., j, None] for j in range(6)).reshape(psi.shape)

    def M(self, psi):
        return self._blocks(self.A, psi)

    def Minv(self, psi):
        return self._blocks(self.inverse(), psi)

    def hop_dir(self, psi, d):
        """d < 4: the term from x + mu, d >= 4: from x - mu, with its -1/2."""
        mu = d & 3
        u = self.U[..., mu, :, :]
        if d < 4:
            v = _colour(u, _shift(psi, mu, 1))
            return -0.5 * self.w[mu] * (v - _gamma(mu, v))
        v = _shift(_colour(_dag(u), psi), mu, -1)
        return -0.5 * self.w[mu] * (v + _gamma(mu, v))

    def H(self, psi):
        return sum(self.hop_dir(psi, d) for d in range(8))

    def D(self, psi):
        return self.M(psi) + self.H(psi)

    def Dr(self, y):
        y = self.even * y
        return y - self.even * self.H(self.Minv((1 - self.even) * self.H(self.Minv(y))))

    def br(self, b):
        return self.even * (b - self.H(self.Minv((1 - self.even) * b)))

    def solve(self, b):
        """D^{-1} b: BiCGStab on the even-odd reduced system, refined on the residual of D."""
        def dot(p, q):
            return (p.conj() * q).sum(tuple(range(1, q.dim())), keepdim=True)

        def reduced(b):
            x = torch.zeros_like(b)
            r = self.br(b)
            goal = 1e-9 * dot(b, b).real.sqrt()
            rh, p, v = r, torch.zeros_like(r), torch.zeros_like(r)
            rho = al = om = torch.ones_like(goal).to(b.dtype)
            for _ in range(2000):
                new = dot(rh, r)
                p = r + (new / rho) * (al / om) * (p - om * v)
                v, rho = self.Dr(p), new
                al = rho / dot(rh, v)
                s = r - al * v
                t = self.Dr(s)
                om = dot(t, s) / dot(t, t)
                x = x + al * p + om * s
                r = s - om * t
                if bool((dot(r, r).real.sqrt() <= goal).all()):
                    break
            xe = self.even * self.Minv(x)
            return xe + (1 - self.even) * self.Minv(b - self.H(xe))

        x = reduced(b)
        for _ in range(2):
            x = x + reduced(b - self.D(x))
        return x


def _galerkin(c, W, V):
    """The coarse operator of the block-orthonormalised, chirality-split vectors V: (Y, X)."""
    b = [c["bt"], c["bz"], c["by"], c["bx"]]
    n = [L // k for L, k in zip(V.shape[1:5], b)]
    nv, nb = c["nv"], math.prod(b)

    def split(v):      # (m, t, z, y, x, 4, 3) -> (coarse sites, chirality, 6 nb, m)
        m = v.shape[0]
        v = v.reshape(m, n[0], b[0], n[1], b[1], n[2], b[2], n[3], b[3], 2, 6)
        return v.permute(1, 3, 5, 7, 9, 2, 4, 6, 8, 10, 0).reshape(math.prod(n), 2, 6 * nb, m)

    def join(p):       # the inverse of split
        m = p.shape[-1]
        p = p.reshape(n + [2] + b + [6, m]).permute(10, 0, 5, 1, 6, 2, 7, 3, 8, 4, 9)
        return p.reshape((m,) + tuple(V.shape[1:5]) + (4, 3))

    Q, R = torch.linalg.qr(split(V))
    ph = R.diagonal(dim1=-2, dim2=-1)
    P = Q * (ph / ph.abs())[..., None, :]
    pos = torch.meshgrid(*(torch.arange(L, device=V.device) % k for L, k in zip(V.shape[1:5], b)), indexing="ij")
    Y = torch.zeros(math.prod(n), 8, 2 * nv, 2 * nv, dtype=V.dtype, device=V.device)
    X = torch.zeros(math.prod(n), 2 * nv, 2 * nv, dtype=V.dtype, device=V.device)
    for ch in range(2):
        for k0 in range(0, nv, 4):
            col = torch.zeros_like(P[..., k0:k0 + 4])
            col[:, ch] = P[:, ch, :, k0:k0 + 4]
            p = join(col)
            u = W.Minv(p)
            inside = p
            to = slice(ch * nv + k0, ch * nv + min(k0 + 4, nv))

            def project(v):
                return (P.transpose(-1, -2).conj() @ split(v)).reshape(math.prod(n), 2 * nv, -1)

            for d in range(8):
                mu, ax = d & 3, 3 - (d & 3)
                face = pos[ax] == (b[ax] - 1 if d < 4 else 0)
                face = (face & (n[ax] > 1)).to(V.dtype)[..., None, None]
                w = W.hop_dir(u, d)
                inside = inside + (1 - face) * w
                Y[:, d, :, to] = project(face * w)
            X[:, :, to] = project(inside)
    return Y.reshape(n + [8, 2 * nv, 2 * nv]), X.reshape(n + [2 * nv, 2 * nv])


def _link_gradient(W_of, U, lam, psi):
    """d/dRe U + i d/dIm U of -Re <lam, D(U) psi>."""
    U = U.detach().clone().requires_grad_(True)
    f = -(lam.conj() * W_of(U).D(psi[None])[0]).real.sum()
    return torch.autograd.grad(f, U)[0]


def exact(c, seed):
    st = _inputs(c, seed)
    U, k = st["U"], c["kind"]

    def wilson(u):
        if c.get("aniso"):
            return Wilson(u, c["m0"], CSW, ANISO_W, ANISO_CSW_T)
        return Wilson(u, c["m0"], CSW)

    if k == "force":
        g = _link_gradient(wilson, U, st["lam"], st["psi"])
        if not c["su3"]:
            return g
        h = 1j * _mm(U, _dag(g))
        h = 0.5 * (h + _dag(h))
        tr = h.diagonal(dim1=-2, dim2=-1).sum(-1) / 3
        return 0.5 * (h - tr[..., None, None] * torch.eye(3, dtype=h.dtype, device=h.device))
    W = wilson(U)
    if k == "remass":
        return _galerkin(c, W, st["V"])
    eta = st["eta"] if st["eta"].dim() == 7 else st["eta"][None]
    if k == "op":
        f = {"D": W.D, "DP": lambda x: x + W.H(W.Minv(x)), "DR": W.Dr, "BR": W.br, "M": W.M, "MINV": W.Minv, "HOP": W.H}
        return torch.cat([f[c["op"]](eta[i:i + 1]) for i in range(eta.shape[0])]).reshape(st["eta"].shape)
    if c["eps"] < 1.0:
        # the nearly free field at a negative mass: the spectrum surrounds the origin and no plain
        # Krylov solver converges
        return None
    psi = W.solve(eta)
    if k != "grad":
        return psi.reshape(st["eta"].shape)
    g5 = torch.tensor([1.0, 1.0, -1.0, -1.0], dtype=torch.float64, device=U.device)[:, None]
    lam = g5 * W.solve(g5 * st["chi"][None])
    return psi[0], lam[0], _link_gradient(wilson, U, lam[0], psi[0])
