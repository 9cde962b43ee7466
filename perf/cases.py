"""Performance cases of the DD-alpha-AMG library: what a user of the package has it do,
through the binding's public entry points, from the smallest call to a whole propagator.

A case is a dict of plain values.  Its lattice is t x x x y x z; eps, kappa, c_sw and mu are those
of the benchmark's workloads at the nearest size.  Kinds of pass:

* apply_d    ddtm_apply_D on canonical FP64 spinors (a residual check of a user's program);
* chain_d    `applies` applications of D(+mu), D(-mu), ... between two device-resident fields
             (what a user's own Krylov or spectral method does), then the export;
* sap        the red-black SAP smoother on a device-resident batch, then the export;
* sap_canon  the same on canonical spinors, one call;
* transfer   restriction to the coarse lattice and prolongation back;
* coarse     the coarse operator D_c on a batch of coarse vectors;
* rebuild    a new gauge field under the kept test vectors: load, Galerkin product, one D_c
             application (the HMC usage without inverse iterations);
* solve      D(mu) x = b with a hierarchy in hand (two or three levels);
* propagator adaptive setup and the solve.

Results come in the type of the computation that was asked for: FP64 operators and solves as
complex128, FP32 ones as complex64, FP16-storage ones as complex32.  The library exports FP64 only;
a program that keeps many such fields keeps them in the precision they have.
"""

import math

import torch

from paper_1610_02370_gb300 import ddtm, synth

F64, F32, F16 = ddtm.PREC_F64, ddtm.PREC_F32, ddtm.PREC_F16
OUT = {F64: torch.complex128, F32: torch.complex64, F16: torch.complex32}

# ensembles of the benchmark, by lattice size: (sites up to, eps, kappa, mu); c_sw 1.5755 for all
ENSEMBLES = ((1 << 18, 0.2, 0.1340, 0.003), (1 << 20, 0.15, 0.1370, 0.002), (1 << 40, 0.12, 0.1372, 0.0015))
C_SW = 1.5755
# the benchmark's multigrid parameters
MG = dict(n_setup=6, post_smooth=2, nmr=3, outer_restart=30, outer_tol=1e-10)


def _dims(c):
    return (c["t"], c["x"], c["y"], c["z"])


def _block(c):
    return (c["bt"], c["bx"], c["by"], c["bz"])


def _sites(c):
    return c["t"] * c["x"] * c["y"] * c["z"]


def _case(kind, dims, nrhs, block=(4, 4, 4, 4), **more):
    c = dict(kind=kind, t=dims[0], x=dims[1], y=dims[2], z=dims[3], bt=block[0], bx=block[1], by=block[2], bz=block[3],
             nrhs=nrhs)
    c.update(more)
    return c


def listed():
    L16, L24, L32 = (32, 16, 16, 16), (48, 24, 24, 24), (64, 32, 32, 32)
    named = [
        # the smallest call: one FP64 application on a small lattice, where launches and allocations count
        ("apply_d_f64_16x8x8x8", _case("apply_d", (16, 8, 8, 8), 1, prec=F64)),
        # one field, FP32: the operator of a single-source Krylov method
        ("chain_d_f32_24x24x24x48", _case("chain_d", L24, 1, prec=F32, applies=4)),
        # the 12 sources of a propagator in one batch, in both storage precisions
        ("chain_d_f32_24x24x24x48_12rhs", _case("chain_d", L24, 12, prec=F32, applies=4)),
        ("chain_d_f16_32x32x32x64_12rhs", _case("chain_d", L32, 12, prec=F16, applies=4)),
        # the smoother as the solver runs it: 2 cycles of 3 MR steps, FP16 storage, 12 sources
        ("sap_f16_24x24x24x48_12rhs", _case("sap", L24, 12, prec=F16, cycles=2, nmr=3)),
        # the smoother on one FP32 vector of a small lattice, one call on canonical spinors
        ("sap_f32_16x8x8x8", _case("sap_canon", (16, 8, 8, 8), 1, prec=F32, cycles=3, nmr=4)),
        # grid transfers of a propagator's batch
        ("transfer_24x24x24x48_12rhs", _case("transfer", L24, 12, nv=24)),
        # the coarse operator on the tensor cores
        ("coarse_f16_32x32x32x64_12rhs", _case("coarse", L32, 12, nv=24, coarse_prec=F16)),
        # a trajectory's new gauge field: operator and hierarchy rebuilt
        ("rebuild_16x16x16x32", _case("rebuild", L16, 12, nv=24, coarse_prec=F16)),
        # a single source on a small lattice: latency of the whole solver
        ("solve_16x8x8x8", _case("solve", (16, 8, 8, 8), 1, nv=24, nv1=0)),
        # the 12 sources of a propagator with the hierarchy in hand
        ("solve_24x24x24x48_12rhs", _case("solve", L24, 12, nv=24, nv1=0)),
        # a whole propagator: adaptive setup and 12 sources
        ("propagator_16x16x16x32", _case("propagator", L16, 12, nv=24, nv1=0)),
    ]
    return [dict(c, name=n) for n, c in named]


def _draw_dims(rng, lo, hi, unit=8):
    """A lattice of lo to hi sites, spread over the logarithm: every extent a multiple of `unit`."""
    target = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    while True:
        d = [unit * rng.randint(1, max(1, 64 // unit)) for _ in range(4)]
        v = math.prod(d)
        if lo <= v <= hi and 0.6 * target <= v <= 1.6 * target:
            return tuple(d)


def draw(rng):
    kind = rng.choice(("apply_d", "chain_d", "chain_d", "sap", "sap", "sap_canon", "transfer", "coarse", "rebuild", "solve",
                       "solve", "propagator"))
    nrhs = rng.choice((1, 2, 3, 4, 5, 7, 8, 11, 12, 12, 16, 24))
    nv = rng.choice((8, 12, 16, 20, 21, 24, 24, 28, 32))
    if kind in ("apply_d", "sap_canon"):
        small = rng.random() < 0.3  # blocks smaller than 4^4, on lattices they fit
        block = rng.choice(((2, 2, 2, 2), (4, 2, 4, 2), (2, 4, 4, 4))) if small else (4, 4, 4, 4)
        dims = _draw_dims(rng, 8 ** 4, 8 ** 5 if small else 32 * 16 ** 3)
        prec = rng.choice((F64, F32, F16))
        steps = {} if kind == "apply_d" else dict(cycles=rng.randint(1, 4), nmr=rng.randint(2, 5))
        return _case(kind, dims, min(nrhs, 4), block, prec=prec, **steps)
    if kind == "chain_d":
        dims = _draw_dims(rng, 8 ** 4, min(1, 4 / nrhs) * 64 * 32 ** 3)
        return _case(kind, dims, nrhs, prec=rng.choice((F32, F16)), applies=rng.randint(2, 4))
    if kind == "sap":
        dims = _draw_dims(rng, 8 ** 4, 48 * 24 ** 3 * 12 // max(nrhs, 12))
        return _case(kind, dims, nrhs, prec=rng.choice((F32, F16, F16)), cycles=rng.randint(1, 4), nmr=rng.randint(2, 5))
    if kind == "transfer":
        return _case(kind, _draw_dims(rng, 8 ** 4, 48 * 24 ** 3 * 12 // max(nrhs, 12)), nrhs, nv=nv)
    if kind == "coarse":
        return _case(kind, _draw_dims(rng, 8 ** 4, 48 * 24 ** 3), nrhs, nv=nv, coarse_prec=rng.choice((F32, F16, F16)))
    if kind == "rebuild":
        return _case(kind, _draw_dims(rng, 8 ** 4, 32 * 16 ** 3), min(nrhs, 12), nv=nv, coarse_prec=rng.choice((F32, F16, F16)))
    nrhs = min(nrhs, 12)
    # three levels need an even number of 2^4 blocks of the 4^4 aggregates in every direction
    three = kind == "solve" and rng.random() < 0.25
    dims = _draw_dims(rng, 16 ** 4, 32 * 16 ** 3, 16) if three else _draw_dims(rng, 8 ** 4, 32 * 16 ** 3)
    return _case(kind, dims, nrhs, nv=rng.choice((20, 24, 24, 28)), nv1=rng.choice((24, 32)) if three else 0)


# ---- inputs ---------------------------------------------------------------------------------

def _ensemble(c):
    for top, eps, kappa, mu in ENSEMBLES:
        if _sites(c) <= top:
            return eps, kappa, mu
    raise ValueError("lattice too large")


def _lat(c):
    return (c["t"], c["z"], c["y"], c["x"])


def _coarse_lat(c):
    return (c["t"] // c["bt"], c["z"] // c["bz"], c["y"] // c["by"], c["x"] // c["bx"])


def _links(c, seed):
    """U_mu(x) = exp(i eps H), H traceless Hermitian Gaussian as in synth.gauge_field, the exponential by
    16 Taylor terms in Horner form (|eps H| is about 1 at most: remainder below 1e-14)."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    a = torch.randn(_lat(c) + (4, 3, 3, 2), generator=g, dtype=torch.float64, device="cuda")
    A = torch.view_as_complex(a)
    H = 0.5 * (A + A.mH)
    eye = torch.eye(3, dtype=H.dtype, device=H.device)
    H = 1j * _ensemble(c)[0] * (H - torch.diagonal(H, dim1=-2, dim2=-1).sum(-1)[..., None, None] / 3.0 * eye)
    U = eye.expand(H.shape)
    for k in range(16, 0, -1):
        U = eye + sum(H[..., :, b, None] * U[..., None, b, :] for b in range(3)) / k
    return U.contiguous()


def _spinors(c, seed):
    return synth.gaussian_spinor(_dims(c), seed=seed + 1, nrhs=c["nrhs"], device="cuda")


def _test_vectors(c, seed):
    return synth.gaussian_vectors((c["nv"],) + _lat(c) + (4, 3), seed=seed + 2, device="cuda")


def _coarse_vectors(c, seed):
    return synth.gaussian_vectors((c["nrhs"],) + _coarse_lat(c) + (2 * c["nv"],), seed=seed + 3, device="cuda")


def _sources(c, seed):
    """Spin-colour point sources at a site drawn from the seed, scaled to distinct norms."""
    g = torch.Generator()
    g.manual_seed(seed + 4)
    site = tuple(int(torch.randint(0, n, (1,), generator=g)) for n in _dims(c))
    scale = 0.5 + torch.rand(12, generator=g, dtype=torch.float64)
    b = synth.point_sources(_dims(c), site=site, device="cuda")
    b *= scale.to("cuda").view(12, 1, 1, 1, 1, 1, 1)
    return b[: c["nrhs"]].contiguous()


class _State:
    """The library handles of one state; they are given back with it."""

    def __init__(self, c):
        self.case, self.ctx, self.fields = c, ddtm.ddtm_create(_dims(c), _block(c), 0), []

    def field(self):
        f = ddtm.ddtm_field_create(self.ctx, self.case["prec"], self.case["nrhs"])
        self.fields.append(f)
        return f

    def params(self, **kw):
        p = ddtm.ddtm_get_params(self.ctx)
        for k, v in kw.items():
            setattr(p, k, v)
        if self.case.get("nv1"):
            p.n_levels = 3
            p.nv[1] = self.case["nv1"]
        if "nv" in self.case:
            p.nv[0] = self.case["nv"]
        ddtm.ddtm_set_params(self.ctx, p)

    def __del__(self):
        if self.ctx:
            for f in self.fields:
                ddtm.ddtm_field_destroy(f)
            ddtm.ddtm_destroy(self.ctx)
            self.ctx = None


def prepare(case, seed):
    s = _State(case)
    kind = case["kind"]
    _, kappa, s.mu = _ensemble(case)
    s.seed = seed
    s.U = _links(case, seed)
    ddtm.ddtm_load_gauge(s.ctx, s.U, kappa, C_SW)
    s.kappa = kappa
    if kind in ("transfer", "coarse", "rebuild"):
        s.params(coarse_prec=case.get("coarse_prec", F16))
        ddtm.ddtm_set_test_vectors(s.ctx, 0, _test_vectors(case, seed), case["nv"])
    if kind in ("solve", "propagator"):
        s.params(smoother_prec=F16, coarse_prec=F16, **MG)
    if kind in ("apply_d", "sap_canon"):
        s.x = _spinors(case, seed)
        s.y = torch.zeros_like(s.x)
    elif kind in ("chain_d", "sap"):
        x = _spinors(case, seed)
        s.fx, s.fy = s.field(), s.field()
        s.fz = s.field() if kind == "chain_d" else None
        ddtm.ddtm_field_import(s.ctx, s.fx, x)
        s.y = x
    elif kind == "transfer":
        s.x = _spinors(case, seed)
        s.y = torch.zeros_like(s.x)
        s.c = torch.zeros_like(_coarse_vectors(case, seed))
    elif kind in ("coarse", "rebuild"):
        s.x = _coarse_vectors(case, seed)
        s.y = torch.zeros_like(s.x)
        if kind == "rebuild":
            s.U = _links(case, seed + 1000003)
    else:
        s.x = _sources(case, seed)
        s.y = torch.zeros_like(s.x)
        if kind == "solve":
            ddtm.ddtm_setup(s.ctx, s.mu, seed)
    if kind != "rebuild":
        s.U = None
    torch.cuda.synchronize()
    return s


def run(s):
    c, kind = s.case, s.case["kind"]
    n = c["nrhs"]
    if kind == "apply_d":
        ddtm.ddtm_apply_D(s.ctx, s.y, s.x, n, s.mu, c["prec"])
        return s.y.to(OUT[c["prec"]])
    if kind == "sap_canon":
        ddtm.ddtm_sap(s.ctx, s.y, s.x, n, s.mu, c["cycles"], c["nmr"], c["prec"])
        return s.y.to(OUT[c["prec"]])
    if kind == "chain_d":
        src, dst = s.fx, s.fy
        for k in range(c["applies"]):
            ddtm.ddtm_apply_D_field(s.ctx, dst, src, s.mu if k % 2 == 0 else -s.mu)
            src, dst = dst, (s.fz if dst is s.fy else s.fy)
        ddtm.ddtm_field_export(s.ctx, src, s.y)
        return s.y.to(OUT[c["prec"]])
    if kind == "sap":
        ddtm.ddtm_sap_field(s.ctx, s.fy, s.fx, s.mu, c["cycles"], c["nmr"])
        ddtm.ddtm_field_export(s.ctx, s.fy, s.y)
        return s.y.to(OUT[c["prec"]])
    if kind == "transfer":
        ddtm.ddtm_restrict(s.ctx, 0, s.c, s.x, n)
        ddtm.ddtm_prolong(s.ctx, 0, s.y, s.c, n)
        return {"coarse": s.c.to(torch.complex64), "fine": s.y.to(torch.complex64)}
    if kind == "coarse":
        ddtm.ddtm_apply_Dc(s.ctx, 1, s.y, s.x, n, s.mu)
        return s.y.to(OUT[c["coarse_prec"]])
    if kind == "rebuild":
        ddtm.ddtm_load_gauge(s.ctx, s.U, s.kappa, C_SW)
        ddtm.ddtm_build_coarse(s.ctx)
        ddtm.ddtm_apply_Dc(s.ctx, 1, s.y, s.x, n, s.mu)
        return s.y.to(OUT[c["coarse_prec"]])
    if kind == "propagator":
        ddtm.ddtm_setup(s.ctx, s.mu, s.seed)
    ddtm.ddtm_solve(s.ctx, s.y, s.x, n, s.mu)
    return s.y


# ---- what a pass cannot do without -------------------------------------------------------------

def _dslash_flops(sites):
    """8 hops (projection, two 3x3 products, reconstruction), the clover term and the twist."""
    return 1920.0 * sites


def work(case):
    V, R, kind = float(_sites(case)), case["nrhs"], case["kind"]
    Nc = V / math.prod(_block(case))
    canon = 192.0 * V * R
    size = {F64: 16.0, F32: 8.0, F16: 4.0}
    if kind == "apply_d":
        op = 72 * V * size[case["prec"]]
        return {"bytes": 2 * canon + op, "flops": _dslash_flops(V) * R}
    if kind == "chain_d":
        sp = size[case["prec"]]
        field = 12 * V * R * sp
        return {"bytes": case["applies"] * (72 * V * sp + 2 * field) + 2 * field, "flops": case["applies"] * _dslash_flops(V) * R}
    if kind in ("sap", "sap_canon"):
        sp = size[case["prec"]]
        field, op = 12 * V * R * sp, 108 * V * sp  # links, clover, even-site inverses
        ends = 2 * canon if kind == "sap_canon" else 2 * field
        # per cycle both colours once; each reads the operator and the right-hand side of its blocks and
        # the whole of x, and writes its half of x
        return {"bytes": case["cycles"] * (op + 4 * field) + ends,
                "flops": case["cycles"] * (case["nmr"] + 1) * _dslash_flops(V) * R}
    if kind == "transfer":
        P = 12 * V * case["nv"] * 8
        return {"bytes": 2 * P + 2 * canon, "flops": 2 * 8 * 12 * V * case["nv"] * R}
    n = 2 * case["nv"]
    cvec = 16 * Nc * n * R
    if kind == "coarse":
        return {"bytes": 9 * Nc * n * n * size[case["coarse_prec"]] + 2 * cvec, "flops": 9 * 8 * Nc * n * n * R}
    galerkin = n * _dslash_flops(V) / 2 + 8 * n * n * 6 * V * (1 + sum(2.0 / b for b in _block(case)))
    if kind == "rebuild":
        return {"bytes": 36 * 16 * V * 3 + 2 * 12 * V * case["nv"] * 8 + 9 * Nc * n * n * size[case["coarse_prec"]] + 2 * cvec,
                "flops": galerkin + 9 * 8 * Nc * n * n * R}
    # solve: a nominal 20 outer iterations, each one D, the smoother and the transfers on every
    # source, plus the FP64 residuals; the coarsest solve is left out (its work depends on the field)
    it = 20 * (MG["post_smooth"] * (MG["nmr"] + 1) + 1 + 0.1 * case["nv"]) * _dslash_flops(V) * R
    if kind == "propagator":
        it += MG["n_setup"] * galerkin + (MG["n_setup"] - 1) * MG["post_smooth"] * (MG["nmr"] + 1) * _dslash_flops(V) * case["nv"]
    return {"bytes": 20 * (108 * V * 4 + 12 * V * case["nv"] * 8 + 6 * 12 * V * R * 4) + 2 * canon, "flops": it}


# ---- the same results in 64 bits, by plain torch -------------------------------------------------

AXIS = (0, 3, 2, 1)  # array axis of direction t, x, y, z in (T, Z, Y, X, ...)


def _gammas():
    s = torch.zeros(3, 2, 2, dtype=torch.complex128)
    s[0, 0, 1] = s[0, 1, 0] = 1
    s[1, 0, 1], s[1, 1, 0] = -1j, 1j
    s[2, 0, 0], s[2, 1, 1] = 1, -1
    g = torch.zeros(4, 4, 4, dtype=torch.complex128)
    g[0, :2, 2:] = g[0, 2:, :2] = torch.eye(2)
    for k in range(3):
        g[k + 1, :2, 2:], g[k + 1, 2:, :2] = 1j * s[k], -1j * s[k]
    return g


def _roll(f, mu, sign):
    """F(x) = f(x + sign mu)."""
    return torch.roll(f, -sign, AXIS[mu])


class _Exact:
    """D(mu), SAP, aggregation and coarse operator of Sec. 2 of arXiv:1610.02370 in complex128."""

    def __init__(self, c, U, kappa):
        self.c, self.U = c, [U[..., m, :, :].contiguous() for m in range(4)]
        g = _gammas()
        self.proj = [[(torch.eye(4, dtype=torch.complex128) - d * g[m]).to(U.device) for d in (1, -1)] for m in range(4)]
        self.Ub = [_roll(self.U[m], m, -1).mH.contiguous() for m in range(4)]  # U_mu(x - mu)^+
        S = torch.zeros(U.shape[:4] + (4, 3, 4, 3), dtype=torch.complex128, device=U.device)
        for s in range(4):
            for a in range(3):
                S[..., s, a, s, a] = 1.0 / (2 * kappa)  # m + 4
        for mu in range(4):
            for nu in range(mu + 1, 4):
                Q = self._leaves(mu, nu)
                F = Q - Q.mH
                gg = (g[mu] @ g[nu]).to(U.device)
                for s in range(4):
                    for t in range(4):
                        if abs(complex(gg[s, t])) > 0:
                            S[..., s, :, t, :] -= C_SW / 16 * gg[s, t] * F
        self.S = S.reshape(U.shape[:4] + (12, 12))

    def _leaves(self, mu, nu):
        a, b, r = self.U[mu], self.U[nu], _roll
        am, bm = r(a, mu, -1), r(b, mu, -1)
        an, bn = r(a, nu, -1), r(b, nu, -1)
        return (a @ r(b, mu, 1) @ r(a, nu, 1).mH @ b.mH + b @ r(am, nu, 1).mH @ bm.mH @ am
                + am.mH @ r(bm, nu, -1).mH @ r(am, nu, -1) @ bn + bn.mH @ an @ r(bn, mu, 1) @ a.mH)

    def hop(self, psi, inside=None):
        """-1/2 sum over the 8 hops; `inside`: masks of the hops that stay in their block."""
        out = torch.zeros_like(psi)
        for mu in range(4):
            for d, sign in enumerate((1, -1)):
                p = torch.einsum("st,...ta->...sa", self.proj[mu][d], _roll(psi, mu, sign))
                M = self.U[mu] if sign > 0 else self.Ub[mu]
                w = sum(M[..., None, :, b] * p[..., :, b, None] for b in range(3))
                if inside is not None:
                    w *= inside[mu][d]
                out += w
        return out.mul_(-0.5)

    def site(self, psi, mu):
        out = (self.S @ psi.reshape(psi.shape[:4] + (12, 1))).reshape(psi.shape)
        out[..., :2, :] += 1j * mu * psi[..., :2, :]
        out[..., 2:, :] -= 1j * mu * psi[..., 2:, :]
        return out

    def D(self, psi, mu):
        return self.site(psi, mu) + self.hop(psi)

    def _coords(self):
        lat = _lat(self.c)
        at = torch.meshgrid(*[torch.arange(k, device=self.S.device) for k in lat], indexing="ij")
        return [at[AXIS[m]] for m in range(4)]

    def to_blocks(self, f):
        """(T, Z, Y, X, ...) -> (blocks, sites of a block, ...), blocks in canonical order."""
        c, n = self.c, _coarse_lat(self.c)
        rest = f.shape[4:]
        f = f.reshape((n[0], c["bt"], n[1], c["bz"], n[2], c["by"], n[3], c["bx"]) + rest)
        f = f.permute((0, 2, 4, 6, 1, 3, 5, 7) + tuple(range(8, 8 + len(rest))))
        return f.reshape((math.prod(n), math.prod(_block(c))) + rest)

    def from_blocks(self, f):
        c, n = self.c, _coarse_lat(self.c)
        rest = f.shape[2:]
        f = f.reshape(n + (c["bt"], c["bz"], c["by"], c["bx"]) + rest)
        f = f.permute((0, 4, 1, 5, 2, 6, 3, 7) + tuple(range(8, 8 + len(rest))))
        return f.reshape(_lat(c) + rest)

    def sap(self, b, mu, cycles, nmr):
        x, B = self._coords(), _block(self.c)
        one = torch.ones_like(x[0], dtype=torch.float64)[..., None, None]
        inside = [[one * (x[m] % B[m] != (B[m] - 1 if d == 0 else 0))[..., None, None] for d in range(2)] for m in range(4)]
        even = one * (sum(x) % 2 == 0)[..., None, None]
        odd = 1 - even
        colour = sum(x[m] // B[m] for m in range(4)) % 2
        A = self.S.reshape(self.S.shape[:4] + (2, 6, 2, 6))
        inv = []
        for h in range(2):
            M = A[..., h, :, h, :] + (1j * mu if h == 0 else -1j * mu) * torch.eye(6, dtype=A.dtype, device=A.device)
            inv.append(torch.linalg.inv(M))

        def ainv(v):
            w = v.reshape(v.shape[:4] + (2, 6, 1))
            return torch.stack([inv[h] @ w[..., h, :, :] for h in range(2)], dim=4).reshape(v.shape)

        z = torch.zeros_like(b)
        for _ in range(cycles):
            for col in range(2):
                m = one * (colour == col)[..., None, None]
                r = (b - self.D(z, mu)) * m
                te = ainv(r * even) * even
                rho = (r - self.hop(te, inside)) * odd
                eo = torch.zeros_like(rho)
                for _ in range(nmr):
                    t = ainv(self.hop(rho, inside)) * even
                    p = (self.site(rho, mu) - self.hop(t, inside)) * odd
                    pp, pr = self._block_dot(p, p).real, self._block_dot(p, rho)
                    alpha = torch.where(pp > 0, pr / torch.where(pp > 0, pp, torch.ones_like(pp)), torch.zeros_like(pr))
                    eo += alpha * rho
                    rho = rho - alpha * p
                z += eo + ainv((r - self.hop(eo, inside)) * even) * even
        return z

    def _block_dot(self, p, q):
        d = self.to_blocks((p.conj() * q).sum((-1, -2)))
        d = d.sum(1, keepdim=True).expand(-1, math.prod(_block(self.c)))
        return self.from_blocks(d)[..., None, None]

    def aggregate(self, v):
        """P per aggregate half: (2, blocks, 6 sites, nv), the QR factor with positive diagonal."""
        halves = []
        for s in range(2):
            cols = [self.to_blocks(v[i][..., 2 * s:2 * s + 2, :]).flatten(1) for i in range(v.shape[0])]
            M = torch.stack(cols, dim=2)
            for _ in range(2):  # Cholesky QR, twice
                C = torch.linalg.cholesky(M.mH @ M)
                M = torch.linalg.solve_triangular(C.mH, M, upper=True, left=False)
            halves.append(M)
        self.P = halves

    def restrict(self, f):
        parts = [(self.P[s].mH @ self.to_blocks(f[..., 2 * s:2 * s + 2, :]).flatten(1)[..., None])[..., 0] for s in range(2)]
        return torch.cat(parts, dim=1).reshape(_coarse_lat(self.c) + (-1,))

    def prolong(self, e):
        nv, e = self.c["nv"], e.reshape(-1, 2 * self.c["nv"])
        out = []
        for s in range(2):
            f = (self.P[s] @ e[:, s * nv:(s + 1) * nv, None])[..., 0]
            out.append(self.from_blocks(f.reshape(f.shape[0], -1, 2, 3)))
        return torch.cat(out, dim=4)

    def coarse(self, e, mu):
        y = self.restrict(self.D(self.prolong(e), 0.0))
        nv = self.c["nv"]
        y[..., :nv] += 1j * mu * e[..., :nv]
        y[..., nv:] -= 1j * mu * e[..., nv:]
        return y

    def solve(self, b, mu, tol=1e-13, most=600):
        """Conjugate gradients on D^+ D, restarted from the true residual; D^+ = Gamma5 D(-mu) Gamma5."""
        g5 = torch.tensor([1.0, 1.0, -1.0, -1.0], dtype=torch.float64, device=b.device)[:, None]

        def dag(v):
            return g5 * self.D(g5 * v, -mu)

        x = torch.zeros_like(b)
        nb = float(torch.linalg.vector_norm(b))
        for _ in range(4):
            res = b - self.D(x, mu)
            if float(torch.linalg.vector_norm(res)) <= tol * nb:
                break
            r = dag(res)
            p, rr, r0 = r.clone(), float(torch.linalg.vector_norm(r)) ** 2, float(torch.linalg.vector_norm(r))
            for _ in range(most):
                q = self.D(p, mu)
                a = rr / float(torch.linalg.vector_norm(q)) ** 2
                x += a * p
                r -= a * dag(q)
                new = float(torch.linalg.vector_norm(r)) ** 2
                if math.sqrt(new) <= 1e-8 * r0:
                    break
                p = r + (new / rr) * p
                rr = new
        return x


def exact(case, seed):
    kind, R = case["kind"], case["nrhs"]
    if kind in ("solve", "propagator") and _sites(case) * R > 16 * 8 ** 3 * 12:
        return None  # 64-bit solutions of larger systems take too long
    _, kappa, mu = _ensemble(case)
    E = _Exact(case, _links(case, seed + 1000003 if kind == "rebuild" else seed), kappa)
    if kind == "apply_d":
        return torch.stack([E.D(v, mu) for v in _spinors(case, seed)])
    if kind in ("sap", "sap_canon"):
        return torch.stack([E.sap(v, mu, case["cycles"], case["nmr"]) for v in _spinors(case, seed)])
    if kind == "chain_d":
        out = _spinors(case, seed)
        for r in range(R):
            v = out[r]
            for k in range(case["applies"]):
                v = E.D(v, mu if k % 2 == 0 else -mu)
            out[r] = v
        return out
    if kind in ("transfer", "coarse", "rebuild"):
        E.aggregate(_test_vectors(case, seed))
        if kind == "transfer":
            c = torch.stack([E.restrict(v) for v in _spinors(case, seed)])
            return {"coarse": c, "fine": torch.stack([E.prolong(e) for e in c])}
        return torch.stack([E.coarse(e, mu) for e in _coarse_vectors(case, seed)])
    return torch.stack([E.solve(v, mu) for v in _sources(case, seed)])
