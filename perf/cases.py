"""Performance cases: what programs built on this package call, over its range of sizes and options.

Each case is a dict of plain values.  listed() holds the fixed ones, draw() one more
of the same ranges; prepare() makes a program's inputs and handles, run() is one pass
through the public entry points, work() and tolerance() state what a pass needs and
how far a correct implementation may differ, and exact() gives the results in 64-bit
torch arithmetic from the definitions of the operator, the smoother and the force.

Kinds of case:
  dslash    the operator D, D^dagger (dagger) or QWS's A = C^-1 D on packed fields, as
            a Krylov loop calls it
  smoother  the SAP smoother with MR, even-odd MR ("eo") or Jacobi-on-A ("A") domain
            solves: on packed fields from zero, as a preconditioner calls it, or
            from a guess on canonical fields, as a relaxation of its own
  solve     D x = b to 1e-10 for one or several right-hand sides, any method
  batch     several lattices with several right-hand sides each, solved at once
  action    the fermion action and its gradient with respect to the links from a new
            gauge field: one force evaluation of a molecular-dynamics step
  multigrid a solve with a two-level multigrid that was set up before
"""
from __future__ import annotations

import math

import torch

from paper_2112_00501_gb300 import api
from paper_2112_00501_gb300.autograd import fermion_action

GAUSS = 0.5 ** 0.5
DEVICE = "cuda"


# ------------------------------------------------------------------ the cases
def _case(kind, dims, block=(4, 4, 4, 4), **kw):
    names = "xyzt"
    c = {"kind": kind}
    c.update({f"L{names[k]}": int(dims[k]) for k in range(4)})
    c.update({f"B{names[k]}": int(block[k]) for k in range(4)})
    c.update({"eps": 0.4, "kappa": 0.1355, "csw": 1.0, "prec": 32, "compress": 18, "nrhs": 1})
    c.update(kw)
    return c


def listed():
    heavy = {"eps": 0.5, "kappa": 0.1370, "prec": 16, "compress": 12}
    return [
        # the operator of a preconditioner's Krylov loop at the smallest storage, full lattice
        _case("dslash", (32, 32, 32, 64), name="dslash_fp16_32x32x32x64", dagger=False, op="D", **heavy),
        # D^dagger on several right-hand sides, odd block counts' worth of ragged extents
        _case("dslash", (20, 12, 28, 36), (2, 2, 2, 2), name="dslash_dagger_fp32_20x12x28x36_3rhs", dagger=True,
              op="D", nrhs=3, kappa=0.13),
        # the operator in full precision: residuals, eigenvalue and force codes
        _case("dslash", (24, 24, 24, 48), name="dslash_fp64_24x24x24x48", dagger=False, op="D", prec=64),
        # one preconditioner call (4 sweeps of 4 MR steps from zero) of the largest solve
        _case("smoother", (32, 32, 32, 64), name="smoother_fp16_32x32x32x64", solver="mr", n_cy=4, n_it=4,
              guess=False, **heavy),
        # relaxing a guess in single precision on a lattice that fits in the cache
        _case("smoother", (16, 16, 16, 32), name="smoother_fp32_guess_16x16x16x32", solver="mr", n_cy=2, n_it=4,
              guess=True, compress=12),
        # the even-odd preconditioned domain solver of the multigrid's literature
        _case("smoother", (24, 16, 16, 40), name="smoother_eo_fp32_24x16x16x40", solver="eo", n_cy=2, n_it=4,
              guess=False),
        # the ordinary large solve: half-precision smoother, single inner, double outer
        _case("solve", (32, 32, 32, 64), name="solve_mixed_32x32x32x64", method=2, guess=False, **heavy),
        # the smallest solve in use: latency, launches and host reads
        _case("solve", (8, 8, 8, 8), name="solve_fp32_8x8x8x8", method=2, guess=False),
        # everything in double precision, the reference solve of a validation run
        _case("solve", (16, 16, 16, 32), name="solve_fp64_16x16x16x32", method=0, guess=False, prec=64),
        # twelve sources of a propagator with ensembles of smaller lattices beside it
        _case("batch", (16, 16, 16, 32), name="batch_solve_fp32_12_4_8_systems", nrhs=12, L4_nrhs=4, L8_nrhs=8),
        # the fermion force of a molecular-dynamics step on a new gauge field
        _case("action", (24, 24, 24, 48), name="action_gradient_24x24x24x48"),
        # a solve with a multigrid kept from an earlier setup
        _case("multigrid", (24, 24, 24, 48), name="multigrid_solve_24x24x24x48", nvec=16, Ax=8, Ay=4, Az=4, At=4),
    ]


def _extent(rng, step, lo, hi):
    """a multiple of step in [lo, hi], even over its logarithm"""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min(max(step, round(v / step) * step), hi // step * step)


def _dims(rng, block, vmin, vmax):
    while True:
        top = 64
        d = [_extent(rng, 2 * b, max(4, 2 * b), top) for b in block]
        if vmin <= d[0] * d[1] * d[2] * d[3] <= vmax:
            return tuple(d)


def _storage(rng):
    prec = rng.choice((32, 32, 16, 64))
    return prec, (18 if prec == 64 else rng.choice((12, 18)))


def draw(rng):
    kind = rng.choice(("dslash", "dslash", "smoother", "smoother", "solve", "solve", "solve", "batch", "action",
                       "multigrid"))
    phys = {"eps": round(rng.uniform(0.4, 0.5), 3), "kappa": round(rng.uniform(0.125, 0.1365), 4),
            "csw": rng.choice((1.0, 1.0, 0.0))}
    block = rng.choice(((4, 4, 4, 4), (4, 4, 4, 4), (4, 4, 4, 4), (2, 2, 2, 2), (4, 2, 4, 8), (8, 4, 4, 4)))
    if kind == "dslash":
        prec, comp = _storage(rng)
        nrhs = rng.choice((1, 1, 2, 3, 5))
        op = rng.choice(("D", "D", "A"))
        return _case(kind, _dims(rng, block, 256, 2**20 // nrhs), block, prec=prec, compress=comp, nrhs=nrhs,
                     dagger=op == "D" and rng.random() < 0.4, op=op, **phys)
    if kind == "smoother":
        prec, comp = _storage(rng)
        solver = rng.choice(("mr", "mr", "eo", "A"))
        # the staged domain solvers of single and half precision hold one domain in shared memory
        if math.prod(block) > 256:
            block = (4, 4, 4, 4)
        return _case(kind, _dims(rng, block, 256, 2**19), block, prec=prec, compress=comp, solver=solver,
                     n_cy=rng.choice((1, 2, 4)), n_it=rng.choice((3, 4, 5)), guess=rng.random() < 0.4, **phys)
    if kind == "solve":
        method = rng.choice((2, 2, 0, 1, 3))
        prec, comp = _storage(rng)
        if method in (2, 3) and prec == 64:
            prec, comp = 32, 18
        if math.prod(block) > 256:
            block = (4, 4, 4, 4)
        return _case(kind, _dims(rng, block, 256, 2**17), block, prec=prec, compress=comp, method=method,
                     guess=rng.random() < 0.3, nrhs=rng.choice((1, 1, 2)), **phys)
    if kind == "batch":
        prec, comp = rng.choice(((32, 18), (32, 12), (16, 12)))
        return _case(kind, _dims(rng, (4, 4, 4, 4), 4096, 2**16), prec=prec, compress=comp,
                     nrhs=rng.randint(1, 6), L4_nrhs=rng.randint(0, 3), L8_nrhs=rng.randint(1, 6), **phys)
    if kind == "action":
        return _case(kind, _dims(rng, (4, 4, 4, 4), 4096, 2**18), prec=rng.choice((32, 16)), **phys)
    dims = _dims(rng, (4, 4, 4, 4), 4096, 2**17)
    return _case(kind, dims, prec=rng.choice((32, 16)), nvec=rng.choice((8, 12, 16)), Ax=4, Ay=4, Az=4, At=4, **phys)


def _geometry(case):
    return tuple(case[f"L{k}"] for k in "xyzt"), tuple(case[f"B{k}"] for k in "xyzt")


def _lattices(case):
    """(dims, right-hand sides) of every lattice of a case; a batch has a 16^4 and an 8^4 one beside its own"""
    dims, _ = _geometry(case)
    out = [(dims, case["nrhs"])]
    if case["kind"] == "batch":
        out += [((16,) * 4, case["L4_nrhs"])] * (case["L4_nrhs"] > 0)
        out += [((8,) * 4, case["L8_nrhs"])] * (case["L8_nrhs"] > 0)
    return out


# ------------------------------------------------------------------ inputs
def _generator(seed):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(int(seed) * 7919 + 13)
    return g


def _gauge_field(dims, eps, g):
    """Disordered SU(3) links exp(i eps H), H traceless Hermitian with unit-variance entries, reunitarised."""
    n = 4 * math.prod(dims)
    out = torch.empty((n, 3, 3), dtype=torch.complex128, device=DEVICE)
    chunk = 1 << 20
    for lo in range(0, n, chunk):
        m = min(chunk, n - lo)
        d = torch.randn((m, 3), dtype=torch.float64, device=DEVICE, generator=g)
        o = torch.randn((m, 3, 2), dtype=torch.float64, device=DEVICE, generator=g) * GAUSS
        h = torch.zeros((m, 3, 3), dtype=torch.complex128, device=DEVICE)
        oc = torch.view_as_complex(o)
        for k, (a, b) in enumerate(((0, 1), (0, 2), (1, 2))):
            h[:, a, b] = oc[:, k]
            h[:, b, a] = oc[:, k].conj()
        d = d - d.mean(dim=1, keepdim=True)
        for a in range(3):
            h[:, a, a] = d[:, a].to(torch.complex128)
        # Taylor series of exp(i eps H / 16), squared four times
        h = h * (1j * eps / 16)
        u = torch.eye(3, dtype=torch.complex128, device=DEVICE).expand(m, 3, 3)
        for k in range(9, 0, -1):
            u = torch.eye(3, dtype=torch.complex128, device=DEVICE) + _mm(h, u) / k
        for _ in range(4):
            u = _mm(u, u)
        r0 = u[:, 0] / torch.linalg.vector_norm(u[:, 0], dim=1, keepdim=True)
        r1 = u[:, 1] - (r0.conj() * u[:, 1]).sum(1, keepdim=True) * r0
        r1 = r1 / torch.linalg.vector_norm(r1, dim=1, keepdim=True)
        out[lo:lo + m, 0] = r0
        out[lo:lo + m, 1] = r1
        out[lo:lo + m, 2] = torch.linalg.cross(r0, r1, dim=1).conj()
    return out.reshape(-1, 4, 3, 3)


def _spinor(dims, g, nrhs=None):
    shape = (math.prod(dims), 4, 3, 2) if nrhs is None else (nrhs, math.prod(dims), 4, 3, 2)
    return torch.view_as_complex(torch.randn(shape, dtype=torch.float64, device=DEVICE, generator=g) * GAUSS)


def _fields(case, seed):
    """Per lattice: the links, the sources (nrhs, V, 4, 3) and a guess for each."""
    g = _generator(seed)
    out = []
    for dims, nrhs in _lattices(case):
        U = _gauge_field(dims, case["eps"], g)
        b = _spinor(dims, g, nrhs)
        out.append((dims, U, b, _spinor(dims, g, nrhs) if case.get("guess") else None))
    return out


def _operator(case, dims, U):
    block = _geometry(case)[1]
    lat = api.Lattice(dims, block, -1)
    gauge = api.Gauge(lat, U, storage_prec=case["prec"], compress=case["compress"])
    return api.CloverOperator(gauge, case["kappa"], case["csw"])


def _params(case, **kw):
    """solver parameters; the domain solves' precision is the storage's"""
    return dict(smoother_prec=case["prec"], **kw)


def prepare(case, seed):
    kind, prec = case["kind"], case["prec"]
    st = {"case": case}
    fields = _fields(case, seed)
    dims, U, b, x0 = fields[0]
    if kind == "action":
        # a new gauge field per step: the lattice is what a program keeps
        st["lat"] = api.Lattice(dims, _geometry(case)[1], -1)
        st["U"] = U.requires_grad_(True)
        st["phi"] = b[0]
        return st
    ops = [_operator(case, d, u) for d, u, _, _ in fields]
    op = st["op"] = ops[0]
    if kind == "batch":
        st["batch"] = api.Batch(ops, [f[2].shape[0] for f in fields])
        st["b"] = [f[2] for f in fields]
        st["x"] = [torch.empty_like(f[2]) for f in fields]
    elif kind == "dslash" or (kind == "smoother" and x0 is None):
        st["b"] = op.lattice.pack(b, prec)
        st["x"] = op.lattice.empty_packed(prec, case["nrhs"])
    elif kind == "smoother":
        st["b"], st["x0"] = b[0], x0[0]
    else:
        st["b"] = b if case["nrhs"] > 1 else b[0]
        if x0 is not None:
            st["x0"] = x0 if case["nrhs"] > 1 else x0[0]
        else:
            st["x"] = torch.empty_like(st["b"])
    if kind == "multigrid":
        mg = st["mg"] = api.Multigrid(op, tuple(case[f"A{k}"] for k in "xyzt"), case["nvec"])
        eta = _spinor(dims, _generator(seed + 1000003), case["nvec"])
        st["mgp"] = api.mg_params(smoother_prec=prec, n_adapt=2)
        mg.setup(eta, st["mgp"])
    return st


# ------------------------------------------------------------------ one pass
def _packed_views(buf, prec, sites):
    """A packed field as numbers: doubles, floats, or halves with their sites' scales."""
    if prec == 64:
        return buf.view(torch.float64)
    if prec == 32:
        return buf.view(torch.float32)
    return {"values": buf[:48 * sites].view(torch.float16), "scale": buf[48 * sites:52 * sites].view(torch.float32)}


def run(state):
    case = state["case"]
    kind, prec, nrhs = case["kind"], case["prec"], case["nrhs"]
    if kind == "action":
        S = fermion_action(state["U"], state["phi"], state["lat"], case["kappa"], case["csw"], **_params(case))
        (g,) = torch.autograd.grad(S, state["U"])
        return {"action": S.detach(), "gradient": g}
    op = state["op"]
    sites = nrhs * op.lattice.volume
    if kind == "dslash":
        f = op.apply_A if case["op"] == "A" else op.apply_Ddag if case["dagger"] else op.apply_D
        return _packed_views(f(state["b"], prec, nrhs, out=state["x"]), prec, sites)
    if kind == "smoother":
        if "x0" in state:
            f = {"mr": op.sap, "eo": op.sap_eo, "A": op.sap_A}[case["solver"]]
            return f(state["b"], prec, case["n_cy"], case["n_it"], x0=state["x0"])
        f = {"mr": op.sap_smooth, "eo": op.sap_smooth_eo, "A": op.sap_smooth_A}[case["solver"]]
        x = state["x"].zero_()
        return _packed_views(f(state["b"], x, prec, nrhs, case["n_cy"], case["n_it"], x_is_zero=True), prec, sites)
    if kind == "batch":
        xs, _ = state["batch"].solve(state["b"], out=state["x"], **_params(case))
        return xs
    if kind == "multigrid":
        x, _ = state["mg"].solve(state["b"], mg=state["mgp"], out=state["x"])
        return x
    x, _ = op.solve(state["b"], x0=state.get("x0"), out=state.get("x"), **_params(case, method=case["method"]))
    return x


# ------------------------------------------------------------------ what a pass needs
HOP, CLOVER, AXPY = 1320, 504, 48  # flops per site


def _site_bytes(prec, compress):
    spinor = {64: 192, 32: 96, 16: 52}[prec]
    links = 576 if prec == 64 else {32: 288, 16: 144}[prec] * compress // 18
    clover = {64: 576, 32: 288, 16: 148}[prec]
    return spinor, links, clover


def work(case):
    """Each input read once, each output written once; conventional flop counts.  A solve is
    counted with the preconditioned iterations that its system needs (about six at these masses)."""
    spinor, links, clover = _site_bytes(case["prec"], case["compress"])
    kind = case["kind"]
    sites = sum(math.prod(d) * n for d, n in _lattices(case))
    volume = sum(math.prod(d) for d, _ in _lattices(case))
    dirac = HOP + CLOVER + AXPY
    block = _geometry(case)[1]
    inside = sum(1 - 1 / b for b in block) / 4  # hops that stay in a domain

    def sweeps(n_cy, n_it):
        return n_cy * (dirac + n_it * (inside * HOP + CLOVER + AXPY + 336))

    if kind == "dslash":
        return {"bytes": 2.0 * spinor * sites + (links + clover) * volume, "flops": float(dirac * sites)}
    if kind == "smoother":
        vectors = 3 * 192 if case["guess"] else 2 * spinor
        return {"bytes": float(vectors * sites + (links + clover) * volume),
                "flops": float(sweeps(case["n_cy"], case["n_it"]) * sites)}
    solve = 6 * (dirac + sweeps(4, 4)) + 2 * dirac
    if kind == "action":
        # links and source in, gradient out; two solves, the leaves and their derivative
        return {"bytes": 576.0 * volume + 192 * sites + 576 * volume, "flops": float((2 * solve + 40000) * volume)}
    if kind == "multigrid":
        solve = 4 * 2 * (dirac + sweeps(2, 4) + 4 * 16 * 96)
    return {"bytes": 2.0 * 192 * sites + (links + clover) * volume, "flops": float(solve * sites)}


def tolerance(case):
    """About four times the distance from exact() (FP64 1.5e-16 to 2.1e-16, FP32 1e-7 to 1.5e-7, FP16 storage
    3.5e-4 to 4.3e-4, solves 3e-11 to 2.1e-10), with room for sums in another order."""
    kind, prec = case["kind"], case["prec"]
    if kind == "dslash":
        return {"rel": {64: 1e-15, 32: 5e-7, 16: 1.5e-3}[prec]}
    if kind == "smoother":
        return {"rel": {64: 1e-14, 32: 7e-7, 16: 2e-3}[prec]}
    # iterates that stop at a residual of 1e-10
    return {"rel": 1e-9}


# ------------------------------------------------------------------ 64-bit results from the definitions
def _mm(a, b):
    """Products of stacks of 3x3 matrices, entry by entry."""
    return sum(a[..., :, k:k + 1] * b[..., k:k + 1, :] for k in range(3))


def _gammas():
    s = [torch.tensor(m, dtype=torch.complex128) for m in
         (((0, 1), (1, 0)), ((0, -1j), (1j, 0)), ((1, 0), (0, -1)))]
    g = torch.zeros((4, 4, 4), dtype=torch.complex128)
    for k in range(3):
        g[k, :2, 2:] = -1j * s[k]
        g[k, 2:, :2] = 1j * s[k]
    g[3, :2, 2:] = -torch.eye(2)
    g[3, 2:, :2] = -torch.eye(2)
    return g.to(DEVICE)


class _Reference:
    """D = C - kappa H and the SAP smoothers on fields (Lt, Lz, Ly, Lx, ...) in complex128."""

    def __init__(self, case, dims, U):
        self.dims, self.block = dims, _geometry(case)[1]
        self.kappa, self.csw = case["kappa"], case["csw"]
        self.shape = tuple(dims[::-1])
        self.gam = _gammas()
        self.U = U.reshape(*self.shape, 4, 3, 3)
        self.bc = torch.ones((dims[3], 1, 1, 1, 1, 1), dtype=torch.complex128, device=DEVICE)
        self.bc[-1] = -1.0  # antiperiodic: the hop from t = Lt - 1 to 0
        self.C = self.clover(self.U)
        self._cinv = None

    def field(self, psi):
        return psi.reshape(*self.shape, 4, 3)

    @staticmethod
    def shift(f, mu, n):
        """f(x + n mu)"""
        return torch.roll(f, -n, dims=3 - mu)

    def clover(self, U):
        """The two chiral 6x6 blocks (..., 2, 6, 6) of C = 1 + i kappa csw sum sigma F."""
        sh, dag = self.shift, lambda m: m.conj().transpose(-1, -2)
        C = torch.eye(6, dtype=torch.complex128, device=DEVICE).expand(*self.shape, 2, 6, 6)
        if self.csw == 0:
            return C
        for mu in range(4):
            for nu in range(mu + 1, 4):
                a, b = U[..., mu, :, :], U[..., nu, :, :]
                # plaquette from x along mu, then nu; its four leaves at x
                ab = _mm(a, sh(b, mu, 1))
                ba = _mm(b, sh(a, nu, 1))
                q = _mm(ab, dag(ba))
                ax, bx = sh(a, mu, -1), sh(b, nu, -1)
                # nu, then -mu: U_nu(x) U_mu(x+nu-mu)^+ U_nu(x-mu)^+ U_mu(x-mu)
                q = q + _mm(_mm(_mm(b, dag(sh(ax, nu, 1))), dag(sh(b, mu, -1))), ax)
                # -mu, then -nu: U_mu(x-mu)^+ U_nu(x-mu-nu)^+ U_mu(x-mu-nu) U_nu(x-nu)
                q = q + _mm(_mm(_mm(dag(ax), dag(sh(bx, mu, -1))), sh(ax, nu, -1)), bx)
                # -nu, then mu: U_nu(x-nu)^+ U_mu(x-nu) U_nu(x-nu+mu) U_mu(x)^+
                q = q + _mm(_mm(_mm(dag(bx), sh(a, nu, -1)), sh(bx, mu, 1)), dag(a))
                F = (q - dag(q)) / 8
                sigma = 0.5j * (self.gam[mu] @ self.gam[nu] - self.gam[nu] @ self.gam[mu])
                for chi in range(2):
                    s = sigma[2 * chi:2 * chi + 2, 2 * chi:2 * chi + 2]
                    t = (1j * self.kappa * self.csw) * torch.einsum("st,...ab->...satb", s, F).reshape(
                        *self.shape, 6, 6)
                    C = C + torch.stack([t, torch.zeros_like(t)] if chi == 0 else [torch.zeros_like(t), t], dim=-3)
        return C

    def apply_C(self, C, psi):
        v = psi.reshape(*self.shape, 2, 6)
        return sum(C[..., k] * v[..., k:k + 1] for k in range(6)).reshape(*self.shape, 4, 3)

    @property
    def cinv(self):
        if self._cinv is None:
            self._cinv = torch.linalg.inv(self.C)
        return self._cinv

    def hop(self, psi, U=None, keep=None, dagger=False):
        """H psi; keep[mu] (0 or 1) masks the forward hops that a domain operator keeps."""
        U = self.U if U is None else U
        sgn = -1.0 if dagger else 1.0
        out = torch.zeros_like(psi)
        for mu in range(4):
            u = U[..., mu, :, :]
            m = self.bc if mu == 3 else 1.0
            if keep is not None:
                m = m * keep[mu]
            f = self.shift(psi, mu, 1)
            f = f - sgn * torch.einsum("st,...tc->...sc", self.gam[mu], f)
            out = out + m * sum(u[..., None, :, k] * f[..., k:k + 1] for k in range(3))
            g = psi + sgn * torch.einsum("st,...tc->...sc", self.gam[mu], psi)
            g = m * sum(u[..., None, k, :].conj() * g[..., k:k + 1] for k in range(3))
            out = out + self.shift(g, mu, -1)
        return out

    def D(self, psi, dagger=False):
        return self.apply_C(self.C, psi) - self.kappa * self.hop(psi, dagger=dagger)

    def A(self, psi):
        return self.apply_C(self.cinv, self.D(psi))

    # -- smoothers
    def domains(self):
        """per-site masks of the kept forward hops, the domain index, domain colour and site parity"""
        ax = [torch.arange(n, device=DEVICE) for n in self.shape]
        t, z, y, x = torch.meshgrid(*ax, indexing="ij")
        c = (x, y, z, t)
        keep = [((c[k] % self.block[k]) != self.block[k] - 1).to(torch.float64)[..., None, None] for k in range(4)]
        idx, colour = torch.zeros_like(x), torch.zeros_like(x)
        for k in range(3, -1, -1):
            idx = idx * (self.dims[k] // self.block[k]) + c[k] // self.block[k]
            colour = colour + c[k] // self.block[k]
        parity = (x + y + z + t) % 2
        return keep, idx, (colour % 2)[..., None, None], parity[..., None, None]

    def smooth(self, b, x, solver, n_cy, n_it):
        keep, idx, colour, parity = self.domains()
        nd = int(idx.max()) + 1
        ci = self.cinv if solver != "mr" else None
        even, odd = (parity == 0).to(torch.float64), (parity == 1).to(torch.float64)

        def dot(p, q):
            s = (p.conj() * q).sum(dim=(-1, -2)).reshape(-1)
            o = torch.zeros(nd, dtype=torch.complex128, device=DEVICE).index_add_(0, idx.reshape(-1), s)
            return o

        def steps(apply, r):
            e = torch.zeros_like(r)
            for _ in range(n_it):
                p = apply(r)
                a = dot(p, r) / (dot(p, p) + 1e-300)
                a = a[idx][..., None, None]
                e, r = e + a * r, r - a * p
            return e

        hop_b = lambda v: self.hop(v, keep=keep)  # noqa: E731
        for _ in range(n_cy):
            for col in range(2):
                on = (colour == col).to(torch.float64)
                if solver == "A":
                    r = on * (b - self.A(x))
                    e = r
                    for _ in range(1, n_it):
                        e = r + self.kappa * self.apply_C(ci, hop_b(e))
                elif solver == "mr":
                    e = steps(lambda v: self.apply_C(self.C, v) - self.kappa * hop_b(v), on * (b - self.D(x)))
                else:
                    r = on * (b - self.D(x))
                    rho = even * (r + self.kappa * hop_b(odd * self.apply_C(ci, r)))

                    def schur(v):
                        y = odd * self.apply_C(ci, self.kappa * hop_b(v))
                        return even * (self.apply_C(self.C, v) - self.kappa * hop_b(y))

                    e = steps(schur, rho)
                    e = e + odd * self.apply_C(ci, r + self.kappa * hop_b(e))
                x = x + on * e
        return x

    # -- solves
    def solve(self, b, dagger=False, tol=2e-14):
        """D x = b (D^dagger x = b) by restarted BiCGStab."""
        A = lambda v: self.D(v, dagger)  # noqa: E731
        norm = lambda v: float(torch.linalg.vector_norm(v))  # noqa: E731
        bn, x = norm(b), torch.zeros_like(b)
        for _ in range(6):
            r = b - A(x)
            if norm(r) <= tol * bn:
                break
            target = max(tol * bn * 0.5, 1e-9 * norm(r))
            r0, p = r.clone(), r.clone()
            rho = torch.vdot(r0.reshape(-1), r.reshape(-1))
            for _ in range(200):
                v = A(p)
                alpha = rho / torch.vdot(r0.reshape(-1), v.reshape(-1))
                s = r - alpha * v
                t = A(s)
                omega = torch.vdot(t.reshape(-1), s.reshape(-1)) / torch.vdot(t.reshape(-1), t.reshape(-1))
                x = x + alpha * p + omega * s
                r = s - omega * t
                if norm(r) <= target:
                    break
                new = torch.vdot(r0.reshape(-1), r.reshape(-1))
                p = r + (new / rho) * (alpha / omega) * (p - omega * v)
                rho = new
        return x

    def action(self, phi):
        """S = |D^-dagger phi|^2 and dS/dU = -2 Re Y^+ (dD/dU) X."""
        Y = self.solve(phi, dagger=True)
        X = self.solve(Y)
        U = self.U.detach().clone().requires_grad_(True)
        f = self.apply_C(self.clover(U), X) - self.kappa * self.hop(X, U=U)
        s = -2 * (Y.conj() * f).real.sum()
        (g,) = torch.autograd.grad(s, U)
        return (Y.abs() ** 2).sum(), g


def _packed(fields, dims, block, prec):
    """Canonical fields (nrhs, V, 4, 3) in the packed order: domain by domain (x fastest), even sites
    of a domain before odd ones, planes of 16 bytes."""
    ax = [torch.arange(d, device=DEVICE) for d in dims[::-1]]
    t, z, y, x = (a.reshape(-1) for a in torch.meshgrid(*ax, indexing="ij"))
    c = (x, y, z, t)
    blk, loc = torch.zeros_like(x), torch.zeros_like(x)
    for k in range(3, -1, -1):
        blk = blk * (dims[k] // block[k]) + c[k] // block[k]
        loc = loc * block[k] + c[k] % block[k]
    vb = math.prod(block)
    order = torch.argsort((blk * 2 + (x + y + z + t) % 2) * vb + loc)
    r = torch.view_as_real(fields[:, order].contiguous()).reshape(fields.shape[0], -1, vb, 24)
    per = {64: 2, 32: 4, 16: 8}[prec]

    def planes(v):
        return v.reshape(*v.shape[:3], 24 // per, per).transpose(2, 3).reshape(-1)

    if prec != 16:
        return planes(r)
    scale = r.abs().amax(dim=-1, keepdim=True)
    return {"values": planes(r / scale), "scale": scale.reshape(-1)}


def exact(case, seed):
    """What run() returns, in 64-bit torch."""
    kind = case["kind"]
    block = _geometry(case)[1]
    outs = []
    with torch.no_grad():
        fields = _fields(case, seed)
    for dims, U, b, x0 in fields:
        ref = _Reference(case, dims, U)
        if kind == "action":
            S, g = ref.action(ref.field(b[0]))
            return {"action": S, "gradient": g.reshape(-1, 4, 3, 3)}
        with torch.no_grad():
            if kind == "dslash":
                f = ref.A if case["op"] == "A" else lambda v: ref.D(v, case["dagger"])
                x = torch.stack([f(ref.field(v)).reshape(-1, 4, 3) for v in b])
                return _packed(x, dims, block, case["prec"])
            if kind == "smoother":
                x = torch.zeros_like(b[0]) if x0 is None else x0[0]
                x = ref.smooth(ref.field(b[0]), ref.field(x), case["solver"], case["n_cy"], case["n_it"])
                x = x.reshape(1, -1, 4, 3)
                return x[0] if x0 is not None else _packed(x, dims, block, case["prec"])
            x = torch.stack([ref.solve(ref.field(v)).reshape(-1, 4, 3) for v in b])
            outs.append(x)
    if kind == "batch":
        return outs
    return outs[0] if case["nrhs"] > 1 else outs[0][0]
