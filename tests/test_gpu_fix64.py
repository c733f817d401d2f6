"""The FP64 operator's block fixed-point path: its error, the fields it leaves
to FP64 instructions, and the batched operator's agreement with it.

Bound in the 2-norm: the fixed-point sum is good to 5e-17, the result's rounding
and the reference, the oracle's FP64 sum, to 2e-16; 6e-16 leaves a factor two.
Bounds of single components are stated at the tests of graded, wide and sparse
fields.
"""
import numpy as np
import pytest

from helpers import fields, rel
from oracle import oracle as O
from paper_2112_00501_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _op(name, U=None, kappa=None, tbc=-1, csw=1.0):
    from paper_2112_00501_gb300 import api

    dims, block, eps, kap, _, U0, psi = fields(name)
    lat = api.Lattice(dims, block, tbc)
    g = api.Gauge(lat, torch.from_numpy(U0 if U is None else U).cuda(), storage_prec=64)
    return api.CloverOperator(g, kap if kappa is None else kappa, csw)


def _scaled(psi, p):
    return np.ldexp(np.ascontiguousarray(psi).view(np.float64), p).view(np.complex128)


def _check(name, psi, tol=6e-16, U=None, kappa=None, dagger=False, p=0):
    dims, block, eps, kap, csw, U0, _ = fields(name)
    U, kappa = U0 if U is None else U, kap if kappa is None else kappa
    got = _op(name, U, kappa).D(torch.from_numpy(_scaled(psi, p)).cuda(), prec=64, dagger=dagger).cpu().numpy()
    got = _scaled(got, -p)
    ref = O.dirac(dims, -1, kappa, U, O.clover(dims, kappa, csw, U), psi, dagger=dagger)
    assert rel(got, ref) < tol
    return got, ref


@pytest.mark.parametrize("name", ["c0_4^4", "ragged_8x4x12x8", "mid_8^4"])
@pytest.mark.parametrize("dagger", [False, True])
@pytest.mark.parametrize("kappa", [0.0, 1e-6, 0.01, 0.13, -0.13, 0.8, 70.0])  # 0 and 1e-6 run on FP64 instructions
def test_error(name, dagger, kappa):
    _check(name, fields(name)[6], kappa=kappa, dagger=dagger)


@pytest.mark.parametrize("p", [-1000, -900, -890, -400, 400, 955, 964])
def test_scales_of_the_whole_field(p):
    _check("ragged_8x4x12x8", fields("ragged_8x4x12x8")[6], p=p)


def _terms(dims, kappa, U, C, psi):
    """The magnitudes |re| + |im| of the terms that enter each component of D psi (or D^dagger psi)."""
    mag = lambda z: np.abs(z.real) + np.abs(z.imag)
    shape = tuple(dims[::-1])
    m = mag(psi).reshape(shape + (4, 3))
    u = mag(U).reshape(shape + (4, 3, 3))
    out = np.einsum("sij,sj->si", mag(C), mag(psi).reshape(-1, 12)).reshape(m.shape)
    for mu in range(4):
        # gamma_mu pairs spins 0, 1 with 3, 2 (x, y) or 2, 3 (z, t)
        h = m + m[..., [3, 2, 1, 0] if mu < 2 else [2, 3, 0, 1], :]
        f = np.einsum("...ab,...sb->...sa", u[..., mu, :, :], np.roll(h, -1, 3 - mu))
        g = np.roll(np.einsum("...ba,...sb->...sa", u[..., mu, :, :], h), 1, 3 - mu)
        out += abs(kappa) * (f + g)
    return out.reshape(psi.shape)


@pytest.mark.parametrize("eps", [None, 0.0])
@pytest.mark.parametrize("kind", ["sites", "neighbours", "components", "zeros", "point", "one_spin", "nothing"])
def test_wide_and_sparse_fields(kind, eps):
    """Every component against the terms that enter it, on disordered and on unit links: the
    fixed-point sum's error is 1.2 units in the mean square, 5 at most in practice, for terms of 2^53
    units at least; FP64 sums of some 60 terms, the oracle's among them, stay within 2 u of the terms
    (u = 2^-53): 8 u.  Components without terms are exactly zero."""
    name = "mid_8^4"
    dims, _, _, kappa, csw, U, psi = fields(name)
    U = U if eps is None else np.broadcast_to(np.eye(3), U.shape).astype(complex).copy()
    psi = psi.copy()
    r = np.random.default_rng(3)
    V = psi.shape[0]
    if kind == "sites":  # neighbours up to 2^24 apart: inside the fixed-point range
        psi *= np.exp2(r.integers(-12, 13, V))[:, None, None]
    if kind == "neighbours":  # beyond it
        psi *= np.exp2(r.integers(-60, 61, V))[:, None, None]
    if kind == "components":
        psi *= np.exp2(r.integers(-40, 41, psi.shape))
    if kind == "zeros":
        psi[r.random(V) < 0.5] = 0
    if kind == "point":
        psi[:] = 0
        psi[77, 2, 1] = 1.5 - 0.25j
    if kind == "one_spin":
        psi[:, 1:] = 0
    if kind == "nothing":
        psi[:] = 0
    op = _op(name, U)
    C = op.export_clover().cpu().numpy()
    for dagger in (False, True):
        got = op.D(torch.from_numpy(psi).cuda(), prec=64, dagger=dagger).cpu().numpy()
        ref = O.dirac(dims, -1, kappa, U, C, psi, dagger=dagger)
        err = np.abs(got - ref)
        assert (err <= 8 * 2.0**-53 * _terms(dims, kappa, U, C, psi)).all()
        assert kind == "nothing" or rel(got, ref) < 6e-16


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_non_finite_propagates(bad):
    name = "mid_8^4"
    dims, block, eps, kappa, csw, U, psi = fields(name)
    psi = psi.copy()
    psi[100, 1, 2] = bad
    got = _op(name).D(torch.from_numpy(psi).cuda(), prec=64).cpu().numpy()
    clean = O.dirac(dims, -1, kappa, U, O.clover(dims, kappa, csw, U), fields(name)[6])
    hit = ~np.isfinite(got).all(axis=(1, 2))
    assert hit.sum() == 9 and hit[100]  # the site and its eight neighbours
    assert rel(got[~hit], clean[~hit]) < 6e-16


def test_links_that_are_not_unitary():
    name = "mid_8^4"
    U = fields(name)[5].copy()
    U[5, 2] *= 1.01  # no fixed-point copy: FP64 instructions
    _check(name, fields(name)[6], U=U)
    U = fields(name)[5].copy()
    U[5, 2] *= 1 + 1e-5  # within the copy's bound
    _check(name, fields(name)[6], U=U)


@pytest.mark.parametrize("kappa", [0.12, 0.13])
def test_links_with_dependent_rows(kappa):
    """Rows and columns of norm 1 that are not orthogonal: no fixed-point copy.  C and D to the
    FP64 path's roundings of a sum of 16 link products each up to 3 (1e-15 leaves a factor 4)."""
    name = "mid_8^4"
    dims, block, eps, _, csw, U, psi = fields(name)
    r = np.random.default_rng(0)
    J = np.exp(2j * np.pi * r.random((U.shape[0], 4, 1, 1))) * np.ones((3, 3)) / np.sqrt(3)
    _check(name, psi, U=J, kappa=kappa, tol=1e-15)
    C = _op(name, J, kappa).export_clover().cpu().numpy()
    assert rel(C, O.clover(dims, kappa, csw, J).reshape(C.shape)) < 1e-15


def _worst_component(a, b):
    """The largest relative 2-norm error of a spin and colour over the lattice."""
    return (np.linalg.norm(a - b, axis=0) / np.linalg.norm(b, axis=0)).max()


def _graded(psi, axis, p):
    """One colour (or one spin) of psi scaled by 2^-p."""
    psi = psi.copy()
    if axis == "colour":
        psi[:, :, 2] *= 2.0**-p
    else:
        psi[:, 1] *= 2.0**-p
    return psi


@pytest.mark.parametrize("eps", [0.0, 1e-5, 0.02])
@pytest.mark.parametrize("axis", ["colour", "spin"])
def test_graded_components(eps, axis):
    """Links that hardly mix the colours: every spin and colour of D, D^dagger and A, with the
    operator's own C and C^-1, on its own.
    A component's error in fixed point is 2^-53 of the terms that enter it where the site is accepted,
    its rounding and the oracle's sum 1.5e-16 each: 4e-16; C^-1 adds a few roundings."""
    name = "mid_8^4"
    dims, block, _, kappa, csw, _, psi = fields(name)
    U = synth.gauge_field(dims, eps, 41)
    op = _op(name, U)
    Cl = op.export_clover().cpu().numpy()
    Ci = op.export_clover(inverse=True).cpu().numpy()
    for p in (0, 1, 2, 3, 4, 5, 7, 10, 15, 20, 25, 40):
        v = _graded(psi, axis, p)
        x = torch.from_numpy(v).cuda()
        for dagger in (False, True):
            ref = O.dirac(dims, -1, kappa, U, Cl, v, dagger=dagger)
            assert _worst_component(op.D(x, prec=64, dagger=dagger).cpu().numpy(), ref) < 4e-16, (p, dagger)
        ref = O.apply_A(dims, -1, kappa, U, Cl, Ci, v)
        assert _worst_component(op.A(x, 64).cpu().numpy(), ref) < 1e-15, p


def test_copies_leave_room_for_workspaces():
    """With 2 GB free an operator on 16^3 x 32 makes no copies (152 MB, which want 20 times as much
    left) and gives the same results."""
    from paper_2112_00501_gb300 import api

    dims, block, _, kappa, csw, U, psi = fields("c1_16^3x32")
    g = api.Gauge(api.Lattice(dims, block, -1), torch.from_numpy(U).cuda(), storage_prec=64)
    x = torch.from_numpy(psi).cuda()

    def create():
        before = torch.cuda.mem_get_info()[0]
        op = api.CloverOperator(g, kappa, csw)
        return before - torch.cuda.mem_get_info()[0], op.D(x, prec=64).cpu().numpy()

    create()  # the kernels' local memory
    torch.cuda.empty_cache()
    roomy, y = create()
    torch.cuda.empty_cache()
    hold = torch.empty(torch.cuda.mem_get_info()[0] - (2 << 30), dtype=torch.uint8, device="cuda")
    tight, z = create()
    del hold
    torch.cuda.empty_cache()
    assert roomy - tight > 0.9 * 1160 * psi.shape[0]
    assert rel(z, y) < 6e-16


def test_batch_is_bit_identical():
    """A batch of one lattice with a fixed-point copy and one without."""
    from paper_2112_00501_gb300 import api

    name = "mid_8^4"
    V = fields(name)[6].shape[0]
    bent = fields(name)[5].copy()
    bent[5, 2] *= 1.01
    ops = [_op(name), _op(name, bent)]
    g = torch.Generator(device="cuda").manual_seed(5)
    xs = [torch.view_as_complex(torch.randn((n, V, 4, 3, 2), dtype=torch.float64, device="cuda", generator=g))
          for n in (3, 1)]
    ps = [op.lattice.pack(x, 64) for op, x in zip(ops, xs)]
    batch = api.Batch(ops, [3, 1])
    for dagger in (False, True):
        for fast in (0, 1):
            batch.set_shape(64, 1, 128, fast, 0)
            out = batch.apply_D(ps, 64, dagger=dagger)
            for op, p, n, o in zip(ops, ps, (3, 1), out):
                assert torch.equal(o, (op.apply_Ddag if dagger else op.apply_D)(p, 64, n))


def test_batch_shape_with_copies():
    """A launch with copies has one shape, whatever is pinned; a batch without is tuned over all."""
    from paper_2112_00501_gb300 import api

    name = "mid_8^4"
    bent = fields(name)[5].copy()
    bent[5, 2] *= 1.01
    op, plain = _op(name), _op(name, bent)
    x = op.lattice.pack(torch.from_numpy(np.stack([fields(name)[6]] * 3)).cuda(), 64)
    for ops in ([op, op], [op, plain], [plain, plain]):
        batch = api.Batch(ops, [3, 3])
        t = batch.tune(64)
        assert plain is ops[0] or (t["rhs_per_thread"], t["threads"]) == (1, 128)
        ref = [o.apply_D(x, 64, 3) for o in ops]
        for shape in ((1, 128), (2, 256), (4, 128)):
            batch.set_shape(64, *shape, 1, 0)
            assert all(torch.equal(a, b) for a, b in zip(batch.apply_D([x, x], 64), ref))


def _check_sap(name, b, kappa=None, n_cy=2, n_mr=4, x0=None, p=0, tol=2e-15):
    dims, block, eps, kap, csw, U, _ = fields(name)
    kappa = kap if kappa is None else kappa
    xg = None if x0 is None else torch.from_numpy(_scaled(x0, p)).cuda()
    got = _op(name, kappa=kappa).sap(torch.from_numpy(_scaled(b, p)).cuda(), 64, n_cy, n_mr, x0=xg).cpu().numpy()
    ref = O.sap(dims, block, -1, kappa, U, O.clover(dims, kappa, csw, U), b, x0=x0, ncy=n_cy, nmr=n_mr)
    assert rel(_scaled(got, -p), ref) < tol
    return got


# the domain solves' sums differ in order from the oracle's: a few 1e-16 each,
# over two sweeps of four steps below 2e-15
@pytest.mark.parametrize("name", ["c0_4^4", "ragged_8x4x12x8", "mid_8^4"])
@pytest.mark.parametrize("kappa", [0.0002, 0.02, 0.13, -0.11, 0.2])  # 0.0002 runs on FP64 instructions
def test_sap(name, kappa):
    psi = fields(name)[6]
    _check_sap(name, psi, kappa)
    _check_sap(name, psi, kappa, x0=np.roll(psi, 7, axis=0))


@pytest.mark.parametrize("n_mr", [1, 3, 40])
def test_sap_step_counts(n_mr):
    _check_sap("ragged_8x4x12x8", fields("ragged_8x4x12x8")[6], n_cy=1, n_mr=n_mr)


@pytest.mark.parametrize("kappa,n_mr", [(0.02, 4), (0.05, 4), (0.1355, 12)])
def test_sap_second_sweep_residuals(kappa, n_mr):
    """Residuals that the first sweep leaves at the faces of the domains: every component of the second
    sweep's result to the bound of test_sap_graded_components."""
    name = "mid_8^4"
    dims, block, _, _, csw, U, b = fields(name)
    op = _op(name, kappa=kappa)
    got = op.sap(torch.from_numpy(b).cuda(), 64, 2, n_mr).cpu().numpy()
    ref = O.sap(dims, block, -1, kappa, U, op.export_clover().cpu().numpy(), b, ncy=2, nmr=n_mr)
    assert _worst_component(got, ref) < 1e-14


@pytest.mark.parametrize("p", [-880, -400, 400, 955])
def test_sap_scales(p):
    _check_sap("mid_8^4", fields("mid_8^4")[6], p=p)


def test_sap_sparse_and_zero_domains():
    name = "mid_8^4"
    b = np.zeros_like(fields(name)[6])
    b[77, 2, 1] = 1.5 - 0.25j
    got = _check_sap(name, b, n_cy=1)
    assert (got == 0).any()
    b = fields(name)[6].copy()
    b *= np.exp2(np.random.default_rng(3).integers(-40, 41, b.shape[0]))[:, None, None]
    _check_sap(name, b)


@pytest.mark.parametrize("eps", [0.0, 1e-5])
@pytest.mark.parametrize("axis", ["colour", "spin"])
@pytest.mark.parametrize("n_cy,n_mr,guess", [(1, 1, False), (2, 4, False), (1, 4, True)])
def test_sap_graded_components(eps, axis, n_cy, n_mr, guess):
    """As test_graded_components, for the smoother.  Every component carries alpha's error: the oracle
    adds a domain's N = 3072 products one after another, a random walk of sqrt(N) u = 6e-15 in <p, r>
    and in <p, p>, together 9e-15.  (Without a test of the sizes a colour at 2^-20 was off by 2e-11.)"""
    name = "mid_8^4"
    dims, block, _, kappa, csw, _, psi = fields(name)
    U = synth.gauge_field(dims, eps, 41)
    op = _op(name, U)
    Cl = op.export_clover().cpu().numpy()
    for p in (0, 1, 2, 3, 4, 5, 7, 10, 15, 20, 25, 40, 60):
        b = _graded(psi, axis, p)
        x0 = np.roll(b, 7, axis=0) if guess else None
        xg = torch.from_numpy(x0).cuda() if guess else None
        got = op.sap(torch.from_numpy(b).cuda(), 64, n_cy, n_mr, x0=xg).cpu().numpy()
        ref = O.sap(dims, block, -1, kappa, U, Cl, b, x0=x0, ncy=n_cy, nmr=n_mr)
        assert _worst_component(got, ref) < 1e-14, p


def test_sap_non_finite():
    b = fields("mid_8^4")[6].copy()
    b[100, 1, 2] = np.nan
    x = _op("mid_8^4").sap(torch.from_numpy(b).cuda(), 64, 1, 4)
    assert bool(torch.isnan(x.real).any())


@pytest.mark.parametrize("name", ["c0_4^4", "ragged_8x4x12x8", "mid_8^4"])
@pytest.mark.parametrize("kappa,csw,bent", [(0.13, 1.0, False), (0.13, 4.0, False), (0.13, 30.0, False),
                                            (-0.13, 1.7, False), (0.13, 1.0, True), (1e-6, 1.0, False)])
def test_clover_build(name, kappa, csw, bent):
    """Blocks that are positive definite and (large c_SW) not; links with and without a fixed-point
    copy.  C to a few roundings of its largest entries; C C^-1 = 1 to the residual bound of an
    elimination on 6 x 6 complex blocks, 10 n u cond = 6.7e-15 cond (u = 1.1e-16); the blocks that
    are not definite go through Gauss-Jordan elimination, whose residual carries the condition twice."""
    from paper_2112_00501_gb300 import api

    dims, block, eps, _, _, U, psi = fields(name)
    U = U.copy()
    if bent:
        U[5, 2] *= 1.01
    lat = api.Lattice(dims, block, -1)
    op = api.CloverOperator(api.Gauge(lat, torch.from_numpy(U).cuda(), storage_prec=64), kappa, csw)
    C, Ci = op.export_clover().cpu().numpy(), op.export_clover(inverse=True).cpu().numpy()
    ref = O.clover(dims, kappa, csw, U).reshape(C.shape)
    assert rel(C, ref) < 5e-16
    cond = np.linalg.norm(ref, axis=(1, 2)) * np.linalg.norm(np.linalg.inv(ref), axis=(1, 2))
    err = np.linalg.norm(np.einsum("sij,sjk->sik", C, Ci) - np.eye(12), axis=(1, 2))
    assert (err < 6.7e-15 * cond * (cond if csw > 4 else 1.0)).all()


@pytest.mark.parametrize("eps", [0.4, 0.2, 0.1, 0.05, 1e-2, 1e-4, 1e-6])
def test_clover_build_weak_fields(eps):
    """The field strength of exp(i eps H): every off-diagonal entry of C, relative to its size over the
    lattice.  An entry adds up to three planes' Q - Q^+, each four leaves of products whose FP64 sums,
    here or the oracle's, are good to about 2e-16: 8e-16 for the two."""
    name = "mid_8^4"
    dims, block, _, kappa, csw, _, _ = fields(name)
    U = synth.gauge_field(dims, eps, 43)
    C = _op(name, U).export_clover().cpu().numpy()
    ref = O.clover(dims, kappa, csw, U).reshape(C.shape)
    off = (np.abs(ref).max(axis=0) > 0) & ~np.eye(12, dtype=bool)
    assert off.sum() == 60
    assert _worst_component(C[:, off], ref[:, off]) < 8e-16


@pytest.mark.parametrize("kappa", [0.125, 0.1])
def test_singular_clover_block_is_refused(kappa):
    """A plaquette of diag(i, -i, 1) in every (x, y) plane gives C = 1 -+ kappa c_SW diag(1, -1, 0) in
    FP64 without rounding, singular at kappa c_SW = 1 (0.1 * 10 is 1 after rounding too)."""
    from paper_2112_00501_gb300 import _lib, api

    dims, block = (8, 4, 4, 4), (4, 2, 2, 2)
    x = np.arange(512) % 8
    U = np.broadcast_to(np.eye(3), (512, 4, 3, 3)).astype(complex).copy()
    U[:, 1, 0, 0] = np.array([1, 1j, -1, -1j])[x % 4]
    U[:, 1, 1, 1] = U[:, 1, 0, 0].conj()
    g = api.Gauge(api.Lattice(dims, block, -1), torch.from_numpy(U).cuda(), storage_prec=64)
    with pytest.raises(_lib.MgcError) as e:
        api.CloverOperator(g, kappa, round(1 / kappa))
    assert e.value.status == _lib.MGC_ERR_BREAKDOWN
    api.CloverOperator(g, kappa, 0.5 / kappa)


@pytest.mark.parametrize("csw", [1.0, 3.0, 4.5])
def test_clover_inverse_of_definite_blocks(csw):
    """C^-1 against extended precision, over the positive definite blocks, no further off than an
    elimination with pivoting; at the larger c_SW with blocks whose C - 1 has eigenvalues beyond 1
    among them, where a refining step with C - 1 would not help."""
    C, Ci = (_op("mid_8^4", csw=csw).export_clover(inverse=i).cpu().numpy() for i in (False, True))
    blocks = np.concatenate([C[:, :6, :6], C[:, 6:, 6:]])
    inv = np.concatenate([Ci[:, :6, :6], Ci[:, 6:, 6:]])
    ev = np.linalg.eigvalsh(blocks)
    ok = ev[:, 0] > 0.1
    assert ok.any() and (csw < 4 or (ev[ok, -1] > 2).any())
    blocks, inv = blocks[ok], inv[ok]
    lu = np.linalg.inv(blocks)
    ref, B = lu.astype(np.clongdouble), blocks.astype(np.clongdouble)
    for _ in range(2):
        ref = ref + np.einsum("nij,njk->nik", ref, np.eye(6) - np.einsum("nij,njk->nik", B, ref))
    assert np.linalg.norm(abs(inv - ref).ravel()) < np.linalg.norm(abs(lu - ref).ravel())


@pytest.mark.parametrize("p", [-455, -400, 400, 470])
def test_force_scales(p):
    """dS/dU of 2^p phi is 2^(2p) times that of phi: the solves commute with powers of two, and the
    matrix products do too but for the scales that run on FP64 instructions (p = -455: below 2^-894),
    whose sums round differently: 1e-13."""
    from paper_2112_00501_gb300 import api

    name = "c4_8^4"
    dims, block, eps, kappa, csw, U, phi = fields(name)
    lat = api.Lattice(dims, block, -1)
    op = api.CloverOperator(api.Gauge(lat, torch.from_numpy(U).cuda(), storage_prec=32), kappa, csw)
    g0, _, _ = op.force(torch.from_numpy(phi).cuda())
    g1, _, _ = op.force(torch.from_numpy(_scaled(phi, p)).cuda())
    assert rel(_scaled(g1.cpu().numpy(), -2 * p), g0.cpu().numpy()) < 1e-13


def test_force_graded_components():
    """Diagonal links leave the colours apart: with one colour of phi scaled by 2^-p its row and column
    of the force scale by 2^-p and 4^-p, to the solves' 1e-13 (1e-11 leaves a factor for the condition)."""
    from paper_2112_00501_gb300 import api

    name = "c4_8^4"
    dims, block, _, _, csw, _, phi = fields(name)
    th = np.random.default_rng(9).uniform(-0.6, 0.6, (phi.shape[0], 4, 3))
    th -= th.mean(axis=2, keepdims=True)
    U = np.zeros((phi.shape[0], 4, 3, 3), complex)
    U[..., range(3), range(3)] = np.exp(1j * th)
    lat = api.Lattice(dims, block, -1)
    op = api.CloverOperator(api.Gauge(lat, torch.from_numpy(U).cuda(), storage_prec=64), 0.12, csw)
    par = dict(method=0, smoother_prec=64, tol=1e-13, max_iter=2000)
    g0 = op.force(torch.from_numpy(phi).cuda(), **par)[0].cpu().numpy()
    for p in (1, 2, 3, 5, 8, 12, 20, 30, 60):
        g = op.force(torch.from_numpy(_graded(phi, "colour", p)).cuda(), **par)[0].cpu().numpy()
        g[..., 2, :] *= 2.0**p
        g[..., :, 2] *= 2.0**p
        err = np.linalg.norm(g - g0, axis=(0, 1)) / np.linalg.norm(g0, axis=(0, 1))
        assert err.max() < 1e-11, (p, err)


@pytest.mark.parametrize("name", ["c0_4^4", "c4_8^4"])
def test_force_links_without_fixed_point_copy(name):
    """Bent links: the force's FP64 products, to the solves' tolerance against the oracle's force."""
    dims, block, _, kappa, csw, U, phi = fields(name)
    U = U.copy()
    U[5, 2] *= 1.01
    g, _, _ = _op(name, U).force(torch.from_numpy(phi).cuda(), method=0, smoother_prec=64, tol=1e-13, max_iter=2000)
    X, Y = O.force_solves(dims, block, -1, kappa, U, O.clover(dims, kappa, csw, U), phi, tol=1e-13)
    assert rel(g.cpu().numpy(), O.force(dims, -1, kappa, csw, U, X, Y)) < 1e-9


@pytest.mark.parametrize("name", ["c0_4^4", "ragged_8x4x12x8", "mid_8^4"])
@pytest.mark.parametrize("kappa,kind", [(0.13, "plain"), (-0.2, "plain"), (0.13, "zeros"), (0.13, "point"),
                                        (1e-6, "plain")])
def test_apply_A(name, kappa, kind):
    """A = C^-1 D; C^-1 on FP64 instructions adds a few of its roundings: 1e-15."""
    dims, block, eps, _, csw, U, psi = fields(name)
    psi = psi.copy()
    if kind == "zeros":
        psi[np.random.default_rng(3).random(psi.shape[0]) < 0.5] = 0
    if kind == "point":
        psi[:] = 0
        psi[77, 2, 1] = 1.5 - 0.25j
    two = np.stack([psi, np.roll(psi, 5, axis=0)])
    got = _op(name, kappa=kappa).A(torch.from_numpy(two).cuda(), 64).cpu().numpy()
    Cl = O.clover(dims, kappa, csw, U)
    Ci = O.clover_inverse(dims, Cl)
    for k in range(2):
        assert rel(got[k], O.apply_A(dims, -1, kappa, U, Cl, Ci, two[k])) < 1e-15
