"""The even-odd domain solver over domain shapes (cubic, elongated, the smallest and
the largest) against the oracle, to the FP32 and FP16 storages' bars."""
import numpy as np
import pytest

from helpers import TOL, rel
from oracle import oracle as O
from paper_2112_00501_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("dims,block", [((4, 4, 4, 4), (2, 2, 2, 2)), ((8, 4, 4, 8), (4, 2, 2, 2)),
                                        ((4, 8, 4, 16), (2, 4, 2, 8)), ((8, 4, 8, 16), (4, 2, 4, 8)),
                                        ((8, 8, 8, 8), (4, 4, 4, 4))])
@pytest.mark.parametrize("prec,compress", [(32, 18), (32, 12), (16, 18), (16, 12)])
@pytest.mark.parametrize("n_mr", [1, 4])
def test_shapes(dims, block, prec, compress, n_mr):
    from paper_2112_00501_gb300 import api

    kappa, csw = 0.13, 1.0
    U = synth.gauge_field(dims, 0.4, 21)
    b, x0 = synth.gaussian_spinor(dims, 22), synth.gaussian_spinor(dims, 23)
    lat = api.Lattice(dims, block, -1)
    op = api.CloverOperator(api.Gauge(lat, torch.from_numpy(U).cuda(), storage_prec=prec, compress=compress), kappa,
                            csw)
    Cl = O.clover(dims, kappa, csw, U)
    Ci = O.clover_inverse(dims, Cl)
    for guess in (None, x0):
        g = None if guess is None else torch.from_numpy(guess).cuda()
        got = op.sap_eo(torch.from_numpy(b).cuda(), prec=prec, n_cy=2, n_mr=n_mr, x0=g).cpu().numpy()
        ref = O.sap_eo(dims, block, -1, kappa, U, Cl, Ci, b, x0=guess, ncy=2, nmr=n_mr)
        assert rel(got, ref) < TOL[prec]


@pytest.mark.parametrize("prec", [32, 16])
@pytest.mark.parametrize("p", [-60, -64])
def test_small_sources(prec, p):
    """2^p b gives 2^p times b's correction to the storages' bars, while the last steps' <p, p> lie
    below FP32's normal range (2^-126; multiples of 2^-149 keep 1e-4 of them, of a small last step)."""
    from paper_2112_00501_gb300 import api

    dims, block, kappa, csw = (8, 4, 12, 8), (2, 2, 2, 2), 0.13, 1.0
    U, b = synth.gauge_field(dims, 0.4, 21), synth.gaussian_spinor(dims, 22)
    lat = api.Lattice(dims, block, -1)
    op = api.CloverOperator(api.Gauge(lat, torch.from_numpy(U).cuda(), storage_prec=prec), kappa, csw)
    Cl = O.clover(dims, kappa, csw, U)
    got = op.sap_eo(torch.from_numpy(b * 2.0**p).cuda(), prec=prec, n_cy=1, n_mr=4).cpu().numpy() * 2.0**-p
    ref = O.sap_eo(dims, block, -1, kappa, U, Cl, O.clover_inverse(dims, Cl), b, ncy=1, nmr=4)
    assert rel(got, ref) < TOL[prec]
