"""Several right-hand sides in either order of the thread blocks (fields beyond and
within the L2's size) give each the single right-hand side's bits."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("dims,block", [((4, 4, 4, 4), (2, 2, 2, 2)), ((8, 4, 8, 16), (4, 2, 4, 8)),
                                        ((8, 8, 8, 8), (4, 4, 4, 4))])
@pytest.mark.parametrize("prec,compress", [(32, 18), (32, 12), (16, 18), (16, 12)])
def test_orders_agree(dims, block, prec, compress):
    from paper_2112_00501_gb300 import api, synth

    lat = api.Lattice(dims, block, -1)
    U = torch.from_numpy(synth.gauge_field(dims, 0.4, 31)).cuda()
    op = api.CloverOperator(api.Gauge(lat, U, storage_prec=prec, compress=compress), 0.13, 1.0)
    V, site = lat.volume, {32: 96, 16: 52}[prec]
    many = int(116e6 / (2 * site * V)) + 1  # the first count past the rule's line
    g = torch.Generator(device="cuda").manual_seed(7)
    x = torch.view_as_complex(torch.randn((many, V, 4, 3, 2), dtype=torch.float64, device="cuda", generator=g))
    for apply in (op.apply_D, op.apply_Ddag):
        for nrhs in (2, many):
            y = lat.unpack(apply(lat.pack(x[:nrhs], prec), prec, nrhs), prec, nrhs)
            for k in {0, 1, nrhs // 2, nrhs - 1}:
                one = lat.unpack(apply(lat.pack(x[k:k + 1], prec), prec, 1), prec, 1)
                assert torch.equal(y[k], one.reshape(y[k].shape))
