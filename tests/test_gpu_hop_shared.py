"""The stencil kernels that share a site among several threads (FP64, double-float, small
FP32 lattices) at the edges of their site blocks and of their size ranges, against the
oracle and against the split-site kernel, which takes the same inputs through other code."""
import pytest
import torch

import pfmp_inputs as pin
from _util import Gpu, oracle_gauge, rel_l2

pytestmark = pytest.mark.gpu

# sites per parity: 8 (one block), 2424 and 2440 (either side of the 8-site-block range,
# both 8 mod 16), 2808 (a half-filled last 16-site block), 24192 and 24448 (either side of
# the FP32 range)
LATTICES = [(2, 2, 2, 2), (2, 2, 6, 202), (2, 2, 2, 610), (6, 6, 6, 26), (12, 12, 12, 28), (4, 4, 4, 764)]


@pytest.fixture(scope="module", params=LATTICES, ids=lambda d: "x".join(map(str, d)))
def setup(request):
    from paper_1609_02652_gb300 import capi

    lat, U = oracle_gauge(request.param, 0.4, 5)
    g = Gpu(lat, U)
    yield lat, U, g, capi
    g.close()


@pytest.mark.parametrize("prec,bar", [(0, 1e-13), (1, 1e-6)], ids=["f64", "f32"])
def test_operator(setup, prec, bar):
    from oracle.dirac import WilsonClover, hop

    lat, U, g, capi = setup
    W = WilsonClover(lat, U, 0.125, 1.0)
    op, other = g.op(0.125, 1.0), g.op(0.125, 1.0)
    capi.pfmp_op_set_split(other, prec, 2)
    psi = torch.tensor(pin.spinor(lat.dims, 9)).reshape(*lat.shape, 4, 3)
    e, o = g.pack(lat.even * psi, prec, 0), g.pack(lat.odd * psi, prec, 1)
    out, ref = g.buf(prec), g.buf(prec)
    for dagger, want in [(0, W.mhat(lat.even * psi)), (1, W.mhat_dag(lat.even * psi))]:
        capi.pfmp_mhat(op, prec, out, e, dagger)
        capi.pfmp_mhat(other, prec, ref, e, dagger)
        assert rel_l2(lat.even * g.unpack(out, prec, 0), want) < bar
        assert rel_l2(out, ref) < bar
    nrm, nref = capi.pfmp_kop(op, prec, out, e, True), capi.pfmp_kop(other, prec, ref, e, True)
    assert rel_l2(out, ref) < bar and abs(nrm - nref) < 10 * bar * nref
    for parity, src, mask in [(0, o, lat.even), (1, e, lat.odd)]:
        for dagger in (0, 1):
            capi.pfmp_dslash(op, prec, out, src, parity, dagger)
            capi.pfmp_dslash(other, prec, ref, src, parity, dagger)
            assert rel_l2(out, ref) < bar
        assert rel_l2(mask * g.unpack(out, prec, parity), mask * hop(lat, U, (1 - mask) * psi, adjoint=True)) < bar


def test_double_float_residual(setup):
    """r = b - K x with K in double-float: every operation is good to a few 2^-48 of its
    operands and a component is a sum of about 100 products, so 2^-42 |K x| bounds it."""
    lat, U, g, capi = setup
    op = g.op(0.125, 1.0)
    x, b = (g.pack(lat.even * torch.tensor(pin.spinor(lat.dims, s)).reshape(*lat.shape, 4, 3), 0, 0) for s in (3, 4))
    rd, rf, kx = g.buf(0), g.buf(0), g.buf(0)
    capi.pfmp_kop(op, 0, kx, x)
    capi.pfmp_true_residual(op, capi.PFMP_DF, rd, x, b)
    capi.pfmp_true_residual(op, capi.PFMP_F64, rf, x, b)
    assert float(torch.linalg.vector_norm(rd - rf)) < 2.0 ** -42 * float(torch.linalg.vector_norm(kx))
    assert rel_l2(rf, b - kx) < 1e-13
