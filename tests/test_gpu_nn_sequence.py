"""Networks whose channels return to 1 between two layers: each layer has a tensor-core form, the
sequence has none, so the tensor-core path refuses them and the FP32 kernels take them."""
import pytest
import torch

import pfmp_inputs as pin
from _util import Gpu, oracle_gauge, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ch", [[1, 8, 1, 8, 1], [1, 8, 8, 1, 8, 1]], ids=lambda c: "-".join(map(str, c)))
def test_channels_back_to_one(ch):
    from oracle import nn
    from paper_1609_02652_gb300 import capi

    lat, U = oracle_gauge((4, 4, 4, 4), 0.4, 61)
    g = Gpu(lat, U)
    net = capi.pfmp_nn_create(g.ctx, ch, capi.PFMP_F32)
    try:
        ws = nn.init_weights(ch, 7)
        capi.pfmp_nn_set_weights(net, [w.numpy() for w in ws])
        b = lat.even * torch.tensor(pin.spinor(lat.dims, 81)).reshape(*lat.shape, 4, 3)
        b32, out = g.pack(b, 1, 0), g.buf(1)
        with pytest.raises(capi.PfmpError) as e:
            capi.pfmp_nn_apply(net, 1, out, b32)
        assert e.value.status == capi.PFMP_E_INVALID
        assert float(out.abs().max()) == 0.0
        prm = capi.SolverParams(method=0, tol=1e-8, max_iter=100, delta=1e-3, check_every=8, restart=8)
        with pytest.raises(capi.PfmpError) as e:
            capi.pfmp_solve_fgcr(g.op(0.12, 1.0), net, prm, g.buf(0), g.pack(b, 0, 0))
        assert e.value.status == capi.PFMP_E_INVALID
        capi.pfmp_nn_set_tensor_cores(net, 0)
        capi.pfmp_nn_apply(net, 1, out, b32)
        # five FP32 layers, as the bar of the FP32 kernels elsewhere
        assert rel_l2(lat.even * g.unpack(out, 1, 0), nn.network_apply(lat, U, ws, b)) < 1e-5
    finally:
        capi.pfmp_nn_destroy(net)
        g.close()
