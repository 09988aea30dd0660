"""The tensor-core network at the edges of its tiles: fewer sites than a tile or an
activation block, remainders of both, extents of two (both neighbours the same site), many
tiles per block, and two to five layers; antiperiodic and periodic time."""
import pytest
import torch

import pfmp_inputs as pin

pytestmark = pytest.mark.gpu

# unit roundoff of FP16 operands, two per product and layer (see test_gpu_nn.TC_BAR)
U16 = 2.0 ** -11


@pytest.mark.parametrize("layers", [2, 3, 5])
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (2, 4, 6, 2), (6, 10, 14, 18), (16, 16, 16, 32)],
                         ids=lambda d: "x".join(map(str, d)))
def test_tensor_core_network_tiles(dims, layers):
    from paper_1609_02652_gb300 import capi

    if layers > 3 and dims[0] == 16:
        pytest.skip("three layers cover the many-tile case")
    V = dims[0] * dims[1] * dims[2] * dims[3]
    gen = torch.Generator(device="cuda").manual_seed(5)
    ctx = capi.pfmp_ctx_create(dims, 1 if layers == 3 else -1, None)
    net = capi.pfmp_nn_create(ctx, [1] + [8] * (layers - 1) + [1], capi.PFMP_F32)
    try:
        h = torch.randn(V, 4, 8, generator=gen, dtype=torch.float64, device="cuda")
        capi.pfmp_gauge_from_algebra(ctx, h, 0.5, capi.PFMP_DEVICE)
        capi.pfmp_nn_set_weights(net, pin.nn_weights([1] + [8] * (layers - 1) + [1], 9))
        n = capi.pfmp_spinor_bytes(ctx, capi.PFMP_F32) // 4
        b = torch.randn(n, generator=gen, dtype=torch.float32, device="cuda")
        out, ref = torch.zeros_like(b), torch.zeros_like(b)
        capi.pfmp_nn_apply(net, capi.PFMP_F32, out, b)
        capi.pfmp_nn_set_tensor_cores(net, 0)
        capi.pfmp_nn_apply(net, capi.PFMP_F32, ref, b)
        torch.cuda.synchronize()
        err = float((out - ref).double().norm() / ref.double().norm())
        assert err < 2 * U16 * layers, err
    finally:
        capi.pfmp_nn_destroy(net)
        capi.pfmp_ctx_destroy(ctx)
