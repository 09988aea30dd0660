"""The norm that K applications return, on FP32 fields whose sums need more than FP32 pairs hold,
or more than FP32's range.  kappa = 1e-30 and c_sw = 0 make M-hat the identity in FP32, so <v, K v>
is the sum of |v|^2 over values that FP32 holds exactly."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(4, 4, 4, 8), (8, 8, 8, 32), (16, 16, 16, 32), (24, 24, 24, 48)],
                         ids=lambda d: "x".join(map(str, d)))
@pytest.mark.parametrize("split", [1, 2])
def test_norm_of_identity(dims, split):
    from paper_1609_02652_gb300 import capi

    V = dims[0] * dims[1] * dims[2] * dims[3]
    Vh = V // 2
    gen = torch.Generator(device="cuda").manual_seed(2)
    ctx = capi.pfmp_ctx_create(dims, -1, None)
    try:
        capi.pfmp_gauge_from_algebra(ctx, torch.randn(V, 4, 8, generator=gen, dtype=torch.float64, device="cuda"), 0.4,
                                     capi.PFMP_DEVICE)
        op = capi.pfmp_op_create(ctx, 1e-30, 0.0)
        capi.pfmp_op_set_split(op, capi.PFMP_F32, split)
        v, out = (torch.zeros(6, Vh, 4, dtype=torch.float32, device="cuda") for _ in range(2))
        # |v|^2 per site: 2^24 + 1 + 10 x 2^-25; each FP64 addition of the lattice sum (at most 64
        # on the way of a value) rounds by 2^-53 of the total, so it is right to 2^-47 of it,
        # while 2^-46 of it would be lost with pairs
        v[..., 0] = v[..., 1] = v[..., 2] = v[..., 3] = 2.0 ** -13
        v[0, :, 0], v[0, :, 1], v[0, :, 2], v[0, :, 3] = 2.0 ** 12, 0.0, 1.0, 0.0
        nrm = capi.pfmp_kop(op, capi.PFMP_F32, out, v, True)
        torch.cuda.synchronize()
        assert torch.equal(out, v)
        want = Vh * (2.0 ** 24 + 1 + 10 * 2.0 ** -25)
        assert abs(nrm - want) < 2.0 ** -47 * want, (nrm - want) / want
        # twelve terms of 1e38: each fits FP32, their sum does not
        v[...] = 0.0
        v[..., 0] = v[..., 2] = 1e19
        nrm = capi.pfmp_kop(op, capi.PFMP_F32, out, v, True)
        torch.cuda.synchronize()
        want = float((v[..., 0] ** 2 + v[..., 2] ** 2).double().sum())
        assert torch.equal(out, v) and abs(nrm - want) < 1e-12 * want, (nrm, want)
        capi.pfmp_op_destroy(op)
    finally:
        capi.pfmp_ctx_destroy(ctx)
