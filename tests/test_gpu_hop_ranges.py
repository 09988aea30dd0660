"""The FP32 stencil on both sides of each of its size ranges (several threads per site; 2, 4
and 7 resident blocks per SM; blocks that go over the lattice once, twice and more when they
sum), against the split-site kernel, which takes the same inputs through other code."""
import pytest
import torch

pytestmark = pytest.mark.gpu

# sites per parity: 4864 | 4872, 38912 | 38976, 77824 | 77888, 136192 | 136256 (ragged last
# blocks among them), 155648 + 64, 331776
DIMS = [(4, 4, 4, 152), (2, 2, 6, 406), (4, 16, 16, 76), (2, 8, 12, 406), (8, 16, 16, 76), (2, 16, 4, 1217 * 2 // 2 * 2),
        (16, 16, 14, 76), (4, 4, 8, 2130), (24, 24, 24, 48)]


@pytest.mark.parametrize("dims", DIMS, ids=lambda d: "x".join(map(str, d)))
def test_operator_and_norm(dims):
    from paper_1609_02652_gb300 import capi

    V = dims[0] * dims[1] * dims[2] * dims[3]
    gen = torch.Generator(device="cuda").manual_seed(2)
    ctx = capi.pfmp_ctx_create(dims, -1, None)
    try:
        capi.pfmp_gauge_from_algebra(ctx, torch.randn(V, 4, 8, generator=gen, dtype=torch.float64, device="cuda"), 0.4,
                                     capi.PFMP_DEVICE)
        ops = [capi.pfmp_op_create(ctx, 0.12, 1.0) for _ in range(2)]
        capi.pfmp_op_set_split(ops[1], capi.PFMP_F32, 2)
        n = capi.pfmp_spinor_bytes(ctx, capi.PFMP_F32) // 4
        v = torch.randn(n, generator=gen, dtype=torch.float32, device="cuda")
        out = [torch.zeros_like(v) for _ in ops]
        nrm = [capi.pfmp_kop(op, capi.PFMP_F32, o, v, True) for op, o in zip(ops, out)]
        torch.cuda.synchronize()
        # FP32 rounding of sums of ~100 products; the norm's terms average it out
        assert float((out[0] - out[1]).double().norm() / out[1].double().norm()) < 1e-6
        assert abs(nrm[0] - nrm[1]) < 1e-6 * nrm[1]
        assert abs(nrm[0] - float((v.double() * out[0].double()).sum())) < 1e-5 * nrm[0]
        plain = torch.zeros_like(v)
        capi.pfmp_kop(ops[0], capi.PFMP_F32, plain, v)
        torch.cuda.synchronize()
        assert float((plain - out[0]).double().norm() / out[0].double().norm()) < 1e-6
        for op in ops:
            capi.pfmp_op_destroy(op)
    finally:
        capi.pfmp_ctx_destroy(ctx)
