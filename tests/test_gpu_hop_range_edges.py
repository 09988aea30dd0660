"""The one-thread-per-site stencils around every change of their resident-block bound: FP32 at the
first size past its four-block range, FP16 storage on both sides of each of its ranges (2, 4 and 6
blocks), with and without the sum."""
import pytest
import torch

pytestmark = pytest.mark.gpu

# sites per parity: 38912 | 38976 (2, 4 blocks), 77824 | 77888 (4, 6; FP32: 4, 7), 116736 | 116800
# (6, 4), 331776 (6)
DIMS = {38912: (4, 16, 16, 76), 38976: (2, 8, 12, 406), 77824: (8, 16, 16, 76), 77888: (2, 16, 2, 2434),
        116736: (8, 16, 12, 152), 116800: (8, 10, 20, 146), 331776: (24, 24, 24, 48)}
H16_BAR = 7.8e-3  # 16 roundings of FP16, as in test_gpu_operator


@pytest.mark.parametrize("vh", sorted(DIMS))
def test_fp32_and_fp16_storage(vh):
    from paper_1609_02652_gb300 import capi

    dims = DIMS[vh]
    V = dims[0] * dims[1] * dims[2] * dims[3]
    assert V == 2 * vh
    gen = torch.Generator(device="cuda").manual_seed(2)
    ctx = capi.pfmp_ctx_create(dims, -1, None)
    try:
        capi.pfmp_gauge_from_algebra(ctx, torch.randn(V, 4, 8, generator=gen, dtype=torch.float64, device="cuda"), 0.4,
                                     capi.PFMP_DEVICE)
        op, other = (capi.pfmp_op_create(ctx, 0.12, 1.0) for _ in range(2))
        capi.pfmp_op_set_split(other, capi.PFMP_F32, 2)
        n = capi.pfmp_spinor_bytes(ctx, capi.PFMP_F32) // 4
        v = torch.randn(n, generator=gen, dtype=torch.float32, device="cuda")
        out, ref, plain, back = (torch.zeros_like(v) for _ in range(4))
        torch.cuda.synchronize()
        nrm, nref = capi.pfmp_kop(op, capi.PFMP_F32, out, v, True), capi.pfmp_kop(other, capi.PFMP_F32, ref, v, True)
        capi.pfmp_kop(op, capi.PFMP_F32, plain, v)
        torch.cuda.synchronize()
        rel = lambda a, b: float((a - b).double().norm() / b.double().norm())  # noqa: E731
        assert rel(out, ref) < 1e-6 and rel(plain, ref) < 1e-6 and abs(nrm - nref) < 1e-6 * nref
        h_in, h_out = (torch.zeros(capi.pfmp_spinor_bytes(ctx, capi.PFMP_H16), dtype=torch.uint8, device="cuda")
                       for _ in range(2))
        torch.cuda.synchronize()
        capi.pfmp_convert(ctx, h_in, capi.PFMP_H16, v, capi.PFMP_F32)
        nh = capi.pfmp_kop(op, capi.PFMP_H16, h_out, h_in, True)
        capi.pfmp_convert(ctx, back, capi.PFMP_F32, h_out, capi.PFMP_H16)
        torch.cuda.synchronize()
        assert rel(back, ref) < H16_BAR and abs(nh - nref) < H16_BAR * nref
        h_out.zero_()
        torch.cuda.synchronize()
        capi.pfmp_kop(op, capi.PFMP_H16, h_out, h_in)
        capi.pfmp_convert(ctx, plain, capi.PFMP_F32, h_out, capi.PFMP_H16)
        torch.cuda.synchronize()
        assert rel(plain, ref) < H16_BAR
        for o in (op, other):
            capi.pfmp_op_destroy(o)
    finally:
        capi.pfmp_ctx_destroy(ctx)
