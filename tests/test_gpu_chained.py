"""Kernels launched with programmatic edges: many dependent ones in a row, on two contexts with
streams of their own at once, give the bits of the same ones with a wait after each."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1], ids=["f64", "f32"])
@pytest.mark.parametrize("dims", [(4, 4, 4, 8), (8, 8, 8, 8)], ids=lambda d: "x".join(map(str, d)))
def test_chained_applications(dims, prec):
    from paper_1609_02652_gb300 import capi

    V = dims[0] * dims[1] * dims[2] * dims[3]
    gen = torch.Generator(device="cuda").manual_seed(4)
    h = torch.randn(V, 4, 8, generator=gen, dtype=torch.float64, device="cuda")
    ctxs = [capi.pfmp_ctx_create(dims, -1, None) for _ in range(2)]
    try:
        ops = []
        for c in ctxs:
            capi.pfmp_gauge_from_algebra(c, h, 0.4, capi.PFMP_DEVICE)
            ops.append(capi.pfmp_op_create(c, 0.12, 1.0))
        dt = torch.float32 if prec else torch.float64
        n = capi.pfmp_spinor_bytes(ctxs[0], prec) // (4 if prec else 8)
        v = torch.randn(n, generator=gen, dtype=dt, device="cuda")
        torch.cuda.synchronize()

        def chain(sync):
            bufs = [[v.clone(), torch.zeros_like(v)] for _ in ops]
            torch.cuda.synchronize()
            for k in range(40):
                for op, b in zip(ops, bufs):
                    capi.pfmp_kop(op, prec, b[(k + 1) & 1], b[k & 1])
                    if sync:
                        torch.cuda.synchronize()
            torch.cuda.synchronize()
            return [b[0] for b in bufs]

        want, got = chain(True), chain(False)
        assert bool(torch.isfinite(want[0]).all())
        for a in want + got:
            assert torch.equal(a, want[0])
        for op in ops:
            capi.pfmp_op_destroy(op)
    finally:
        for c in ctxs:
            capi.pfmp_ctx_destroy(c)
