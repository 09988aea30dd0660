"""What a filter force keeps on the device between calls: at most a quarter of the free memory
beyond the chain itself, and the same force with all, some or none of the chain's images kept."""
import pytest
import torch

from test_gpu_force_chains import _action

pytestmark = pytest.mark.gpu


def test_images_take_a_quarter_of_the_free_memory():
    from paper_1609_02652_gb300 import capi

    dims, order = (24, 24, 24, 24), 64
    V = 24 ** 4
    field = V // 2 * 24 * 4
    gen = torch.Generator(device="cuda").manual_seed(3)
    ctx = capi.pfmp_ctx_create(dims, -1, None)
    acts, hog = [], None
    try:
        capi.pfmp_gauge_from_algebra(ctx, torch.randn(V, 4, 8, generator=gen, dtype=torch.float64, device="cuda"), 0.4,
                                     capi.PFMP_DEVICE)
        phi = torch.randn(V, 4, 3, 2, generator=gen, dtype=torch.float64, device="cuda")
        F = [torch.zeros(V, 4, 8, dtype=torch.float64, device="cuda") for _ in range(3)]
        for k, left in enumerate((None, 9 * 10 ** 9, 3 * 10 ** 9)):
            acts.append(_action(capi, ctx, capi.PFMP_F32, order, capi.PFMP_SCHEME_1PF))
            capi.pfmp_action_set_phi(acts[k], 0, phi, capi.PFMP_DEVICE)
            if left:
                torch.cuda.empty_cache()
                hog = torch.empty(torch.cuda.mem_get_info()[0] - left, dtype=torch.uint8, device="cuda")
            before = torch.cuda.mem_get_info()[0]
            capi.pfmp_action_force(acts[k], 2, F[k], capi.PFMP_DEVICE)
            after = torch.cuda.mem_get_info()[0]
            # the chain (order fields), the contractions' fields (40) and an FP32 copy of phi, each in
            # pages of 2 MB
            if left:
                assert before - after <= before // 4 + (order + 44) * (field + 2 ** 21), (before, after)
            capi.pfmp_action_force(acts[k], 2, F[k], capi.PFMP_DEVICE)
            assert torch.cuda.mem_get_info()[0] == after  # the second call takes nothing more
            hog = None
        assert float(F[0].norm()) > 0
        assert torch.equal(F[0], F[1]) and torch.equal(F[0], F[2])
    finally:
        hog = None
        torch.cuda.empty_cache()
        for A in acts:
            capi.pfmp_action_destroy(A)
        capi.pfmp_ctx_destroy(ctx)
