"""The filter force's chains (images kept or recomputed, more factors than pending
contractions) and the correction force's conjugate pairs."""
import numpy as np
import pytest
import torch

import pfmp_inputs as pin
from _util import Gpu, canon, oracle_gauge, rel_l2

pytestmark = pytest.mark.gpu


def _action(capi, ctx, prec, order, scheme):
    d = capi.ActionDef()
    d.beta, d.csw, d.nkappa = 5.5, 1.0, 2
    d.kappa[0], d.kappa[1] = 0.120, 0.110
    d.mu, d.nu, d.tol, d.max_iter = 1.2, 0.9, 1e-12, 5000
    d.force_prec, d.md_tol = prec, (1e-6 if prec == capi.PFMP_F32 else 0.0)
    capi.pfmp_action_scheme(scheme, 0, order, d)
    return capi.pfmp_action_create_def(ctx, d)


@pytest.mark.parametrize("order", [2, 10, 18])
def test_filter_orders(order):
    """Up to 18 factors and nine pole pairs (four pairs of contractions are pending at most). The
    bars are those of the other FP64 force tests (1e-11 for products, 1e-9 through solves at
    1e-12), times ten for the chains' length."""
    from oracle.action import PFMP, PFMPParams
    from paper_1609_02652_gb300 import capi

    dims = (4, 2, 4, 6)
    lat, U = oracle_gauge(dims, 0.3, 8)
    g = Gpu(lat, U)
    A = _action(capi, g.ctx, capi.PFMP_F64, order, capi.PFMP_SCHEME_PFMP)
    act = PFMP(lat, PFMPParams(beta=5.5, kappa=0.120, kappa_h=0.110, csw=1.0, n=order, mu=1.2, nu=0.9, tol=1e-12))
    try:
        phi = [lat.even * torch.tensor(pin.spinor(dims, 20 + i)).reshape(*lat.shape, 4, 3) for i in range(2)]
        F = np.zeros(lat.V * 32)
        for i, (ref, bar) in enumerate([(act.F_poly(U, phi[0]), 1e-10), (act.F_polycorr(U, phi[1]), 1e-8)]):
            capi.pfmp_action_set_phi(A, i, canon(phi[i]))
            capi.pfmp_action_force(A, 2 + i, F)
            assert rel_l2(torch.tensor(F).reshape(*lat.shape, 4, 8), ref) < bar
    finally:
        capi.pfmp_action_destroy(A)
        g.close()


def test_filter_force_with_little_free_memory():
    """The chain's images recomputed (4 GB of them against 5 GB free) instead of kept: the same
    kernels on the same fields, so the same bits."""
    from paper_1609_02652_gb300 import capi

    dims = (24, 24, 24, 24)
    V = 24 ** 4
    gen = torch.Generator(device="cuda").manual_seed(3)
    ctx = capi.pfmp_ctx_create(dims, -1, None)
    acts, hog = [], None
    try:
        capi.pfmp_gauge_from_algebra(ctx, torch.randn(V, 4, 8, generator=gen, dtype=torch.float64, device="cuda"), 0.4,
                                     capi.PFMP_DEVICE)
        phi = torch.randn(V, 4, 3, 2, generator=gen, dtype=torch.float64, device="cuda")
        F = [torch.zeros(V, 4, 8, dtype=torch.float64, device="cuda") for _ in range(2)]
        for k in range(2):
            acts.append(_action(capi, ctx, capi.PFMP_F32, 64, capi.PFMP_SCHEME_1PF))
            capi.pfmp_action_set_phi(acts[k], 0, phi, capi.PFMP_DEVICE)
            if k == 1:
                torch.cuda.empty_cache()
                free = torch.cuda.mem_get_info()[0]
                hog = torch.empty(max(free - 5 * 10 ** 9, 1), dtype=torch.uint8, device="cuda")
            capi.pfmp_action_force(acts[k], 2, F[k], capi.PFMP_DEVICE)
        assert float(F[0].norm()) > 0
        assert torch.equal(F[0], F[1])
    finally:
        del hog
        torch.cuda.empty_cache()
        for A in acts:
            capi.pfmp_action_destroy(A)
        capi.pfmp_ctx_destroy(ctx)
