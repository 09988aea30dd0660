"""The FP64 gauge force on both sides of the change from a thread per leaf to a thread per link
(768 sites per parity), ragged last blocks among them, against the oracle; and its time on a large
lattice against the FP64 pipe's."""
import time

import numpy as np
import pytest
import torch

from _util import Gpu, oracle_gauge, rel_l2

pytestmark = pytest.mark.gpu


def _action(capi, ctx):
    d = capi.ActionDef()
    d.beta, d.csw, d.nkappa, d.nterms = 5.5, 0.0, 1, 1
    d.kappa[0] = 0.12
    d.term[0] = capi.Term(capi.PFMP_KIND_GAUGE, 0, 0, 0, 0)
    d.mu, d.nu, d.tol, d.max_iter = 1.2, 0.9, 1e-12, 5000
    d.solver, d.force_prec, d.md_tol = capi.PFMP_SOLVER_CG64, capi.PFMP_F64, 0.0
    return capi.pfmp_action_create_def(ctx, d)


# 8, 760 | 768, 776 (8 past a block), 1296 sites per parity
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (2, 2, 10, 38), (4, 4, 4, 24), (2, 2, 2, 194), (6, 6, 6, 12)],
                         ids=lambda d: "x".join(map(str, d)))
def test_against_oracle(dims):
    from oracle.action import PFMP, PFMPParams
    from paper_1609_02652_gb300 import capi

    lat, U = oracle_gauge(dims, 0.4, 8)
    g = Gpu(lat, U)
    A = _action(capi, g.ctx)
    try:
        F = np.zeros(lat.V * 32)
        capi.pfmp_action_force(A, 0, F)
        ref = PFMP(lat, PFMPParams(beta=5.5, kappa=0.120, kappa_h=0.110, csw=0.0, n=2, mu=1.2, nu=0.9, tol=1e-12)).F_gauge(U)
        assert rel_l2(torch.tensor(F).reshape(*lat.shape, 4, 8), ref) < 1e-12
    finally:
        capi.pfmp_action_destroy(A)
        g.close()


def test_time_is_the_pipes():
    """52 colour products per site, 108 multiply-adds each, at the measured FP64 rate."""
    from paper_1609_02652_gb300 import capi

    dims = (16, 16, 16, 32)
    V = 16 ** 3 * 32
    gen = torch.Generator(device="cuda").manual_seed(1)
    ctx = capi.pfmp_ctx_create(dims, -1, None)
    try:
        capi.pfmp_gauge_from_algebra(ctx, torch.randn(V, 4, 8, generator=gen, dtype=torch.float64, device="cuda"), 0.4,
                                     capi.PFMP_DEVICE)
        A = _action(capi, ctx)
        F = torch.zeros(V, 4, 8, dtype=torch.float64, device="cuda")

        def once():
            torch.cuda.synchronize()
            t = time.perf_counter()
            for _ in range(10):
                capi.pfmp_action_force(A, 0, F, capi.PFMP_DEVICE)
            torch.cuda.synchronize()
            return (time.perf_counter() - t) / 10

        once()
        pipe = V * 52 * 108 * 2 / (capi.pfmp_fma_rate(ctx, capi.PFMP_F64) * 1e12)
        best = min(once() for _ in range(3))
        print("FP64 gauge force %.0f us, pipe %.0f us" % (best * 1e6, pipe * 1e6))
        assert best < 1.5 * pipe
        capi.pfmp_action_destroy(A)
    finally:
        capi.pfmp_ctx_destroy(ctx)
