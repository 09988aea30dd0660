"""The force kernels on lattices that take their other forms: FP32 forces with one thread per
link (half-filled last blocks included) against the FP64 forces, and FP64 forces on ragged
lattices against the oracle."""
import numpy as np
import pytest
import torch

import pfmp_inputs as pin
from _util import Gpu, canon, oracle_gauge, rel_l2

pytestmark = pytest.mark.gpu

NAMES = ["gauge", "det", "filter", "filtercorr", "ratio"]


def _action(capi, g, prec, csw=1.0):
    d = capi.ActionDef()
    d.beta, d.csw, d.nkappa = 5.5, csw, 2
    d.kappa[0], d.kappa[1] = 0.120, 0.110
    d.mu, d.nu, d.tol, d.max_iter = 1.2, 0.9, 1e-11, 5000
    d.force_prec, d.md_tol = prec, (1e-6 if prec == capi.PFMP_F32 else 0.0)
    capi.pfmp_action_scheme(capi.PFMP_SCHEME_PFMP, 0, 6, d)
    return capi.pfmp_action_create_def(g.ctx, d)


# sites per parity: 9720 and 9736 (either side of the small-lattice range of the FP32 force
# kernels, 24 and 8 mod 32), 10920
@pytest.mark.parametrize("dims", [(2, 6, 6, 270), (2, 2, 2, 2434), (6, 10, 14, 26)], ids=lambda d: "x".join(map(str, d)))
def test_fp32_forces_follow_fp64(dims):
    """FP32 products are good to ~1e-6 of the force; a chain of filter factors amplifies that
    ~1e2, a solve stopped at 1e-6 leaves cond(K) x 1e-6 (~5e-5 at kappa = 0.12)."""
    from paper_1609_02652_gb300 import capi

    lat, U = oracle_gauge(dims, 0.3, 7)
    g = Gpu(lat, U)
    acts = [_action(capi, g, p) for p in (capi.PFMP_F64, capi.PFMP_F32)]
    try:
        xi = np.concatenate([canon(lat.even * torch.tensor(pin.spinor(dims, 10 + i)).reshape(*lat.shape, 4, 3)) for i in range(3)])
        F = [np.zeros(lat.V * 32) for _ in acts]
        for A in acts:
            capi.pfmp_action_heatbath(A, xi)
        for t, bar in enumerate([1e-5, 1e-5, 1e-4, 5e-4, 5e-4]):
            for A, f in zip(acts, F):
                capi.pfmp_action_force(A, t, f)
            assert rel_l2(torch.tensor(F[1]), torch.tensor(F[0])) < bar, NAMES[t]
    finally:
        for A in acts:
            capi.pfmp_action_destroy(A)
        g.close()


@pytest.mark.parametrize("dims,csw", [((6, 4, 4, 6), 1.0), ((2, 4, 6, 4), 1.0), ((4, 2, 2, 6), 0.0)])
def test_fp64_forces_ragged(dims, csw):
    from oracle.action import PFMP, PFMPParams
    from paper_1609_02652_gb300 import capi

    lat, U = oracle_gauge(dims, 0.3, 8)
    g = Gpu(lat, U)
    A = _action(capi, g, capi.PFMP_F64, csw)
    act = PFMP(lat, PFMPParams(beta=5.5, kappa=0.120, kappa_h=0.110, csw=csw, n=6, mu=1.2, nu=0.9, tol=1e-12))
    try:
        phi = [lat.even * torch.tensor(pin.spinor(dims, 20 + i)).reshape(*lat.shape, 4, 3) for i in range(3)]
        for i in range(3):
            capi.pfmp_action_set_phi(A, i, canon(phi[i]))
        refs = [act.F_gauge(U), act.F_det(U) if csw else None, act.F_poly(U, phi[0]), act.F_polycorr(U, phi[1]),
                act.F_hasen(U, phi[2])]
        F = np.zeros(lat.V * 32)
        for t, (ref, bar) in enumerate(zip(refs, [1e-12, 1e-11, 1e-11, 1e-9, 1e-9])):
            if ref is None:
                continue
            capi.pfmp_action_force(A, t, F)
            assert rel_l2(torch.tensor(F).reshape(*lat.shape, 4, 8), ref) < bar, NAMES[t]
    finally:
        capi.pfmp_action_destroy(A)
        g.close()
