"""Multi-shift CG stopped by its iteration cap inside, at and beyond a block of iterations
(the shifts' vectors are updated once per block): the residual of every shift stays a
multiple of the seed system's, b - (K + sigma) x = zeta r, exactly when x holds every
iteration that ran and no other."""
import numpy as np
import pytest
import torch

import pfmp_inputs as pin
from _util import Gpu, oracle_gauge

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ns", [1, 17, 40])
@pytest.mark.parametrize("cap", [1, 7, 8, 9, 21])
def test_capped_residuals_are_collinear(ns, cap):
    from paper_1609_02652_gb300 import capi

    lat, U = oracle_gauge((4, 4, 4, 6), 0.4, 3)
    g = Gpu(lat, U)
    try:
        op = g.op(0.125, 1.0)
        b = g.pack(lat.even * torch.tensor(pin.spinor(lat.dims, 4)).reshape(*lat.shape, 4, 3), 0, 0)
        # the seed itself (sigma = 0) and shifts from slow to fast convergence
        sigma = np.array([0.0] + [0.02 * k * np.exp(0.3j * (k % 5)) for k in range(1, ns)])
        x = [g.buf(0) for _ in sigma]
        with pytest.raises(capi.PfmpError) as e:
            capi.pfmp_solve_multishift(op, sigma, x, b, 1e-13, cap, want_info=False)
        assert e.value.status == capi.PFMP_E_NOT_CONVERGED
        res, kx = [], g.buf(0)
        for s, v in zip(sigma, x):
            capi.pfmp_kop(op, 0, kx, v)
            res.append(torch.view_as_complex((b - kx).view(-1, 2)) - complex(s) * torch.view_as_complex(v.view(-1, 2)))
        seed = res[0]
        nb = float(torch.linalg.vector_norm(b))
        assert float(torch.linalg.vector_norm(seed)) < nb
        for r in res[1:]:
            zeta = torch.vdot(seed, r) / torch.vdot(seed, seed)
            # what is left after the multiple: the solver's rounding, some 1e-15 |b| an iteration
            assert float(torch.linalg.vector_norm(r - zeta * seed)) < 1e-12 * nb
    finally:
        g.close()
