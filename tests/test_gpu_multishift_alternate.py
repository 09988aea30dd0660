"""Multi-shift solves with different numbers of shifts in turn on one operator: the same solutions
as on an operator of their own, and no preparation repeated because the number changed."""
import time

import numpy as np
import pytest
import torch

import pfmp_inputs as pin
from _util import Gpu, oracle_gauge

pytestmark = pytest.mark.gpu

SIGMA = {3: [0.0, 0.5 + 0.5j, 2.0], 5: [0.3, 1.0 - 0.4j, 1.0 + 0.4j, 4.0, 7.0], 1: [1.5], 17: [0.25 * k for k in range(17)]}


@pytest.mark.parametrize("prec", [0, 1], ids=["f64", "f32"])
def test_solutions(prec):
    from paper_1609_02652_gb300 import capi

    lat, U = oracle_gauge((4, 4, 4, 6), 0.4, 3)
    g = Gpu(lat, U)
    try:
        b = g.pack(lat.even * torch.tensor(pin.spinor(lat.dims, 4)).reshape(*lat.shape, 4, 3), prec, 0)

        def solve(op, n, cap):
            x = [g.buf(prec) for _ in range(n)]
            try:
                capi.pfmp_solve_multishift_prec(op, prec, np.array(SIGMA[n]), x, b, 1e-6, cap)
            except capi.PfmpError as e:
                assert e.status == capi.PFMP_E_NOT_CONVERGED and cap < 100
            torch.cuda.synchronize()
            return x

        shared = g.op(0.125, 1.0)
        for n, cap in [(5, 500), (3, 500), (5, 11), (1, 500), (17, 500), (3, 3), (3, 500), (17, 500), (1, 500)]:
            for a, r in zip(solve(shared, n, cap), solve(g.op(0.125, 1.0), n, cap)):
                assert torch.equal(a, r) and float(a.abs().max()) > 0, (n, cap)
    finally:
        g.close()


def test_no_capture_per_change():
    """A solve of some 0.2 ms: one that captures its chunk anew takes several times as long."""
    from paper_1609_02652_gb300 import capi

    lat, U = oracle_gauge((4, 4, 4, 4), 0.4, 3)
    g = Gpu(lat, U)
    try:
        op = g.op(0.1, 1.0)
        b = g.pack(lat.even * torch.tensor(pin.spinor(lat.dims, 4)).reshape(*lat.shape, 4, 3), 1, 0)
        x = [g.buf(1) for _ in range(5)]
        torch.cuda.synchronize()

        def once(n):
            t = time.perf_counter()
            capi.pfmp_solve_multishift_prec(op, 1, np.array(SIGMA[n]) + 4.0, x[:n], b, 1e-3, 100)
            return time.perf_counter() - t

        for n in (5, 3, 5, 5):
            once(n)
        same = np.median([once(5) for _ in range(40)])
        turn = np.median([once(5) for _ in range(40) if once(3)])
        print("5 shifts after 5: %.0f us, after 3: %.0f us" % (same * 1e6, turn * 1e6))
        assert turn < 1.5 * same, (same, turn)
    finally:
        g.close()
