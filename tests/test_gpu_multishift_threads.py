"""First multi-shift solves (those that prepare a chunk's graph) while another thread keeps
synchronising the device, which no stream capture survives."""
import threading

import numpy as np
import pytest
import torch

import pfmp_inputs as pin
from _util import Gpu, oracle_gauge

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1], ids=["f64", "f32"])
def test_first_solves_beside_device_synchronisation(prec):
    from paper_1609_02652_gb300 import capi

    lat, U = oracle_gauge((4, 4, 4, 4), 0.4, 3)
    g = Gpu(lat, U)
    stop, errors = threading.Event(), []

    def other():
        try:
            while not stop.is_set():
                torch.cuda.synchronize()
        except Exception as e:  # noqa: BLE001
            errors.append(repr(e))

    thread = threading.Thread(target=other)
    try:
        b = g.pack(lat.even * torch.tensor(pin.spinor(lat.dims, 4)).reshape(*lat.shape, 4, 3), prec, 0)
        sigma = np.array([0.1, 0.5 + 0.5j, 2.0])
        ops = [g.op(0.12, 1.0) for _ in range(41)]
        xs = [[g.buf(prec) for _ in sigma] for _ in ops]
        torch.cuda.synchronize()
        capi.pfmp_solve_multishift_prec(ops[0], prec, sigma, xs[0], b, 1e-6, 500)
        thread.start()
        for op, x in zip(ops[1:], xs[1:]):
            capi.pfmp_solve_multishift_prec(op, prec, sigma, x, b, 1e-6, 500)
        stop.set()
        thread.join()
        assert not errors, errors
        for x in xs[1:]:
            for a, r in zip(x, xs[0]):
                assert torch.equal(a, r) and float(a.abs().max()) > 0
    finally:
        stop.set()
        if thread.is_alive():
            thread.join()
        g.close()
