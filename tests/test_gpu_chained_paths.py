"""The kernels launched with programmatic edges beyond K itself, on two contexts with streams of
their own, driven by a thread each: an FP32 multi-shift solve above the size whose chunks are
graphs, K, the norms and copies of a mixed solve, FP32 forces with the clover terms of a new gauge
field, and an MD step.  The bits are those of a process that waits after every launch."""
import os
import subprocess
import sys
import threading

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _drive(dims, stream, out):
    import numpy as np
    import torch

    from paper_1609_02652_gb300 import capi

    def wait():  # not the device: a solve of the other thread may be capturing its chunk
        torch.cuda.current_stream().synchronize()
        stream.synchronize()

    V = dims[0] * dims[1] * dims[2] * dims[3]
    gen = torch.Generator(device="cuda").manual_seed(11)
    h = [torch.randn(V, 4, 8, generator=gen, dtype=torch.float64, device="cuda") for _ in range(3)]
    xi = torch.randn(V, 4, 3, 2, generator=gen, dtype=torch.float64, device="cuda")
    ctx = capi.pfmp_ctx_create(dims, -1, stream.cuda_stream)
    n = capi.pfmp_spinor_bytes(ctx, capi.PFMP_F32) // 4
    b = torch.randn(n, generator=gen, dtype=torch.float32, device="cuda")
    b64 = torch.randn(n, generator=gen, dtype=torch.float64, device="cuda")
    wait()
    capi.pfmp_gauge_from_algebra(ctx, h[0], 0.4, capi.PFMP_DEVICE)
    op = capi.pfmp_op_create(ctx, 0.12, 1.0)
    xs = [torch.zeros_like(b) for _ in range(3)]
    v = [b.clone(), torch.zeros_like(b)]
    x = torch.zeros_like(b64)
    wait()
    capi.pfmp_solve_multishift_prec(op, capi.PFMP_F32, np.array([0.0, 0.3 + 0.4j, 1.5 - 0.2j]), xs, b, 1e-6, 200)
    for k in range(8):
        capi.pfmp_kop(op, capi.PFMP_F32, v[(k + 1) & 1], v[k & 1])
    capi.pfmp_solve(op, capi.SolverParams(method=capi.PFMP_SOLVER_CG_MIXED, tol=1e-9, max_iter=500, delta=1e-2,
                                          check_every=8), x, b64)
    d = capi.ActionDef()
    d.beta, d.csw, d.nkappa = 5.5, 1.0, 2
    d.kappa[0], d.kappa[1] = 0.120, 0.110
    d.mu, d.nu, d.tol, d.max_iter = 1.2, 0.9, 1e-12, 5000
    d.force_prec, d.md_tol = capi.PFMP_F32, 1e-6
    capi.pfmp_action_scheme(capi.PFMP_SCHEME_PFMP, 0, 6, d)
    A = capi.pfmp_action_create_def(ctx, d)
    for i in range(3):
        capi.pfmp_action_set_phi(A, i, xi, capi.PFMP_DEVICE)
    forces = []
    for eps in (0.4, 0.3):  # a new gauge field: links, field strength, clover terms
        capi.pfmp_gauge_from_algebra(ctx, h[1], eps, capi.PFMP_DEVICE)
        capi.pfmp_action_refresh(A)
        for term in range(5):
            F = torch.zeros(V, 4, 8, dtype=torch.float64, device="cuda")
            wait()
            capi.pfmp_action_force(A, term, F, capi.PFMP_DEVICE)
            forces.append(F)
    T, S = capi.pfmp_schedule_2mn(1, 0.05, 0.19)
    P = h[2]
    capi.pfmp_md(A, T, np.array([S]), [0] * 5, P, capi.PFMP_DEVICE)
    wait()
    for i, t in enumerate(xs + [v[0], x] + forces + [P]):
        out[f"{'x'.join(map(str, dims))}_{i}"] = t.cpu().numpy()
    capi.pfmp_action_destroy(A)
    capi.pfmp_op_destroy(op)
    capi.pfmp_ctx_destroy(ctx)


def _main(path):
    import numpy as np
    import torch

    sys.path.insert(0, ROOT)
    out, errors = {}, []

    def run(dims):
        try:
            _drive(dims, torch.cuda.Stream(), out)
        except Exception as e:  # noqa: BLE001
            errors.append(repr(e))

    torch.zeros(1, device="cuda")
    threads = [threading.Thread(target=run, args=(d,)) for d in ((16, 16, 16, 18), (4, 4, 4, 8))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    if errors:
        sys.exit("; ".join(errors))
    np.savez(path, **out)


@pytest.mark.gpu
def test_same_bits_as_with_waits(tmp_path):
    import numpy as np

    res = []
    for wait in ("1", "0"):
        path = str(tmp_path / f"out{wait}.npz")
        env = dict(os.environ, CUDA_LAUNCH_BLOCKING=wait)
        r = subprocess.run([sys.executable, os.path.abspath(__file__), path], env=env, capture_output=True, text=True,
                           timeout=300, cwd=ROOT)
        assert r.returncode == 0, r.stderr[-2000:]
        res.append(np.load(path))
    assert sorted(res[0].files) == sorted(res[1].files) and len(res[0].files) == 2 * 16
    for k in res[0].files:
        assert np.isfinite(res[0][k]).all(), k
        assert np.array_equal(res[0][k], res[1][k]), k
        assert np.abs(res[0][k]).max() > 0, k


if __name__ == "__main__":
    _main(sys.argv[1])
