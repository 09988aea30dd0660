"""Cases that time the library through its public entry points (capi), over the range of
lattices, precisions and steps of the method that a user's program calls:

    kop         out = K in = M-hat^dag M-hat in, the operator itself
    solve       x = K^{-1} b (CG in FP64, mixed, or on FP16 storage)
    multishift  x_k = (K + sigma_k)^{-1} b for the poles of a filter correction
    force       the FP64 force of one action term
    trajectory  heatbath, both Hamiltonians, MD and accept step on a small lattice
    md          molecular dynamics of the multi-filter action with FP32 forces
    nn          one application of the learned preconditioner
    batch       many systems with several right-hand sides each in one call

Fields are synthetic: links exp(i eps H) with Gaussian algebra coefficients (eps = 0.5 has
about the plaquette of a thermalised field at beta = 5.5), Gaussian spinors and momenta.
The reference values (exact) are plain torch in complex128 and share nothing with the
library but the conventions of include/pfmp.h.
"""
import math

import numpy as np
import torch

from paper_1609_02652_gb300 import capi

LAMBDA_2MN = 0.1931833275037836
PREC = {"f64": capi.PFMP_F64, "f32": capi.PFMP_F32}
METHOD = {"cg64": capi.PFMP_SOLVER_CG64, "mixed": capi.PFMP_SOLVER_CG_MIXED, "half": capi.PFMP_SOLVER_CG_HALF}


def listed():
    return [
        # the smallest call: K on a tuning-size lattice, four launches of one to two blocks
        {"name": "kop_f32_4x8", "kind": "kop", "dims": "4,4,4,8", "prec": "f32", "eps": 0.3, "kappa": 0.12, "csw": 1.0},
        # the operator at the size where it streams from HBM
        {"name": "kop_f32_32x64", "kind": "kop", "dims": "32,32,32,64", "prec": "f32", "eps": 0.5, "kappa": 0.13, "csw": 1.0},
        # FP64 operator on the benchmark lattice: filter products, heatbath, true residuals
        {"name": "kop_f64_16x32", "kind": "kop", "dims": "16,16,16,32", "prec": "f64", "eps": 0.5, "kappa": 0.13, "csw": 1.0},
        # the benchmark's solve
        {"name": "solve_mixed_16x32", "kind": "solve", "method": "mixed", "dims": "16,16,16,32", "eps": 0.5, "kappa": 0.13,
         "csw": 1.0, "tol": 1e-10, "delta": 1e-4},
        # a measurement's solve on the largest lattice, on FP16 storage
        {"name": "solve_half_32x64", "kind": "solve", "method": "half", "dims": "32,32,32,64", "eps": 0.5, "kappa": 0.13,
         "csw": 1.0, "tol": 1e-10, "delta": 0.03},
        # the action's default solver, at the actions' tolerance
        {"name": "solve_cg64_12x24", "kind": "solve", "method": "cg64", "dims": "12,12,12,24", "eps": 0.4, "kappa": 0.128,
         "csw": 1.0, "tol": 1e-12, "delta": 0.1},
        # the correction force's solve inside a production MD: 13 poles, FP32
        {"name": "multishift_f32_24x48", "kind": "multishift", "dims": "24,24,24,48", "prec": "f32", "eps": 0.5,
         "kappa": 0.12, "csw": 1.0, "order": 12, "tol": 1e-6},
        # the FP64 force of a filter correction on a ragged lattice
        {"name": "force_f64_6x10x14x18", "kind": "force", "dims": "6,10,14,18", "eps": 0.4, "kappa": 0.11, "csw": 1.0,
         "order": 12, "tol": 1e-12},
        # a whole PF-MP trajectory on the smallest lattice: latency and launches
        {"name": "trajectory_4x4", "kind": "trajectory", "dims": "4,4,4,4", "eps": 0.3, "kappa": 0.12, "kappa_h": 0.11,
         "csw": 1.0, "order": 8, "steps": 2, "tau": 0.125, "tol": 1e-12},
        # the production MD (two filters, two mass ratios, four time scales), FP32 forces
        {"name": "md_f32_24x48", "kind": "md", "dims": "24,24,24,48", "eps": 0.5, "csw": 1.0, "p1": 12, "p2": 64,
         "steps": 1, "tau": 0.1},
        # the learned preconditioner of the benchmark
        {"name": "nn_16x32", "kind": "nn", "dims": "16,16,16,32", "eps": 0.5, "hidden": 2},
        # many systems at once: two each on three lattices, one to eight right-hand sides
        {"name": "batch_6", "kind": "batch", "systems": 6, "eps": 0.4, "kappa": 0.122, "csw": 1.0, "tol": 1e-10,
         "delta": 1e-4},
    ]


def _draw_dims(rng, vmin, vmax):
    """Even extents whose volume is near a log-uniform target in [vmin, vmax]."""
    target = math.exp(rng.uniform(math.log(vmin), math.log(vmax)))
    while True:
        d = [2 * round(math.exp(rng.uniform(math.log(2), math.log(16)))) for _ in range(3)]
        d.append(2 * round(math.exp(rng.uniform(math.log(2), math.log(32)))))
        v = d[0] * d[1] * d[2] * d[3]
        if vmin <= v <= vmax and target / 1.4 <= v <= target * 1.4:
            return ",".join(str(x) for x in d)


def draw(rng):
    kind = rng.choice(["kop", "kop", "kop", "solve", "solve", "solve", "multishift", "force", "force", "trajectory", "md",
                       "nn", "batch"])
    c = {"kind": kind}
    if kind == "kop":
        c |= {"dims": _draw_dims(rng, 256, 2 ** 21), "prec": rng.choice(["f32", "f64"]), "eps": 0.5,
              "kappa": round(rng.uniform(0.11, 0.134), 4), "csw": rng.choice([0.0, 1.0, 1.0, 1.6])}
        if c["prec"] == "f64":
            c["dims"] = _draw_dims(rng, 256, 2 ** 19)
    elif kind == "solve":
        m = rng.choice(["mixed", "half", "cg64"])
        c |= {"method": m, "dims": _draw_dims(rng, 512, 2 ** 17 if m == "cg64" else 2 ** 20),
              "eps": round(rng.uniform(0.4, 0.5), 3), "kappa": round(rng.uniform(0.118, 0.128), 4),
              "csw": 1.0, "tol": 1e-12 if m == "cg64" else 1e-10, "delta": {"mixed": 1e-4, "half": 0.03, "cg64": 0.1}[m]}
    elif kind == "multishift":
        p = rng.choice(["f32", "f64"])
        c |= {"dims": _draw_dims(rng, 1024, 2 ** 19 if p == "f32" else 2 ** 16), "prec": p, "eps": 0.5,
              "kappa": round(rng.uniform(0.11, 0.122), 4), "csw": 1.0, "order": rng.choice([4, 8, 12, 16]),
              "tol": 1e-6 if p == "f32" else 1e-12}
    elif kind == "force":
        c |= {"dims": _draw_dims(rng, 512, 2 ** 15), "eps": 0.4, "kappa": round(rng.uniform(0.105, 0.118), 4),
              "csw": rng.choice([0.0, 1.0, 1.0]), "order": rng.choice([4, 8, 12]), "tol": 1e-12}
    elif kind == "trajectory":
        c |= {"dims": _draw_dims(rng, 256, 4096), "eps": 0.3, "kappa": round(rng.uniform(0.115, 0.122), 4), "kappa_h": 0.11,
              "csw": 1.0, "order": rng.choice([4, 8]), "steps": rng.choice([1, 2]), "tau": 0.125, "tol": 1e-12}
    elif kind == "md":
        c |= {"dims": _draw_dims(rng, 8192, 2 ** 18), "eps": 0.5, "csw": rng.choice([1.0, 1.2]), "p1": 4, "p2": 24,
              "steps": 1, "tau": 0.1}
    elif kind == "nn":
        c |= {"dims": _draw_dims(rng, 4096, 2 ** 18), "eps": 0.5, "hidden": rng.choice([1, 2])}
    else:
        c |= {"systems": rng.choice([2, 3, 4, 5]), "eps": round(rng.uniform(0.35, 0.45), 3),
              "kappa": round(rng.uniform(0.118, 0.124), 4), "csw": 1.0, "tol": 1e-10, "delta": 1e-4}
    return c


# ------------------------------------------------------------------ inputs
def _dims(text):
    return tuple(int(v) for v in text.split(","))


def _volume(dims):
    return dims[0] * dims[1] * dims[2] * dims[3]


def _generator(seed, stream):
    return torch.Generator(device="cuda").manual_seed((int(seed) * 1000003 + stream) % (2 ** 63))


def _normal(seed, stream, *shape):
    return torch.randn(*shape, generator=_generator(seed, stream), dtype=torch.float64, device="cuda")


def _algebra(dims, seed, stream=1):
    return _normal(seed, stream, _volume(dims), 4, 8)


def _noise(dims, seed, stream, *batch):
    """Canonical Gaussian spinors [batch][V][4][3] complex, density exp(-xi^dag xi)."""
    return _normal(seed, stream, *batch, _volume(dims), 4, 3, 2) * math.sqrt(0.5)


class _System:
    """A context with its gauge field and the operators, actions and networks on it."""

    def __init__(self, dims, seed, eps, stream=1):
        self.dims = dims
        self.handles = []
        self.ctx = capi.pfmp_ctx_create(dims, -1, None)
        capi.pfmp_gauge_from_algebra(self.ctx, _algebra(dims, seed, stream), eps, capi.PFMP_DEVICE)

    def op(self, kappa, csw):
        return self.own(capi.pfmp_op_create(self.ctx, kappa, csw), capi.pfmp_op_destroy)

    def own(self, handle, destroy):
        self.handles.append((handle, destroy))
        return handle

    def field(self, prec):
        dt = torch.float64 if prec == capi.PFMP_F64 else torch.float32
        return torch.zeros(capi.pfmp_spinor_bytes(self.ctx, prec) // dt.itemsize, dtype=dt, device="cuda")

    def packed(self, xi, prec):
        f = self.field(prec)
        capi.pfmp_spinor_pack(self.ctx, f, prec, xi, capi.PFMP_DEVICE, 0)
        return f

    def __del__(self):
        for handle, destroy in reversed(self.handles):
            destroy(handle)
        capi.pfmp_ctx_destroy(self.ctx)


def _poles(order):
    """Chebyshev roots z_1..z_n of P_n, (mu, nu) = (1.2, 0.9), and the pole at zero."""
    mu, nu = 1.2, 0.9
    t = 2 * np.pi * np.arange(1, order + 1) / (order + 1)
    z = mu * (1 - np.cos(t)) - 1j * math.sqrt(mu * mu - nu * nu) * np.sin(t)
    return np.concatenate([z, [0.0]]), 1.0 / (mu * np.prod(mu - z)).real


def _params(c):
    return capi.SolverParams(method=METHOD[c.get("method", "mixed")], tol=c["tol"], max_iter=20000, delta=c["delta"],
                             check_every=8)


def _schedule(tau, steps):
    return capi.pfmp_schedule_merge([capi.pfmp_schedule_2mn(n, tau, LAMBDA_2MN) for n in steps])


def _batch_systems(c):
    lattices = [(8, 8, 8, 8), (12, 12, 12, 24), (16, 16, 16, 32)]
    return [(lattices[s % 3], c["kappa"] + 0.001 * s, 1 + (5 * s + 2) % 8) for s in range(c["systems"])]


def prepare(case, seed):
    c = dict(case)
    s = {"case": c}
    if c["kind"] == "batch":
        s["sys"], s["ops"], s["b"], s["x"], s["nrhs"] = [], [], [], [], []
        for k, (dims, kappa, nrhs) in enumerate(_batch_systems(c)):
            y = _System(dims, seed, c["eps"], 100 + k)
            s["sys"].append(y)
            s["ops"].append(y.op(kappa, c["csw"]))
            s["nrhs"].append(nrhs)
            for r in range(nrhs):
                s["b"].append(y.packed(_noise(dims, seed, 1000 + 10 * k + r), capi.PFMP_F64))
                s["x"].append(y.field(capi.PFMP_F64))
        # the first system owns the batch, so the operators outlive it
        last = s["sys"][-1]
        s["batch"] = last.own(capi.pfmp_batch_create(s["ops"], s["nrhs"]), capi.pfmp_batch_destroy)
        return s
    dims = _dims(c["dims"])
    y = s["sys"] = _System(dims, seed, c["eps"])
    if c["kind"] == "kop":
        s["op"] = y.op(c["kappa"], c["csw"])
        s["in"], s["out"] = y.packed(_noise(dims, seed, 2), PREC[c["prec"]]), y.field(PREC[c["prec"]])
    elif c["kind"] == "solve":
        s["op"] = y.op(c["kappa"], c["csw"])
        s["b"], s["x"] = y.packed(_noise(dims, seed, 2), capi.PFMP_F64), y.field(capi.PFMP_F64)
    elif c["kind"] == "multishift":
        s["op"] = y.op(c["kappa"], c["csw"])
        s["sigma"] = -_poles(c["order"])[0]
        s["b"] = y.packed(_noise(dims, seed, 2), PREC[c["prec"]])
        s["x"] = [y.field(PREC[c["prec"]]) for _ in s["sigma"]]
    elif c["kind"] == "force":
        d = capi.ActionDef()
        d.beta, d.csw, d.nkappa, d.nterms = 5.5, c["csw"], 1, 1
        d.kappa[0] = c["kappa"]
        d.term[0] = capi.Term(capi.PFMP_KIND_FILTERCORR, 0, 0, 0, c["order"])
        d.mu, d.nu, d.tol, d.max_iter = 1.2, 0.9, c["tol"], 20000
        s["action"] = y.own(capi.pfmp_action_create_def(y.ctx, d), capi.pfmp_action_destroy)
        capi.pfmp_action_set_phi(s["action"], 0, _noise(dims, seed, 2), capi.PFMP_DEVICE)
        s["F"] = torch.zeros(_volume(dims), 4, 8, dtype=torch.float64, device="cuda")
    elif c["kind"] in ("trajectory", "md"):
        if c["kind"] == "trajectory":
            p = capi.ActionParams(beta=5.5, kappa=c["kappa"], kappa_h=c["kappa_h"], csw=c["csw"], n=c["order"], mu=1.2,
                                  nu=0.9, tol=c["tol"], max_iter=5000)
            s["action"] = y.own(capi.pfmp_action_create(y.ctx, p), capi.pfmp_action_destroy)
            s["levels"] = [1, 1, 1, 0, 0]
            steps = (c["steps"], 2 * c["steps"])
        else:
            d = capi.ActionDef()
            d.beta, d.csw, d.nkappa, d.nterms = 5.5, c["csw"], 3, 7
            d.kappa[0], d.kappa[1], d.kappa[2] = 0.130, 0.115, 0.125
            terms = [(capi.PFMP_KIND_GAUGE, 0, 0, 0, 0), (capi.PFMP_KIND_DET, 0, 0, 0, 0),
                     (capi.PFMP_KIND_FILTER, 1, 0, 0, c["p1"]), (capi.PFMP_KIND_FILTER, 1, 0, c["p1"], c["p2"]),
                     (capi.PFMP_KIND_FILTERCORR, 1, 0, 0, c["p2"]), (capi.PFMP_KIND_RATIO, 1, 2, 0, 0),
                     (capi.PFMP_KIND_RATIO, 2, 0, 0, 0)]
            for k, t in enumerate(terms):
                d.term[k] = capi.Term(*t)
            d.mu, d.nu, d.tol, d.max_iter = 1.44, 1.08, 1e-10, 20000
            d.solver, d.force_prec, d.md_tol = capi.PFMP_SOLVER_CG_MIXED, capi.PFMP_F32, 1e-6
            s["action"] = y.own(capi.pfmp_action_create_def(y.ctx, d), capi.pfmp_action_destroy)
            s["levels"] = [0, 0, 1, 2, 3, 3, 3]
            n = c["steps"]
            steps = (6 * n, 3 * n, 2 * n, n)
        s["T"], s["S"] = _schedule(c["tau"], steps)
        s["npf"] = capi.pfmp_action_counts(s["action"])[1]
        s["xi"] = _noise(dims, seed, 2, s["npf"])
        s["mom0"] = _algebra(dims, seed, 3)
        s["mom"] = torch.empty_like(s["mom0"])
        s["U0"] = torch.empty(_volume(dims), 4, 3, 3, 2, dtype=torch.float64, device="cuda")
        s["U"] = torch.empty_like(s["U0"])
        capi.pfmp_gauge_get(y.ctx, s["U0"], capi.PFMP_DEVICE)
        if c["kind"] == "md":
            capi.pfmp_action_heatbath(s["action"], s["xi"], capi.PFMP_DEVICE)
            del s["xi"]
    elif c["kind"] == "nn":
        s["nn"] = y.own(capi.pfmp_nn_create(y.ctx, _channels(c)), capi.pfmp_nn_destroy)
        capi.pfmp_nn_set_weights(s["nn"], _weights(c, seed))
        s["in"], s["out"] = y.packed(_noise(dims, seed, 2), capi.PFMP_F32), y.field(capi.PFMP_F32)
    return s


def _channels(c):
    return [1] + [8] * (c["hidden"] + 1) + [1]


def _weights(c, seed):
    """Gaussian weights with the identity on the on-site block, a network before training."""
    r, out = np.random.RandomState(int(seed) % (2 ** 31)), []
    for ci, co in zip(_channels(c)[:-1], _channels(c)[1:]):
        w = (r.standard_normal((9, co, ci, 4, 4)) + 1j * r.standard_normal((9, co, ci, 4, 4))) * (0.3 / (4 * math.sqrt(9 * ci)))
        for k in range(min(ci, co)):
            w[0, k, k] += np.eye(4)
        out.append(w)
    return out


# ------------------------------------------------------------------ one pass
def run(s):
    c = s["case"]
    if c["kind"] == "kop":
        capi.pfmp_kop(s["op"], PREC[c["prec"]], s["out"], s["in"])
        return s["out"]
    if c["kind"] == "solve":
        capi.pfmp_solve(s["op"], _params(c), s["x"], s["b"])
        return s["x"]
    if c["kind"] == "multishift":
        capi.pfmp_solve_multishift_prec(s["op"], PREC[c["prec"]], s["sigma"], s["x"], s["b"], c["tol"], 20000)
        return s["x"]
    if c["kind"] == "force":
        capi.pfmp_action_force(s["action"], 0, s["F"], capi.PFMP_DEVICE)
        return s["F"]
    if c["kind"] == "nn":
        capi.pfmp_nn_apply(s["nn"], capi.PFMP_F32, s["out"], s["in"])
        return s["out"]
    if c["kind"] == "batch":
        capi.pfmp_batch_solve(s["batch"], _params(c), s["x"], s["b"])
        return s["x"]
    # from a stored configuration and momenta, as a program that runs or reverses a trajectory
    ctx, act = s["sys"].ctx, s["action"]
    capi.pfmp_gauge_set(ctx, s["U0"], capi.PFMP_DEVICE)
    capi.pfmp_action_refresh(act)
    if c["kind"] == "trajectory":
        info = capi.pfmp_trajectory(act, s["T"], s["S"], s["levels"], s["mom0"], s["xi"], 0.0, capi.PFMP_DEVICE)
        capi.pfmp_gauge_get(ctx, s["U"], capi.PFMP_DEVICE)
        return {"U": s["U"], "S0": np.array(info.S0[:5]), "S1": np.array(info.S1[:5]), "H": np.array([info.H0, info.H1])}
    s["mom"].copy_(s["mom0"])
    capi.pfmp_md(act, s["T"], s["S"], s["levels"], s["mom"], capi.PFMP_DEVICE)
    capi.pfmp_gauge_get(ctx, s["U"], capi.PFMP_DEVICE)
    # forces in FP32 leave the fields with that accuracy: stored in single precision
    return {"U": s["U"].float(), "mom": s["mom"].float()}


# ------------------------------------------------------------------ what a pass cannot do without
_K_FLOPS = 4 * 1896        # per half-lattice site: four hops and four clover multiplications
_K_REALS = 96 + 144        # per half-lattice site: 8 links of 12 reals, the clover of both parities


def _k_bytes(prec, vh):
    return (_K_REALS + 48) * (8 if prec == "f64" else 4) * vh


def _solve_iters(kappa):
    """CG iterations to 1e-10, nominal."""
    return 40 + 50 * max(0.0, (kappa - 0.11) / 0.02)


def work(case):
    c = case
    if c["kind"] == "batch":
        n = [(_volume(d) // 2, r, _solve_iters(k)) for d, k, r in _batch_systems(c)]
        return {"bytes": sum(v * (_K_REALS * 4 + r * 384) for v, r, _ in n), "flops": sum(v * r * i * _K_FLOPS for v, r, i in n)}
    vh = _volume(_dims(c["dims"])) // 2
    if c["kind"] == "kop":
        return {"bytes": _k_bytes(c["prec"], vh), "flops": _K_FLOPS * vh}
    if c["kind"] == "solve":
        # every iteration needs the operator and three vectors; FP16 storage halves the operator
        per = {"cg64": 8 * (_K_REALS + 144), "mixed": 4 * (_K_REALS + 144), "half": 2 * _K_REALS + 4 * 96 + 2 * 48}[c["method"]]
        n = _solve_iters(c["kappa"]) * (1.2 if c["method"] == "cg64" else 1.0)
        return {"bytes": n * per * vh, "flops": n * _K_FLOPS * vh}
    if c["kind"] == "multishift":
        n = 0.6 * _solve_iters(c["kappa"])
        b = 8 if c["prec"] == "f64" else 4
        return {"bytes": vh * b * (n * (_K_REALS + 96) + (c["order"] + 1) * 24), "flops": n * _K_FLOPS * vh}
    if c["kind"] == "force":
        n, m = 1.2 * _solve_iters(c["kappa"]), c["order"] + 1
        return {"bytes": 8 * vh * (72 + 144 + 24 + 64), "flops": vh * (n * _K_FLOPS + m * (2 * _K_FLOPS + 16 * 400))}
    if c["kind"] == "nn":
        ch = _channels(c)
        v = 2 * vh
        mix = sum(9 * ci * co * 4 * 4 * 3 * 8 for ci, co in zip(ch[:-1], ch[1:]))
        act = sum(2 * 48 * k for k in ch[1:-1])
        return {"bytes": v * (4 * 48 + act) + vh * 192, "flops": v * mix}
    # per trajectory: links, momenta and pseudofermions in and out; the products of the terms
    if c["kind"] == "trajectory":
        k = 4 * c["steps"] * 2 * c["order"] + 300 * (2 + 2 * c["steps"])
        return {"bytes": vh * 8 * 2 * (288 + 64), "flops": k * _K_FLOPS * vh}
    k = 12 * c["steps"] * c["p1"] * 4 + 4 * c["steps"] * c["p2"] * 5 + 2 * c["steps"] * (4 * c["p2"] + 400)
    return {"bytes": vh * (8 * 2 * (288 + 64) + 2 * _K_REALS * 4), "flops": k * _K_FLOPS * vh}


# ------------------------------------------------------------------ the same in 64 bits, plain torch
def _gammas():
    i = 1j
    g = [[[0, 0, 0, i], [0, 0, i, 0], [0, -i, 0, 0], [-i, 0, 0, 0]], [[0, 0, 0, -1], [0, 0, 1, 0], [0, 1, 0, 0], [-1, 0, 0, 0]],
         [[0, 0, i, 0], [0, 0, 0, -i], [-i, 0, 0, 0], [0, i, 0, 0]], [[0, 0, 1, 0], [0, 0, 0, 1], [1, 0, 0, 0], [0, 1, 0, 0]]]
    return torch.tensor(g, dtype=torch.complex128, device="cuda")


def _generators():
    lam = torch.zeros(8, 3, 3, dtype=torch.complex128, device="cuda")
    for a, (i, j) in enumerate([(0, 1), (0, 2), (1, 2)]):
        n = (0, 3, 5)[a]
        lam[n, i, j] = lam[n, j, i] = 1
        lam[n + 1, i, j], lam[n + 1, j, i] = -1j, 1j
    lam[2, 0, 0], lam[2, 1, 1] = 1, -1
    lam[7] = torch.diag(torch.tensor([1.0, 1.0, -2.0], dtype=torch.complex128)) / math.sqrt(3)
    return lam / 2


class _Exact:
    """M-hat and K on full-lattice fields [Lt][Lz][Ly][Lx][4][3], zero on odd sites."""

    def __init__(self, dims, U, kappa=0.0, csw=0.0):
        self.dims, self.kappa, self.G = dims, kappa, _gammas()
        self.shape = (dims[3], dims[2], dims[1], dims[0])
        x = torch.meshgrid(*[torch.arange(n, device="cuda") for n in self.shape], indexing="ij")
        self.parity = (x[0] + x[1] + x[2] + x[3]) % 2
        self.even = (self.parity == 0).to(torch.float64)[..., None, None]
        self.U = [U[..., mu, :, :] for mu in range(4)]
        self.A = self.Ainv = None
        if kappa:
            A = torch.eye(12, dtype=torch.complex128, device="cuda").expand(*self.shape, 12, 12)
            if csw:
                for mu in range(4):
                    for nu in range(mu + 1, 4):
                        sig = 0.5j * (self.G[mu] @ self.G[nu] - self.G[nu] @ self.G[mu])
                        A = A - kappa * csw * torch.einsum("rs,...ab->...rasb", sig, self._strength(mu, nu)).reshape(*self.shape, 12, 12)
            # the clover term is block diagonal in chirality
            self.A = [A[..., :6, :6].contiguous(), A[..., 6:, 6:].contiguous()]
            self.Ainv = [torch.linalg.inv(b) for b in self.A]

    @staticmethod
    def shift(f, mu, d, tail):
        """f(x + d mu-hat) of a field with `tail` trailing dimensions."""
        return torch.roll(f, -d, dims=f.dim() - tail - 1 - mu)

    def _strength(self, mu, nu):
        m, n, S = self.U[mu], self.U[nu], lambda f, k, d: self.shift(f, k, d, 2)
        H = lambda f: f.mH  # noqa: E731
        mm, nm, nn, mn = S(m, mu, -1), S(n, mu, -1), S(n, nu, -1), S(m, nu, -1)
        Q = m @ S(n, mu, 1) @ H(S(m, nu, 1)) @ H(n) + n @ H(S(mm, nu, 1)) @ H(nm) @ mm
        Q = Q + H(mm) @ H(S(nm, nu, -1)) @ S(mm, nu, -1) @ nn + H(nn) @ mn @ S(nn, mu, 1) @ H(m)
        F = (Q - H(Q)) / 8j
        return F - (F.diagonal(dim1=-2, dim2=-1).sum(-1) / 3)[..., None, None] * torch.eye(3, dtype=F.dtype, device=F.device)

    def fshift(self, psi, mu, d):
        """A shifted spinor field, antiperiodic in time."""
        f = self.shift(psi, mu, d, 2)
        if mu == 3:
            sgn = torch.ones(self.shape[0], 1, 1, 1, 1, 1, dtype=torch.float64, device="cuda")
            sgn[-1 if d > 0 else 0] = -1
            f = f * sgn
        return f

    def hop(self, psi, s=1.0):
        """H psi (s = 1) or H^dag psi (s = -1)."""
        out = torch.zeros_like(psi)
        for mu in range(4):
            f = self.fshift(psi, mu, 1) @ self.U[mu].transpose(-1, -2)
            b = self.fshift(psi @ self.U[mu].conj(), mu, -1)
            out = out + f + b - s * (self.G[mu] @ (f - b))
        return out

    @staticmethod
    def blocks(B, psi):
        v = psi.reshape(*psi.shape[:-2], 2, 6, 1)
        return torch.stack([B[0] @ v[..., 0, :, :], B[1] @ v[..., 1, :, :]], -3).reshape(psi.shape)

    def mhat(self, psi, s=1.0):
        t = (1 - self.even) * self.blocks(self.Ainv, self.hop(psi, s))
        return self.even * (self.blocks(self.A, psi) - self.kappa ** 2 * self.hop(t, s))

    def K(self, psi):
        return self.mhat(self.mhat(psi), -1.0)

    def cg(self, b, tol=1e-14, most=2000):
        x, r = torch.zeros_like(b), b.clone()
        p, rr = r.clone(), _norm2(r)
        stop = tol * tol * rr
        while rr > stop and most:
            q = self.K(p)
            a = rr / _dot(p, q).real
            x, r = x + a * p, r - a * q
            new = _norm2(r)
            p, rr, most = r + (new / rr) * p, new, most - 1
        return x

    def shifted(self, sigma, b, tol=1e-14):
        """(K + sigma_k)^{-1} b for every shift, from one Krylov space."""
        n = len(sigma)
        x = [torch.zeros_like(b) for _ in range(n)]
        ps, z0, z1 = [b.clone() for _ in range(n)], [1.0 + 0j] * n, [1.0 + 0j] * n
        r, p, rr = b.clone(), b.clone(), _norm2(b)
        stop, a0, b0 = tol * tol * rr, 1.0, 0.0
        for _ in range(2000):
            q = self.K(p)
            a = rr / _dot(p, q).real
            r = r - a * q
            new = _norm2(r)
            be = new / rr
            live = False
            for k in range(n):
                if abs(z1[k]) ** 2 * rr < stop:
                    continue
                live = True
                z2 = z1[k] * z0[k] * a0 / (a0 * z0[k] * (1 + a * sigma[k]) + a * b0 * (z0[k] - z1[k]))
                f = z2 / z1[k]
                x[k] = x[k] + complex(a * f) * ps[k]
                ps[k] = complex(z2) * r + complex(be * f * f) * ps[k]
                z0[k], z1[k] = z1[k], z2
            p, rr, a0, b0 = r + be * p, new, a, be
            if not live:
                break
        return x

    def field(self, xi):
        """The even sites of a canonical spinor."""
        return torch.view_as_complex(xi).reshape(*self.shape, 4, 3) * self.even

    def layout(self, psi, prec):
        """A full field's even sites in the library's device order: words of one (FP64) or
        two (FP32) complex numbers, sites fastest."""
        v = psi.reshape(-1, 12)[(self.parity == 0).reshape(-1)]
        per = 1 if prec == "f64" else 2
        return torch.view_as_real(v.reshape(-1, 12 // per, per).transpose(0, 1).contiguous()).reshape(-1)


def _dot(x, y):
    return complex(torch.vdot(x.reshape(-1), y.reshape(-1)))


def _norm2(x):
    return _dot(x, x).real


def _exact_links(dims, seed, eps, stream=1):
    T = _generators()
    h = _algebra(dims, seed, stream).reshape(-1, 8)
    U = torch.cat([torch.linalg.matrix_exp(1j * eps * torch.einsum("na,aij->nij", p.to(T.dtype), T)) for p in h.split(1 << 20)])
    return U.reshape(dims[3], dims[2], dims[1], dims[0], 4, 3, 3)


def exact(case, seed):
    c = dict(case)
    if c["kind"] in ("trajectory", "md"):
        return None
    if c["kind"] == "batch":
        out = []
        for k, (dims, kappa, nrhs) in enumerate(_batch_systems(c)):
            small = _volume(dims) < 100000
            E = _Exact(dims, _exact_links(dims, seed, c["eps"], 100 + k), kappa, c["csw"]) if small else None
            for r in range(nrhs):
                out.append(E.layout(E.cg(E.field(_noise(dims, seed, 1000 + 10 * k + r))), "f64") if small else None)
        return out
    dims = _dims(c["dims"])
    if c["kind"] != "kop" and _volume(dims) > 300000:
        return None
    U = _exact_links(dims, seed, c["eps"])
    if c["kind"] == "nn":
        return _exact_network(c, _Exact(dims, U), seed)
    if c["kind"] == "force":
        return _exact_force(c, dims, U, seed)
    E = _Exact(dims, U, c["kappa"], c["csw"])
    b = E.field(_noise(dims, seed, 2))
    if c["kind"] == "kop":
        return E.layout(E.K(b), c["prec"])
    if c["kind"] == "solve":
        return E.layout(E.cg(b), "f64")
    return [E.layout(x, c["prec"]) for x in E.shifted(list(-_poles(c["order"])[0]), b)]


def _exact_network(c, E, seed):
    a = [E.field(_noise(E.dims, seed, 2))]
    for w in _weights(c, seed):
        w = torch.tensor(w, device="cuda")
        out = [0] * w.shape[1]
        for i, v in enumerate(a):
            hops = [v] + [E.fshift(v, mu, 1) @ E.U[mu].transpose(-1, -2) for mu in range(4)]
            hops += [E.fshift(v @ E.U[mu].conj(), mu, -1) for mu in range(4)]
            for o in range(len(out)):
                for d in range(9):
                    out[o] = out[o] + w[d, o, i] @ hops[d]
        a = out
    return E.layout(E.even * a[0], "f32")


def _exact_force(c, dims, U, seed):
    """The force of phi^dag [J P_n(J)]^{-1} phi = sum_i r_i phi^dag (J - z_i)^{-1} phi: the
    gradient of -Re sum_i eta_i^dag J(U) chi_i at fixed chi_i = r_i (J - z_i)^{-1} phi and
    eta_i = (J - z_i^*)^{-1} phi, along U -> exp(i w T_a) U."""
    z, a_n = _poles(c["order"])
    E = _Exact(dims, U, c["kappa"], c["csw"])
    x = E.shifted(list(-z), E.field(_noise(dims, seed, 2)))
    U = U.detach().clone().requires_grad_(True)
    E = _Exact(dims, U, c["kappa"], c["csw"])
    L = 0.0
    for i in range(len(z)):
        r = 1.0 / (a_n * np.prod([z[i] - z[j] for j in range(len(z)) if j != i]))
        conj = min(range(len(z)), key=lambda j: abs(z[j] - z[i].conjugate()))
        L = L - (E.mhat(x[conj]).conj() * E.mhat(complex(r) * x[i])).sum().real
    G, = torch.autograd.grad(L, U)
    # dL = Re sum conj(G) dU with dU = i T_a U
    W = (U.detach() @ G.mH).reshape(-1, 4, 3, 3)
    return torch.einsum("smij,aji->sma", 1j * W, _generators()).real.contiguous()
