"""Measured workloads of the library, each through its public entry points.

A case is a dict of plain values; ``prepare`` makes its inputs on the GPU (or
in page-locked host memory where the entry point takes host data), ``run`` does
one pass as a user's program does it, ``work`` says what the pass cannot do
without and ``exact`` evaluates it in 64 bits with plain torch.

The kinds:

``update``   gsm_update, the batched implicit-Euler material update.
``host``     gsm_update_host, the same on page-locked host arrays.
``ode``      gsm_update_ode23, the adaptive update of the force-potential form.
``scheme``   ms_run, the basic scheme over a load history on a planned context.
``serve``    a batch of homogenization jobs through the serving engine.
``adjoint``  ms_run_taped + ms_adjoint, the gradient of the effective stress.
"""
import math

import numpy as np
import torch

import paper_2006_04391_gb300 as G

# The repository's matrix law (E, nu, sigma0, edot0, n) without its exponent, its
# stiff inclusion and its soft fibre (E, nu).
MATRIX = (70.0, 0.3, 0.1, 1.0)
INCLUSION = (400.0, 0.2)
FIBRE = (72.0, 0.22)

PRECISION = {"fp64": 0, "fix": 1, "fp32": 2}
SCHEME_EVALS_PER_SERVED_STEP = 60  # a served step's material evaluations, for work() only


def listed():
    return [
        # a few integration points of a finite-element patch: the launch and the
        # latency of one voxel decide (4096 + 5 voxels is the smoke check's batch)
        {"name": "update_small", "kind": "update", "n": 4101, "precision": "fix", "tangent": False, "exponent": 5.0,
         "h": 0.01},
        # the benchmark's material-law batch: 2^24 voxels, FP32 search and FP64 correction
        {"name": "update_bulk", "kind": "update", "n": 1 << 24, "precision": "fix", "tangent": False, "exponent": 5.0,
         "h": 0.01},
        # the full-precision update on a ragged batch, the fibre composite's exponent
        {"name": "update_fp64", "kind": "update", "n": 3000017, "precision": "fp64", "tangent": False,
         "exponent": 10.0, "h": 0.1},
        # the update with the consistent tangent (the derivative direction: a Newton
        # solver's or the reference medium's call), a ragged batch
        {"name": "update_tangent", "kind": "update", "n": 1000003, "precision": "fp64", "tangent": True,
         "exponent": 5.0, "h": 0.01},
        # the FP32 update (FP32 in, out and arithmetic)
        {"name": "update_fp32", "kind": "update", "n": 5000011, "precision": "fp32", "tangent": False,
         "exponent": 3.0, "h": 0.01},
        # fields that live in host memory (a CPU elasticity solver, as in the paper)
        {"name": "update_host", "kind": "host", "n": 2000003, "precision": "fix", "exponent": 5.0, "h": 0.01},
        # the adaptive Runge-Kutta update of the force-potential form (rtol 1e-3)
        {"name": "ode23", "kind": "ode", "n": 200003, "exponent": 5.0, "h": 0.1},
        # the first steps of the 16^3 sphere composite, FP64, solved to 1e-8: many tiny iterations
        {"name": "scheme_16", "kind": "scheme", "N": 16, "micro": "sphere", "fraction": 0.1, "exponent": 5.0,
         "precision": "fp64", "steps": 2, "evals": 0, "amplitude": 0.002},
        # the paper's 150^3 grid, fibres, FP64, a bounded number of iterations per step
        {"name": "scheme_fp64", "kind": "scheme", "N": 150, "micro": "fibres", "fraction": 0.15, "exponent": 10.0,
         "precision": "fp64", "steps": 2, "evals": 8, "amplitude": 0.002},
        # the 256^3 fibre composite in FP32 bulk with its FP64 finish
        {"name": "scheme_bulk", "kind": "scheme", "N": 256, "micro": "fibres", "fraction": 0.15, "exponent": 10.0,
         "precision": "bulk", "steps": 1, "evals": 60, "amplitude": 0.001},
        # a burst of small and medium jobs on one server, mixed grids
        {"name": "serve_burst", "kind": "serve", "jobs": 10, "grid_lo": 32, "grid_hi": 64, "steps": 2, "tol": 1e-4},
        # the gradient of the final stress through a short history
        {"name": "adjoint", "kind": "adjoint", "N": 64, "fraction": 0.2, "exponent": 5.0, "steps": 2, "evals": 10,
         "adj_iters": 20},
    ]


def _log_int(rng, lo, hi):
    v = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return max(lo, min(hi, v | 1 if rng.random() < 0.5 else v))


def draw(rng):
    """One more case: every kind over its whole range of sizes, exponents,
    precisions and options (cost at most the largest listed one's)."""
    kind = rng.choice(["update", "update", "update", "update", "scheme", "scheme", "scheme", "ode", "host", "serve",
                       "adjoint"])
    exponent = rng.choice([1.0, 2.0, 3.0, 5.0, 10.0, 20.0])
    h = 10.0 ** rng.uniform(-3.0, -1.0)
    if kind == "update":
        tangent = rng.random() < 0.3
        return {"kind": kind, "n": _log_int(rng, 1, 4000000 if tangent else 1 << 24),
                "precision": rng.choice(["fp64", "fix", "fp32"]), "tangent": tangent, "exponent": exponent, "h": h}
    if kind == "host":
        return {"kind": kind, "n": _log_int(rng, 100000, 2000003), "precision": rng.choice(["fp64", "fix", "fp32"]),
                "exponent": exponent, "h": h}
    if kind == "ode":
        return {"kind": kind, "n": _log_int(rng, 10000, 200003), "exponent": rng.choice([3.0, 5.0]), "h": 0.1}
    if kind == "scheme":
        bulk = rng.random() < 0.5
        N = _log_int(rng, 8, 192 if bulk else 128)
        if rng.random() < 0.5:  # half of them FFT-friendly, the others as they fall
            N = min((8, 12, 16, 20, 24, 32, 40, 48, 60, 64, 80, 96, 100, 120, 128, 160, 192), key=lambda k: abs(k - N))
        return {"kind": kind, "N": N, "micro": rng.choice(["sphere", "fibres"]), "fraction": rng.uniform(0.05, 0.25),
                "exponent": rng.choice([3.0, 5.0, 10.0]), "precision": "bulk" if bulk else "fp64",
                "steps": rng.choice([1, 2, 3]), "evals": rng.randint(6, 20), "amplitude": rng.uniform(0.0005, 0.002)}
    if kind == "serve":
        lo = rng.choice([16, 24, 32])
        return {"kind": kind, "jobs": rng.randint(2, 10), "grid_lo": lo, "grid_hi": lo + rng.choice([8, 16, 32]),
                "steps": rng.choice([1, 2]), "tol": 1e-4}
    return {"kind": kind, "N": _log_int(rng, 12, 64), "fraction": rng.uniform(0.1, 0.3),
            "exponent": rng.choice([3.0, 5.0, 10.0]), "steps": rng.choice([1, 2]), "evals": rng.randint(6, 12),
            "adj_iters": rng.randint(8, 20)}


# ------------------------------------------------------------------- inputs

def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _uniform(gen, shape, amp, dtype=torch.float64):
    return (torch.rand(shape, generator=gen, device="cuda", dtype=dtype) * 2 - 1) * amp


def _internal(gen, n, dtype):
    """Deviatoric internal variables, the independent components U[-0.005, 0.005]."""
    y = _uniform(gen, (5, n), 0.005, dtype)
    return torch.stack([y[0], y[1], -y[0] - y[1], y[2], y[3], y[4]])


def _batch(case, seed):
    """The material-law batch: eps ~ U[-0.02, 0.02]^6, z_n deviatoric."""
    dtype = torch.float32 if case["precision"] == "fp32" else torch.float64
    gen = _generator(seed)
    return _uniform(gen, (6, case["n"]), 0.02, dtype), _internal(gen, case["n"], dtype)


def _ode_batch(case, seed):
    """Load-step-like voxels: strain increments of a fraction of the yield strain."""
    gen = _generator(seed)
    n = case["n"]
    zn = _internal(gen, n, torch.float64)
    eps_n = zn + _uniform(gen, (6, n), 0.002)
    return eps_n, eps_n + _uniform(gen, (6, n), 0.001), zn


def _sphere(N, fraction, rng):
    """One sphere, its centre moved off the grid's centre by less than a voxel."""
    r = (3.0 * fraction * N ** 3 / (4.0 * math.pi)) ** (1.0 / 3.0)
    c = torch.arange(N, device="cuda", dtype=torch.float64) + 0.5 - 0.5 * N
    o = rng.uniform(-0.5, 0.5, 3)
    d2 = ((c - o[0]) ** 2)[:, None, None] + ((c - o[1]) ** 2)[None, :, None] + ((c - o[2]) ** 2)[None, None, :]
    return (d2 <= r * r).to(torch.uint8)


def _fibres(N, fraction, rng):
    """Straight fibres with axes in the x-y plane (aspect ratio 15 on large grids),
    periodic, placed at random until their volumes add up to the fraction."""
    r = max(1.5, 6.0 * N / 256.0)
    length = min(30.0 * r, 0.7 * N)
    count = max(1, int(round(fraction * N ** 3 / (math.pi * r * r * length))))
    c = torch.arange(N, device="cuda", dtype=torch.float32) + 0.5
    ph = torch.zeros((N, N, N), dtype=torch.uint8, device="cuda")
    for _ in range(count):
        x, y, z = rng.uniform(0, N, 3)
        a = rng.uniform(0, math.pi)
        wrap = [torch.remainder(c - v + 0.5 * N, N) - 0.5 * N for v in (float(x), float(y), float(z))]
        dx, dy = wrap[0][:, None], wrap[1][None, :]
        t = (dx * math.cos(a) + dy * math.sin(a)).clamp(-0.5 * length, 0.5 * length)
        d2 = (dx - t * math.cos(a)) ** 2 + (dy - t * math.sin(a)) ** 2
        near = (wrap[2].abs() <= r).nonzero()[:, 0]
        ph[:, :, near] |= (d2[:, :, None] + wrap[2][near][None, None, :] ** 2 <= r * r).to(torch.uint8)
    return ph


def _direction(rng):
    d = rng.normal(size=6)
    return d / np.linalg.norm(d)


def _ramp(steps, end):
    return np.array([(k / steps) * np.asarray(end) for k in range(1, steps + 1)])


def _scheme_inputs(case, seed):
    """Phase field, laws of the phases (kind, parameters) and the load history."""
    rng = np.random.default_rng(seed)
    micro = case.get("micro", "sphere")
    phase = (_sphere if micro == "sphere" else _fibres)(case["N"], case["fraction"], rng)
    spec = [(1, MATRIX + (case["exponent"],)), (0, INCLUSION if micro == "sphere" else FIBRE)]
    E = _ramp(case["steps"], case.get("amplitude", 0.003) * _direction(rng))
    return phase, spec, E, [0.1] * case["steps"]


def _laws(spec, precision):
    return [G.norton(*p, precision=precision) if kind == 1 else G.elastic(*p) for kind, p in spec]


def _serve_jobs(case, seed):
    """Jobs of mixed grids and microstructures, matrix exponents 3, 5 and 10."""
    rng = np.random.default_rng(seed)
    grids = np.linspace(case["grid_lo"], case["grid_hi"], 3).round().astype(int)
    jobs = []
    for k in range(case["jobs"]):
        N = int(grids[k % 3])
        if k % 2:
            phase, fraction = _fibres, rng.uniform(0.10, 0.30)
        else:
            phase, fraction = _sphere, rng.uniform(0.05, 0.25)
        spec = [(1, MATRIX + ((3.0, 5.0, 10.0)[(k // 3) % 3],)), (0, INCLUSION)]
        E = _ramp(case["steps"], 0.001 * case["steps"] * _direction(rng))
        jobs.append({"phase": phase(N, fraction, rng).cpu().numpy(), "spec": spec, "E": E,
                     "h": [0.1] * case["steps"]})
    return jobs


def prepare(case, seed):
    G.load()
    kind = case["kind"]
    if kind == "update":
        eps, zn = _batch(case, seed)
        mat = G.norton(*MATRIX, case["exponent"], precision=PRECISION[case["precision"]])
        tan = torch.empty((21, case["n"]), dtype=eps.dtype, device="cuda") if case["tangent"] else None
        return {"case": case, "mat": mat, "eps": eps, "zn": zn, "sig": torch.empty_like(eps),
                "z": torch.empty_like(eps), "tan": tan}
    if kind == "host":
        eps, zn = (t.cpu().pin_memory() for t in _batch(case, seed))
        mat = G.norton(*MATRIX, case["exponent"], precision=PRECISION[case["precision"]])
        return {"case": case, "mat": mat, "eps": eps, "zn": zn, "sig": torch.empty_like(eps).pin_memory(),
                "z": torch.empty_like(eps).pin_memory()}
    if kind == "ode":
        eps_n, eps, zn = _ode_batch(case, seed)
        return {"case": case, "mat": G.norton(*MATRIX, case["exponent"]), "eps_n": eps_n, "eps": eps, "zn": zn,
                "sig": torch.empty_like(eps), "z": torch.empty_like(eps)}
    if kind in ("scheme", "adjoint"):
        phase, spec, E, h = _scheme_inputs(case, seed)
        bulk = case.get("precision") == "bulk"
        laws = _laws(spec, G.GSM_FP32_FP64FIX if bulk else G.GSM_FP64)
        ctx = G.ms_create(phase, laws, G.MS_PREC_FP32_BULK if bulk else G.MS_PREC_FP64)
        state = {"case": case, "ctx": ctx, "phase": phase, "laws": laws, "E": E, "h": h}
        if kind == "scheme":
            field = torch.empty((6, case["N"] ** 3), dtype=torch.float64, device="cuda")
            state.update(eps=field, z=torch.empty_like(field))
        return state
    jobs = _serve_jobs(case, seed)
    for j in jobs:
        j["laws"] = _laws(j["spec"], G.GSM_FP32_FP64FIX)
    return {"case": case, "server": G.Server(8 << 30, 64), "jobs": jobs}


# ------------------------------------------------------------------ a pass

def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "update":
        G.gsm_update(state["mat"], state["eps"], state["zn"], case["h"], state["sig"], state["z"], state["tan"])
        return [state["sig"], state["z"]] + ([state["tan"]] if case["tangent"] else [])
    if kind == "host":
        # the caller reads the results in host memory: they are there once the stream has passed the call
        G.gsm_update_host(state["mat"], state["eps"], state["zn"], case["h"], state["sig"], state["z"])
        torch.cuda.current_stream().synchronize()
        return [state["sig"], state["z"]]
    if kind == "ode":
        G.gsm_update_ode23(state["mat"], state["eps_n"], state["eps"], state["zn"], case["h"], state["sig"],
                           state["z"])
        return [state["sig"], state["z"]]
    if kind == "scheme":
        evals = [case["evals"]] * case["steps"] if case["evals"] else None
        bulk = case["precision"] == "bulk"
        res = G.ms_run(state["ctx"], state["E"], state["h"], tol=1e-12 if evals else 1e-8, forced_iters=evals,
                       eps=state["eps"], z=state["z"], switch_tol=1e-12 if bulk and evals else 0.0)
        if bulk:
            # FP32 fields, FFTs and laws: the caller keeps the fields in the type they were computed in
            return {"Sigma": res["Sigma"].astype(np.float32), "eps": state["eps"].float(), "z": state["z"].float()}
        # (the equilibrium errors the solve ends with are differences that cancel: their last digits are rounding)
        return {"Sigma": res["Sigma"], "iters": res["iters"], "eps": state["eps"], "z": state["z"]}
    if kind == "adjoint":
        res, tape = G.ms_run_taped(state["ctx"], state["E"], state["h"], tol=1e-12,
                                   forced_iters=[case["evals"]] * case["steps"])
        grads = []
        for w in np.eye(6)[[0, 5]]:  # two of the stress components: the normal and the in-plane shear one
            g, _ = G.ms_adjoint(tape, w, 0, tol=1e-30, max_iter=case["adj_iters"], check=False)
            grads.append(g)
        return {"Sigma": res["Sigma"], "grad": np.stack(grads)}
    server = state["server"]
    ids = [server.submit(j["phase"], j["laws"], j["E"], j["h"], tol=case["tol"]) for j in state["jobs"]]
    while True:
        active, queued, _ = server.tick()
        if not active and not queued:
            break
    # FP32-bulk solves to 1e-4: the effective stresses in the type they were computed in
    return [server.fetch(i)["Sigma"].astype(np.float32) for i in ids]


# ----------------------------------------------------------- what it takes

def _evaluations_work(N, count, size):
    """Material evaluations of the basic scheme: the law reads the strain and z_n
    and writes z (18 values a voxel and its phase id), a 3-D transform that does
    not fit on the chip takes two passes each way (24 values read and written
    as spectra, half of them redundant); FFT 2.5 N log2 N flops each way."""
    v = float(N) ** 3
    return {"bytes": count * v * (1 + 42 * size), "flops": count * v * (2 * 6 * 2.5 * 3 * math.log2(N) + 150 + 60)}


def work(case):
    kind = case["kind"]
    if kind in ("update", "host"):
        size = 4 if case["precision"] == "fp32" else 8
        tangent = case.get("tangent", False)
        # trial strain 13, its norm 8, one power 30, the step 20, stress and z 20; the tangent 60
        return {"bytes": float(case["n"] * size * (24 + (21 if tangent else 0))),
                "flops": float(case["n"] * (91 + (60 if tangent else 0)))}
    if kind == "ode":
        # 23 accepted and 7 rejected substeps of three right-hand sides (50) and an error (60)
        return {"bytes": float(case["n"] * 8 * 30), "flops": float(case["n"] * 30 * 210)}
    if kind == "scheme":
        evals = case["evals"] or 2000  # evaluations of a step solved to 1e-8 at this contrast
        size = 4 if case["precision"] == "bulk" else 8
        return _evaluations_work(case["N"], evals * case["steps"], size)
    if kind == "adjoint":
        # a forward evaluation and a conjugate-gradient iteration each take a transform each way
        return _evaluations_work(case["N"], (case["evals"] + 2 * case["adj_iters"]) * case["steps"], 8)
    parts = [_evaluations_work(N, SCHEME_EVALS_PER_SERVED_STEP * case["steps"], 4)
             for N in np.linspace(case["grid_lo"], case["grid_hi"], 3)[np.arange(case["jobs"]) % 3]]
    return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}


# ------------------------------------------------- the same in plain 64 bits

def _lame(E, nu):
    return E * nu / ((1.0 + nu) * (1.0 - 2.0 * nu)), E / (2.0 * (1.0 + nu))


def _norton_exact(prm, eps, zn, h, tangent=False):
    """The implicit-Euler step of the Norton law as a radial return, 64 bits.

    With the deviatoric trial strain e the flow is theta e; the von Mises stress
    s of the step solves s + 3 mu h edot0 (s / sigma0)^n = s_trial, in the
    variable ln s by bracketed Newton."""
    E, nu, s0, e0, n = prm
    lam, mu = _lame(E, nu)
    kappa = lam + 2.0 * mu / 3.0
    zn = zn.clone()
    zn[2] = -zn[0] - zn[1]
    tr = eps[:3].sum(0)
    dev = eps - zn
    dev[:3] -= tr / 3.0
    norm2 = (dev[:3] ** 2).sum(0) + 0.5 * (dev[3:] ** 2).sum(0)   # e : e on the tensor
    s_trial = 2.0 * mu * torch.sqrt(1.5 * norm2)
    c = 3.0 * mu * h * e0
    # x = s / sigma0 solves sigma0 x + c x^n = s_trial; start above the root
    pos = s_trial > 0
    st = torch.where(pos, s_trial, torch.ones_like(s_trial))
    u = torch.minimum(torch.log(st / s0), torch.log(st / c) / n)
    for _ in range(60):
        a, b = s0 * torch.exp(u), c * torch.exp(n * u)
        du = (a + b - st) / (a + n * b)
        u = u - du
        if float(du.abs().max()) < 1e-15:
            break
    a, b = s0 * torch.exp(u), c * torch.exp(n * u)
    rest = torch.where(pos, a / (a + b), torch.ones_like(a))      # s / s_trial
    flow = torch.where(pos, b / (a + b), torch.zeros_like(a))     # theta
    z = zn + flow * dev
    z[2] = -z[0] - z[1]
    w = torch.tensor([2.0, 2.0, 2.0, 1.0, 1.0, 1.0], dtype=eps.dtype, device=eps.device)[:, None] * mu
    sig = w * rest * dev
    sig[:3] += kappa * tr
    if not tangent:
        return sig, z
    # sigma = kappa tr 1 + 2 mu rest(e:e) e, and d(rest)/de from the scalar equation
    p = 1.0 / n
    slope = -(1.0 - p) * flow * rest / (p * rest + flow)          # d ln-slope times rest
    t = w / mu * 0.5 * dev                                        # tensor components of e
    inv = torch.where(norm2 > 0, 1.0 / torch.where(norm2 > 0, norm2, torch.ones_like(norm2)),
                      torch.zeros_like(norm2))
    out = torch.empty((21,) + eps.shape[1:], dtype=eps.dtype, device=eps.device)
    k = 0
    for i in range(6):
        for j in range(i, 6):
            v = 2.0 * mu * slope * inv * t[i] * t[j]
            if i < 3 and j < 3:
                v = v + kappa + 2.0 * mu * rest * ((1.0 if i == j else 0.0) - 1.0 / 3.0)
            elif i == j:
                v = v + mu * rest
            out[k] = v
            k += 1
    return sig, z, out


def _elastic_exact(prm, eps):
    lam, mu = _lame(*prm)
    sig = mu * eps
    sig[:3] = 2.0 * mu * eps[:3] + lam * eps[:3].sum(0)
    return sig


def _ode23_exact(prm, eps_n, eps, zn, h, rtol=1e-3, atol=1e-6):
    """The Bogacki-Shampine 3(2) integration with the stress-driven step control."""
    E, nu, s0, e0, n = prm
    lam, mu = _lame(E, nu)
    de = eps - eps_n
    z = zn.clone()
    z[2] = -z[0] - z[1]

    def stress(theta, z):
        return _elastic_exact((E, nu), eps_n + theta * de - z)

    def rate(theta, z):
        s = stress(theta, z)
        d = s.clone()
        d[:3] -= s[:3].mean(0)
        eq = torch.sqrt(1.5 * ((d[:3] ** 2).sum(0) + 2.0 * (d[3:] ** 2).sum(0)))
        r = 1.5 * e0 / s0 * (eq / s0) ** (n - 1.0) * d
        r[3:] *= 2.0
        return r

    t = torch.zeros_like(eps[0])
    dt = torch.full_like(t, h)
    done = torch.zeros_like(t, dtype=torch.bool)
    rejected = torch.zeros_like(done)
    k1, old = rate(0.0, z), stress(0.0, z)
    for _ in range(20000):
        clip = t + dt >= h
        dt = torch.where(clip, h - t, dt)
        tn = torch.where(clip, torch.full_like(t, h), t + dt)
        k2 = rate((t + 0.5 * dt) / h, z + 0.5 * dt * k1)
        k3 = rate((t + 0.75 * dt) / h, z + 0.75 * dt * k2)
        z3 = z + dt * (2.0 * k1 + 3.0 * k2 + 4.0 * k3) / 9.0
        k4 = rate(tn / h, z3)
        z2 = z + dt * (7.0 / 24.0 * k1 + 0.25 * k2 + k3 / 3.0 + 0.125 * k4)
        hi, lo = stress(tn / h, z3), stress(tn / h, z2)
        e = (hi - lo) / (atol + rtol * torch.maximum(old.abs(), hi.abs()))
        err = torch.sqrt((e * e).mean(0))
        err = torch.where(torch.isfinite(err), err, torch.full_like(err, 1e300))
        f = torch.where(err == 0, torch.full_like(err, 1e300), 0.9 * err ** (-1.0 / 3.0))
        most = torch.where(rejected, torch.ones_like(f), torch.full_like(f, 5.0))
        ok = (err <= 1.0) & ~done
        z, k1, old = torch.where(ok, z3, z), torch.where(ok, k4, k1), torch.where(ok, hi, old)
        t = torch.where(ok, tn, t)
        rejected = torch.where(done, rejected, ~ok)
        done = done | (ok & clip)
        dt = torch.where(done, dt, dt * torch.minimum(most, f.clamp(min=0.2)))
        if bool(done.all()):
            break
    return old, z


class _Scheme:
    """The basic scheme in 64 bits on torch fields [6, N, N, N]."""

    def __init__(self, phase, spec):
        self.N = N = phase.shape[0]
        self.phase, self.spec = phase, spec
        lm = [_lame(p[0], p[1]) for _, p in spec]
        self.lam0 = 0.5 * (min(a for a, _ in lm) + max(a for a, _ in lm))
        self.mu0 = 0.5 * (min(b for _, b in lm) + max(b for _, b in lm))
        f = torch.fft.fftfreq(N, d=1.0 / N, device="cuda", dtype=torch.float64).round()
        fr = torch.arange(N // 2 + 1, device="cuda", dtype=torch.float64)
        self.k = [f[:, None, None], f[None, :, None], fr[None, None, :]]
        some = sum((k != 0).to(torch.int8) for k in self.k)
        skip = some == 0
        if N % 2 == 0:
            edge = (self.k[0].abs() == N // 2) | (self.k[1].abs() == N // 2) | (self.k[2].abs() == N // 2)
            skip = skip | (edge & (some >= 2))
        self.keep = (~skip).to(torch.float64)
        self.weight = torch.full_like(fr, 2.0)
        self.weight[0] = 1.0
        if N % 2 == 0:
            self.weight[-1] = 1.0
        self.masks = [(phase.reshape(-1) == p).nonzero()[:, 0] for p in range(len(spec))]

    def law(self, eps, zn, h):
        e, z0 = eps.reshape(6, -1), zn.reshape(6, -1)
        sig, z = torch.empty_like(e), torch.zeros_like(e)
        for (kind, prm), at in zip(self.spec, self.masks):
            if kind == 1:
                sig[:, at], z[:, at] = _norton_exact(prm, e[:, at], z0[:, at], h)
            else:
                sig[:, at] = _elastic_exact(prm, e[:, at])
        return sig.reshape(eps.shape), z.reshape(eps.shape)

    def update(self, sig, eps, E):
        """(equilibrium error, the next strain)."""
        N, k = self.N, self.k
        mean = sig.mean(dim=(1, 2, 3))
        s = [torch.fft.rfftn(sig[c]) for c in range(6)]
        rows = ((0, 5, 4), (5, 1, 3), (4, 3, 2))
        q = [sum(s[c] * k[j] for j, c in enumerate(row)) * self.keep for row in rows]
        power = sum((x.real ** 2 + x.imag ** 2) for x in q)
        num = 2.0 * math.pi * math.sqrt(float((power * self.weight).sum())) / N ** 3
        m = mean.tolist()
        den = math.sqrt(sum((1.0 if c < 3 else 2.0) * m[c] ** 2 for c in range(6)))
        k2 = k[0] ** 2 + k[1] ** 2 + k[2] ** 2
        k2 = torch.where(k2 == 0, torch.ones_like(k2), k2)
        kq = (k[0] * q[0] + k[1] * q[1] + k[2] * q[2]) * (self.lam0 + self.mu0) / (
            self.mu0 * (self.lam0 + 2.0 * self.mu0)) / k2 ** 2
        out = torch.empty_like(eps)
        for c, (i, j) in enumerate(((0, 0), (1, 1), (2, 2), (1, 2), (0, 2), (0, 1))):
            d = (k[j] * q[i] + k[i] * q[j]) / (2.0 * self.mu0 * k2) - kq * k[i] * k[j]
            d[0, 0, 0] = 0.0
            step = torch.fft.irfftn(d, s=(N, N, N)) * (1.0 if c < 3 else 2.0)
            out[c] = eps[c] - step
            out[c] += E[c] - out[c].mean()
        return num / max(den, 1e-6 * self.mu0), out, m

    def solve(self, E, h, evals, tol):
        N = self.N
        eps = torch.zeros((6, N, N, N), dtype=torch.float64, device="cuda")
        zn = torch.zeros_like(eps)
        prev = np.zeros(6)
        Sigma, iters = [], []
        for Ek, hk in zip(E, h):
            eps = eps + torch.tensor(Ek - prev, device="cuda")[:, None, None, None]
            count = 0
            while True:
                sig, z = self.law(eps, zn, hk)
                count += 1
                e, nxt, mean = self.update(sig, eps, Ek)
                if count >= evals if evals else (e < tol or count >= 10000):
                    break
                eps = nxt
            zn, prev = z, Ek
            Sigma.append(mean)
            iters.append(count)
        flat = [t.reshape(6, -1) for t in (eps, zn)]
        return np.array(Sigma), np.array(iters, dtype=np.int32), flat[0], flat[1]


def exact(case, seed):
    kind = case["kind"]
    if kind in ("update", "host"):
        eps, zn = (t.double() for t in _batch(case, seed))
        return list(_norton_exact(MATRIX + (case["exponent"],), eps, zn, case["h"],
                                  tangent=case.get("tangent", False)))
    if kind == "ode":
        return list(_ode23_exact(MATRIX + (case["exponent"],), *_ode_batch(case, seed), case["h"]))
    if kind in ("scheme", "adjoint"):
        phase, spec, E, h = _scheme_inputs(case, seed)
        Sigma, iters, eps, z = _Scheme(phase, spec).solve(E, h, case["evals"], 1e-8)
        if kind == "adjoint":
            return {"Sigma": Sigma, "grad": None}
        if case["precision"] == "bulk":
            return {"Sigma": Sigma, "eps": eps, "z": z}
        return {"Sigma": Sigma, "iters": iters, "eps": eps, "z": z}
    out = []
    for j in _serve_jobs(case, seed):
        solver = _Scheme(torch.from_numpy(j["phase"]).cuda(), j["spec"])
        out.append(solver.solve(j["E"], j["h"], 0, case["tol"])[0])
    return out
