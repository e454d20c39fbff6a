"""The work a user of this framework has it do, as cases to time.

Each case is one call chain through the public entry points of
``paper_1808_04406_gb300`` (``lbm.Simulation``, ``lbm.HermiteSimulation``,
``lbm.Batch``, ``closure.Trainer``) on seeded synthetic input:

  tp       a single D2Q9 / D3Q27 run advanced by ``step(n)``
  h37      a single 37-velocity run advanced by ``step(n)``
  wave     a wave-decay measurement on a caller-supplied Hermite lattice
  batch    many independent D2Q9 runs advanced together
  learned  a D3Q27 run with the learned closure in its sweep
  train    Adam steps of the closure's network
  logged   a whole short run: host fields in, totals logged every step, host
           fields out

Runs advance by an even number of steps, after which the populations' storage
buffer holds f_i(x) in slot (i, x); ``exact`` restates every run in FP64 torch.
"""
import math

import numpy as np
import torch

from paper_1808_04406_gb300 import closure, gen_rules, lbm

DEV = "cuda"
CS2 = 1.0 / 3.0
STORAGES = {"f64": torch.float64, "f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
BYTES = {"f64": 8, "f32": 4, "f16": 2, "bf16": 2}
LATTICE_DQ = {"D2Q9": (2, 9), "D3Q27": (3, 27)}
# FP operations of one node update with the per-axis transforms (D2Q9, D3Q27) and
# with transforms that use the lattice's reflections (37 and 17 velocities)
FLOPS = {"D2Q9": 160, "D3Q27": 720, "D2Q37": 900, 17: 400, 37: 900}
MLP_FLOPS = 2 * (20 * 64 + 64 * 64 + 64 * 6)


def listed():
    return [
        # the FP64 correctness run: a 2D Taylor-Green vortex small enough that launches and latency count
        {"name": "tg_d2q9_f64_128", "kind": "tp", "lattice": "D2Q9", "nx": 128, "ny": 128, "nz": 1, "storage": "f64",
         "steps": 100},
        # one chunk of a stability run: thermal double shear layer, FP32, as the maximum-Ma search steps it
        {"name": "dsl_d2q37_f32_128", "kind": "h37", "nx": 128, "ny": 128, "storage": "f32", "thermal": True,
         "theta0": 1.0, "flow": "dsl", "steps": 256},
        # one measurement of the grid-convergence study: FP64 shear wave on a minimal quadrature
        {"name": "wave_e9a_f64_80", "kind": "wave", "rule": "E9-A", "n": 80, "storage": "f64", "records": 40},
        # the headline configuration: 3D Taylor-Green vortex, FP32 populations far larger than L2
        {"name": "tgv_d3q27_f32_256", "kind": "tp", "lattice": "D3Q27", "nx": 256, "ny": 256, "nz": 256,
         "storage": "f32", "steps": 20},
        # the same with 16-bit offsets
        {"name": "tgv_d3q27_f16_256", "kind": "tp", "lattice": "D3Q27", "nx": 256, "ny": 256, "nz": 256,
         "storage": "f16", "steps": 20},
        # a ragged box with odd sides, as geometry rather than the hardware dictates them
        {"name": "box_d3q27_f32_odd", "kind": "tp", "lattice": "D3Q27", "nx": 161, "ny": 95, "nz": 77,
         "storage": "f32", "steps": 20},
        # the thermal benchmark: 37 velocities, FP16 offsets
        {"name": "thermal_d2q37_f16_1024", "kind": "h37", "nx": 1024, "ny": 1024, "storage": "f16", "thermal": True,
         "theta0": 1.2, "flow": "wave", "steps": 20},
        # a thermal run at the accuracy FP32 storage takes by default
        {"name": "thermal_d2q37_f32_512", "kind": "h37", "nx": 512, "ny": 512, "storage": "f32", "thermal": True,
         "theta0": 1.2, "flow": "wave", "steps": 20},
        # the ensemble benchmark: 512 independent decaying-turbulence runs of sides 64 to 512
        {"name": "batch512_bf16", "kind": "batch", "runs": 512, "lo": 64, "hi": 512, "sizes_seed": 0,
         "storage": "bf16", "steps": 20},
        # the coarse run with the learned closure
        {"name": "learned_128", "kind": "learned", "nx": 128, "ny": 128, "nz": 128, "steps": 20},
        # training of the closure: Adam steps on mini-batches
        {"name": "train_65536", "kind": "train", "samples": 1 << 20, "batch": 65536, "iters": 20},
        # a whole run as a user writes it: pinned host fields in and out, totals logged every step
        {"name": "logged_d3q27_f32_128", "kind": "logged", "lattice": "D3Q27", "nx": 128, "ny": 128, "nz": 128,
         "storage": "f32", "steps": 20},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["tp", "tp", "tp", "h37", "h37", "wave", "batch", "learned", "train", "logged"])
    if kind in ("tp", "logged"):
        if rng.random() < 0.4:
            lat, nz, storage = "D2Q9", 1, rng.choice(["f64", "f32", "f16", "bf16"])
            nx, ny = _log_int(rng, 48, 1024), _log_int(rng, 48, 1024)
            steps = 2 * _log_int(rng, 10, 50)
        else:
            lat, storage = "D3Q27", rng.choice(["f32", "f32", "f16", "bf16"])
            nx, ny, nz = (_log_int(rng, 24, 250) for _ in range(3))
            steps = 2 * _log_int(rng, 4, 10)
        if rng.random() < 0.6:
            nx += nx & 1
        return {"kind": kind, "lattice": lat, "nx": nx, "ny": ny, "nz": nz, "storage": storage, "steps": steps}
    if kind == "h37":
        storage = rng.choice(["f64", "f32", "f16", "bf16"])
        nx, ny = (_log_int(rng, 48, 320 if storage == "f64" else 1000) for _ in range(2))
        if rng.random() < 0.6:
            nx += nx & 1
        return {"kind": "h37", "nx": nx, "ny": ny, "storage": storage, "thermal": rng.random() < 0.7, "theta0": 1.0,
                "flow": "wave", "steps": 2 * _log_int(rng, 4, 10)}
    if kind == "wave":
        return {"kind": "wave", "rule": rng.choice(["E9-A", "E9-C", "E7-D", "E7-A"]), "n": _log_int(rng, 20, 80),
                "storage": rng.choice(["f64", "f64", "f32"]), "records": 40}
    if kind == "batch":
        return {"kind": "batch", "runs": _log_int(rng, 8, 256), "lo": 64, "hi": _log_int(rng, 128, 512),
                "sizes_seed": rng.randrange(1 << 20), "storage": rng.choice(["bf16", "f16", "f32"]),
                "steps": 2 * _log_int(rng, 4, 10)}
    if kind == "learned":
        nx, ny, nz = (_log_int(rng, 24, 128) for _ in range(3))
        return {"kind": "learned", "nx": nx, "ny": ny, "nz": nz, "steps": 2 * _log_int(rng, 4, 10)}
    return {"kind": "train", "samples": _log_int(rng, 1 << 14, 1 << 20), "batch": _log_int(rng, 1 << 10, 1 << 16),
            "iters": _log_int(rng, 5, 20)}


# ---- seeded input ----------------------------------------------------------------------------

def _modes(dims, seed, fields, kmax, count=6, velocity=False):
    """fields smooth periodic fields [fields, N] (FP64, on the GPU, x fastest, each of unit RMS): sums of `count`
    products of low Fourier modes with random wavenumbers, phases and amplitudes.  velocity: the last ones are the
    components of a velocity, each constant along its own axis, so that it has no divergence."""
    g = np.random.default_rng(seed)
    out = []
    for j in range(fields):
        axes = []
        for a, n in enumerate(reversed(dims)):
            if velocity and len(dims) - 1 - a == j - (fields - len(dims)):
                axes.append(torch.ones(count, n, dtype=torch.float64, device=DEV))
                continue
            x = torch.arange(n, dtype=torch.float64, device=DEV) * (2.0 * math.pi / n)
            k = torch.as_tensor(g.integers(1, min(kmax, max(1, n // 8)) + 1, count), dtype=torch.float64, device=DEV)
            p = torch.as_tensor(g.uniform(0, 2 * math.pi, count), device=DEV)
            axes.append(torch.cos(k[:, None] * x[None, :] + p[:, None]))
        a = torch.as_tensor(g.uniform(0.3, 1.0, count), device=DEV)
        f = torch.einsum("m,ma,mb->ab", a, *axes) if len(dims) == 2 else torch.einsum("m,ma,mb,mc->abc", a, *axes)
        f = f.reshape(-1)
        out.append(f / f.square().mean().sqrt().clamp_min(1e-3))
    return torch.stack(out)


def _coords(dims):
    """2 pi x_d / n_d at every node, x fastest."""
    D = len(dims)
    out = []
    for d, n in enumerate(dims):
        x = torch.arange(n, dtype=torch.float64, device=DEV) * (2.0 * math.pi / n)
        shape = [1] * D
        shape[D - 1 - d] = n
        out.append(x.view(shape).expand(*reversed(dims)).reshape(-1))
    return out


def _dims(case):
    return tuple(case[k] for k in ("nx", "ny", "nz") if k != "nz" or case.get("lattice", "D3Q27") == "D3Q27")


def _tp_fields(case, seed):
    """A Taylor-Green vortex at Ma 0.1 with seeded phases and a smooth perturbation of a tenth of it."""
    dims = _dims(case)
    g = np.random.default_rng(seed)
    X = [x + g.uniform(0, 2 * math.pi) for x in _coords(dims)]
    u0 = 0.1 / math.sqrt(3.0)
    c = torch.cos(X[2]) if len(dims) == 3 else 1.0
    u = [u0 * torch.sin(X[0]) * torch.cos(X[1]) * c, -u0 * torch.cos(X[0]) * torch.sin(X[1]) * c]
    if len(dims) == 3:
        u.append(torch.zeros_like(u[0]))
    pert = _modes(dims, seed + 1, len(dims) + 1, 4, velocity=True)
    return 1.0 + 0.002 * pert[0], (torch.stack(u) + 0.1 * u0 * pert[1:]).contiguous()


def _tp_taus(case):
    if case["lattice"] == "D2Q9":
        return [0.6, 1.0, 1.0]
    t2 = 0.5 + 3.0 * (0.1 / math.sqrt(3.0)) * (256 / (2 * math.pi)) / 1600.0  # the 256^3 vortex at Re 1600
    return [t2, 1.0, t2, 1.0, t2]


def _h37_fields(case, seed):
    dims = (case["nx"], case["ny"])
    g = np.random.default_rng(seed)
    X, Y = _coords(dims)
    th0 = case["theta0"]
    pert = _modes(dims, seed + 1, 4, 4)  # density, velocity, temperature
    if case["flow"] == "dsl":  # double shear layer at Ma 0.2
        u0 = 0.2 / _C37
        y = Y / (2 * math.pi)
        ux = torch.where(y <= 0.5, u0 * torch.tanh(80 * (y - 0.25)), u0 * torch.tanh(80 * (0.75 - y)))
        uy = 0.05 * u0 * torch.sin(X + g.uniform(0, 2 * math.pi))
        u = torch.stack([ux, uy]) + 0.01 * u0 * pert[1:3]
        return torch.ones_like(X), u.contiguous(), torch.full_like(X, th0)
    s = torch.sin(10 * X + g.uniform(0, 2 * math.pi)) if case["nx"] >= 160 else torch.sin(X + g.uniform(0, 6.28))
    theta = th0 + 1e-3 * s + 1e-4 * pert[3]
    if not case["thermal"]:
        theta = torch.ones_like(X)
    u = torch.stack([1e-4 * pert[1], 1e-3 * s + 1e-4 * pert[2]])
    return th0 / theta if case["thermal"] else 1.0 + 1e-3 * pert[0], u.contiguous(), theta


def _h37_taus(case):
    if case["flow"] == "dsl":  # Re 1e4, Pr 1
        t2 = 0.5 + 0.2 * _C37 * case["nx"] / 1e4
        return [t2, t2, t2]
    t2 = 0.5 + 0.1 / case["theta0"]
    return [t2, 0.5 + (t2 - 0.5) / 0.71, t2]


def _batch_runs(case):
    g = np.random.default_rng(case["sizes_seed"])
    sides = [int(s) for s in g.integers(case["lo"], case["hi"] + 1, case["runs"])]
    re = 10.0 ** g.uniform(2.0, 3.5, case["runs"])  # resolved: no run diverges, however long it is advanced
    u_rms = 0.1 / math.sqrt(3.0)
    return sides, [[0.5 + 3.0 * u_rms * s / r, 1.0, 1.0] for s, r in zip(sides, re)]


def _batch_fields(case, seed):
    out = []
    for r, s in enumerate(_batch_runs(case)[0]):
        m = _modes((s, s), seed * 1000 + r, 2, 6, 4, velocity=True)
        out.append((torch.ones(s * s, dtype=torch.float64, device=DEV), (0.1 / math.sqrt(3.0)) * m))
    return out


LEARNED_RANGE = (0.5, 1.98)


def _learned_taus():
    nu = closure.taylor_scale_viscosity(512, 4.0, 0.04, 100.0) / 4.0  # Re_lambda 100 of the 512^3 run, on 128^3
    t2 = 0.5 + 3.0 * nu
    return [t2, 1.0, t2, 1.0, t2]


def _learned_net(seed):
    """Seeded random hidden layers and a small output layer around the plain model's rates: every node evaluates
    the network and the run stays stable."""
    taus = _learned_taus()
    P = closure.init_params(seed, DEV)
    lo, hi = LEARNED_RANGE
    om = [1.02, 1.02, 1.0 / taus[0], 1.0 / taus[0], 1.02, 1.0 / taus[0]]
    q = torch.tensor([(min(max(o, lo + 1e-3), hi - 1e-3) - lo) / (hi - lo) for o in om], device=DEV)
    P[5504:5888] *= 0.05
    P[5888:] = torch.log(q / (1 - q))
    norm = torch.zeros(40, device=DEV)
    norm[20:] = 30.0  # the scaled moments are of the order of the velocity gradients
    return P, norm


def _learned_fields(case, seed):
    dims = _dims(case)
    m = _modes(dims, seed, 3, 6, 8, velocity=True)
    return torch.ones(m.shape[1], dtype=torch.float64, device=DEV), 0.04 * m


def _wave_setup(case):
    e, w, c, order = gen_rules.rule(case["rule"])
    taus = [0.6, 0.7, 0.6]
    k = 2 * math.pi / case["n"]
    steps = int(0.7 / (0.1 * k * k / c ** 2))
    return (e, w, c, order), taus, max(1, steps // (case["records"] - 1))


def _wave_fields(case, seed):
    n = case["n"]
    p = np.random.default_rng(seed).uniform(0, 2 * math.pi)
    x = np.tile(np.arange(n) * (2 * math.pi / n), n)
    u = np.zeros((2, n * n))
    u[1] = 1e-3 * np.sin(x + p)
    return np.ones(n * n), u, np.ones(n * n)


# ---- the calls --------------------------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind == "tp":
        s["sim"] = lbm.Simulation(case["lattice"], _dims(case), _tp_taus(case), storage=case["storage"])
        s["sim"].init_fields(*_tp_fields(case, seed))
    elif kind == "h37":
        flags = lbm.LBM_THERMAL if case["thermal"] else 0
        s["sim"] = lbm.Simulation("D2Q37", (case["nx"], case["ny"]), _h37_taus(case), storage=case["storage"],
                                  flags=flags, theta_ref=case["theta0"])
        s["sim"].init_fields(*_h37_fields(case, seed))
    elif kind == "wave":
        rule, taus, s["stride"] = _wave_setup(case)
        s["sim"] = lbm.HermiteSimulation(rule, (case["n"], case["n"]), taus, storage=case["storage"],
                                         flags=lbm.LBM_THERMAL)
        s["fields"] = _wave_fields(case, seed)
    elif kind == "batch":
        sides, taus = _batch_runs(case)
        b = lbm.Batch([(n, n) for n in sides], taus, storage=case["storage"])
        b.pop.zero_()  # the gaps between the runs' slices are compared too
        fields = _batch_fields(case, seed)
        torch.cuda.synchronize()  # the batch has its own stream
        b.init_runs(fields)
        b.use_graph(True)
        s["batch"] = b
    elif kind == "learned":
        s["sim"] = lbm.Simulation("D3Q27", _dims(case), _learned_taus(), storage="f32")
        s["sim"].init_fields(*_learned_fields(case, seed))
        s["sim"].set_closure(*_learned_net(seed), *LEARNED_RANGE)
    elif kind == "train":
        g = torch.Generator(device=DEV).manual_seed(seed)
        n = case["samples"]
        s["X"] = torch.randn(n, 20, generator=g, device=DEV)
        k = torch.randn(n, 6, generator=g, device=DEV)
        ks = -0.2 * k * torch.tanh(s["X"][:, :6]) + 0.3 * torch.randn(n, 6, generator=g, device=DEV)
        s["abc"] = torch.stack([k * k, k * ks, ks * ks], dim=2).reshape(n, 18).contiguous()
        s["cw"] = closure.class_weights(s["abc"])
        s["trainer"] = closure.Trainer(closure.init_params(seed, DEV), case["batch"])
        s["seed"] = seed
    else:
        rho, u = _tp_fields(case, seed)
        s["sim"] = lbm.Simulation(case["lattice"], _dims(case), _tp_taus(case), storage=case["storage"])
        s["rho"], s["u"] = rho.float().cpu().pin_memory(), u.float().cpu().pin_memory()
        s["rho_out"] = torch.empty_like(s["rho"], pin_memory=True)
        s["u_out"] = torch.empty_like(s["u"], pin_memory=True)
        s["totals"] = torch.empty(case["steps"], 5, dtype=torch.float64, pin_memory=True)
    return s


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind in ("tp", "h37", "learned"):
        s["sim"].step(case["steps"])
        return s["sim"].raw_populations()
    if kind == "wave":
        s["sim"].init_fields(*s["fields"])
        fit, amps = s["sim"].mode_history(2, (1, 0), case["records"], s["stride"])
        return {"fit": fit, "amplitudes": amps, "populations": s["sim"].populations(on_device=True)}
    if kind == "batch":
        b = s["batch"]
        b.step(case["steps"])
        return b.pop.view(STORAGES[case["storage"]])
    if kind == "train":
        t = s["trainer"]
        losses = t.train(s["X"], s["abc"], s["cw"], case["iters"], 2e-3, s["seed"])
        return {"losses": losses, "params": t.params, "m": t.m, "v": t.v}
    sim = s["sim"]
    sim.init_fields(s["rho"], s["u"])
    p = s["totals"].data_ptr()
    for k in range(case["steps"]):
        sim.step_totals_async(p + 40 * k)
    lbm.lbm_moments(sim.handle, s["rho_out"].data_ptr(), s["u_out"].data_ptr(), 0, lbm.LBM_DTYPE_F32, 0)
    return {"rho": s["rho_out"], "u": s["u_out"], "totals": s["totals"]}


def work(case):
    """State (or fields) read once and written once a pass, whatever the number of steps; the operations of every
    step."""
    kind = case["kind"]
    if kind in ("tp", "logged", "learned"):
        lat = case.get("lattice", "D3Q27")
        N, (D, Q) = case["nx"] * case["ny"] * case["nz"], LATTICE_DQ[lat]
        fl = FLOPS[lat] + (MLP_FLOPS if kind == "learned" else 0)
        b = 2 * 4 * (1 + D) * N if kind == "logged" else 2 * Q * BYTES[case.get("storage", "f32")] * N
        return {"bytes": b, "flops": fl * N * case["steps"]}
    if kind == "h37":
        N = case["nx"] * case["ny"]
        return {"bytes": 2 * 37 * BYTES[case["storage"]] * N, "flops": FLOPS["D2Q37"] * N * case["steps"]}
    if kind == "wave":
        rule, _, stride = _wave_setup(case)
        q, N = len(rule[1]), case["n"] ** 2
        return {"bytes": (4 + q) * 8 * N, "flops": FLOPS[q] * N * stride * (case["records"] - 1)}
    if kind == "batch":
        N = sum(n * n for n in _batch_runs(case)[0])
        return {"bytes": 18 * BYTES[case["storage"]] * N, "flops": FLOPS["D2Q9"] * N * case["steps"]}
    n = case["batch"] * case["iters"]
    return {"bytes": n * 38 * 4, "flops": 3 * MLP_FLOPS * n}


# ---- FP64 restatements ------------------------------------------------------------------------

def _axis_view(f, D, d):
    """[..., 3, ..., N] views of the three e_d = -1, 0, +1 (or alpha_d = 0, 1, 2) groups along axis d."""
    g = f.view(*([3] * D), -1)
    return [g.select(D - 1 - d, k) for k in range(3)]


def _central(f, u, D):
    """Central moments [Q, N] about u, index sum_d alpha_d 3^d."""
    f = f.clone()
    for d in range(D):
        m, z, p = _axis_view(f, D, d)
        a, b, c = -1.0 - u[d], -u[d], 1.0 - u[d]
        k0, k1, k2 = m + z + p, a * m + b * z + c * p, a * a * m + b * b * z + c * c * p
        m.copy_(k0), z.copy_(k1), p.copy_(k2)
        del k0, k1, k2
    return f


def _populations(k, u, D):
    """The inverse of _central, in place."""
    for d in range(D):
        a, b, c = _axis_view(k, D, d)
        m1 = b + u[d] * a
        m2 = c + 2 * u[d] * b + u[d] * u[d] * a
        m0 = a.clone()
        a.copy_(0.5 * (m2 - m1)), b.copy_(m0 - m2), c.copy_(0.5 * (m2 + m1))
    return k


def _tp_tables(D):
    a = [[(i // 3 ** d) % 3 for d in range(D)] for i in range(3 ** D)]
    w = torch.tensor([math.prod((1 / 6, 2 / 3, 1 / 6)[x] for x in r) for r in a], dtype=torch.float64, device=DEV)
    meq = torch.tensor([math.prod((1.0, 0.0, CS2)[x] for x in r) for r in a], dtype=torch.float64, device=DEV)
    e = torch.tensor([[x - 1.0 for x in r] for r in a], dtype=torch.float64, device=DEV)
    return a, w, meq, e


def _stream(f, e, dims):
    for i in range(f.shape[0]):
        g = f[i].view(*reversed(dims))
        f[i] = torch.roll(g, shifts=tuple(int(x) for x in reversed(e[i])), dims=tuple(range(len(dims)))).reshape(-1)
    return f


def _tp_init(rho, u, D):
    _, _, meq, _ = _tp_tables(D)
    return _populations(meq[:, None] * rho[None, :], u, D)


def _tp_step(f, dims, taus, rates=None):
    """One collide-and-stream step of absolute populations f [Q, N]; rates(k1 scaled) gives orders 3 and up."""
    D = len(dims)
    al, w, meq, e = _tp_tables(D)
    rho = f.sum(0)
    u = (e.T @ f) / rho
    k = _central(f, u, D)
    over = rates(k, rho, al, meq) if rates else {}
    for i, a in enumerate(al):
        n = sum(a)
        if n >= 2:
            om = over.get(i, 1.0 / (taus[n - 2] if n - 2 < len(taus) else 1.0))
            k[i] += om * (meq[i] * rho - k[i])
    return _stream(_populations(k, u, D), e, dims), rho, u


def _offsets(f, w, storage):
    d = f - w[:, None]
    return d / w[:, None] if storage in ("f16", "bf16") else d


def _learned_rates(P, norm):
    lo, hi = LEARNED_RANGE
    P = P.double()
    cut, at = [], 0
    for shape in ((20, 64), (64,), (64, 64), (64,), (64, 6), (6,)):
        n = math.prod(shape)
        cut.append(P[at:at + n].view(shape))
        at += n
    W1, b1, W2, b2, W3, b3 = cut
    mean, inv = norm.double()[:20], norm.double()[20:]
    classes = {(2, 1, 0): 0, (1, 1, 1): 1, (2, 2, 0): 2, (2, 1, 1): 3, (2, 2, 1): 4, (2, 2, 2): 5}
    tau2 = _learned_taus()[0]

    def rates(k, rho, al, meq):
        x = [(k[i] - meq[i] * rho) / (rho * CS2 ** (0.5 * sum(a))) for i, a in enumerate(al) if 2 <= sum(a) <= 4]
        x.append(torch.full_like(rho, tau2 - 0.5))
        X = (torch.stack(x, 1) - mean) * inv
        h = torch.relu(torch.relu(X @ W1 + b1) @ W2 + b2)
        om = (lo + (hi - lo) * torch.sigmoid(h @ W3 + b3)).T
        return {i: om[classes[tuple(sorted(a, reverse=True))]] for i, a in enumerate(al) if sum(a) >= 3}

    return rates


# the 37-velocity rule of degree 9 in the storage's velocity order (opposites at i and 36 - i): its scale and, by
# |e|^2, its weights
_C37 = 1.1969797703930745
_EX37 = (-1, 0, -1, -1, -2, 0, -2, -2, -1, -1, -2, -2, -3, 0, -3, -3, -1, -1, 0, 1, 1, 3, 3, 0, 3, 2, 2, 1, 1, 2, 2, 0,
         2, 1, 1, 0, 1)
_EY37 = (0, -1, -1, 1, 0, -2, -1, 1, -2, 2, -2, 2, 0, -3, -1, 1, -3, 3, 0, -3, 3, -1, 1, 3, 0, -2, 2, -2, 2, -1, 1, 2,
         0, -1, 1, 1, 0)
_W37 = {0: 0.23315066913235249, 1: 0.107306091542219, 2: 0.05766785988879488, 4: 0.01420821615845075,
        5: 0.0053530490005137751, 8: 0.0010119375926735754, 9: 0.00024530102775771736, 10: 0.00028341425299419824}


def _he(n, x):
    return (1.0 + 0 * x, x, x * x - 1, x * x * x - 3 * x, x * x * x * x - 6 * x * x + 3)[n]


class _H37:
    """The 37-velocity model in FP64: Hermite truncation 4, every central moment of order n >= 2 of the truncated
    distribution's non-equilibrium part relaxed at 1 / tau_n."""

    def __init__(self, taus, thermal):
        self.e = np.stack([_EX37, _EY37], 1)
        self.w = torch.tensor([_W37[x * x + y * y] for x, y in self.e], dtype=torch.float64, device=DEV)
        xi = torch.tensor(self.e * _C37, dtype=torch.float64, device=DEV)
        self.pq = [(p, q) for p in range(5) for q in range(5) if p + q <= 4]
        self.H = torch.stack([_he(p, xi[:, 0]) * _he(q, xi[:, 1]) for p, q in self.pq])
        self.R = torch.stack([self.w * h / (math.factorial(p) * math.factorial(q))
                              for h, (p, q) in zip(self.H, self.pq)], 1)
        self.at = {pq: k for k, pq in enumerate(self.pq)}
        self.om = [0.0, 0.0] + [1.0 / t for t in taus]
        self.thermal = thermal

    def a0(self, rho, u, th):
        g = [[1.0 + 0 * v, v, v * v + th - 1, v ** 3 + 3 * v * (th - 1),
              v ** 4 + 6 * v * v * (th - 1) + 3 * (th - 1) ** 2] for v in u]
        return torch.stack([rho * g[0][p] * g[1][q] for p, q in self.pq])

    def equilibrium(self, rho, u, th):
        return self.R @ self.a0(rho, u, th)

    def macro(self, a):
        rho = a[self.at[0, 0]]
        u = (a[self.at[1, 0]] / rho, a[self.at[0, 1]] / rho)
        if not self.thermal:
            return rho, u, torch.ones_like(rho)
        tr = a[self.at[2, 0]] + a[self.at[0, 2]]
        return rho, u, 1 + 0.5 * (tr / rho - u[0] ** 2 - u[1] ** 2)

    def _shift(self, a, u, axis, inverse):
        """Hermite coefficients to central moments of one axis about u (and back): binomials times the Gaussian's
        moments about u, whose inverse series is the Hermite polynomials'."""
        v = u[axis]
        mu = ([_he(m, v) for m in range(5)] if inverse else
              [1.0 + 0 * v, -v, v * v + 1, -(v ** 3 + 3 * v), v ** 4 + 6 * v * v + 3])
        out = []
        for p, q in self.pq:
            n, s = (p, q)[axis], 0.0
            for k in range(n + 1):
                s = s + math.comb(n, k) * mu[n - k] * a[self.at[(k, q) if axis == 0 else (p, k)]]
            out.append(s)
        return torch.stack(out)

    def step(self, f, dims):
        a = self.H @ f
        rho, u, th = self.macro(a)
        k = self._shift(self._shift(a - self.a0(rho, u, th), u, 0, False), u, 1, False)
        k = k * torch.tensor([-self.om[p + q] for p, q in self.pq], dtype=torch.float64, device=DEV)[:, None]
        a = a + self._shift(self._shift(k, u, 0, True), u, 1, True)
        return _stream(self.R @ a, self.e, dims)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("tp", "learned", "logged"):
        dims = _dims(case)
        D = len(dims)
        _, w, _, e = _tp_tables(D)
        rho, u = _learned_fields(case, seed) if kind == "learned" else _tp_fields(case, seed)
        if kind == "logged":
            rho, u = rho.float().double(), u.float().double()
        taus = _learned_taus() if kind == "learned" else _tp_taus(case)
        rates = _learned_rates(*_learned_net(seed)) if kind == "learned" else None
        f = _tp_init(rho, u, D)
        totals = []
        for _ in range(case["steps"]):
            f, rho, u = _tp_step(f, dims, taus, rates)
            if kind == "logged":
                j = [float((rho * v).sum()) for v in u] + [0.0] * (3 - D)
                totals.append([float((rho - 1).sum())] + j + [float((0.5 * rho * (u * u).sum(0)).sum())])
        if kind == "logged":
            rho = f.sum(0)
            return {"rho": rho, "u": (e.T @ f) / rho, "totals": torch.tensor(totals, dtype=torch.float64)}
        return _offsets(f, w, case.get("storage", "f32"))
    if kind == "h37":
        dims = (case["nx"], case["ny"])
        M = _H37(_h37_taus(case), case["thermal"])
        rho, u, th = _h37_fields(case, seed)
        f = M.equilibrium(rho, u * _C37, th)
        one = torch.ones(1, dtype=torch.float64, device=DEV)
        ref = M.equilibrium(one, (0 * one, 0 * one), case["theta0"] * one)
        for _ in range(case["steps"]):
            f = M.step(f, dims)
        d = f - ref
        return d / M.w[:, None] if case["storage"] in ("f16", "bf16") else d
    if kind == "wave":
        if case["rule"] != "E9-A":
            return None
        n, (rule, taus, stride) = case["n"], _wave_setup(case)
        M = _H37(taus, True)
        rho, u, th = (torch.as_tensor(x, device=DEV) for x in _wave_fields(case, seed))
        f = M.equilibrium(rho, u * _C37, th)
        ph = torch.exp(-2j * math.pi * torch.arange(n, device=DEV, dtype=torch.float64) / n)
        amps = []
        for r in range(case["records"]):
            for _ in range(stride if r else 0):
                f = M.step(f, (n, n))
            rho, u, _ = M.macro(M.H @ f)
            amps.append(((u[1] / _C37).view(n, n).sum(0) * ph).sum())
        A = torch.stack(amps).cpu().numpy()
        t = np.arange(case["records"]) * float(stride)
        ln, arg = np.polyfit(t, np.log(np.abs(A)), 1), np.polyfit(t, np.unwrap(np.angle(A)), 1)
        order = {tuple(x): i for i, x in enumerate(M.e.tolist())}
        pops = f[[order[int(x), int(y)] for x, y in rule[0]]]
        return {"fit": np.array([-ln[0], arg[0], ln[1], arg[1]]), "amplitudes": A, "populations": pops}
    if kind == "batch":
        sides, taus = _batch_runs(case)
        _, w, _, _ = _tp_tables(2)
        flat = []
        for n, t, (rho, u) in zip(sides, taus, _batch_fields(case, seed)):
            f = _tp_init(rho, u, 2)
            for _ in range(case["steps"]):
                f = _tp_step(f, (n, n), t)[0]
            f = _offsets(f, w, case["storage"]).reshape(-1)
            flat.append(torch.nn.functional.pad(f, (0, -f.numel() % 64)))  # slices start at multiples of 64 values
        flat = torch.cat(flat)
        return torch.nn.functional.pad(flat, (0, -flat.numel() % (256 // BYTES[case["storage"]])))
    return None
