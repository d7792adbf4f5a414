"""What the performance of this framework is measured on.

The cases are the work that its users have it do, through the calls of
paper_2605_07083_gb300 that they make: time steps of one diode and of batches
of diodes (the 5 mm production diode, the 64-diode emission-flux sweep, the
paper's own 10 cm diode with its late-time profiles, the 1 mm diode whose steps
are bound by launches), the surrogate's PIC data runs, the loading of a state
and its charge and field, the sort by cell, and the surrogate network's
training step, gradient and prediction.  Sizes are those of workloads.py,
bench.py, surrogate.py and the tests.

listed() is the fixed list, draw(rng) one more case of the same ranges,
prepare(case, seed) what a program holds before the call, run(state) one pass,
work(case) the bytes and operations a pass cannot do without, and
exact(case, seed) the outputs in 64 bits by plain torch.

Step cases keep their handle, as a program that advances a diode does, so a
pass continues from where the last one ended; their populations are close to
stationary over the passes of a measurement.  They have no exact(): a pass
starts from the result of hundreds of Monte Carlo steps, and a 64-bit run
would take other collision branches and hold other particles.
"""
import ctypes as C
import math

import numpy as np
import torch

from paper_2605_07083_gb300 import pic, surrogate
from paper_2605_07083_gb300 import workloads as W

PUSH_BYTES = 20              # a particle-step: read z, v_z, id, write z, v_z
PARTICLE_BYTES = 20          # z, v_x, v_y, v_z, id
MLP_MACS = 5 * 128 + 2 * 128 * 128 + 128 * 4
MLP_LAYERS = ((5, 128), (128, 128), (128, 128), (128, 4))


# ------------------------------------------------------------------ the list
def listed():
    return [
        # a program that looks at the charge and the field after every step of
        # the 1 mm, 128-cell diode: launches and host reads are all of it
        {"name": "small_diode_each_step", "kind": "diode", "cells": 128, "gap_mm": 1.0,
         "flight": 20000, "pairs": 0, "fill": False, "settle": 2000, "steps": 1, "sort": 0,
         "fields": True},
        # the 1 mm diode run on between two looks at it (bench.py's small diode)
        {"name": "small_diode_run", "kind": "diode", "cells": 128, "gap_mm": 1.0, "flight": 20000,
         "pairs": 0, "fill": False, "settle": 2000, "steps": 250, "sort": 0, "fields": False},
        # the production diode of bench.py: 6M emitted electrons, 2M e-He+ pairs
        {"name": "production_diode", "kind": "diode", "cells": 2048, "gap_mm": 5.0,
         "flight": 6000000, "pairs": 2000000, "fill": True, "settle": 64, "steps": 100, "sort": 0,
         "fields": False},
        # a mid-size diode, odd sizes, kept sorted by cell (pic_tune sort_period)
        {"name": "sorted_diode", "kind": "diode", "cells": 1021, "gap_mm": 2.55,
         "flight": 1500007, "pairs": 300011, "fill": True, "settle": 64, "steps": 100, "sort": 25,
         "fields": False},
        # the 64-diode emission-flux sweep in one handle (bench.py)
        {"name": "flux_sweep", "kind": "sweep", "diodes": 64, "flight_max": 4000000, "settle": 64,
         "steps": 250},
        # the Table 2 scan of the paper's diode (flux_scan.py): 11 diodes, late-time profiles
        {"name": "paper_scan", "kind": "paper", "diodes": 11, "ppc": 250, "period": 100,
         "settle": 64, "steps": 200},
        # one batch of the surrogate's PIC data, from empty diodes to diagnostics
        {"name": "surrogate_batch", "kind": "surrogate", "diodes": 128, "flight": 20000.0,
         "steps": 1000},
        # a 10M-particle state loaded from device arrays; its charge, field and particles read back
        {"name": "load_state", "kind": "load", "cells": 2048, "emitted": 6000000,
         "pairs": 2000000},
        # the allocation-free sort by cell, close to its limit of 4.19M over 2048 cells
        {"name": "sort_by_cell", "kind": "sort", "n": 4000037, "cells": 2048},
        # a training step of the surrogate on its 4096 samples
        {"name": "mlp_train_step", "kind": "mlp_train", "batch": 4096},
        # loss and gradient of a small ragged batch
        {"name": "mlp_grad_small", "kind": "mlp_grad", "batch": 100},
        # the search's prediction grid: 256 settings x 161 fluxes
        {"name": "mlp_predict_grid", "kind": "mlp_forward", "batch": 41216},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["diode", "diode", "diode", "sweep", "paper", "surrogate", "load", "sort",
                       "mlp_train", "mlp_grad", "mlp_forward"])
    if kind == "diode":
        cells = _log(rng, 128, 2048)
        flight = _log(rng, 20000, 6000000)
        fill = flight > 100000 or rng.random() < 0.5
        steps = rng.choice([1, 50, 97])
        return {"kind": kind, "cells": cells, "gap_mm": cells * 2.5e-3, "flight": flight,
                "pairs": _log(rng, 1000, flight / 3) if fill else 0, "fill": fill,
                "settle": 64 if fill else 2000, "steps": steps,
                "sort": rng.choice([0, 0, 25]) if steps > 1 else 0, "fields": steps == 1}
    if kind == "sweep":
        return {"kind": kind, "diodes": rng.randint(2, 64), "flight_max": _log(rng, 200000, 4000000),
                "settle": 64, "steps": rng.randint(50, 150)}
    if kind == "paper":
        return {"kind": kind, "diodes": rng.randint(1, 11), "ppc": _log(rng, 20, 250),
                "period": rng.choice([25, 50, 100]), "settle": 64, "steps": 100}
    if kind == "surrogate":
        return {"kind": kind, "diodes": _log(rng, 4, 128), "flight": float(_log(rng, 5000, 30000)),
                "steps": rng.randint(200, 600)}
    if kind == "load":
        emitted = _log(rng, 20000, 6000000)
        return {"kind": kind, "cells": _log(rng, 128, 4096), "emitted": emitted,
                "pairs": _log(rng, 1000, emitted / 3)}
    if kind == "sort":
        cells = _log(rng, 128, 4096)
        return {"kind": kind, "n": _log(rng, 10000, min(4000000, 8192 * ((1 << 20) // cells))),
                "cells": cells}
    if kind == "mlp_forward":
        return {"kind": kind, "batch": _log(rng, 1, 41216)}
    return {"kind": kind, "batch": _log(rng, 32, 4096)}


# ------------------------------------------------------------------ inputs
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _inside(z, L):
    """FP32 positions strictly inside [0, L)."""
    top = float(np.nextafter(np.float32(L), np.float32(0)))
    return z.clamp_(0.0, top)


def _emitted(g, n, L, T_wall_K):
    """n emitted-type electrons: uniform in z, flux-weighted T_w velocities
    (the recipe of workloads.emitted_fill, drawn on the device)."""
    s = math.sqrt(W.K_B * T_wall_K / W.M_E)
    z = _inside(torch.rand(n, generator=g, device="cuda") * L, L)
    vx, vy = (torch.randn(n, generator=g, device="cuda") * s for _ in range(2))
    u = torch.rand(n, generator=g, device="cuda").clamp_(min=1e-7)
    return z, vx, vy, s * torch.sqrt(-2.0 * torch.log(u))


def _plasma(g, n, L, T_eV, mass):
    """n particles uniform in z, Maxwellian at T_eV (workloads.uniform_plasma)."""
    s = math.sqrt(W.E_CHARGE * T_eV / mass)
    z = _inside(torch.rand(n, generator=g, device="cuda") * L, L)
    return (z, *(torch.randn(n, generator=g, device="cuda") * s for _ in range(3)))


def _loaded_state(g, p, n_emit, n_pairs):
    return {0: _emitted(g, n_emit, p["L"], p["T_wall_K"]),
            1: _plasma(g, n_pairs, p["L"], p["T_e0_eV"], W.M_E),
            2: _plasma(g, n_pairs, p["L"], p["T_i0_eV"], p["m_ion"])}


def _room(n):
    return int(2.2 * n) + 400000


def _diode_params(case, seed):
    """A diode of the single-diode workloads (He, 10 V, T_w 2500 K) at the
    case's gap, cells and population."""
    cells = case["cells"]
    p = W.single_diode_small(seed=seed) if cells <= 128 else W.single_diode_production(seed=seed)
    L = case["gap_mm"] * 1e-3
    # the production preload is 6M of the 8M emitted electrons in flight its weight is sized for
    flight = case["flight"] * (4.0 / 3.0 if case["fill"] else 1.0)
    p.update(L=L, Nz=cells, weight=W.weight_for_in_flight(p["gamma_emit"], L, p["V"], flight),
             window_start=0)
    p["capacity"] = (_room(case["flight"]), _room(case["pairs"]), _room(case["pairs"]))
    return p


def _buffers(params):
    """Device buffers for z, v_x, v_y, v_z, id of all diodes' particles."""
    n = sum(sum(p["capacity"]) for p in params)
    return ([torch.zeros(n, dtype=torch.float32, device="cuda") for _ in range(4)]
            + [torch.zeros(n, dtype=torch.int32, device="cuda")])


def _kept(d, case):
    """A handle that a program keeps: settled, its graphs captured."""
    d.step(case["settle"])
    d.prepare(case["steps"])
    buffers = _buffers(d.params)
    torch.cuda.synchronize()
    return {"diode": d, "buffers": buffers}


def _load(d, species, arrays, instance=0):
    """Inject arrays drawn on the current stream: the handle has its own."""
    torch.cuda.current_stream().synchronize()
    d.inject(species, *arrays, instance=instance)


def _prepare_diode(case, seed):
    g = _generator(seed)
    p = _diode_params(case, seed)
    d = pic.Diode(p)
    if case["fill"]:
        for sp, arrays in _loaded_state(g, p, case["flight"], case["pairs"]).items():
            _load(d, sp, arrays)
    if case["sort"]:
        d.tune(sort_period=case["sort"])
    return _kept(d, case)


def _prepare_sweep(case, seed):
    g = _generator(seed)
    ps = W.batched_sweep(n_instances=case["diodes"], seed=1000)
    scale = case["flight_max"] / 4.0e6
    counts = []
    for p in ps:
        n = max(1000, int(p["target_in_flight"] * scale))
        p["weight"] = W.weight_for_in_flight(p["gamma_emit"], p["L"], p["V"], n)
        p["window_start"] = 0
        p["seed"] += 100000 * seed
        p["capacity"] = (_room(n), 131072, 131072)
        counts.append(n)
    d = pic.Diode(ps)
    for i, (p, n) in enumerate(zip(ps, counts)):
        _load(d, 0, _emitted(g, n, p["L"], p["T_wall_K"]), instance=i)
    return _kept(d, case)


def _prepare_paper(case, seed):
    g = _generator(seed)
    ps = W.paper_flux_scan(W.TABLE2_FLUXES[:case["diodes"]], ppc=case["ppc"], window_start=0,
                           seed=3 + 100 * seed)
    d = pic.Diode(ps)
    for i, p in enumerate(ps):
        n = p["ppc"] * p["Nz"]
        _load(d, 1, _plasma(g, n, p["L"], p["T_e0_eV"], W.M_E), instance=i)
        _load(d, 2, _plasma(g, n, p["L"], p["T_i0_eV"], p["m_ion"]), instance=i)
    d.set_profile_period(case["period"])
    return _kept(d, case)


def _mlp_parameters(seed):
    """Parameters of a network in training (He initialisation as Surrogate
    has it, small biases) and its Adam moments, as FP32 numpy arrays."""
    rng = np.random.default_rng(1000 + seed)
    theta = (rng.standard_normal(pic.MLP_PARAMS) * 0.05).astype(np.float32)
    at = 0
    for i, o in MLP_LAYERS:
        theta[at:at + o * i] = rng.standard_normal(o * i) * math.sqrt(2.0 / i)
        at += o * i + o
    m = (rng.standard_normal(pic.MLP_PARAMS) * 1e-3).astype(np.float32)
    v = (rng.uniform(0.5, 2.0, pic.MLP_PARAMS) * 1e-5).astype(np.float32)
    return theta, m, v


def _mlp_data(seed, n):
    """Normalised settings in [-1, 1] and targets of the diagnostics' size."""
    rng = np.random.default_rng(5000 + seed)
    x = rng.uniform(-1.0, 1.0, (n, 5)).astype(np.float32)
    back = 1.0 / (1.0 + np.exp(-4.0 * x[:, 0] + x[:, 4]))
    t = np.stack([back, 1.0 - back, 0.9 * (1.0 - back), 0.9 - 0.3 * back + 0.1 * x[:, 1]], 1)
    return x, t.astype(np.float32)


def _ptr(t):
    return C.c_void_p(t.data_ptr())


def _ok(rc, what):
    if rc != 0:
        raise pic.PicError(rc, what)


ADAM_STEP, LR, BETA1, BETA2, EPS = 1000, 1e-3, 0.9, 0.999, 1e-8


def _prepare_mlp(case, seed):
    lib = pic.load()
    n = case["batch"]
    theta, m, v = _mlp_parameters(seed)
    x, t = _mlp_data(seed, n)
    s = {"lib": lib, "n": n, "step": ADAM_STEP, "master": torch.from_numpy(theta).cuda(),
         "w": torch.empty(pic.MLP_PARAMS, dtype=torch.bfloat16, device="cuda"),
         "x": torch.from_numpy(x).cuda()}
    _ok(lib.pic_mlp_cast_bf16(_ptr(s["master"]), _ptr(s["w"]), None), "cast")
    if case["kind"] == "mlp_forward":
        s["y"] = torch.empty((n, 4), dtype=torch.float32, device="cuda")
        return s
    s["t"] = torch.from_numpy(t).cuda()
    s["bytes"] = lib.pic_mlp_scratch_bytes(n)
    s["scratch"] = torch.empty(s["bytes"] // 4 + 1, dtype=torch.float32, device="cuda")
    s["loss"] = torch.empty(1, dtype=torch.float32, device="cuda")
    if case["kind"] == "mlp_grad":
        s["grad"] = torch.empty(pic.MLP_PARAMS, dtype=torch.float32, device="cuda")
    else:
        s["m"], s["v"] = torch.from_numpy(m).cuda(), torch.from_numpy(v).cuda()
    return s


def _sort_input(case, seed):
    p = W.single_diode_production()
    return _emitted(_generator(seed), case["n"], p["L"], p["T_wall_K"]), p["L"]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "diode":
        return case, _prepare_diode(case, seed)
    if kind == "sweep":
        return case, _prepare_sweep(case, seed)
    if kind == "paper":
        return case, _prepare_paper(case, seed)
    if kind == "surrogate":
        settings = W.sobol_settings(case["diodes"], seed)
        return case, {"settings": settings, "seed0": seed * 100003}
    if kind == "load":
        p = _load_params(case, seed)
        s = {"params": p, "stream": torch.cuda.Stream(), "state": _load_input(case, seed, p),
             "buffers": _buffers([p])}
        torch.cuda.current_stream().synchronize()
        return case, s
    if kind == "sort":
        particles, L = _sort_input(case, seed)
        ids = torch.arange(case["n"], dtype=torch.int32, device="cuda")
        out = [torch.empty_like(a) for a in particles] + [torch.empty_like(ids)]
        return case, {"lib": pic.load(), "in": [*particles, ids], "out": out, "L": L}
    return case, _prepare_mlp(case, seed)


def _load_params(case, seed):
    p = W.single_diode_production(seed=seed)
    p["Nz"] = case["cells"]
    p["capacity"] = (_room(case["emitted"]), _room(case["pairs"]), _room(case["pairs"]))
    return p


def _load_input(case, seed, p):
    return _loaded_state(_generator(seed), p, case["emitted"], case["pairs"])


# ------------------------------------------------------------------ one pass
def _diagnostics(d):
    rows = [d.diagnostics(i) for i in range(d.n_instances)]
    return {k: np.array([r[k] for r in rows]) for k in rows[0]}


def _particles(d, buffers):
    """The live particles of every diode and species into the program's own
    device buffers, each species at its place; the diagnostics' n_live says
    how many of a place are live."""
    lib, n, at = pic.load(), C.c_int64(), 0
    for i, p in enumerate(d.params):
        for sp in range(3):
            cap = p["capacity"][sp]
            _ok(lib.pic_get_state(d.handle, i, sp, *[C.c_void_p(b.data_ptr() + 4 * at)
                                                     for b in buffers], cap, C.byref(n), 1), "state")
            at += cap
    return buffers


def run(state):
    case, s = state
    kind = case["kind"]
    if kind in ("diode", "sweep", "paper"):
        d = s["diode"]
        d.step(case["steps"])
        out = {"diagnostics": _diagnostics(d), "particles": _particles(d, s["buffers"])}
        if kind == "diode" and case["fields"]:
            out["rho"] = d.rho_fixed()
            out["phi"], out["E"] = d.field()
        if kind == "paper":
            prof = [d.profiles(i) for i in range(d.n_instances)]
            out["profiles"] = {k: np.stack([q[k] for q in prof])
                               for k in ("phi", "density", "counts")}
        return out
    if kind == "surrogate":
        rows, _, pushed = surrogate.run_settings(s["settings"], n_flight=case["flight"],
                                                 seed0=s["seed0"], n_steps=case["steps"])
        return {"rows": {k: np.array([r[k] for r in rows]) for k in rows[0]}, "pushed": pushed}
    if kind == "load":
        d = pic.Diode(s["params"], stream=s["stream"])
        for sp in range(3):
            d.inject(sp, *s["state"][sp])
        rho = d.rho_fixed()
        phi, E = d.field()
        particles = _particles(d, s["buffers"])
        d.close()
        return {"rho": rho, "phi": phi, "E": E, "particles": particles}
    stream = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    lib = s["lib"]
    if kind == "sort":
        _ok(lib.pic_sort_by_cell_static(*[_ptr(a) for a in s["in"]], case["n"], case["cells"],
                                        s["L"], *[_ptr(a) for a in s["out"]], stream), "sort")
        return s["out"]
    if kind == "mlp_forward":
        _ok(lib.pic_mlp_forward(_ptr(s["master"]), _ptr(s["w"]), _ptr(s["x"]), s["n"],
                                _ptr(s["y"]), stream), "forward")
        return s["y"]
    if kind == "mlp_grad":
        _ok(lib.pic_mlp_grad(_ptr(s["master"]), _ptr(s["w"]), _ptr(s["x"]), _ptr(s["t"]), s["n"],
                             _ptr(s["grad"]), _ptr(s["loss"]), _ptr(s["scratch"]), s["bytes"],
                             stream), "grad")
        return {"grad": s["grad"], "loss": s["loss"]}
    _ok(lib.pic_mlp_train_step(_ptr(s["master"]), _ptr(s["w"]), _ptr(s["m"]), _ptr(s["v"]),
                               s["step"], LR, BETA1, BETA2, EPS, _ptr(s["x"]), _ptr(s["t"]),
                               s["n"], _ptr(s["loss"]), _ptr(s["scratch"]), s["bytes"], stream),
        "train")
    s["step"] += 1
    return {k: s[k] for k in ("master", "w", "m", "v", "loss")}


# ------------------------------------------------------------------ floors
def work(case):
    kind = case["kind"]
    if kind == "diode":
        n = case["flight"] + 2 * case["pairs"]
        return {"bytes": PUSH_BYTES * n * case["steps"] + 2 * PARTICLE_BYTES * n, "flops": 0}
    if kind == "sweep":
        ps = W.batched_sweep(n_instances=case["diodes"], seed=1000)
        n = sum(p["target_in_flight"] for p in ps) * case["flight_max"] / 4.0e6
        return {"bytes": PUSH_BYTES * n * case["steps"] + 2 * PARTICLE_BYTES * n, "flops": 0}
    if kind == "paper":
        n = 2 * case["diodes"] * case["ppc"] * 4096
        return {"bytes": PUSH_BYTES * n * case["steps"] + 2 * PARTICLE_BYTES * n, "flops": 0}
    if kind == "surrogate":
        # the diodes start empty and fill within about a transit time: half of it on average
        return {"bytes": PUSH_BYTES * 0.5 * case["flight"] * case["diodes"] * case["steps"],
                "flops": 0}
    if kind == "load":
        n = case["emitted"] + 2 * case["pairs"]
        return {"bytes": n * (16 + 2 * PARTICLE_BYTES), "flops": 0}
    if kind == "sort":
        return {"bytes": 2 * PARTICLE_BYTES * case["n"], "flops": 0}
    n, params = case["batch"], 4 * pic.MLP_PARAMS
    if kind == "mlp_forward":
        return {"bytes": n * 36 + params // 2, "flops": 2 * MLP_MACS * n}
    if kind == "mlp_grad":
        return {"bytes": n * 36 + params // 2 + params, "flops": 6 * MLP_MACS * n}
    return {"bytes": n * 36 + 7 * params, "flops": 6 * MLP_MACS * n}


# ------------------------------------------------------------------ 64 bits
def _exact_load(p, state):
    """The fixed-point charge by its rule (the cell and fraction of the FP32
    product z * (Nz / L)) and the potential and field of the difference
    equations, in 64-bit numbers; the particles as they were given, with the
    ids in order."""
    Nz, dz = p["Nz"], p["L"] / p["Nz"]
    inv = float(np.float32(Nz / p["L"]))
    rho = torch.zeros(Nz + 1, dtype=torch.int64, device="cuda")
    for sp, (z, *_) in state.items():
        s = z * torch.tensor(inv, dtype=torch.float32, device="cuda")
        j = s.floor().clamp_(0, Nz - 1)
        q = ((s - j).double() * 16777216.0).floor().long()
        j = j.long()
        sign = 1 if sp == 2 else -1
        rho.index_add_(0, j, sign * (16777216 - q))
        rho.index_add_(0, j + 1, sign * q)
    rho = rho.cpu().numpy()
    kappa = dz * W.E_CHARGE * p["weight"] / (16777216.0 * 8.8541878128e-12)
    G = np.concatenate([[0], np.cumsum(rho[1:Nz])])
    d = (p["V"] + kappa * float(G.sum())) / Nz - kappa * G.astype(np.float64)
    phi = np.concatenate([[0.0], np.cumsum(d)])
    E = -np.concatenate([d[:1], 0.5 * (d[1:] + d[:-1]), d[-1:]]) / dz
    particles = _buffers([p])
    at = next_id = 0
    for sp in range(3):
        n = state[sp][0].numel()
        for k in range(4):
            particles[k][at:at + n] = state[sp][k]
        particles[4][at:at + n] = torch.arange(next_id, next_id + n, device="cuda")
        at, next_id = at + p["capacity"][sp], next_id + n
    return {"rho": rho, "phi": phi, "E": E, "particles": particles}


def _exact_network(w, x):
    """Pre-activations and activations of every layer, float64."""
    at, a, layers, pre, act = 0, x, [], [], [x]
    for k, (i, o) in enumerate(MLP_LAYERS):
        Wk, b = w[at:at + o * i].view(o, i), w[at + o * i:at + o * i + o]
        at += o * i + o
        z = a @ Wk.T + b
        a = 0.5 * z * (1.0 + torch.erf(z / math.sqrt(2.0))) if k < 3 else z
        layers.append(Wk)
        pre.append(z)
        act.append(a)
    return layers, pre, act


def _exact_gradient(w, x, t):
    layers, pre, act = _exact_network(w, x)
    diff = act[-1] - t
    delta, grads = 2.0 * diff / diff.numel(), []
    for k in range(3, -1, -1):
        grads = [delta.T @ act[k], delta.sum(0)] + grads
        if k:
            z = pre[k - 1]
            slope = (0.5 * (1.0 + torch.erf(z / math.sqrt(2.0)))
                     + z * torch.exp(-0.5 * z * z) / math.sqrt(2.0 * math.pi))
            delta = (delta @ layers[k]) * slope
    return torch.cat([g.reshape(-1) for g in grads]), (diff * diff).mean().reshape(1)


def _bf16_weights(theta):
    """FP64 parameters with the weights (not the biases) rounded to bfloat16."""
    w, at = theta.double().clone(), 0
    for i, o in MLP_LAYERS:
        w[at:at + o * i] = theta[at:at + o * i].to(torch.bfloat16).double()
        at += o * i + o
    return w


def exact(case, seed):
    kind = case["kind"]
    if kind == "load":
        p = _load_params(case, seed)
        return _exact_load(p, _load_input(case, seed, p))
    if kind == "sort":
        particles, L = _sort_input(case, seed)
        inv = torch.tensor(float(np.float32(case["cells"] / L)), dtype=torch.float32, device="cuda")
        cell = (particles[0] * inv).floor().clamp_(0, case["cells"] - 1)
        order = torch.sort(cell, stable=True).indices
        return [a[order].double() for a in particles] + [order.int()]
    if not kind.startswith("mlp"):
        return None
    theta, m, v = (torch.from_numpy(a).cuda() for a in _mlp_parameters(seed))
    x, t = (torch.from_numpy(a).cuda().double() for a in _mlp_data(seed, case["batch"]))
    w = _bf16_weights(theta)
    if kind == "mlp_forward":
        return _exact_network(w, x)[2][-1]
    grad, loss = _exact_gradient(w, x, t)
    if kind == "mlp_grad":
        return {"grad": grad, "loss": loss}
    m = BETA1 * m.double() + (1.0 - BETA1) * grad
    v = BETA2 * v.double() + (1.0 - BETA2) * grad * grad
    step = LR * (m / (1.0 - BETA1 ** ADAM_STEP)) / (torch.sqrt(v / (1.0 - BETA2 ** ADAM_STEP)) + EPS)
    master = theta.double() - step
    return {"master": master, "w": master, "m": m, "v": v, "loss": loss}
