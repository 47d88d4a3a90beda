"""The work that programs built on this library have it do, as cases that can be timed.

Particle state, fields and rates are returned as FP32: the library keeps them in FP64
buffers, but the pair sums and the kick behind them are FP32 by design (`include/md.h`).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1307_3711_gb300 import md, synth


def listed():
    return [
        # a paper-sized cluster (Fig. 2 and 7: some thousand macro-particles, thousands of
        # steps): what counts is the cost of one small step, replayed from the graph
        {"name": "step_2k", "kind": "step", "n": 2000, "z": 1, "steps": 32, "pol": 0,
         "env": 1, "boundary": 0, "tuned": False},
        # a mid-sized run with a record count that fills no block, circular polarisation, a
        # Gaussian pulse and the mixed boundary, stepped a few at a time
        {"name": "step_19k", "kind": "step", "n": 19003, "z": 2, "steps": 6, "pol": 1,
         "env": 0, "boundary": 2, "tuned": False},
        # the throughput workload: 50k Xe3+ and 150k electrons, autotuned as the README does
        {"name": "step_200k", "kind": "step", "n": 200000, "z": 3, "steps": 1, "pol": 0,
         "env": 1, "boundary": 0, "tuned": True},
        # a parameter scan: uneven clusters of 1k to 30k records advanced together
        {"name": "scan_32", "kind": "scan", "clusters": 32, "n_min": 1000, "n_max": 30000,
         "steps": 4},
        # a diagnosed step of a production run (energies and momentum every few steps)
        {"name": "diag_50k", "kind": "diag", "n": 50000, "z": 3},
        # a plasma filling a periodic box, forces through the nearest images
        {"name": "image_12k", "kind": "image", "n": 12000, "steps": 2},
        # a few thousand atoms through the pulse, an ionization pass before every step (the
        # long runs behind the ion energy spectra)
        {"name": "ionize_4k", "kind": "ionize", "atoms": 4000, "steps": 16},
        # a large ionizing cluster: 50k argon atoms, some 420k live records
        {"name": "ionize_50k", "kind": "ionize", "atoms": 50000, "steps": 1},
        # field and potential at a few hundred probe points of a large cluster
        {"name": "field_probe", "kind": "field", "nt": 300, "ns": 150000, "phi": True,
         "alloc": True},
        # a small field evaluation inside another program's loop that may not allocate
        {"name": "field_small", "kind": "field", "nt": 1000, "ns": 4001, "phi": False,
         "alloc": False},
        # ionization rates of the ions of a large cluster from the surrogate
        {"name": "rates_mlp", "kind": "rates", "n": 200000},
        # one minibatch of surrogate training: loss and gradient
        {"name": "grad_8k", "kind": "grad", "n": 8192},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "scan", "diag", "image", "ionize", "field",
                       "field", "rates", "grad"])
    if kind == "step":
        n = _log_uniform(rng, 500, 190000)
        most = max(1, min(40, int(3e10 / (float(n) * n))))
        return {"kind": kind, "n": n, "z": rng.randint(1, 8), "steps": rng.randint(1, most),
                "pol": rng.randint(0, 1), "env": rng.randint(0, 3),
                "boundary": rng.randint(0, 2), "tuned": False}
    if kind == "scan":
        lo = _log_uniform(rng, 300, 3000)
        return {"kind": kind, "clusters": rng.randint(3, 40), "n_min": lo,
                "n_max": _log_uniform(rng, 2 * lo, 25000), "steps": rng.randint(1, 4)}
    if kind == "diag":
        return {"kind": kind, "n": _log_uniform(rng, 1000, 120000), "z": rng.randint(1, 8)}
    if kind == "image":
        return {"kind": kind, "n": _log_uniform(rng, 1000, 30000), "steps": rng.randint(1, 3)}
    if kind == "ionize":
        atoms = _log_uniform(rng, 500, 40000)
        return {"kind": kind, "atoms": atoms,
                "steps": rng.randint(1, 20) if atoms < 6000 else 1}
    if kind == "field":
        alloc = rng.random() < 0.6
        return {"kind": kind, "nt": _log_uniform(rng, 1, 30000),
                "ns": _log_uniform(rng, 100, 300000), "phi": rng.random() < 0.5,
                "alloc": alloc}
    if kind == "rates":
        return {"kind": kind, "n": _log_uniform(rng, 100, 400000)}
    return {"kind": "grad", "n": _log_uniform(rng, 100, 60000)}


# ------------------------------------------------------------------ inputs --

LAMBDA = 0.8
LAMBDA_AR = 0.806


def _radius(n):
    """Sphere radius (1/k) of n records at the density of 400k in 10 nm."""
    return synth.nm_to_len(10.0 * (n / 400000.0) ** (1.0 / 3.0))


def _step_inputs(c, seed):
    """Ions of charge z with their electrons (10 eV) in a sphere, near the envelope's peak."""
    ni = max(1, int(round(c["n"] / (1 + c["z"]))))
    ne = max(0, c["n"] - ni)
    r0 = _radius(c["n"])
    cl = synth.make_cluster(seed, ni, ne, r0, c["z"], synth.MASS_XE, kT_e_ev=10.0)
    tau = synth.fs_to_time(100.0)
    env = c.get("env", 1)
    tau = synth.sin2_length_from_fwhm(tau) if env == synth.ENV_SIN2 else tau
    peak = tau / 2 if env == synth.ENV_SIN2 else (0.0 if env == synth.ENV_FLAT else 2 * tau)
    dt = 0.02
    t0 = peak + 0.9
    p = {"a0": 0.07, "tau": tau, "t0": t0, "dt": dt, "softening": synth.nm_to_len(0.1),
         "lambda_um": LAMBDA, "polarization": c.get("pol", 0), "envelope": env,
         "boundary": c.get("boundary", 0), "box": 20 * r0 if c.get("boundary", 0) else 0.0,
         "t_switch": t0 + 2.5 * dt, "min_image": 0}
    return [(p, cl)]


def _scan_entries(c):
    return synth.batched_scan(c["clusters"], 0, c["n_min"], c["n_max"])


def _scan_inputs(c, seed):
    out = []
    for e in _scan_entries(c):  # the sizes are the case's, the records the seed's
        e.seed += 7919 * seed
        p = {"a0": e.a0, "tau": e.tau, "t0": e.tau / 2 + 0.9, "dt": 0.02,
             "softening": synth.nm_to_len(0.1), "lambda_um": LAMBDA, "polarization": 0,
             "envelope": synth.ENV_SIN2, "boundary": 0, "box": 0.0, "t_switch": 0.0,
             "min_image": 0}
        out.append((p, synth.scan_cluster(e)))
    return out


def _image_inputs(c, seed):
    """A singly charged plasma filling its periodic cube."""
    rng = np.random.default_rng(seed)
    n, ni = c["n"], c["n"] // 2
    box = synth.nm_to_len(16.0) * (n / 400000.0) ** (1.0 / 3.0)
    x = rng.uniform(-0.5 * box, 0.5 * box, (n, 3))
    u = rng.normal(size=(n, 3)) * synth.thermal_sigma_u(10.0, 1.0)
    u[:ni] = 0.0
    z = np.where(np.arange(n) < ni, 1, -1).astype(np.int32)
    mass = np.where(np.arange(n) < ni, synth.MASS_AR, 1.0)
    cl = synth.Cluster(x, u, z, mass, np.ones(n), np.ones(n, np.uint8), ni, n - ni)
    p = {"a0": 0.07, "tau": 1.0, "t0": 0.9, "dt": 0.02, "softening": synth.nm_to_len(0.1),
         "lambda_um": LAMBDA, "polarization": 0, "envelope": synth.ENV_FLAT, "boundary": 1,
         "box": box, "t_switch": 0.0, "min_image": 1}
    return [(p, cl)]


_INPUTS = {"step": _step_inputs, "diag": _step_inputs, "scan": _scan_inputs,
           "image": _image_inputs}


def _ionize_inputs(c, seed):
    """Argon past the pulse's peak: ions of charge 7 and 8, their electrons (100 eV) around
    them in the first slots, the remaining slots free."""
    rng = np.random.default_rng(seed)
    n = c["atoms"]
    r0 = synth.nm_to_len(8.0 * (n / 200000) ** (1 / 3), LAMBDA_AR)
    z = rng.integers(7, 9, n).astype(np.int32)
    ne, slots = int(z.sum()), 8 * n
    rw = synth.nm_to_len(synth.ARGON["r_w_nm"], LAMBDA_AR)
    x = np.zeros((n + slots, 3))
    u = np.zeros((n + slots, 3))
    x[:n] = synth.uniform_sphere(rng, n, r0)
    x[n:n + ne] = np.repeat(x[:n], z, axis=0) + synth.uniform_sphere(rng, ne, rw)
    u[n:n + ne] = rng.normal(size=(ne, 3)) * synth.thermal_sigma_u(100.0, 1.0)
    zz = np.zeros(n + slots, np.int32)
    zz[:n], zz[n:n + ne] = z, -1
    mass = np.ones(n + slots)
    mass[:n] = synth.ARGON["mass"]
    kind = np.full(n + slots, md.KIND_INACTIVE, np.uint8)
    kind[:n], kind[n:n + ne] = md.KIND_ION, md.KIND_ELECTRON
    tau = synth.sin2_length_from_fwhm(synth.fs_to_time(100.0, LAMBDA_AR))
    cfg = md.make_config(a0=0.0617, tau=tau, t0=0.62 * tau, dt=0.02,
                         softening=synth.nm_to_len(0.1, LAMBDA_AR), lambda_um=LAMBDA_AR,
                         envelope=synth.ENV_SIN2, rate_model=md.RATES_PLAIN, ionize_every=1,
                         zmax=8, n_ions=n, slot_base=n, seed=seed + 17, r_loc=3 * rw, r_create=rw,
                         species=synth.ARGON)
    return cfg, md.HostParticles(x, u, zz, mass, np.ones(n + slots), kind)


def _host_records(n):
    """Page-locked host arrays for the read-back of n records."""
    pin = lambda shape, t: torch.zeros(shape, dtype=t, pin_memory=True).numpy()  # noqa: E731
    return md.HostParticles(pin((n, 3), torch.float64), pin((n, 3), torch.float64),
                            pin(n, torch.int32), pin(n, torch.float64), pin(n, torch.float64),
                            pin(n, torch.uint8))


def _field_inputs(c, seed):
    rng = np.random.default_rng(seed)
    ns, nt = c["ns"], c["nt"]
    r0 = _radius(ns)
    src = np.zeros((ns, 4), np.float32)
    src[:, :3] = synth.uniform_sphere(rng, ns, r0)
    q = np.where(np.arange(ns) < ns // 4, 3.0, -1.0)
    src[:, 3] = md.coulomb_constant(LAMBDA) * q
    tgt = np.zeros((nt, 4), np.float32)
    tgt[:, :3] = synth.uniform_sphere(rng, nt, 1.5 * r0)
    return src, tgt, float(np.float32(synth.nm_to_len(0.1) ** 2))


def _mlp_params(rng):
    """Parameters of the 4 -> 64 -> 64 -> 8 network: uniform weights, small biases."""
    u = lambda fi, fo: rng.uniform(-1, 1, fi * fo) * math.sqrt(6.0 / (fi + fo))  # noqa: E731
    b = lambda n: rng.uniform(-0.1, 0.1, n)  # noqa: E731
    return np.concatenate([u(4, 64), b(64), u(64, 64), b(64), u(64, 8), b(8)]).astype(np.float32)


def _rates_inputs(c, seed):
    rng = np.random.default_rng(seed)
    n = c["n"]
    logu = lambda lo, hi: 10.0 ** rng.uniform(math.log10(lo), math.log10(hi), n)  # noqa: E731
    return (_mlp_params(rng), logu(2e-3, 0.5), rng.integers(0, 8, n).astype(np.int32),
            logu(1e17, 1e23), logu(1.0, 1e3))


def _grad_inputs(c, seed):
    rng = np.random.default_rng(seed)
    n = c["n"]
    return (_mlp_params(rng), rng.uniform(-1, 1, (n, 4)).astype(np.float32),
            rng.integers(0, 8, n).astype(np.int32), rng.uniform(0, 1, n).astype(np.float32))


def _cuda(*arrays):
    return [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in arrays]


def prepare(case, seed):
    k = case["kind"]
    if k in _INPUTS:
        ins = _INPUTS[k](case, seed)
        ctx = md.Context([md.make_config(**p) for p, _ in ins],
                         [md.HostParticles.from_cluster(c) for _, c in ins])
        if case.get("tuned"):
            ctx.autotune()
        ctx.sync()
        return {"case": case, "ctx": ctx, "out": [_host_records(c.n) for _, c in ins]}
    if k == "ionize":
        cfg, p = _ionize_inputs(case, seed)
        ctx = md.Context([cfg], [p])
        ctx.sync()
        return {"case": case, "ctx": ctx, "out": [_host_records(p.n)]}
    stream = torch.cuda.current_stream().cuda_stream
    if k == "field":
        src, tgt, eps2 = _field_inputs(case, seed)
        s, t = _cuda(src, tgt)
        e = torch.empty((case["nt"], 3), dtype=torch.float64, device="cuda")
        phi = torch.empty(case["nt"], dtype=torch.float64, device="cuda") if case["phi"] else None
        return {"case": case, "src": s, "tgt": t, "eps2": eps2, "e": e, "phi": phi,
                "stream": stream}
    if k == "rates":
        w, emag, z, ne, te = _cuda(*_rates_inputs(case, seed))
        nu = torch.empty(case["n"], dtype=torch.float64, device="cuda")
        return {"case": case, "cfg": md.mlp_train_config(synth.ARGON), "in": (w, emag, z, ne, te),
                "nu": nu, "stream": stream}
    w, f, z, t = _cuda(*_grad_inputs(case, seed))
    return {"case": case, "in": (w, f, z, t),
            "grad": torch.empty(5000, dtype=torch.float32, device="cuda"),
            "loss": torch.empty(1, dtype=torch.float32, device="cuda"), "stream": stream}


def _f32(a):
    return torch.from_numpy(a).float()


def run(state):
    c = state["case"]
    k = c["kind"]
    if k in ("step", "scan", "image"):
        ctx = state["ctx"]
        ctx.step(c["steps"])
        got = [ctx.get_particles(i, out) for i, out in enumerate(state["out"])]
        if k == "scan":  # the frames of a scan, all clusters one after the other
            return {"x": torch.cat([_f32(p.x) for p in got]),
                    "u": torch.cat([_f32(p.u) for p in got])}
        return {"x": _f32(got[0].x), "u": _f32(got[0].u)}
    if k == "diag":
        ctx = state["ctx"]
        d = ctx.step_diag()[0]
        p = ctx.get_particles(0, state["out"][0])
        return {"energy": np.array([d["ke"], d["ke_ions"], d["ke_electrons"], d["pe"], d["total"],
                                    *d["p"]], np.float32),
                "count": np.concatenate([[d["n_active"], d["n_nonfinite"]], d["charge_count"]]),
                "x": _f32(p.x), "u": _f32(p.u)}
    if k == "ionize":
        ctx = state["ctx"]
        ctx.step(c["steps"])
        p = ctx.get_particles(0, state["out"][0])
        ion = ctx.ionization(0)
        return {"x": _f32(p.x), "u": _f32(p.u), "z": p.z, "kind": p.kind,
                "emag": _f32(ion["emag"]), "ne": _f32(ion["ne"]), "te": _f32(ion["te"])}
    if k == "field":
        f = md.coulomb_field_device if c["alloc"] else md.coulomb_field_device_noalloc
        e, phi = state["e"], state["phi"]
        f(state["src"].data_ptr(), c["ns"], state["tgt"].data_ptr(), c["nt"], state["eps2"], -1,
          e.data_ptr(), phi.data_ptr() if c["phi"] else None, state["stream"])
        return {"e": e.float(), "phi": phi.float() if c["phi"] else None}
    if k == "rates":
        w, emag, z, ne, te = state["in"]
        md.ion_rates_device(state["cfg"], md.RATES_MLP, w.data_ptr(), emag.data_ptr(),
                            z.data_ptr(), ne.data_ptr(), te.data_ptr(), c["n"],
                            state["nu"].data_ptr(), state["stream"])
        return state["nu"].float()
    w, f, z, t = state["in"]
    md.mlp_loss_grad_device(w.data_ptr(), f.data_ptr(), z.data_ptr(), t.data_ptr(), c["n"],
                            state["grad"].data_ptr(), state["loss"].data_ptr(), state["stream"])
    return {"grad": state["grad"], "loss": state["loss"]}


# ------------------------------------------------------------------- work --

PAIR_FLOPS = 18   # 3 differences, 3 squares added, 1/r^3 from 1/r, 3 products added
RECORD_BYTES = 69  # one record read or written by the host (x, u, z, mass, w, kind)


def _sizes(case):
    if case["kind"] == "scan":
        return [e.n_total for e in _scan_entries(case)]
    if case["kind"] == "ionize":
        return [int(8.5 * case["atoms"])]
    return [case["n"]]


def work(case):
    k = case["kind"]
    if k in _INPUTS or k == "ionize":
        ns, steps = _sizes(case), case.get("steps", 1)
        pairs = float(sum(n * n for n in ns)) * steps
        state = sum(ns) * 130.0 * steps  # the integrator state read and written each step
        return {"flops": PAIR_FLOPS * pairs, "bytes": state + RECORD_BYTES * sum(ns)}
    if k == "field":
        out = 24 + (8 if case["phi"] else 0)
        return {"flops": PAIR_FLOPS * float(case["nt"]) * case["ns"],
                "bytes": 16.0 * (case["nt"] + case["ns"]) + out * case["nt"]}
    n = float(case["n"])
    if k == "rates":
        return {"flops": 2 * (4 * 64 + 64 * 64 + 64) * n, "bytes": 36 * n + 20000}
    return {"flops": 6 * (4 * 64 + 64 * 64 + 64) * n, "bytes": 24 * n + 40000}


# ------------------------------------------------------------------ exact --

def _field64(x, q, eps, box=0.0):
    """Softened Coulomb field and potential at the records x (their own term left out)."""
    n = x.shape[0]
    e, phi = torch.empty_like(x), torch.empty(n, dtype=x.dtype, device=x.device)
    chunk = max(1, int(6e7 // n))
    self_phi = q / eps
    for i in range(0, n, chunk):
        d = [x[i:i + chunk, None, c] - x[None, :, c] for c in range(3)]
        if box:
            d = [v - box * torch.round(v / box) for v in d]
        r2 = d[0] * d[0]
        r2.addcmul_(d[1], d[1]).addcmul_(d[2], d[2]).add_(eps * eps)
        s = r2.rsqrt_()
        phi[i:i + chunk] = s @ q
        s = s * s * s * q
        for c in range(3):
            e[i:i + chunk, c] = (d[c] * s).sum(1)
    return e, phi - self_phi


def _laser64(p, t):
    env, tau = p["envelope"], p["tau"]
    if env == synth.ENV_SIN2:
        a = math.sin(math.pi * t / tau) ** 2 if 0.0 <= t <= tau else 0.0
    elif env == synth.ENV_FLAT:
        a = 1.0
    else:
        a = math.exp(-(2.0 * math.log(2.0) if env == synth.ENV_GAUSS else 2.77)
                     * ((t - 2 * tau) / tau) ** 2)
    a *= p["a0"]
    c = -a * math.cos(t) if p["polarization"] else 0.0
    return [a * math.sin(t), c, 0.0], [-c, a * math.sin(t), 0.0]


def _kick64(u, e, b, qm, dt):
    h = (0.5 * dt * qm)[:, None]
    um = u + h * e
    t = h * b / torch.sqrt(1.0 + (um * um).sum(1, keepdim=True))
    s = 2.0 * t / (1.0 + (t * t).sum(1, keepdim=True))
    return um + torch.linalg.cross(um + torch.linalg.cross(um, t), s) + h * e


def _steps64(p, cl, steps):
    """x, u after `steps` steps and the (energies, momentum) at the start of the last."""
    x, u, z, mass, w = _cuda(cl.x, cl.u, cl.z.astype(np.float64), cl.mass, cl.w)
    kc = 2.0 * math.pi * 2.8179403262e-15 / (p["lambda_um"] * 1e-6)
    diag = None
    for n in range(steps):
        t = p["t0"] + n * p["dt"]
        t1 = p["t0"] + (n + 1) * p["dt"]
        e, phi = _field64(x, kc * w * z, p["softening"], p["box"] if p["min_image"] else 0.0)
        le, lb = (torch.tensor(v, dtype=x.dtype, device=x.device) for v in _laser64(p, t))
        un = _kick64(u, e + le, lb.expand_as(u), z / mass, p["dt"])
        m = 0.5 * (u + un)
        uu = (m * m).sum(1)
        ke = w * mass * uu / (torch.sqrt(1.0 + uu) + 1.0)
        pe = (0.5 * w * z * phi).sum()
        ion = z >= 0
        diag = torch.stack([ke.sum(), ke[ion].sum(), ke[~ion].sum(), pe, ke.sum() + pe,
                            *(w * mass) @ m])
        u = un
        x = x + p["dt"] * u / torch.sqrt(1.0 + (u * u).sum(1, keepdim=True))
        if p["boundary"] == 1 or (p["boundary"] == 2 and t1 < p["t_switch"]):
            x = x - p["box"] * torch.floor((x + 0.5 * p["box"]) / p["box"])
    return x, u, diag


def _mlp64(w, f, z):
    """Output of charge state z of the network, parameters and features in FP64."""
    o = [0, 256, 320, 4416, 4480, 4992, 5000]
    w1, b1, w2, b2, w3, b3 = (w[o[i]:o[i + 1]] for i in range(6))
    silu = torch.nn.functional.silu
    h = silu(f @ w1.reshape(64, 4).T + b1)
    h = silu(h @ w2.reshape(64, 64).T + b2)
    y = h @ w3.reshape(8, 64).T + b3
    return y.gather(1, z.long()[:, None])[:, 0]


def exact(case, seed):
    k = case["kind"]
    if k == "ionize":
        return None  # the draws decide which records exist
    if k in _INPUTS:
        steps = case.get("steps", 1)
        if sum(n * n for n in _sizes(case)) * steps > 6e10:
            return None
        got = [_steps64(p, cl, steps) for p, cl in _INPUTS[k](case, seed)]
        out = {"x": torch.cat([g[0] for g in got]), "u": torch.cat([g[1] for g in got])}
        if k == "diag":
            out["energy"] = got[0][2]
            out["count"] = None
        return out
    if k == "field":
        src, tgt, eps2 = _field_inputs(case, seed)
        s, t = (v.double() for v in _cuda(src, tgt))
        e, phi = [], []
        for i in range(0, case["nt"], 128):
            d = t[i:i + 128, None, :3] - s[None, :, :3]
            r = torch.rsqrt((d * d).sum(2) + eps2)
            phi.append(r @ s[:, 3])
            e.append((d * (s[:, 3] * r ** 3)[:, :, None]).sum(1))
        return {"e": torch.cat(e), "phi": torch.cat(phi) if case["phi"] else None}
    if k == "rates":
        w, emag, z, ne, te = _cuda(*_rates_inputs(case, seed))
        ip = torch.tensor(synth.ARGON["ip_ev"], dtype=torch.float64, device="cuda")[z.long()]
        k_si = 2.0 * math.pi / (LAMBDA * 1e-6)
        fau = emag.clamp(min=1e-6) * 510998.95 * k_si / 5.14220674763e11
        f0 = (2.0 * ip / 27.211386245988) ** 1.5
        f = torch.stack([(torch.log10(fau / f0) + 1.4) / 1.5, z / 8.0,
                         (torch.log10(ne.clamp(min=1e15)) - 19.5) / 4.5,
                         (torch.log10(te.clamp(min=0.1) / ip) + 0.2) / 3.0], 1).double()
        y = _mlp64(w.double(), f, z)
        return (10.0 ** (6.0 * y - 6.0) - 1e-12).clamp(min=0.0)
    w, f, z, t = _cuda(*_grad_inputs(case, seed))
    w = w.double().requires_grad_()
    loss = ((_mlp64(w, f.double(), z) - t.double()) ** 2)
    loss.mean().backward()
    # the call reports the sum of the squared errors beside the gradient of their mean
    return {"grad": w.grad, "loss": loss.sum().detach()[None]}
