"""The work that is timed: passes through the public entry points over the range that users run.

Sizes and settings are those of the repository's own workloads (``inputs.py``), tests and benchmark:
head-on runs of one species and energy, the species x energy sweep, thermal baths, the mixed-parameter
sweep as a CUDA graph, batches in parts, differentiation, device-drawn initial conditions and ensemble
statistics. Trajectory lengths are heavy-tailed, so every batch of trajectories carries an attempt cap,
as the benchmark's side measurements do (their smaller cap, 8,192 attempted steps, and four times it).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2509_15117_gb300 import binding as Bd
from paper_2509_15117_gb300 import inputs as I
from paper_2509_15117_gb300 import schedule as Sch
from paper_2509_15117_gb300.autograd import observables

KINDS = ("run", "thermal", "sweep", "queue", "graph", "tangent", "autograd", "sample", "stats")
ENERGIES_K = (1.5e-6,) + I.C2_ENERGIES_K
SAMPLERS = {"head_on": Bd.IA_SAMPLE_HEAD_ON, "sphere": Bd.IA_SAMPLE_SPHERE, "disk": Bd.IA_SAMPLE_DISK}


def listed():
    return [
        # One trajectory looked at by hand: host arrays in, observables and the final state out.
        {"name": "run_one", "kind": "run", "n": 1, "species": "Rb", "E_K": 1.5e-6, "cap": 8192, "y_final": True},
        # The head-on map of Fig. 1 at its 32 x 32 sampling, directions uniform on the octant.
        {"name": "run_map_1024", "kind": "run", "n": 1024, "species": "Rb", "E_K": 1.5e-6, "cap": 32768,
         "y_final": False},
        # A large batch of short trajectories (1 mK, mostly single bounces): throughput.
        {"name": "run_rb_1mK_262144", "kind": "run", "n": 262144, "species": "Rb", "E_K": 1e-3, "cap": 32768,
         "y_final": False},
        # Thermal run of Fig. 3: initial conditions drawn on the device, integrated, reduced to statistics.
        {"name": "thermal_rb_100uK_49999", "kind": "thermal", "n": 49999, "species": "Rb", "T_K": 1e-4, "De_K": 1.0,
         "sampler": "sphere", "cap": 8192},
        # The species x energy sweep on a coarse grid: 40 systems in one launch, costliest first.
        {"name": "sweep_40x41x41", "kind": "sweep", "grid": 41, "cap": 8192, "order": True},
        # The same sweep as one batch in four parts, as long runs are split.
        {"name": "queue_40x32x32", "kind": "queue", "grid": 32, "parts": 4, "cap": 32768},
        # All 250 cells of the mixed-parameter sweep: one CUDA graph, launch and per-cell statistics.
        {"name": "graph_mixed_250", "kind": "graph", "inv_scale": 256, "cap": 8192},
        # Derivatives along (theta, phi, E, q) and the Lyapunov exponent.
        {"name": "tangent_4dir_3001", "kind": "tangent", "n": 3001, "ndir": 4, "cap": 8192},
        # A differentiable call: observables, and gradients by the adjoint kernel.
        {"name": "autograd_1000", "kind": "autograd", "n": 1000, "cap": 8192},
        # Initial conditions of a large head-on run and of a Monte Carlo bath.
        {"name": "sample_head_on_16M", "kind": "sample", "sampler": "head_on", "n": 1 << 24},
        {"name": "sample_disk_4194301", "kind": "sample", "sampler": "disk", "n": 4194301},
        # Statistics of a large ensemble, one cell per system of the mixed sweep.
        {"name": "stats_4M_250", "kind": "stats", "n": 1 << 22, "cells": 250},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(KINDS)
    c = {"kind": kind}
    if kind == "run":
        # slow collisions make long complexes: large batches of them run for minutes, so the size falls with 1/E
        E = rng.choice(ENERGIES_K)
        c.update(n=_log(rng, 1, 262144 if E > 1e-4 else 30000), species=rng.choice(I.C2_SPECIES), E_K=E,
                 cap=rng.choice((8192, 32768)), y_final=rng.random() < 0.5)
    elif kind == "thermal":
        c.update(n=_log(rng, 100, 60000), species=rng.choice(I.C2_SPECIES), T_K=rng.choice(I.FIG3_TEMPS_K),
                 De_K=rng.choice(I.FIG3_DEPTHS_K), sampler=rng.choice(("sphere", "disk")), cap=8192)
    elif kind == "sweep":
        c.update(grid=_log(rng, 1, 50), cap=8192, order=rng.random() < 0.5)
    elif kind == "queue":
        c.update(grid=_log(rng, 2, 36), parts=rng.randint(1, 8), cap=rng.choice((8192, 32768)))
    elif kind == "graph":
        c.update(inv_scale=_log(rng, 256, 8192), cap=8192)
    elif kind == "tangent":
        c.update(n=_log(rng, 1, 4000), ndir=rng.randint(1, 4), cap=8192)
    elif kind == "autograd":
        c.update(n=_log(rng, 1, 1200), cap=8192)
    elif kind == "sample":
        c.update(sampler=rng.choice(tuple(SAMPLERS)), n=_log(rng, 1, 1 << 22))
    else:
        c.update(n=_log(rng, 1, 1 << 22), cells=rng.choice((1, 1, 3, 30, 40, 250, 500)))
    return c


# ---------------------------------------------------------------------------------------------

def _octant(n, seed):
    return I.octant_random(n, seed)


def _run_inputs(case, seed):
    sysd = I.make_system(case["species"], De_K=1.0, q=0.1, E_K=case["E_K"], max_attempts=case["cap"],
                         r0=I.r0_rule(I.SPECIES[case["species"]]["alpha"], I.kelvin(case["E_K"])))
    th, ph = _octant(case["n"], seed)
    y0 = I.head_on(th, ph, sysd.r0, I.speed_for_energy(I.kelvin(case["E_K"]), sysd.m_atom))
    return sysd.as_dict(), y0, np.zeros(case["n"])


def _sweep_inputs(case, seed):
    """The sweep's systems on a grid whose cells are sampled at random points, with a random rf phase."""
    systems, y0, _, sid = I.c2_workload(case["grid"])
    rng = np.random.default_rng(seed)
    speed = np.linalg.norm(y0[:, 9:12], axis=1)
    r0 = np.array([s.r0 for s in systems])[sid]
    u = rng.normal(size=(len(sid), 3))
    u = np.abs(u) / np.linalg.norm(u, axis=1, keepdims=True)
    y0[:, 6:9] = r0[:, None] * u
    y0[:, 9:12] = -speed[:, None] * u
    for s in systems:
        s.max_attempts = case["cap"]
    return systems, y0, I.random_phase(len(sid), seed), sid


def _order(systems, sid):
    speeds = [s.atol_vel / 1e-10 for s in systems]
    return torch.from_numpy(Sch.order_by_cost(sid, Sch.system_cost(systems, speeds))).cuda()


def _thermal_system(case):
    m_a = I.SPECIES[case["species"]]["mass_amu"] * I.AMU_TO_ME
    return I.make_system(case["species"], De_K=case["De_K"], q=0.1, r0=5000.0,
                         v_scale=math.sqrt(I.kelvin(case["T_K"]) / m_a), max_attempts=case["cap"]).as_dict()


def _sampler_args(kind, T_K=1e-4):
    if kind == "head_on":
        return {"E": I.kelvin(1.5e-6)}
    kw = {"kT": I.kelvin(T_K), "kT_ion": I.kelvin(1e-5)}
    return dict(kw, b_max=2000.0, micromotion=True) if kind == "disk" else kw


def _c5(n, seed, cap, ndir=4):
    """The differentiation workload with the last ndir of its seed directions (theta, phi, E, q)."""
    sysd, y0, phi0, seeds, dq = I.c5_workload(n, seed=seed)
    sysd.max_attempts = cap
    dy0 = np.concatenate([seeds, np.zeros((n, 1, 12))], axis=1)
    return sysd.as_dict(), y0, phi0, dy0[:, 4 - ndir:], dq[4 - ndir:]


def prepare(case, seed):
    k = case["kind"]
    if k == "run":
        d, y0, phi0 = _run_inputs(case, seed)
        return {"case": case, "S": Bd.System([d]), "y0": y0, "phi0": phi0}
    if k == "thermal":
        d = _thermal_system(case)
        n = case["n"]
        return {"case": case, "S": Bd.System([d]), "out": Bd.alloc_obs(n), "stats": Bd.alloc_stats(1),
                "smp": Bd.make_sampler(SAMPLERS[case["sampler"]], d, seed, **_sampler_args(case["sampler"], case["T_K"])),
                "y": torch.empty((12, n), dtype=torch.float64, device="cuda"),
                "phi": torch.empty(n, dtype=torch.float64, device="cuda")}
    if k in ("sweep", "queue"):
        systems, y0, phi0, sid = _sweep_inputs(case, seed)
        S = Bd.System([s.as_dict() for s in systems])
        y, p, d = Bd.to_device_soa(y0, phi0, sid)
        st = {"case": case, "S": S, "y": y, "phi": p, "sid": d, "out": Bd.alloc_obs(len(sid)), "order": None}
        if k == "queue" or case["order"]:
            st["order"] = _order(systems, sid)
        if k == "queue":
            st["Q"] = Bd.Queue(S.handle, len(sid))
        return st
    if k == "graph":
        systems, y0, phi0, sid = I.c4_workload(scale=1.0 / case["inv_scale"], seed=seed)
        for s in systems:
            s.max_attempts = case["cap"]
        S = Bd.System([s.as_dict() for s in systems])
        y, p, d = Bd.to_device_soa(y0, phi0, sid)
        out, stats, stream = Bd.alloc_obs(len(sid)), Bd.alloc_stats(len(systems)), torch.cuda.Stream()
        torch.cuda.synchronize()
        with torch.cuda.stream(stream):
            G = Bd.Graph(S.handle, y, p, d, out, stream, order=_order(systems, sid), cell_id=d,
                         n_cells=len(systems), stats=stats)
        stream.synchronize()
        return {"case": case, "S": S, "G": G, "out": out, "stats": stats, "stream": stream}
    if k == "tangent":
        d, y0, phi0, dy0, dq = _c5(case["n"], seed, case["cap"], case["ndir"])
        y, p, _ = Bd.to_device_soa(y0, phi0)
        return {"case": case, "S": Bd.System([d]), "y": y, "phi": p, "dq": dq, "out": Bd.alloc_obs(case["n"]),
                "dy0": torch.from_numpy(np.ascontiguousarray(np.transpose(dy0, (1, 2, 0)))).cuda(),
                "tan": Bd.alloc_tangent(case["n"], case["ndir"])}
    if k == "autograd":
        d, y0, phi0, _, _ = _c5(case["n"], seed, case["cap"])
        g = np.random.default_rng(seed).normal(size=(case["n"], 4)) * np.array([1.0, 1e-2, 1e10, 1e-9])
        return {"case": case, "desc": d, "y0": torch.from_numpy(y0).cuda(), "phi": torch.from_numpy(phi0).cuda(),
                "q": torch.tensor(d["q"], dtype=torch.float64), "g": torch.from_numpy(g).cuda()}
    if k == "sample":
        n, d = case["n"], I.make_system("Rb").as_dict()
        return {"case": case, "smp": Bd.make_sampler(SAMPLERS[case["sampler"]], d, seed, **_sampler_args(case["sampler"])),
                "y": torch.empty((12, n), dtype=torch.float64, device="cuda"),
                "phi": torch.empty(n, dtype=torch.float64, device="cuda")}
    S = Bd.System([I.make_system("Rb").as_dict()])
    out, cell = _observables(case, seed)
    return {"case": case, "S": S, "out": out, "cell": cell, "stats": Bd.alloc_stats(case["cells"])}


def _observables(case, seed):
    """Observables of an ensemble as a run leaves them: three in ten complexes with a power-law bounce count and
    lifetime, lengths log-normal, trajectories grouped by cell as the samplers lay them out."""
    n, cells = case["n"], case["cells"]
    g = torch.Generator(device="cuda").manual_seed(seed)

    def u():
        return torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
    out = Bd.alloc_obs(n)
    for f in ("theta_s", "dp", "t_final"):
        out[f].copy_(u())
    cx = u() < 0.3
    nb = torch.where(cx, 1.0 + (u() + 1e-6) ** -0.7, torch.ones_like(out["dp"]))
    out["n_bounce"].copy_(nb.clamp(max=1e6).to(torch.int32))
    out["status"].copy_(torch.where(cx, Bd.ST_COMPLEX, 0).to(torch.int32))
    out["status"].bitwise_or_((u() < 1e-3).to(torch.int32) * Bd.ST_MAX_STEPS)
    out["n_steps"].copy_((700.0 * torch.exp(1.2 * (u() + u() + u() - 1.5).abs() * 2.0)).to(torch.int32))
    out["n_rej"].copy_((out["n_steps"].to(torch.float64) * 0.1 * u()).to(torch.int32))
    out["dE_ion"].copy_(1e-11 * (u() + u() - 1.0) * out["n_bounce"].to(torch.float64).sqrt())
    out["t_first_bounce"].copy_(6e11 * (1.0 + 0.01 * u()))
    out["t_last_bounce"].copy_(out["t_first_bounce"] + torch.where(cx, 4e10 * (u() + 1e-5) ** -0.6, 0.0))
    cell = (torch.arange(n, device="cuda") * cells // n).to(torch.int32) if cells > 1 else None
    return out, cell


def _stats(stats):
    """The two kinds of fields of the statistics records, as views."""
    w = stats.view(torch.int64).view(-1, Bd.STATS_DTYPE.itemsize // 8)
    f = stats.view(torch.float64).view(w.shape)
    return {"counts": w[:, :-2], "sums": f[:, -2:]}


def run(state):
    c, k = state["case"], state["case"]["kind"]
    if k == "run":
        return state["S"].run(state["y0"], state["phi0"], y_final=c["y_final"])
    if k == "thermal":
        Bd.ia_sample_ics(state["smp"], 0, state["y"], state["phi"])
        Bd.ia_launch(state["S"].handle, state["y"], state["phi"], None, state["out"])
        Bd.ia_reduce_stats(state["S"].handle, state["out"], c["n"], None, 1, state["stats"])
        return {"y": state["y"], "phi": state["phi"], "obs": state["out"], "stats": _stats(state["stats"])}
    if k == "sweep":
        Bd.ia_launch(state["S"].handle, state["y"], state["phi"], state["sid"], state["out"], order=state["order"])
        return state["out"]
    if k == "queue":
        Q, n = state["Q"], int(state["phi"].shape[0])
        Q.reset()
        for j in range(c["parts"]):
            Q.launch(state["y"], state["phi"], state["sid"], state["out"],
                     n * (j + 1) // c["parts"] - n * j // c["parts"], order=state["order"])
        return state["out"]
    if k == "graph":
        state["stream"].wait_stream(torch.cuda.current_stream())
        state["G"].launch(state["stream"])
        torch.cuda.current_stream().wait_stream(state["stream"])
        return {"obs": state["out"], "stats": _stats(state["stats"])}
    if k == "tangent":
        Bd.ia_launch_tangent(state["S"].handle, state["y"], state["phi"], None, state["out"], state["dy0"],
                             state["dq"], state["tan"])
        return {"obs": state["out"], "tan": state["tan"]}
    if k == "autograd":
        y0, q = state["y0"].clone().requires_grad_(), state["q"].clone().requires_grad_()
        obs = observables(y0, q, state["phi"], state["desc"])
        gy, gq = torch.autograd.grad(obs, (y0, q), state["g"])
        return {"obs": obs.detach(), "grad_y0": gy, "grad_q": gq}
    if k == "sample":
        Bd.ia_sample_ics(state["smp"], 0, state["y"], state["phi"])
        return {"y": state["y"], "phi": state["phi"]}
    Bd.ia_reduce_stats(state["S"].handle, state["out"], c["n"], state["cell"], c["cells"], state["stats"])
    return _stats(state["stats"])


# ---------------------------------------------------------------------------------------------

FLOPS_ATTEMPT = 884.0    # arithmetic of one attempted step of the method (FMA = 2)
FLOPS_TANGENT = 11680.0  # ... with four tangent directions
FLOPS_ADJOINT = 29670.0  # ... forward, replay and reverse sweep for four objectives
BOUNCE_ATTEMPTS = 750.0  # steps near the ion that the tolerance asks for in one pass
OBS_BYTES, IC_BYTES = 6 * 8 + 4 * 4, 13 * 8
SAMPLE_FLOPS = {"head_on": 40.0, "sphere": 250.0, "disk": 300.0}


def _attempts(sysd, speed, cap):
    """Fewest attempted steps of a trajectory: in and out at the largest step, and one pass near the ion."""
    return min(float(cap), 2.0 * sysd["r0"] / (speed * sysd["h_max"]) + BOUNCE_ATTEMPTS)


def work(case):
    k = case["kind"]
    if k == "run":
        s = I.make_system(case["species"], E_K=case["E_K"],
                          r0=I.r0_rule(I.SPECIES[case["species"]]["alpha"], I.kelvin(case["E_K"]))).as_dict()
        a = _attempts(s, I.speed_for_energy(I.kelvin(case["E_K"]), s["m_atom"]), case["cap"])
        b = case["n"] * (IC_BYTES + OBS_BYTES + (96 if case["y_final"] else 0))
        return {"bytes": b, "flops": case["n"] * a * FLOPS_ATTEMPT}
    if k == "thermal":
        d = _thermal_system(case)
        a = _attempts(d, 2.0 * math.sqrt(I.kelvin(case["T_K"]) / d["m_atom"]), case["cap"])
        return {"bytes": case["n"] * (IC_BYTES + OBS_BYTES) + Bd.STATS_DTYPE.itemsize,
                "flops": case["n"] * (0.25 * a * FLOPS_ATTEMPT + SAMPLE_FLOPS[case["sampler"]])}
    if k in ("sweep", "queue"):
        sy = [(I.speed_for_energy(I.kelvin(E), s.m_atom), s.as_dict()) for _, E, s in I.c2_systems()]
        per = case["grid"] ** 2
        b = len(sy) * per * (IC_BYTES + 4 + OBS_BYTES + (8 if k == "queue" or case["order"] else 0))
        return {"bytes": b, "flops": sum(per * _attempts(d, v, case["cap"]) * FLOPS_ATTEMPT for v, d in sy)}
    if k == "graph":
        b = f = 0.0
        for c in I.c4_cells():
            n = max(1, int(round(c["n"] / case["inv_scale"])))
            d = I.make_system(c["species"], E_K=1.5e-6).as_dict()
            f += n * FLOPS_ATTEMPT * _attempts(d, I.speed_for_energy(I.kelvin(1.5e-6), d["m_atom"]), case["cap"])
            b += n * (IC_BYTES + 4 + 8 + OBS_BYTES) + Bd.STATS_DTYPE.itemsize
        return {"bytes": b, "flops": f}
    if k in ("tangent", "autograd"):
        d = I.make_system("Rb", E_K=1.5e-6).as_dict()
        a = case["n"] * _attempts(d, I.speed_for_energy(I.kelvin(1.5e-6), d["m_atom"]), case["cap"])
        if k == "tangent":
            per = FLOPS_ATTEMPT + (FLOPS_TANGENT - FLOPS_ATTEMPT) * case["ndir"] / 4.0
            return {"bytes": case["n"] * (IC_BYTES + OBS_BYTES + case["ndir"] * (96 + 32) + 8), "flops": a * per}
        return {"bytes": case["n"] * (2 * IC_BYTES + OBS_BYTES + 2 * 32 + 96) + 48,
                "flops": a * (FLOPS_ADJOINT + FLOPS_ATTEMPT)}
    if k == "sample":
        return {"bytes": case["n"] * IC_BYTES, "flops": case["n"] * SAMPLE_FLOPS[case["sampler"]]}
    cells = case["cells"]
    return {"bytes": case["n"] * (4 * 4 + 3 * 8 + (4 if cells > 1 else 0)) + cells * Bd.STATS_DTYPE.itemsize,
            "flops": 6.0 * case["n"]}


# ---------------------------------------------------------------------------------------------
# 64-bit values from plain numpy

def exact(case, seed):
    k = case["kind"]
    if k == "sample" and case["n"] <= 1 << 24:
        y, phi = _exact_sample(case, seed)
        return {"y": y, "phi": phi}
    if k == "stats":
        return _exact_stats(case, seed)
    if k == "run" and case["n"] <= 2:
        return _exact_run(case, seed)
    return None


M64 = np.uint64(0xFFFFFFFF)


def _mulhilo(a, b):
    a0, a1, b0, b1 = a & M64, a >> np.uint64(32), b & M64, b >> np.uint64(32)
    t = a0 * b0
    w = a1 * b0 + (t >> np.uint64(32))
    u = a0 * b1 + (w & M64)
    return a1 * b1 + (w >> np.uint64(32)) + (u >> np.uint64(32)), a * b


def _philox(c0, c1, k0, k1):
    """Philox4x64-10 (Salmon et al., SC'11) on counters (c0, c1, 0, 0)."""
    m0, m1 = np.uint64(0xD2E7470EE14C6C93), np.uint64(0xCA5A826395121157)
    w0, w1 = np.uint64(0x9E3779B97F4A7C15), np.uint64(0xBB67AE8584CAA73B)
    z = np.zeros_like(c0)
    c = [c0, z + np.uint64(c1), z, z]
    k0, k1 = z[:1] + np.uint64(k0), z[:1] + np.uint64(k1)
    for r in range(10):
        if r:
            k0, k1 = k0 + w0, k1 + w1
        h0, l0 = _mulhilo(c[0], z + m0)
        h1, l1 = _mulhilo(c[2], z + m1)
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
    return c


def _exact_sample(case, seed):
    n, kind = case["n"], SAMPLERS[case["sampler"]]
    d, a = I.make_system("Rb").as_dict(), _sampler_args(case["sampler"])
    y, phi = np.zeros((12, n)), np.empty(n)
    for lo in range(0, n, 1 << 18):
        g = np.arange(lo, min(n, lo + (1 << 18)), dtype=np.uint64)
        sl = slice(lo, lo + len(g))
        u = [((w >> np.uint64(11)) | np.uint64(1)).astype(np.float64) * 2.0 ** -53
             for j in range(1 if kind == 0 else 4) for w in _philox(g, j, seed, kind)]
        phi[sl] = 2.0 * math.pi * u[0]
        ct = u[1] if kind == 0 else 2.0 * u[1] - 1.0
        az = (0.5 if kind == 0 else 2.0) * math.pi * u[2]
        st = np.sqrt((1.0 - ct) * (1.0 + ct))
        xh = np.stack([st * np.cos(az), st * np.sin(az), ct])
        if kind == 0:
            y[6:9, sl], y[9:12, sl] = d["r0"] * xh, -math.sqrt(2.0 * a["E"] / d["m_atom"]) * xh
            continue
        z = []
        for q in range(5):
            rho, t = np.sqrt(-2.0 * np.log(u[4 + 2 * q])), 2.0 * math.pi * u[5 + 2 * q]
            z += [rho * np.cos(t), rho * np.sin(t)]
        v = math.sqrt(a["kT"] / d["m_atom"]) * np.stack(z[0:3])
        if kind == 1:
            v = np.where(np.sum(v * xh, axis=0) >= 0.0, -v, v)
            y[6:9, sl] = d["r0"] * xh
        else:
            vh = v / np.sqrt(np.sum(v * v, axis=0))
            ref = np.where(np.abs(vh[2]) < 0.9, np.array([[0.0], [0.0], [1.0]]), np.array([[1.0], [0.0], [0.0]]))
            e1 = np.cross(vh, ref, axis=0)
            e1 /= np.sqrt(np.sum(e1 * e1, axis=0))
            e2 = np.cross(vh, e1, axis=0)
            b, t = a["b_max"] * np.sqrt(u[1]), 2.0 * math.pi * u[2]
            y[6:9, sl] = b * (np.cos(t) * e1 + np.sin(t) * e2) - np.sqrt(d["r0"] ** 2 - b * b) * vh
        y[9:12, sl] = v
        sv = math.sqrt(a["kT_ion"] / d["m_ion"])
        X = sv / (abs(d["q"][0]) * d["Omega"] / (2.0 * math.sqrt(2.0))) * np.stack(z[3:6])
        V = sv * np.stack(z[6:9])
        if kind == 2:
            h = 0.5 * d["rf_sign"] * np.array(d["q"])[:, None]
            f = 1.0 + h * np.cos(phi[sl])
            X, V = X * f, V * f - X * h * d["Omega"] * np.sin(phi[sl])
        y[0:3, sl], y[3:6, sl] = X, V
    return y, phi


def _exact_stats(case, seed):
    out, cell = _observables(case, seed)
    o = {k: v.cpu().numpy() for k, v in out.items()}
    nc = case["cells"]
    cell = cell.cpu().numpy().astype(np.int64) if cell is not None else np.zeros(case["n"], dtype=np.int64)
    s = np.stack([np.bincount(cell, o["dE_ion"], nc),
                  np.bincount(cell, o["dE_ion"] ** 2, nc)], axis=1)
    return {"counts": None, "sums": s}


def _exact_run(case, seed):
    d, y0, phi0 = _run_inputs(case, seed)
    r = [_trajectory(d, y, p) for y, p in zip(y0, phi0)]
    if any(x is None for x in r):
        return None
    out = {f: np.array([x[f] for x in r]) for f in ("theta_s", "dp", "dE_ion", "t_final", "t_first_bounce",
                                                    "t_last_bounce")}
    out.update({f: None for f in ("n_bounce", "status", "n_steps", "n_rej")})
    if case["y_final"]:
        out["y_final"] = np.stack([x["y"] for x in r], axis=1)
    return out


# Dormand & Prince (1980) 5(4)
A = [[], [1 / 5], [3 / 40, 9 / 40], [44 / 45, -56 / 15, 32 / 9],
     [19372 / 6561, -25360 / 2187, 64448 / 6561, -212 / 729],
     [9017 / 3168, -355 / 33, 46732 / 5247, 49 / 176, -5103 / 18656],
     [35 / 384, 0.0, 500 / 1113, 125 / 192, -2187 / 6784, 11 / 84]]
C = [0.0, 1 / 5, 3 / 10, 4 / 5, 8 / 9, 1.0, 1.0]
EB = [71 / 57600, 0.0, -71 / 16695, 71 / 1920, -17253 / 339200, 22 / 525, -1 / 40]


def _dense(s):
    """Weights of the continuous extension (Shampine 1986) at fraction s."""
    return [s * (1.0 + s * (-183 / 64 + s * (37 / 12 - 145 / 128 * s))), 0.0,
            s * s * (1500 / 371 + s * (-1000 / 159 + s * 1000 / 371)),
            s * s * (-125 / 32 + s * (125 / 12 - s * 375 / 64)),
            s * s * (9477 / 3392 + s * (-729 / 106 + s * 25515 / 6784)),
            s * s * (-11 / 7 + s * (11 / 3 - s * 55 / 28)), s * s * (1.5 + s * (-4.0 + s * 2.5))]


def _trajectory(d, y, phase, most=12000):
    """One trajectory by ode45's rules in textbook form; None when it takes more than `most` attempts, is stopped
    by something other than its exit, or bounces again (each bounce amplifies rounding by about 1e7, so that a
    complex has no value that two 64-bit programs share)."""
    mi, ma, Om = d["m_ion"], d["m_atom"], d["Omega"]
    C4 = 0.5 * d["alpha"]
    C8 = C4 * C4 / (4.0 * d["De"])
    av, qv = np.array(d["a"]), np.array(d["q"])

    def trap(t):
        return av + 2.0 * d["rf_sign"] * qv * math.cos(Om * t + phase)

    def f(t, w):
        sep = w[6:9] - w[0:3]
        s = 1.0 / (sep @ sep)
        F = (8.0 * C8 * s * s - 4.0 * C4) * s * s * s * sep
        return np.concatenate([w[3:6], -0.25 * Om * Om * trap(t) * w[0:3] - F / mi, w[9:12], F / ma])

    def energy(t, w):
        return 0.5 * mi * (w[3:6] @ w[3:6]) + mi * Om * Om / 8.0 * (trap(t) @ (w[0:3] ** 2))

    def radial(w):
        return (w[6:9] - w[0:3]) @ (w[9:12] - w[3:6])
    atol = np.repeat([d["atol_pos"], d["atol_vel"], d["atol_pos"], d["atol_vel"]], 3)
    y0, t, rtol = y, 0.0, d["rtol"]
    k1 = f(t, y)
    rh = np.max(np.abs(k1) / np.maximum(np.abs(y), atol / rtol)) / (0.8 * rtol ** 0.2)
    h = min(d["h_max"], d["t_max"])
    h = 1.0 / rh if h * rh > 1.0 else h
    failed, attempts, rd, bounces = False, 0, radial(y), []
    while attempts < min(most, d["max_attempts"]) and t < d["t_max"]:
        if not failed:
            h = min(max(min(h, d["h_max"]), 16.0 * np.spacing(t)), d["t_max"] - t)
        attempts += 1
        k = [k1]
        for j in range(1, 7):
            yn = y + h * sum(c * kk for c, kk in zip(A[j], k) if c)
            k.append(f(t + C[j] * h, yn))
        e = np.max(np.abs(h * sum(c * kk for c, kk in zip(EB, k) if c)) /
                   np.maximum(rtol * np.maximum(np.abs(y), np.abs(yn)), atol))
        if e > 1.0:
            h, failed = max(16.0 * np.spacing(t), h * (0.5 if failed else max(0.1, 0.8 * e ** -0.2))), True
            continue
        rn = radial(yn)
        if rd < 0.0 <= rn:
            bounces.append(t + h)
            if len(bounces) > 1:
                return None
        rd = rn
        sep = yn[6:9] - yn[0:3]
        if rn > 0.0 and sep @ sep >= d["r0"] ** 2:
            def at(s):
                return y + h * sum(c * kk for c, kk in zip(_dense(s), k) if c)
            lo, hi = 0.0, 1.0
            for _ in range(60):
                m = 0.5 * (lo + hi)
                z = at(m)
                lo, hi = (m, hi) if np.sum((z[6:9] - z[0:3]) ** 2) < d["r0"] ** 2 else (lo, m)
            z, tf = at(hi), t + hi * h
            v0, vf = y0[9:12], z[9:12]
            return {"theta_s": math.atan2(np.linalg.norm(np.cross(v0, vf)), v0 @ vf),
                    "dp": ma * np.linalg.norm(vf - v0), "dE_ion": energy(tf, z) - energy(0.0, y0), "t_final": tf,
                    "t_first_bounce": bounces[0] if bounces else 0.0,
                    "t_last_bounce": bounces[-1] if bounces else 0.0, "y": z}
        y, t, k1 = yn, t + h, k[6]
        h = h * min(5.0, 0.8 * max(e, 1e-300) ** -0.2) if not failed else h
        failed = False
    return None
