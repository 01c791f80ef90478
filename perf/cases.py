"""The work a user has this framework do, as cases that can be timed and compared.

Three kinds of call, all through the public entry points:

  fields   pic_field_solve_static: charge deposit, Poisson solve and field from particle
           arrays that the caller owns;
  advance  Simulation.step over a stretch of an RF cycle, then what a run reads afterwards:
           the diagnostics of every discharge (the window is reset, as after each averaging
           window) and the fields of the first;
  restart  a particle state from host arrays (a checkpoint, or a host code's particles) put
           into a simulation, some steps, and the state read back.

Sizes and options are those of `inputs.py` (cfg1 .. cfg4, the 64-discharge grid, the 13.8 Pa
voltage sweep), of the tests and of the benchmark's variants.
"""
import ctypes
import math

import numpy as np
import torch

from paper_0705_0495_gb300 import inputs, o2pic

QE = 1.602176634e-19
EPS0 = 8.8541878128e-12


def _advance(name, **kw):
    """an advance case: one discharge of cfg1's geometry unless told otherwise"""
    c = dict(kind="advance", plan="single", n_cells=128, L=0.025, p_Pa=20.0, U_rf=100.0, steps_per_cycle=1000,
             n0_m3=1e15, n_op=20000, fp64=False, n1=10, n2=0, inter=False, gas_scheme=0, ion_subcycle=1,
             sort_interval=10, capacity_factor=16.0, warm=200, steps=100)
    c.update(kw)
    if name:
        c["name"] = name
    return c


CFG2 = dict(n_cells=512, L=0.04, p_Pa=10.0, U_rf=300.0, steps_per_cycle=3000, n0_m3=1e16, n_op=2_000_000,
            capacity_factor=2.0)
CFG4 = dict(n_cells=4096, L=0.04, p_Pa=20.0, U_rf=400.0, steps_per_cycle=4000, n0_m3=1e16, n_op=25_000_000,
            capacity_factor=1.25)


def listed():
    return [
        # a host framework that owns every allocation asks for the field of a small FP64 discharge
        # (cfg1's 40 thousand particles in no order): the smallest call, where launches count
        dict(name="fields-fp64-cfg1", kind="fields", n_cells=128, n_op=20000, fp64=True, ordered=False),
        # the same call on a large discharge (cfg4's 5e7 particles, ten steps after a cell sort)
        dict(name="fields-fp32-cfg4", kind="fields", n_cells=4096, n_op=25_000_000, fp64=False, ordered=True),
        # a host loop that steps a small discharge once at a time and looks at the fields after each
        # step (a probe, a coupled external circuit): launch and synchronisation latency
        _advance("probe-cfg1", steps=1),
        # a stretch of the plain FP64 reference discharge, the precision of the step-by-step checks
        _advance("cfg1-fp64", fp64=True, warm=100, steps=100),
        # the 13.8 Pa voltage sweep of the paper's Sec. IV: seven small discharges in one handle, Coulomb
        # collisions every ten steps, one RF cycle: the everyday production run
        _advance("volts-cycle", plan="volts", L=0.025, p_Pa=13.8, n2=10, steps=1000),
        # one RF cycle of a middle-sized discharge (cfg2: 4e6 superparticles), diagnostics read per cycle
        _advance("cfg2-cycle", **CFG2, steps=3000),
        # 64 discharges of uneven size in one handle (a parameter study: voltage x pressure x gap)
        _advance("grid64", plan="grid", n_op=15_000_000, steps_per_cycle=2000, n0_m3=1e16, capacity_factor=1.5,
                 warm=20, steps=100),
        # the large discharge of the headline benchmark (cfg4: 5e7 superparticles, 4096 cells)
        _advance("cfg4", **CFG4, warm=100, steps=400),
        # the same in FP64, for runs that are checked step by step
        _advance("cfg4-fp64", **CFG4, fp64=True, warm=20, steps=40),
        # intra- and inter-species Coulomb collisions every ten steps on cfg2
        _advance("cfg2-coulomb-inter", **CFG2, n2=10, inter=True, warm=100, steps=200),
        # the paper's own sequential gas-channel scheme on cfg2
        _advance("cfg2-sequential", **CFG2, gas_scheme=1, warm=100, steps=200),
        # a restart from host arrays with sub-cycled ions on a ragged grid: state in, one schedule of
        # steps, state out (coupling to a host code, checkpoints)
        dict(_advance("restart-ragged", **dict(CFG2, n_cells=501, n_op=499_999), ion_subcycle=5, warm=100, steps=100),
             kind="restart"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    k = rng.random()
    if k < 0.2:
        return dict(kind="fields", n_cells=_log_int(rng, 16, 4096), n_op=_log_int(rng, 2000, 25_000_000),
                    fp64=rng.random() < 0.5, ordered=rng.random() < 0.5)
    if k < 0.3:
        return _advance(None, plan="volts", L=0.025, p_Pa=13.8, n2=10, n_op=_log_int(rng, 5000, 60000),
                        fp64=rng.random() < 0.2, steps=100 * rng.randint(1, 5))
    if k < 0.4:
        return _advance(None, plan="grid", n_op=_log_int(rng, 1_000_000, 15_000_000), steps_per_cycle=2000,
                        n0_m3=1e16, capacity_factor=1.5, warm=20, steps=10 * rng.randint(2, 8) + rng.randint(0, 1))
    n_cells = _log_int(rng, 64, 4096)
    n_op = _log_int(rng, 20000, 25_000_000)
    c = _advance(None, n_cells=n_cells, n_op=n_op, L=round(rng.uniform(0.025, 0.04), 4),
                 p_Pa=round(rng.uniform(5.0, 50.0), 2), U_rf=round(rng.uniform(75.0, 500.0), 1),
                 steps_per_cycle=1000 if n_cells < 256 else (3000 if n_cells < 1024 else 4000),
                 n0_m3=1e15 if n_cells < 256 else 1e16,
                 capacity_factor=24.0 if n_op < 200_000 else (8.0 if n_op < 2_000_000 else 2.0),
                 fp64=rng.random() < 0.3, warm=20, sort_interval=rng.choice((5, 10, 20)), n1=rng.choice((10, 20)))
    option = rng.random()
    if option < 0.25:
        c["n2"] = 10
        # Inter-species chains grow with the particles of a cell: kept to the sizes such runs have.
        c["inter"] = n_op <= 2_000_000 and n_op <= 4000 * n_cells and rng.random() < 0.5
    elif option < 0.4:
        c["gas_scheme"] = 1
    elif option < 0.55:
        c["ion_subcycle"] = rng.choice((2, 5))
    cost = 4e9 / n_op / (8.0 if c["fp64"] else 1.0) / (4.0 if c["n2"] or c["gas_scheme"] else 1.0)
    c["steps"] = max(1, min(150 if c["fp64"] else 1000, int(rng.uniform(0.3, 1.0) * cost)))
    if rng.random() < 0.15 and n_op <= 1_000_000:
        c["kind"] = "restart"
        c["steps"] = min(c["steps"], 100)
    return c


# ------------------------------------------------------------------ particles of a fields call

MOVED = (1.5, 0.02, 0.02)  # rms cells that a species has moved since the last sort


def _particles(case, seed):
    """(cell, offset) of the three species on the GPU, as a simulation holds them: the electrons leave the
    sheaths, a few slots are dead; ordered by cell up to the moves since the last sort, or in no order"""
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    N = case["n_cells"]
    n_op = case["n_op"]
    cells, offs = [], []
    for s, n in enumerate((n_op // 2, n_op - n_op // 2, n_op)):
        x = torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
        if case["ordered"]:
            x += torch.arange(n, device="cuda", dtype=torch.float64)
            x /= max(n, 1)
        if s == 0:
            x = 0.05 + 0.9 * x
        x *= N
        if case["ordered"]:
            x += MOVED[s] * torch.randn(n, generator=g, device="cuda", dtype=torch.float32)
        c = torch.floor(x)
        off = (x - c).to(torch.float64 if case["fp64"] else torch.float32)
        dead = (c < 0) | (c >= N) | (torch.rand(n, generator=g, device="cuda") < 1e-3)
        cells.append(torch.where(dead, -1.0, c).to(torch.int32))
        offs.append(off)
    return cells, offs


def _fields_discharge(case):
    return inputs.Discharge(L=0.04, n_cells=case["n_cells"], U_rf=300.0, n0_m3=1e16, n_op=case["n_op"],
                            fp64=case["fp64"])


def _fields_step(seed):
    return int(seed) % 997 + 1  # the time step whose drive voltage is applied


# ------------------------------------------------------------------ discharges of a simulation

def _discharges(case, seed):
    kw = dict(seed=int(seed) + 1, fp64=case["fp64"], n1=case["n1"], sort_interval=case["sort_interval"],
              capacity_factor=case["capacity_factor"], n2=case["n2"], coulomb_inter=case["inter"],
              gas_scheme=case["gas_scheme"], ion_subcycle=case["ion_subcycle"])
    if case["plan"] == "volts":
        return inputs.sweep_13p8(n_op=case["n_op"], **kw)
    if case["plan"] == "grid":
        return inputs.cfg3_sweep(total=2 * case["n_op"], **kw)
    return [inputs.Discharge(L=case["L"], n_cells=case["n_cells"], p_Pa=case["p_Pa"], U_rf=case["U_rf"],
                             steps_per_cycle=case["steps_per_cycle"], n0_m3=case["n0_m3"], n_op=case["n_op"], **kw)]


def prepare(case, seed):
    if case["kind"] == "fields":
        cells, offs = _particles(case, seed)
        out = [torch.empty(case["n_cells"] + 1, dtype=torch.float64, device="cuda") for _ in range(3)]
        return {"case": case, "cfg": o2pic.make_config(_fields_discharge(case)), "cells": cells, "offs": offs,
                "out": out, "step": _fields_step(seed)}
    ds = _discharges(case, seed)
    # The sequential scheme's n1 dt is coarse for fast electrons: such runs accept clamped probabilities.
    sim = o2pic.Simulation(ds, inputs.xs_tables(), numeric_budget=1.0 if case["gas_scheme"] else None)
    sim.step(case["warm"])
    state = {"case": case, "sim": sim}
    if case["kind"] == "restart":
        state["host"] = [sim.get_state(0, s) for s in range(3)]
        # the caller's host arrays that the state comes back into, as long as the species' capacity
        state["back"] = [[np.zeros(cap) for _ in range(4)] + [np.zeros(cap, dtype=np.int32)]
                         for cap in ds[0].capacity]
    return state


def _state_into(sim, s, arrays):
    """pic_get_state of species s into host arrays of the caller"""
    n = ctypes.c_longlong()
    kinds = [ctypes.c_double] * 4 + [ctypes.c_int]
    rc = sim.lib.pic_get_state(sim.h, 0, s, *[a.ctypes.data_as(ctypes.POINTER(k)) for a, k in zip(arrays, kinds)],
                               len(arrays[0]), ctypes.byref(n))
    if rc:
        raise o2pic.PicError(rc, sim.lib.pic_last_error(sim.h).decode())
    return {"n": n.value, "x": arrays[0], "vx": arrays[1], "vy": arrays[2], "vz": arrays[3], "alive": arrays[4]}


READ = ("n_samples", "dens_sum", "phi_sum", "eedf", "iedf", "fm", "absorbed", "events", "violations", "slots",
        "particle_steps", "candidates")


def run(state):
    case = state["case"]
    if case["kind"] == "fields":
        out = state["out"]
        o2pic.field_solve_static(state["cfg"], state["step"], [t.data_ptr() for t in state["cells"]],
                                 [t.data_ptr() for t in state["offs"]], [t.numel() for t in state["cells"]],
                                 out[0].data_ptr(), out[1].data_ptr(), out[2].data_ptr(),
                                 torch.cuda.current_stream().cuda_stream)
        return {"rho": out[0], "phi": out[1], "E": out[2]}
    sim = state["sim"]
    if case["kind"] == "restart":
        for s, h in enumerate(state["host"]):
            sim.set_state(0, s, h["x"], h["vx"], h["vy"], h["vz"], h["alive"])
        sim.set_step(case["warm"])
        sim.step(case["steps"])
        return {"fields": list(sim.fields(0)), "state": [_state_into(sim, s, a) for s, a in enumerate(state["back"])]}
    sim.step(case["steps"])
    if case["steps"] == 1:
        return {"fields": list(sim.fields(0))}
    diags = [sim.diagnostics(k, reset=True) for k in range(len(sim.discharges))]
    return {"fields": list(sim.fields(0)),
            "diagnostics": {k: np.concatenate([np.ravel(g[k]) for g in diags]) for k in READ}}


def work(case):
    real = 8 if case["fp64"] else 4
    n_op = case["n_op"]
    if case["kind"] == "fields":
        return {"bytes": 2.0 * n_op * (4 + real) + 3 * 8.0 * (case["n_cells"] + 1), "flops": 2.0 * n_op * 6}
    # Per particle and step: cell, offset and vx read and written; per sort: every field read and
    # written; per Coulomb pass and sequential-scheme pass: the velocity read and written.
    particles = 2.0 * n_op * (7 if case["plan"] == "volts" else 1)
    steps = case["steps"]
    ions = 0.75 / case["ion_subcycle"]  # three quarters of the load are ions
    moved = particles * (0.25 + ions) * steps
    sorts = steps / min(case["sort_interval"], case["n1"])
    b = moved * 2 * (4 + 2 * real) + particles * sorts * 2 * (4 + 4 * real)
    f = moved * 30
    if case["n2"]:
        passes = steps / case["n2"] * (2 if case["inter"] else 1)
        b += particles * passes * 6 * real
        f += particles * passes * 60
    if case["gas_scheme"]:
        b += particles * steps / case["n1"] * 2 * 6 * real
        f += particles * steps / case["n1"] * 200
    if case["kind"] == "restart":
        b += particles * 2 * (4 * 8 + 4)  # host arrays in and out
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------ the same in plain 64 bits

def exact(case, seed):
    """The field solve in 64 bits.  A simulated stretch has no such value: its collisions are random
    decisions, and what follows from them is one realisation."""
    if case["kind"] != "fields":
        return None
    d = _fields_discharge(case)
    N, dx = d.n_cells, d.L / d.n_cells
    cells, offs = _particles(case, seed)
    rho = np.zeros(N + 1, dtype=np.longdouble)
    for sign, c, o in zip((-1, -1, 1), cells, offs):
        live = c >= 0
        c, o = c[live].long(), o[live].double()
        node = torch.bincount(c, 1.0 - o, minlength=N + 1) + torch.bincount(c + 1, o, minlength=N + 1)
        rho += sign * node.cpu().numpy().astype(np.longdouble)
    volume = np.full(N + 1, dx)
    volume[[0, N]] = 0.5 * dx
    rho *= QE * d.weight / volume
    phi0 = d.U_rf * math.sin(2.0 * math.pi * d.f_rf * (_fields_step(seed) * d.dt) + d.rf_phase)
    # phi_{i+1} - phi_i falls by s_i = rho_i dx^2 / eps0 from one interval to the next
    s = rho[1:N] * dx * dx / EPS0
    s2 = np.cumsum(np.cumsum(s))
    slope = (s2[-1] - phi0) / N
    phi = np.zeros(N + 1, dtype=np.longdouble)
    phi[0] = phi0
    phi[1:N] = phi0 + np.arange(1, N) * slope
    phi[2:N] -= s2[:-1]
    E = np.empty(N + 1, dtype=np.longdouble)
    E[1:N] = -(phi[2:] - phi[:-2]) / (2 * dx)
    E[0] = -(phi[1] - phi[0]) / dx - rho[0] * dx / (2 * EPS0)
    E[N] = -(phi[N] - phi[N - 1]) / dx + rho[N] * dx / (2 * EPS0)
    return {"rho": rho.astype(np.float64), "phi": phi.astype(np.float64), "E": E.astype(np.float64)}
