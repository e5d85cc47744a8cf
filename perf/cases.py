"""Measured cases of the transport library: what its users have it do.

A pass is one use of the public entry points on a context that the program
keeps: submit events, step until no track is left, read every event's scores;
or one replayed request stream (`Context.serve`).  The range covers both
precisions, every geometry (slab, layered calorimeter with and without a
field, cylinder shells), every step schedule and loop driver, the physics
options, track selection, device and host inputs and outputs, and one to ten
thousand events per call.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2203_09467_gb300 import emt
from paper_2203_09467_gb300 import workloads as W

ELECTRON_MASS = 0.51099895  # MeV
ALL_OPTIONS = 63 | 64 | 128 | 256  # six processes, multiple scattering, angles, Rayleigh

# geometry: setup, FP64 flops of one track-step (add, sub, mul, div and sqrt
# one each, a fused multiply-add two; counted in the scalar form of the
# method) and track-steps per MeV of primary energy (cut 1 MeV)
GEOMETRY = {
    "slab": (W.slab_setup, 59.1, 0.74),
    "calo": (W.calo_setup, 43.1, 2.35),
    "calo_field": (W.calo_field_setup, 968.0, 2.2),
    "cms": (W.cms_setup, 73.5, 0.80),
}


def listed():
    batch = dict(host=False, options=False, select=False, requests_per_s=0, graph_steps=24, block=256)
    return [
        # one 10 GeV electron at a time, for the latency of a single event
        dict(batch, name="event_fp64_persistent", geometry="calo", events=1, primaries=1, e_min=1e4, e_max=1e4,
             precision="fp64", schedule="fused", loop="persistent", graph_steps=256, block=0, slots=1 << 22),
        # a few dozen events through host arrays on a context with the default
        # schedule and driver, as in a first script or a smoke test
        dict(batch, name="few_fp64_default", geometry="calo", events=37, primaries=1, e_min=1e4, e_max=1e4,
             precision="fp64", schedule="fused", loop="plain", graph_steps=12, block=0, slots=1 << 20, host=True),
        # 1,000 x 100 MeV electrons into a lead slab: short showers, few steps
        dict(batch, name="slab_fp64_fused", geometry="slab", events=1000, primaries=1, e_min=100.0, e_max=100.0,
             precision="fp64", schedule="fused", loop="graph", slots=1 << 22),
        # the sampling calorimeter's full batch in both precisions: the headline workload
        dict(batch, name="calo_fp64_pipelined", geometry="calo", events=10000, primaries=1, e_min=1e4, e_max=1e4,
             precision="fp64", schedule="pipelined", loop="graph", slots=1 << 25),
        dict(batch, name="calo_mixed_split", geometry="calo", events=10000, primaries=1, e_min=1e4, e_max=1e4,
             precision="mixed", schedule="split", loop="graph", block=128, slots=1 << 25),
        # every physics option on (multiple scattering, angular distributions,
        # Rayleigh scattering), an odd number of events of mixed primaries
        dict(batch, name="options_fp64_split", geometry="calo", events=777, primaries=1, e_min=1e3, e_max=1e5,
             precision="fp64", schedule="split", loop="graph", graph_steps=12, slots=3000001, options=True),
        # the calorimeter in 2 T (RK4 propagation), e-/e+/gamma of 1-100 GeV
        dict(batch, name="field_fp64_split", geometry="calo_field", events=4000, primaries=1, e_min=1e3, e_max=1e5,
             precision="fp64", schedule="split", loop="graph", slots=1 << 25),
        dict(batch, name="field_mixed_split", geometry="calo_field", events=10000, primaries=1, e_min=1e3, e_max=1e5,
             precision="mixed", schedule="split", loop="graph", slots=1 << 25),
        # uneven events whose showers outgrow a 2^20-slot store: interactions
        # waiting for a slot (FP64), lowest energies first (mixed precision)
        dict(batch, name="batched_fp64_pipelined", geometry="calo_field", events=256, primaries=64, e_min=1e2,
             e_max=1e5, precision="fp64", schedule="pipelined", loop="graph", block=128, slots=1 << 20),
        dict(batch, name="batched_mixed_select", geometry="calo_field", events=256, primaries=64, e_min=1e2,
             e_max=1e5, precision="mixed", schedule="split", loop="graph", slots=1 << 20, select=True),
        # 100 events of 1,000 isotropic 1 GeV photons in six cylinder shells
        dict(batch, name="shells_fp64_split", geometry="cms", events=100, primaries=1000, e_min=1e3, e_max=1e3,
             precision="fp64", schedule="split", loop="graph", graph_steps=12, slots=1 << 25),
        # requests arriving faster than they are finished, admitted into the
        # running step loop (continuous batching)
        dict(batch, name="served_mixed", geometry="calo_field", events=64, primaries=100, e_min=1e3, e_max=5e4,
             precision="mixed", schedule="split", loop="graph", graph_steps=6, block=0, slots=1 << 22, host=True,
             requests_per_s=1000),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    geometry = rng.choice(["slab", "calo", "calo", "calo_field", "calo_field", "cms"])
    precision = rng.choice(["fp64", "mixed"])
    schedule = rng.choice(["fused", "split", "pipelined"])
    loop = rng.choice(["plain", "graph", "graph", "persistent"])
    if loop == "persistent":
        schedule = "fused"
    options = rng.random() < 0.15
    primaries, e_min, e_max = 1, 1e3, 1e5
    if geometry == "slab":
        e_min = e_max = round(_log_uniform(rng, 30.0, 1000.0), 3)
    elif geometry == "cms":
        primaries = int(_log_uniform(rng, 20, 1000))
        e_min = e_max = round(_log_uniform(rng, 300.0, 3000.0), 2)
    elif rng.random() < 0.5:
        e_min = e_max = round(_log_uniform(rng, 1e3, 5e4), 1)
    else:
        primaries = rng.randint(1, 64)
        e_min = 1e2
    case = {"geometry": geometry, "events": 1, "primaries": primaries, "e_min": e_min, "e_max": e_max,
            "precision": precision, "schedule": schedule, "loop": loop, "graph_steps": rng.choice([6, 12, 24]),
            "block": rng.choice([0, 128, 256]), "slots": int(_log_uniform(rng, 1 << 19, 1 << 24)),
            "host": rng.random() < 0.3, "options": options, "requests_per_s": 0,
            "select": schedule == "split" and rng.random() < 0.2}
    # total primary energy: from one event up to a bound that keeps the pass
    # well below the largest listed one (fields and the fused step cost more)
    # and the showers within a few times the track store
    most = {"slab": 1e6, "calo": 6e7, "calo_field": 1.5e7, "cms": 6e7}[geometry]
    if precision == "mixed":
        most *= 2
    if loop != "graph" or schedule == "fused" or options:
        most /= 4
    if case["select"]:
        most /= 2
    most = min(most, 100.0 * case["slots"])
    one = _mean_energy(case)
    case["events"] = max(1, int(_log_uniform(rng, 1.0, max(2.0, min(1e4, most / one)))))
    return case


def _is_mix(case):
    """Primaries e-/e+/gamma of log-uniform energy, rather than a fixed one."""
    return case["e_max"] > case["e_min"]


def _mean_energy(case):
    """Mean primary energy of one event (MeV)."""
    lo, hi = case["e_min"], case["e_max"]
    mean = (hi - lo) / math.log(hi / lo) if hi > lo else lo
    return mean * (case["primaries"] if not _is_mix(case) else 0.5 * (case["primaries"] + 1))


def _primaries(case, seed):
    n = case["events"]
    if case["geometry"] == "slab":
        return W.slab_primaries(n, energy=case["e_min"])
    if case["geometry"] == "cms":
        return W.cms_primaries(n, case["primaries"], energy=case["e_min"], seed=seed)
    if _is_mix(case):
        return W.multi_primaries(n, 1, case["primaries"], case["e_min"], case["e_max"] / case["e_min"], seed=seed)
    return W.calo_primaries(n, energy=case["e_min"], seed=seed)


def prepare(case, seed):
    setup = GEOMETRY[case["geometry"]][0](seed=seed, mask=ALL_OPTIONS if case["options"] else 63)
    prim = _primaries(case, seed)
    n = case["events"]
    more = {"max_active": 3 * case["slots"] // 4, "select": "low_energy"} if case["select"] else {}
    ctx = emt.context_for(setup, precision=case["precision"], schedule=case["schedule"], loop_mode=case["loop"],
                          graph_steps=case["graph_steps"], block_size=case["block"], slot_capacity=case["slots"],
                          max_events=4096 if case["requests_per_s"] else n, **more)
    ids = np.arange(n, dtype=np.uint64) + np.uint64(seed)
    state = {"ctx": ctx, "ids": ids, "prim": prim, "hist": None, "summary": None}
    if case["requests_per_s"]:
        rng = np.random.default_rng(seed)
        state["arrival"] = np.cumsum(rng.exponential(1.0 / case["requests_per_s"], n))
    elif not case["host"]:
        state["prim"] = {k: torch.as_tensor(v).to(ctx.device) for k, v in prim.items()}
        state["hist"] = torch.empty((n, setup.n_bins), dtype=torch.float64, device=ctx.device)
        state["summary"] = torch.empty((n, 6), dtype=torch.float64, device=ctx.device)
    return state


def run(state):
    ctx, out = state["ctx"], {}
    if "arrival" in state:
        _, _, hist, summary = ctx.serve(state["ids"], state["arrival"], state["prim"], mode="continuous",
                                        steps_per_poll=6)
    else:
        ctx.submit(state["ids"], state["prim"])
        out["track_steps"] = ctx.run()["track_steps"]
        hist, summary, _ = ctx.read_all(state["hist"], state["summary"])
    out["hist"] = hist
    for k, field in enumerate(emt.SUMMARY_FIELDS):
        out[field] = summary[:, k]
    return out


def work(case):
    """Primaries read and scores written once; the method's floating-point
    operations on the expected number of track-steps."""
    _, flops, steps_per_mev = GEOMETRY[case["geometry"]]
    n = case["events"]
    n_prim = n * (0.5 * (case["primaries"] + 1) if _is_mix(case) else case["primaries"])
    bins = {"slab": 1, "calo": 100, "calo_field": 100, "cms": 140}[case["geometry"]]
    return {"bytes": 64.0 * n_prim + 8.0 * n * (bins + 6),
            "flops": flops * steps_per_mev * n * _mean_energy(case)}


def exact(case, seed):
    """The energy that entered with each event's primaries; a shower's scores
    have no closed form."""
    prim = _primaries(case, seed)
    rest = np.where(prim["type"] == W.POSITRON, 2.0 * ELECTRON_MASS, 0.0)
    e_in = np.bincount(prim["event"], weights=prim["T"] + rest, minlength=case["events"])
    out = {field: None for field in ("hist",) + emt.SUMMARY_FIELDS}
    out["e_in"] = e_in
    return out
