"""Dose calculations whose speed is tracked, through the package's public calls.

A case is a kind of calculation (phantom, source, options) with its number of
histories and batches.  ``listed()`` holds one of each kind that a planning
system or a research user runs, at the size it is run at; ``draw()`` gives
more of the same kinds over the whole range of sizes, odd ones included.

``prepare`` makes what such a program holds before the call (the context, the
phantom on the device, the cross-section tables and the source), ``run`` is
one calculation with dose, sigma, event counts and the energy ledger.
"""
import functools
import math

import numpy as np
import torch

from paper_1107_3355_gb300 import gdpm as G
from paper_1107_3355_gb300 import workloads as W

# Nominal FP32 operations per source history of each kind of calculation: its
# mean numbers of Woodcock flights (30 operations each), Klein-Nishina events
# (60) and condensed-history electron steps (100).
FLOPS_PER_HISTORY = {
    "pencil_photon": 30 * 10 + 60 * 4.5 + 100 * 2.4,
    "water_electron": 100 * 30,
    "ct": 30 * 10.2 + 60 * 2.7 + 100 * 6.3,
    "slab_photon": 30 * 8.5 + 60 * 3 + 100 * 6.2,
    "slab_electron": 100 * 39.6,
    "matrix": 30 * 8.5 + 60 * 3 + 100 * 6.2,
}

STAT_KEYS = ["n_primary", "ph_created", "ph_terminated", "ph_flights", "ph_real", "compton",
             "photoelectric", "pair", "el_created", "el_terminated", "el_steps", "moller", "brems",
             "annihilations", "local_deposits", "crossings"]
LEDGER_KEYS = ["source_energy", "deposited", "escaped", "discarded"]


def _case(name, kind, plan, histories, batches, shape, tally="fp64"):
    c = {"kind": kind, "plan": plan, "histories": int(histories), "batches": int(batches),
         "nx": shape[0], "ny": shape[1], "nz": shape[2], "tally": tally}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest useful call: a quick look at a 1 MeV pencil in water
        # (the smoke check's problem); launches and host checks count here
        _case("water32_pencil_1e4", "pencil_photon", "pencil", 10_000, 10, (32, 32, 32)),
        # one beamlet of a plan on the patient phantom: the small request of a
        # dose server, thousands of them per plan
        _case("ct_beamlet_1e5", "ct", "beamlet", 100_000, 10, (256, 256, 128)),
        # one fluence-map field of a plan: the middling request of a server
        _case("ct_beam_1e7", "ct", "beam", 10_000_000, 10, (256, 256, 128)),
        # a VMAT arc (180 apertures) whose beamlets are sampled by Metropolis
        _case("ct_arc_metropolis_2e7", "ct", "arc_metropolis", 20_000_000, 10, (256, 256, 128)),
        # the whole 7-field plan with 100 batches: a final dose calculation
        _case("ct_imrt7_1e8", "ct", "imrt7", 100_000_000, 100, (256, 256, 128)),
        # the paper's Sec. 3.1 photon case on its own grid (odd sizes)
        _case("paper_slab_6MV_lung_2.5e8", "slab_photon", "paper_lung", 250_000_000, 10, (61, 61, 150)),
        # the paper's Sec. 3.1 electron case
        _case("paper_slab_e20_bone_2.5e6", "slab_electron", "paper_bone", 2_500_000, 10, (61, 61, 150)),
        # a clinical electron field on the 128^3 slab
        _case("slab128_e20_1e6", "slab_electron", "field", 1_000_000, 100, (128, 128, 128)),
        # a photon field on the 128^3 slab, and the same kind of run with the
        # FP32 compensated tally
        _case("slab128_6MV_1e6", "slab_photon", "field", 1_000_000, 100, (128, 128, 128)),
        _case("slab128_6MV_fp32pair_1e7", "slab_photon", "field", 10_000_000, 20, (128, 128, 128),
              "fp32pair"),
        # the paper's Sec. 4 comparison: 15 MeV electrons in water
        _case("water64_e15_1e6", "water_electron", "pencil", 1_000_000, 10, (64, 64, 64)),
        # a beamlet dose matrix for optimisation: 64 beamlets in one call
        _case("slab128_matrix64", "matrix", "matrix64", 16_000_000, 2, (128, 128, 128)),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["pencil_photon", "water_electron", "ct", "ct", "slab_photon", "slab_photon",
                       "slab_electron", "matrix"])
    if kind == "pencil_photon":
        n = rng.randint(20, 64)
        return _case(None, kind, "pencil", log(1e4, 1e7), rng.randint(5, 100), (n, n, n))
    if kind == "water_electron":
        n = rng.randint(31, 80)
        return _case(None, kind, "pencil", log(1e4, 3e6), rng.randint(5, 40), (n, n, n))
    if kind == "ct":
        plan = rng.choice(["beamlet", "beam", "beam_alias", "arc", "arc_metropolis", "imrt7"])
        lo, hi = {"beamlet": (3e4, 1e6), "imrt7": (1e6, 5e7)}.get(plan, (1e6, 3e7))
        shape = rng.choice([(256, 256, 128), (167, 151, 75)])
        return _case(None, kind, plan, log(lo, hi), rng.randint(5, 50), shape)
    if kind == "slab_photon":
        plan = rng.choice(["paper_lung", "paper_bone", "field"])
        shape = (61, 61, 150) if plan != "field" else tuple(rng.randint(60, 150) for _ in range(3))
        return _case(None, kind, plan, log(1e5, 8e7), rng.randint(5, 60), shape,
                     rng.choice(["fp64", "fp64", "fp32pair"]))
    if kind == "slab_electron":
        plan = rng.choice(["paper_lung", "paper_bone", "field"])
        shape = (61, 61, 150) if plan != "field" else tuple(rng.randint(60, 150) for _ in range(3))
        return _case(None, kind, plan, log(3e4, 4e6), rng.randint(5, 40), shape)
    k = rng.randint(5, 80)
    return _case(None, kind, "matrix%d" % k, k * log(2e4, 4e5), rng.randint(2, 3),
                 tuple(rng.randint(60, 128) for _ in range(3)))


@functools.lru_cache(maxsize=2)
def _ct(shape):
    return W.ct_phantom(shape)


def _problem(case, seed):
    """The Problem of a case; fluence maps, apertures and beamlets from the seed."""
    n, nb, shape = case["histories"], case["batches"], (case["nx"], case["ny"], case["nz"])
    kind, plan = case["kind"], case["plan"]
    rng = np.random.default_rng(seed)
    if kind == "pencil_photon":
        ph = W.homogeneous_phantom(shape, (0.5, 0.5, 0.5), W.WATER, 1.0)
        prob = W.tiny_problem(n, n_batches=nb).with_(phantom=ph, source=W.pencil_source(ph, 1.0))
    elif kind == "water_electron":
        ph = W.homogeneous_phantom(shape, (0.5, 0.5, 0.5), W.WATER, 1.0)
        prob = W.water64_problem(W.ELECTRON, n, nb).with_(phantom=ph,
                                                         source=W.pencil_source(ph, 15.0, W.ELECTRON))
    elif kind == "ct":
        ph = _ct(shape)
        angle = float(rng.uniform(0, 360))
        if plan == "beamlet":
            u, v = rng.uniform(-5, 4, 2)
            src = W.single_beamlet(ph, angle, float(u), float(v), 1.0)
        elif plan in ("beam", "beam_alias"):
            fr = W.beam_frame(angle, tuple(e / 2 for e in ph.extent))
            src = W.beamlet_source(W.fluence_map_rows(fr, rng.uniform(0, 1, (20, 20))), W.kramers_spectrum())
        elif plan in ("arc", "arc_metropolis"):
            src = W.vmat_arc(ph, seed=seed)
        else:
            src = W.imrt_plan(ph, seed=seed)
        src.sampler = {"beam_alias": "alias", "arc_metropolis": "metropolis"}.get(plan, "cdf")
        prob = W.Problem(ph, src, n, nb, eabs_photon=0.05, eabs_electron=0.2, e_min=0.005, e_max=6.5)
    elif kind in ("slab_photon", "slab_electron"):
        particle = W.PHOTON if kind == "slab_photon" else W.ELECTRON
        if plan.startswith("paper_"):
            prob = W.paper_slab_problem(plan[6:], particle, n, nb)
        elif particle == W.PHOTON:
            prob = W.slab_photon_problem(n, n_batches=nb, shape=shape)
        else:
            prob = W.slab_electron_problem(n, n_batches=nb, shape=shape)
    else:
        # one row per beamlet, every beamlet with its own number of histories
        k = int(plan[6:])
        prob = W.beamlet_matrix_problem(k, seed=seed, n_batches=nb, shape=shape)
        share = rng.lognormal(0.0, 1.0, k)
        sub = np.maximum(2000, np.floor(n * share / share.sum())).astype(np.int64)
        prob = prob.with_(sub_histories=tuple(int(v) for v in sub), n_histories=int(sub.sum()))
    return prob.with_(seed=seed)


class _State:
    """A user's handles: the engine (context, phantom, tables, source) and its outputs."""

    def __init__(self, case, seed):
        prob = _problem(case, seed)
        params = {G.GDPM_PARAM_TALLY_MODE: 1} if case["tally"] == "fp32pair" else None
        self.engine = G.Engine(prob, params=params)
        self.rows = prob.sub_histories
        n = prob.phantom.n_voxels
        size = (len(self.rows), n) if self.rows else (n,)
        self.dose = torch.empty(size, dtype=torch.float64, device="cuda")
        self.sigma = torch.empty(size, dtype=torch.float64, device="cuda")


def prepare(case, seed):
    return _State(case, seed)


def run(state):
    e = state.engine
    if state.rows:
        st = G.gdpm_simulate_beamlets(e.ctx, e.phantom, e.tables, state.rows, e.prob.n_batches,
                                      state.dose, state.sigma)
    else:
        st = e.run(dose=state.dose, sigma=state.sigma)[2]
    return {"dose": state.dose, "sigma": state.sigma,
            "events": np.array([st[k] for k in STAT_KEYS], np.int64),
            "ledger": np.array([st[k] for k in LEDGER_KEYS], np.float64),
            "source_energy": float(st["source_energy"])}


def work(case):
    voxels = case["nx"] * case["ny"] * case["nz"]
    grids = int(case["plan"][6:]) if case["kind"] == "matrix" else 1
    # densities and materials read once; dose and sigma written once
    return {"bytes": 5 * voxels + 16 * voxels * grids,
            "flops": FLOPS_PER_HISTORY[case["kind"]] * case["histories"]}


def exact(case, seed):
    """Random histories have no closed form; the energy a monoenergetic source emits has one."""
    energy = {("pencil_photon", "pencil"): 1.0, ("water_electron", "pencil"): 15.0}.get(
        (case["kind"], case["plan"]), 20.0 if case["kind"] == "slab_electron" else None)
    if energy is None:
        return None
    return {"dose": None, "sigma": None, "events": None, "ledger": None,
            "source_energy": energy * case["histories"]}
