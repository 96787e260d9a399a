"""A history's result depends on its id alone: not on how many warps run a
phase, how many particles a warp holds, or which particles share its stack in
shared memory.  The same histories under several launch shapes."""
import numpy as np
import pytest

from paper_1107_3355_gb300 import gdpm as G
from paper_1107_3355_gb300 import workloads as W

pytestmark = pytest.mark.gpu

KEYS = ["n_primary", "ph_created", "ph_terminated", "ph_flights", "ph_real", "compton", "photoelectric",
        "pair", "el_created", "el_terminated", "el_steps", "moller", "brems", "annihilations",
        "local_deposits", "crossings"]


def problem(kind, n):
    if kind == "compton":                       # 1 MeV photons in water
        return W.tiny_problem(n, n_batches=2)
    ph = W.slab_phantom((17, 23, 40), (0.5, 0.5, 0.5))
    if kind == "photoelectric":                 # 60 keV photons, Sauter angles, electrons followed to 20 keV
        return W.Problem(ph, W.pencil_source(ph, 0.06), n, 2, eabs_photon=0.01, eabs_electron=0.02,
                         e_min=0.005, e_max=0.1, flags=W.FLAG_SAUTER)
    if kind == "pair":                          # 15 MeV photons: pairs, positrons, annihilation photons
        return W.Problem(ph, W.pencil_source(ph, 15.0), n, 2, eabs_photon=0.05, eabs_electron=0.2,
                         e_min=0.005, e_max=16.0)
    return W.Problem(ph, W.pencil_source(ph, 12.0, W.ELECTRON), n, 2, eabs_photon=0.05, eabs_electron=0.2,
                     e_min=0.005, e_max=16.0)


# fewer particles than warps, about a warp's worth, more than one per lane of
# the narrow shapes; shapes down to two warps on the whole GPU
@pytest.mark.parametrize("kind", ["compton", "photoelectric", "pair", "electron"])
@pytest.mark.parametrize("n", [2, 33, 4097, 60_000])
def test_results_do_not_depend_on_launch_shape(kind, n):
    prob = problem(kind, n)
    ref = None
    for params in ({}, {G.GDPM_PARAM_BLOCK_THREADS: 64, G.GDPM_PARAM_BLOCKS_PER_SM: 1},
                   {G.GDPM_PARAM_BLOCK_THREADS: 256}, {G.GDPM_PARAM_SOURCE_CHUNK: max(1, n // 3)},
                   {G.GDPM_PARAM_ELECTRON_WALK: 1}, {G.GDPM_PARAM_GRAPH: 1}):
        eng = G.Engine(prob, params=params)
        try:
            d, _, st = eng.run()
            d = d.cpu().numpy()
        finally:
            eng.close()
        events = [st[k] for k in KEYS]
        assert st["ph_created"] == st["ph_terminated"] and st["el_created"] == st["el_terminated"]
        if ref is None:
            ref = d, events
        assert events == ref[1], params
        # the same FP64 deposits in another order
        assert np.all(np.abs(d - ref[0]) <= 1e-11 * ref[0]), params


# A source phase of 9e6 photons fills the wide photon shape; in chunks of half
# of them, every phase runs the narrow one.  A voxel's dose is a sum of up to
# 9e6 positive FP64 deposits, whose order moves it by about sqrt(9e6) half-ulps.
@pytest.mark.parametrize("kind", ["compton", "pair"])
def test_wide_and_narrow_photon_phases(kind):
    n = 9_000_000
    prob = problem(kind, n)
    runs = []
    for params in ({G.GDPM_PARAM_SOURCE_CHUNK: n}, {G.GDPM_PARAM_SOURCE_CHUNK: n // 2}):
        eng = G.Engine(prob, params=params)
        try:
            d, _, st = eng.run()
            runs.append((d.cpu().numpy(), [st[k] for k in KEYS]))
        finally:
            eng.close()
    assert runs[0][1] == runs[1][1]
    assert np.all(np.abs(runs[0][0] - runs[1][0]) <= 1e-11 * runs[0][0])


# Sources in CTAs of 1024 threads, one per SM, from 1024 primaries per SM on;
# in chunks of 50 000 always in CTAs of 256.  Seven batches leave long and
# short ones, and chunks start inside them; half of the field misses the
# phantom.  The same deposits in another order.
@pytest.mark.parametrize("n", [1024 * 152 - 1, 1024 * 152, 200_003])
def test_source_launch_shapes(n):
    ph = W.slab_phantom((17, 23, 40), (0.5, 0.5, 0.5))
    prob = W.Problem(ph, W.field_source(ph, W.kramers_spectrum(), ssd=30.0, field=(14.0, 14.0)), n, 7,
                     eabs_photon=0.05, eabs_electron=0.2, e_min=0.005, e_max=7.0)
    runs = []
    for chunk in (n, 50_000):
        eng = G.Engine(prob, params={G.GDPM_PARAM_SOURCE_CHUNK: chunk})
        try:
            d, s, st = eng.run()
            runs.append((d.cpu().numpy(), s.cpu().numpy(), [st[k] for k in KEYS]))
        finally:
            eng.close()
    assert runs[0][2] == runs[1][2]
    for a, b in zip(runs[0][:2], runs[1][:2]):
        # sigma takes a difference of sums: 1e-11 of its voxel's dose
        assert np.all(np.abs(a - b) <= 1e-11 * runs[0][0])
