"""Electron phases beside the largest tables a context accepts: as fast as
beside the usual ones, and the same events in every launch shape."""
import dataclasses

import pytest

from paper_1107_3355_gb300 import gdpm as G
from paper_1107_3355_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

KEYS = ("el_created", "el_steps", "moller", "brems", "crossings", "local_deposits", "ph_flights")


def problem(n_mat, n_energy):
    prob = W.slab_electron_problem(n_histories=300_000, n_batches=10)
    mats = (list(prob.phantom.materials) * n_mat)[:n_mat]
    return prob.with_(phantom=dataclasses.replace(prob.phantom, materials=mats), n_energy=n_energy)


def electron_ms(prob):
    eng = G.Engine(prob, params={G.GDPM_PARAM_PROFILE: 1})
    try:
        return min(eng.run()[2]["kernel_ms"][1] for _ in range(8))
    finally:
        eng.close()


# The phases are bound by the instructions they issue and the latency of a
# warp's round, both the same whatever the tables; half as much again leaves
# room for tables that miss the L1 more often.  With 4 warps an SM instead of
# 24 they took twice as long.
@pytest.mark.parametrize("n_mat,n_energy", [(8, 512), (4, 1100), (4, 1500), (4, 2048), (8, 1024)])
def test_electron_phases_keep_their_speed(n_mat, n_energy):
    assert electron_ms(problem(n_mat, n_energy)) < 1.5 * electron_ms(problem(4, 512))


# 18 staged warps beside 8 x 512 and 17 beside 4 x 1100, where the step and
# event table moves to global memory; blocks of 256 and 64 threads stage it
# beside 4 x 1100 and, of 64, beside the largest
@pytest.mark.parametrize("n_mat,n_energy", [(8, 512), (4, 1100), (4, 2048), (8, 1024)])
def test_events_do_not_depend_on_launch_shape(n_mat, n_energy):
    prob = problem(n_mat, n_energy)
    runs = []
    for params in ({}, {G.GDPM_PARAM_BLOCK_THREADS: 64, G.GDPM_PARAM_BLOCKS_PER_SM: 1}, {G.GDPM_PARAM_BLOCK_THREADS: 256},
                   {G.GDPM_PARAM_TALLY_MODE: 1}, {G.GDPM_PARAM_GRAPH: 1}):
        eng = G.Engine(prob, params=params)
        try:
            st = eng.run()[2]
            runs.append([st[k] for k in KEYS])
        finally:
            eng.close()
    assert all(r == runs[0] for r in runs)
