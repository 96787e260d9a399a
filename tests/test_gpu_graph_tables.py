"""The device-driven phase loop beside tables of any accepted size: its phase
kernels keep their arguments in shared memory too, and the warps' stacks must
leave room for them."""
import pytest

from paper_1107_3355_gb300 import gdpm as G
from paper_1107_3355_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

KEYS = ("n_primary", "compton", "photoelectric", "pair", "el_steps", "moller", "brems", "crossings",
        "ph_flights", "annihilations", "local_deposits")


def problem(n_mat, n_energy):
    import dataclasses
    prob = W.slab_electron_problem(n_histories=3000, n_batches=2, shape=(32, 32, 64))
    mats = (list(prob.phantom.materials) * n_mat)[:n_mat]
    return prob.with_(phantom=dataclasses.replace(prob.phantom, materials=mats), n_energy=n_energy)


# material and energy counts whose electron (4 x 578 to 7 x 544) or photon
# tables leave the last 0 to 144 of the 227 KB beside whole warp stacks, and
# the largest tables
@pytest.mark.parametrize("n_mat,n_energy", [(4, 578), (4, 654), (7, 544), (4, 1776), (8, 1000), (4, 2000), (8, 1024)])
def test_graph_loop_beside_tables(n_mat, n_energy):
    prob = problem(n_mat, n_energy)
    stats = []
    for graph in (0, 1):
        eng = G.Engine(prob, params={G.GDPM_PARAM_GRAPH: graph})
        try:
            stats.append(eng.run()[2])
        finally:
            eng.close()
    for k in KEYS:
        assert stats[0][k] == stats[1][k], k
    assert stats[1]["deposited"] == pytest.approx(stats[0]["deposited"], rel=1e-9)


def test_autotune_beside_tables():
    prob = problem(7, 544)
    eng = G.Engine(prob)
    try:
        r = G.gdpm_autotune(eng.ctx, eng.phantom, eng.tables, prob.n_histories, prob.n_batches, budget_ms=20000.0)
        assert r["histories_per_s"] > 0
    finally:
        eng.close()
