"""The fold of batches side by side where its chunks of 10 batches end, and
the whole-step electron form, against the other route to the same result."""
import numpy as np
import pytest

from paper_1107_3355_gb300 import gdpm as G
from paper_1107_3355_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# (batches, long batches): chunks of the long and of the short batches that
# are whole, one short and one over
@pytest.mark.parametrize("batches,n_big", [(9, 0), (9, 8), (10, 0), (11, 10), (19, 9), (20, 10), (20, 19), (21, 10),
                                           (21, 11)])
@pytest.mark.parametrize("tally", [0, 1])
def test_side_by_side_fold_at_chunk_edges(batches, n_big, tally):
    ph = W.homogeneous_phantom((13, 11, 9), (0.5, 0.5, 0.5), W.WATER, 1.0)
    prob = W.tiny_problem(batches * 900 + n_big, n_batches=batches).with_(phantom=ph, source=W.pencil_source(ph, 1.0))
    out = {}
    for mode in (1, 2):
        eng = G.Engine(prob, params={G.GDPM_PARAM_BATCH_MODE: mode, G.GDPM_PARAM_TALLY_MODE: tally})
        try:
            for _ in range(2):
                d, s, st = eng.run()
            out[mode] = d.cpu().numpy(), s.cpu().numpy(), st
        finally:
            eng.close()
    (d1, s1, a), (d2, s2, b) = out[1], out[2]
    assert a["el_steps"] == b["el_steps"] and (d1 > 0).any()
    # the same FP64 tallies in another order of addition: a few eps per sum;
    # the variance is a difference of sums, off by a few eps of the mean square
    assert np.all(np.abs(d1 - d2) <= 1e-12 * d1)
    assert np.all(np.abs(s1 ** 2 - s2 ** 2) <= 1e-12 * d1 ** 2 + 1e-12 * s1 ** 2)


KEYS = ("n_primary", "ph_flights", "compton", "pair", "el_created", "el_steps", "moller", "brems", "annihilations",
        "local_deposits", "crossings")


@pytest.mark.parametrize("n", [33, 4097, 60_000])
@pytest.mark.parametrize("air", [False, True])
def test_whole_steps_equal_resumable_steps(n, air):
    ph = W.slab_phantom((17, 23, 40), (0.5, 0.5, 0.5))
    if air:
        ph.rho[len(ph.rho) // 3:] = 0.0012      # steps hundreds of voxels long
    prob = W.Problem(ph, W.pencil_source(ph, 12.0, W.ELECTRON), n, 2, eabs_photon=0.05, eabs_electron=0.2, e_min=0.005,
                     e_max=16.0)
    runs = []
    for walk in (0, 1):
        eng = G.Engine(prob, params={G.GDPM_PARAM_ELECTRON_WALK: walk})
        try:
            d, _, st = eng.run()
            runs.append((d.cpu().numpy(), [st[k] for k in KEYS]))
        finally:
            eng.close()
    assert runs[0][1] == runs[1][1]
    # the same FP64 deposits in another order
    assert np.all(np.abs(runs[0][0] - runs[1][0]) <= 1e-11 * runs[0][0])
