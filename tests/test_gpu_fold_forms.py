"""The fold of batches side by side (one kernel from the tally grids to dose
and sigma) against the fold of batches one after another (per-batch sums, then
the finalize kernel), on the same histories."""
import numpy as np
import pytest

from paper_1107_3355_gb300 import gdpm as G
from paper_1107_3355_gb300 import workloads as W

pytestmark = pytest.mark.gpu


# voxel counts below, at and above a CTA's 256, odd ones; batch counts around
# the 16 read at a time; batches of unequal size (histories % batches != 0)
@pytest.mark.parametrize("shape,batches", [((1, 1, 1), 2), ((5, 17, 3), 15), ((16, 16, 1), 16),
                                           ((13, 11, 9), 17), ((31, 7, 40), 33)])
@pytest.mark.parametrize("tally", [0, 1])
def test_side_by_side_fold_equals_sequential(shape, batches, tally):
    ph = W.homogeneous_phantom(shape, (0.5, 0.5, 0.5), W.WATER, 1.0)
    prob = W.tiny_problem(20_000 + batches // 2, n_batches=batches).with_(
        phantom=ph, source=W.pencil_source(ph, 1.0))
    out = {}
    for mode in (1, 2):
        eng = G.Engine(prob, params={G.GDPM_PARAM_BATCH_MODE: mode, G.GDPM_PARAM_TALLY_MODE: tally})
        try:
            for _ in range(2):          # the second run uses the grids the first one's fold cleared
                d, s, st = eng.run()
            out[mode] = d.cpu().numpy(), s.cpu().numpy(), st
        finally:
            eng.close()
    (d1, s1, a), (d2, s2, b) = out[1], out[2]
    assert a["el_steps"] == b["el_steps"] and a["compton"] == b["compton"]
    # the same FP64 tallies in another order of addition: a few eps per sum;
    # the variance is a difference of sums, off by a few eps of the mean square
    assert np.all(np.abs(d1 - d2) <= 1e-12 * d1)
    assert np.all(np.abs(s1 ** 2 - s2 ** 2) <= 1e-12 * d1 ** 2 + 1e-12 * s1 ** 2)
    assert (d1 > 0).any()
    assert abs(a["deposited"] - b["deposited"]) <= 1e-12 * a["deposited"]
    assert abs(a["sigma_over_dmax"] - b["sigma_over_dmax"]) <= 1e-6 * a["sigma_over_dmax"] + 1e-9


# a dose matrix of one beamlet holds the histories of that beamlet's own
# calculation; up to 4 batches keep their tallies apart until the last kernel
# step, more are summed first
@pytest.mark.parametrize("batches", [2, 3, 4, 5, 11])
@pytest.mark.parametrize("tally", [0, 1])
def test_matrix_fold_equals_calculation(batches, tally):
    ph = W.homogeneous_phantom((19, 23, 29), (0.5, 0.5, 0.5), W.WATER, 1.0)
    n = 10_000 + batches // 2
    src = W.single_beamlet(ph, 0.0, -0.5, -0.5, 1.0)
    prob = W.Problem(ph, src, n, batches, eabs_photon=0.05, eabs_electron=0.2, e_min=0.005, e_max=6.5,
                     sub_histories=(n,))
    eng = G.Engine(prob, params={G.GDPM_PARAM_TALLY_MODE: tally})
    try:
        d1, s1, _ = eng.run()
        for _ in range(2):
            d2, s2, _ = eng.run_beamlets()
        d1, s1, d2, s2 = (t.cpu().numpy().ravel() for t in (d1, s1, d2, s2))
    finally:
        eng.close()
    assert (d1 > 0).any()
    assert np.all(np.abs(d1 - d2) <= 1e-12 * d1)
    assert np.all(np.abs(s1 ** 2 - s2 ** 2) <= 1e-12 * d1 ** 2 + 1e-12 * s1 ** 2)
