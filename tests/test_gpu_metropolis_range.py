"""Metropolis picks at the end of the history range, with as many chains as a
source may have, pick for pick against the oracle."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1107_3355_gb300 import gdpm as G
from paper_1107_3355_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def problem(chains):
    ph = W.homogeneous_phantom((16, 16, 16), (1.0, 1.0, 1.0))
    rng = np.random.default_rng(5)
    fr = W.beam_frame(30.0, (8.0, 8.0, 8.0))
    rows = [W.beamlet_row(fr, i - 18.5, i - 17.5, -0.5, 0.5, float(f)) for i, f in enumerate(rng.uniform(0.1, 1.0, 37))]
    src = W.beamlet_source(rows, W.kramers_spectrum())
    src.sampler, src.chains = "metropolis", chains
    return W.Problem(ph, src, 20_000, 2, eabs_photon=0.05, eabs_electron=0.2, e_min=0.005, e_max=6.5)


def picks(prob, first, n):
    eng = G.Engine(prob)
    try:
        out = torch.full((n,), -1, dtype=torch.int32, device="cuda")
        G.gdpm_debug_beamlets(eng.ctx, first, n, out)
    finally:
        eng.close()
    return out.cpu().numpy()


@pytest.mark.parametrize("chains", [2 ** 24 - 1, 2 ** 24])
@pytest.mark.parametrize("end", [2 ** 32 - 2 ** 24 + 1, 2 ** 32 - 1])
def test_picks_at_the_end_of_the_range(chains, end):
    prob = problem(chains)
    n = 2000
    assert np.array_equal(picks(prob, end - n, n), O.beamlet_picks(prob, end - n, n))


# the last history id there is, one more than a launch's 32-bit count reaches
@pytest.mark.parametrize("sampler", ["metropolis", "alias"])
def test_picks_up_to_the_last_history_id(sampler):
    prob = problem(2 ** 20)
    prob.source.sampler = sampler
    n = 300
    assert np.array_equal(picks(prob, 2 ** 32 - n, n), O.beamlet_picks(prob, 2 ** 32 - n, n))
