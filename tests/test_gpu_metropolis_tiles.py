"""The Metropolis kernel's edges, pick for pick against the oracle: chain
counts around a CTA's 32, histories around its tiles of 56 steps a chain, and
weights outside FP32's range, where every acceptance is decided in FP64."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1107_3355_gb300 import gdpm as G
from paper_1107_3355_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("chains,steps", [(1, 55), (31, 56), (32, 57), (33, 112), (100, 113)])
@pytest.mark.parametrize("weights", ["plain", "wide", "equal"])
def test_picks_at_tile_edges(chains, steps, weights):
    ph = W.homogeneous_phantom((16, 16, 16), (1.0, 1.0, 1.0))
    rng = np.random.default_rng(5)
    k = 37
    f = {"plain": rng.uniform(0.1, 1.0, k), "wide": 10.0 ** rng.uniform(-60, 60, k), "equal": np.full(k, 0.3)}[weights]
    fr = W.beam_frame(30.0, (8.0, 8.0, 8.0))
    rows = [W.beamlet_row(fr, i - k / 2, i + 1 - k / 2, -0.5, 0.5, float(f[i])) for i in range(k)]
    src = W.beamlet_source(rows, W.kramers_spectrum())
    src.sampler, src.chains = "metropolis", chains
    prob = W.Problem(ph, src, 20_000, 2, eabs_photon=0.05, eabs_electron=0.2, e_min=0.005, e_max=6.5)
    n = chains * steps + chains // 2
    eng = G.Engine(prob)
    try:
        out = torch.full((n,), -1, dtype=torch.int32, device="cuda")
        G.gdpm_debug_beamlets(eng.ctx, 3, n, out)
    finally:
        eng.close()
    assert np.array_equal(out.cpu().numpy(), O.beamlet_picks(prob, 3, n))
