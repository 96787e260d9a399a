"""Ranges whose end leaves the integer type are refused like any other range
past the end."""
import pytest

from paper_1107_3355_gb300 import gdpm as G
from paper_1107_3355_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def refused(call):
    with pytest.raises(G.GdpmError) as e:
        call()
    assert e.value.code == G.GDPM_E_ARG


def test_ends_that_wrap_are_refused():
    ph = W.homogeneous_phantom((16, 16, 16), (1.0, 1.0, 1.0))
    prob = W.Problem(ph, W.single_beamlet(ph, 0.0, -0.5, -0.5, 1.0), 10_000, 10, eabs_photon=0.05,
                     eabs_electron=0.2, e_min=0.005, e_max=6.5)
    eng = G.Engine(prob)
    try:
        out = torch.zeros(64, dtype=torch.int32, device="cuda")
        outd = torch.zeros(64 * 8, dtype=torch.float64, device="cuda")
        s = torch.zeros(ph.n_voxels, dtype=torch.float64, device="cuda")
        for first, n in ((2 ** 64 - 10, 20), (2 ** 32 - 1, 2), (2, 2 ** 64 - 1)):
            refused(lambda: G.gdpm_debug_beamlets(eng.ctx, first, n, out))
            refused(lambda: G.gdpm_debug_sources(eng.ctx, eng.phantom, eng.tables, 10_000, 10, first, n, outd))
        for first, n in ((2 ** 31 - 1, 2), (2 ** 31 - 5, 10), (9, 2), (0, 11)):
            refused(lambda: G.gdpm_simulate_part(eng.ctx, eng.phantom, eng.tables, 10_000, 10, first, n, s, s))
    finally:
        eng.close()
