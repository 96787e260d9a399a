"""Dose and sigma from batch sums of any magnitude, in voxels of any size:
both are FP64 results, and neither may depend on a value fitting FP32."""
import numpy as np
import pytest

from paper_1107_3355_gb300 import gdpm as G
from paper_1107_3355_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# relative error: a few roundings of the sums and of q - x^2/(n-1), whose
# terms are within a factor of 4 of each other here, and one FP64 Newton step
# from a 2-ulp FP32 estimate (2^-43): 1e-12 in all
@pytest.mark.parametrize("side", [1e-3, 0.25, 10.0, 100.0])
def test_finalize_over_magnitudes(side):
    nb, rho = 10, 0.7
    mag = 10.0 ** np.arange(-100, 61)
    rng = np.random.default_rng(2)
    x = mag[:, None] * rng.uniform(0.0, 1.0, (mag.size, nb))
    ph = W.homogeneous_phantom((mag.size, 1, 1), (side, side, side), W.WATER, rho)
    eng = G.Engine(W.tiny_problem(1000, n_batches=2).with_(phantom=ph, source=W.pencil_source(ph, 1.0)))
    try:
        d = torch.empty(mag.size, dtype=torch.float64, device="cuda")
        s = torch.empty_like(d)
        G.gdpm_finalize(eng.ctx, eng.phantom, nb, x.sum(1), (x * x).sum(1), d, s)
    finally:
        eng.close()
    f = np.float64(np.float32(side))
    mass = np.float64(np.float32(rho)) * f * f * f
    mean = x.sum(1) / nb
    # the sums as the call got them
    sd = np.sqrt(((x * x).sum(1) - nb * mean * mean) / (nb * (nb - 1)))
    np.testing.assert_allclose(d.cpu().numpy(), mean / mass, rtol=1e-12)
    np.testing.assert_allclose(s.cpu().numpy(), sd / mass, rtol=1e-12)
