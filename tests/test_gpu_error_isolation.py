"""A calculation that fails leaves nothing behind that fails the next one."""
import dataclasses

import pytest

from paper_1107_3355_gb300 import gdpm as G
from paper_1107_3355_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_next_call_after_a_cuda_error():
    # tables after which the graph loop's shared memory is a close fit
    prob = W.slab_electron_problem(n_histories=2000, n_batches=2, shape=(16, 16, 32))
    wide = prob.with_(phantom=dataclasses.replace(prob.phantom, materials=(list(prob.phantom.materials) * 7)[:7]),
                      n_energy=544)
    for p in (wide, prob, wide):
        eng = G.Engine(p, params={G.GDPM_PARAM_GRAPH: 1 if p is wide else 0})
        try:
            st = eng.run()[2]
            assert st["n_primary"] == 2000
        except G.GdpmError as e:
            assert p is wide and e.code == G.GDPM_E_CUDA
        finally:
            eng.close()
