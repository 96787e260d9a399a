"""Source kernels of several host threads: one context's primaries need a few
bytes of shared memory for their tables, another's some 30 KB.  Neither's
launches may depend on what the other asked for last."""
import threading

import pytest

from paper_1107_3355_gb300 import gdpm as G
from paper_1107_3355_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_threads_with_small_and_large_source_tables():
    small = W.tiny_problem(4000, n_batches=2)
    ph = small.phantom
    large = W.Problem(ph, W.field_source(ph, W.kramers_spectrum(), ssd=30.0, field=(6.0, 6.0)), 6000, 120,
                      eabs_photon=0.05, eabs_electron=0.2, e_min=0.005, e_max=7.0)
    failed, counts = [], {0: set(), 1: set()}

    def work(k, prob, calls):
        try:
            eng = G.Engine(prob, params={G.GDPM_PARAM_SOURCE_CHUNK: 100, G.GDPM_PARAM_SPECULATIVE: 4})
            try:
                for _ in range(calls):
                    counts[k].add(eng.run()[2]["ph_flights"])
            finally:
                eng.close()
        except Exception as e:      # reported by the test, not by the thread
            failed.append((k, repr(e)))

    threads = [threading.Thread(target=work, args=(0, small, 150)), threading.Thread(target=work, args=(1, large, 100)),
               threading.Thread(target=work, args=(0, small, 150))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed
    assert len(counts[0]) == 1 and len(counts[1]) == 1


def test_threads_building_graphs_beside_small_and_large_tables():
    """The graph loop's kernels, whose shared memory grows with the tables."""
    base = W.slab_electron_problem(n_histories=500, n_batches=2, shape=(16, 16, 32))
    failed, counts = [], {32: set(), 2048: set()}

    def work(n_energy):
        try:
            # small blocks: the tables are most of a CTA's shared memory
            eng = G.Engine(base.with_(n_energy=n_energy), params={G.GDPM_PARAM_GRAPH: 1, G.GDPM_PARAM_BLOCK_THREADS: 64})
            try:
                for k in range(150):
                    # another walk form is another graph
                    G.gdpm_set_param(eng.ctx, G.GDPM_PARAM_ELECTRON_WALK, k % 2)
                    counts[n_energy].add(eng.run()[2]["el_steps"])
            finally:
                eng.close()
        except Exception as e:
            failed.append((n_energy, repr(e)))

    threads = [threading.Thread(target=work, args=(n,)) for n in (32, 2048, 32)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed
    assert all(len(c) == 1 for c in counts.values())
