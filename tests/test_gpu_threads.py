"""Handles solved from several threads at once: their cooperative grids share
the SMs (a part each while several solves are in progress), beside launches of
the large levels' kernels.  Every result must be the oracle's, whatever else is
running and however many blocks a grid got."""
import threading

import numpy as np
import pytest

import oracle
import paper_2608_03695_gb300 as pkg
from paper_2608_03695_gb300 import synth
from qtol import q_close

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pkg.build()
    oracle.build()


@pytest.mark.parametrize("bound", [None, "30000", "0"])
def test_threads_with_handles_of_their_own(bound, monkeypatch):
    # bound 30000: the larger graphs' level 0 by the large levels' kernels, the rest resident
    if bound is not None:
        monkeypatch.setenv("MSLICE_RESIDENT_MAX_WORK", bound)
    graphs = [synth.planted_partition_temporal(250 * (i + 1), 3, 4, 0.08, 0.01, 0.1, None, 4, i)[0] for i in range(5)]
    graphs += [synth.dcsbm_powerlaw_temporal(900, 4, mean_deg=12.0, size_min=8, size_max=60, seed=1)[0],
               synth.contact_temporal(40, 60, 4, 200, 900, 0.7, 2)[0],
               synth.random_temporal(6, 2, p=0.5, seed=3), synth.random_temporal(70, 5, p=0.1, seed=4)]
    expect = [oracle.leiden(g) for g in graphs]
    start = threading.Barrier(len(graphs))
    bad = []

    def work(i):
        try:
            with pkg.mslice_build(graphs[i]) as h:
                start.wait(60)
                for k in range(4):
                    lab, Q, _ = h.mslice_leiden()
                    if not (np.array_equal(lab, expect[i][0]) and q_close(Q, expect[i][1])):
                        bad.append((i, k))
        except Exception as e:  # noqa: BLE001 (reported below)
            bad.append((i, repr(e)))
            start.abort()

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(graphs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad, bad
