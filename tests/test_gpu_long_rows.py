"""Rows at the edges of the builder's and Q's row classes: 64 and 65 entries
(eight lanes, then a warp), 2,048 and 2,049 (a warp, then blocks of their own),
hubs next to one another in node order, on graphs whose rows get eight lanes
(many short rows), a warp each (long rows on average) and a warp each without
hub blocks (few rows).  Q and the solve must be the oracle's, and a malformed
entry must be refused in whatever class its row is."""
import numpy as np
import pytest

import oracle
import paper_2608_03695_gb300 as pkg
from paper_2608_03695_gb300 import synth
from qtol import q_close

pytestmark = pytest.mark.gpu

DEGREES = (64, 65, 2048, 2049, 4500, 3000, 63, 2047)


@pytest.fixture(scope="module", autouse=True)
def built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pkg.build()
    oracle.build()


def graph(kind):
    """Nodes 0..7 have exactly DEGREES neighbours, all among the others."""
    rng = np.random.default_rng(17)
    n, T, extra = {"lanes": (4901, 2, 6000), "warps": (4900, 2, 165_000), "few": (4800, 2, 6000)}[kind]
    k = len(DEGREES)
    us = [np.full(d, i) for i, d in enumerate(DEGREES)] + [rng.integers(k, n, extra)]
    vs = [rng.choice(np.arange(k, n), d, replace=False) for d in DEGREES] + [rng.integers(k, n, extra)]
    u, v = np.concatenate(us), np.concatenate(vs)
    key = np.unique(np.minimum(u, v) * n + np.maximum(u, v))
    u, v = key // n, key % n
    u, v = u[u != v], v[u != v]
    snaps = [synth.csr_from_edges(n, u, v, rng.integers(1, 9, size=len(u))) for _ in range(T)]
    assert tuple(np.diff(snaps[0].indptr)[:k]) == DEGREES
    rows, entries = n * T, sum(s.nnz for s in snaps)
    assert (rows > 152 * 64) == (kind != "few") and (entries > 64 * rows) == (kind == "warps")
    return snaps


@pytest.mark.parametrize("coupling", ["ordinal", "categorical"])
@pytest.mark.parametrize("kind", ["lanes", "warps", "few"])
def test_q_and_labels(kind, coupling):
    snaps = graph(kind)
    n, T = snaps[0].n, len(snaps)
    labels = np.random.default_rng(3).integers(0, 40, n * T).astype(np.int32)
    with pkg.mslice_build(snaps, coupling=coupling) as h:
        for lab in (labels, np.zeros(n * T, np.int32)):
            assert q_close(h.mslice_modularity(lab, (1, 1), (1, 2)),
                           oracle.modularity(snaps, lab, (1, 1), (1, 2), coupling=coupling))
        got, Q, _ = h.mslice_leiden(n_iterations=1)
    ref, Qref, _ = oracle.leiden(snaps, n_iterations=1, coupling=coupling)
    assert np.array_equal(got, ref) and q_close(Q, Qref)


def test_q_of_a_batch():
    snaps = graph("lanes")
    with pkg.mslice_build(snaps) as h, pkg.Batch() as b:
        for gm in ((1, 1), (3, 2)):
            b.add(h, gm, (1, 2))
        b.run()
        for i, gm in enumerate(((1, 1), (3, 2))):
            lab, Q = b.results(i)
            ref, Qref, _ = oracle.leiden(snaps, gm, (1, 2))
            assert np.array_equal(lab, ref) and q_close(Q, Qref)


@pytest.mark.parametrize("row", range(len(DEGREES)))
@pytest.mark.parametrize("kind", ["lanes", "warps", "few"])
def test_malformed_entries_are_refused(kind, row):
    def refused(change):
        snaps = graph(kind)
        s = snaps[1]
        s.indices, s.weights = s.indices.copy(), s.weights.copy()
        change(s, int(s.indptr[row]), int(s.indptr[row + 1]))
        with pytest.raises(pkg.MsliceError) as e:
            pkg.mslice_build(snaps).close()
        return e.value.code == pkg.MSLICE_EINVAL

    def heavier(s, a, b):
        s.weights[b - 1] += 1

    def repeated(s, a, b):
        s.indices[a + 1] = s.indices[a]

    def out_of_range(s, a, b):
        s.indices[b - 1] = s.n

    def loop(s, a, b):
        s.indices[a] = row

    def weightless(s, a, b):
        s.weights[a] = 0

    for change in (heavier, repeated, out_of_range, loop, weightless):
        assert refused(change), change.__name__
