"""Rounds of local moving that leave settled nodes out, against the oracle.

The library tracks settled nodes on large levels; here every level of small
graphs is tracked (MSLICE_TRACK_MIN_ENTRIES=0), so that pushes, budgets and
rejoining nodes occur next to tie-breaks, singletons and moves to empty
communities.  Small levels run inside one launch per phase; with
MSLICE_RESIDENT_MAX_WORK=0 the same graphs take the large levels' kernels.  Every result must be the oracle's: labels bit-exact, counters
equal, Q within 1e-12 relative.
"""
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


@pytest.fixture(autouse=True)
def tracked(monkeypatch):
    monkeypatch.setenv("MSLICE_TRACK_MIN_ENTRIES", "0")


def graph(seed, kind):
    if kind == "planted":
        return synth.planted_partition_temporal(150 + 37 * seed, 3 + seed % 4, 4, 0.1, 0.02, 0.2, None, 5, seed)[0]
    if kind == "powerlaw":
        return synth.dcsbm_powerlaw_temporal(300 + 61 * seed, 2 + seed % 5, mean_deg=12.0, size_min=8, size_max=60,
                                             seed=seed)[0]
    if kind == "contact":
        return synth.contact_temporal(40 + seed, 60, 4, 200, 900, 0.7, seed)[0]
    return synth.random_temporal(30 + 9 * seed, 1 + seed % 6, p=0.12, w_max=3, seed=seed, p_empty=0.2)


def same(g, o):
    assert np.array_equal(g[0], o[0])
    assert q_close(g[1], o[1]), (g[1], o[1])
    for k in ("iterations", "levels", "lm_rounds", "lm_edges", "lm_moves", "stop_reason", "last_level0_moves"):
        assert g[2][k] == o[2][k], k


@pytest.mark.parametrize("resident", [None, "0"])
@pytest.mark.parametrize("dense", [None, "0"])
@pytest.mark.parametrize("null", ["multislice", "global", "cpm"])
@pytest.mark.parametrize("kind", ["planted", "powerlaw", "contact", "random"])
def test_tracked_solves(kind, null, dense, resident, monkeypatch):
    if resident is not None:
        monkeypatch.setenv("MSLICE_RESIDENT_MAX_WORK", resident)
    if dense is not None:
        monkeypatch.setenv("MSLICE_DENSE_LIMIT", dense)
    for seed in range(4):
        snaps = graph(seed, kind)
        n, T = snaps[0].n, len(snaps)
        kw = dict(K=1 + (seed + 3) % 5, seed=seed, n_iterations=1 + seed % 3)
        if seed % 2:  # start from random labels: heavy movement in a recorded round
            kw["init"] = np.random.default_rng(seed).integers(0, max(n // 4, 1), n * T).astype(np.int32)
        omega = [(1, 1), (1, 10), (7, 3), (0, 1)][seed]
        gamma = (1, 8) if null == "cpm" else [(1, 1), (3, 2), (5, 4), (1, 2)][seed]
        coupling = "categorical" if seed == 2 and T <= 8 else "ordinal"
        with pkg.mslice_build(snaps, omega=omega, coupling=coupling) as h:
            g = h.mslice_leiden(gamma=gamma, omega=omega, null=null, **kw)
        same(g, oracle.leiden(snaps, gamma, omega, null=null, coupling=coupling, **kw))


@pytest.mark.parametrize("resident", [None, "0"])
@pytest.mark.parametrize("shift", [8, 16, 24])
def test_tracked_heavy_weights(shift, resident, monkeypatch):
    """Margins in units coarser than a weight unit, and pushes past the largest."""
    if resident is not None:
        monkeypatch.setenv("MSLICE_RESIDENT_MAX_WORK", resident)
    snaps = graph(2, "powerlaw")
    for s in snaps:
        s.weights = (s.weights.astype(np.int64) << shift).astype(np.int32)
    with pkg.mslice_build(snaps) as h:
        g = h.mslice_leiden(omega=(1 << shift, 3))
    same(g, oracle.leiden(snaps, (1, 1), (1 << shift, 3)))


@pytest.mark.parametrize("theta", [None, (1, 100)])
def test_untracked_large_level_kernels(theta, monkeypatch):
    """The large levels' kernels without tracking, greedy and randomised."""
    monkeypatch.delenv("MSLICE_TRACK_MIN_ENTRIES")
    monkeypatch.setenv("MSLICE_RESIDENT_MAX_WORK", "0")
    for kind in ("planted", "powerlaw", "contact", "random"):
        for dense in ("4194304", "0"):
            monkeypatch.setenv("MSLICE_DENSE_LIMIT", dense)
            snaps = graph(1, kind)
            with pkg.mslice_build(snaps) as h:
                g = h.mslice_leiden(theta=theta)
            same(g, oracle.leiden(snaps, theta=theta))


@pytest.mark.parametrize("resident", [None, "0"])
def test_tracked_batch(resident, monkeypatch):
    """Instances of very different movement in one batch, alone and together."""
    if resident is not None:
        monkeypatch.setenv("MSLICE_RESIDENT_MAX_WORK", resident)
    cases = [(graph(s, k), gm, om) for s, k in ((0, "planted"), (3, "planted"), (1, "powerlaw"), (2, "contact"))
             for gm, om in (((1, 1), (1, 1)), ((3, 2), (10, 1)))]
    handles = [pkg.mslice_build(c[0]) for c in cases]
    with pkg.Batch() as b:
        for h, (_, gm, om) in zip(handles, cases):
            b.add(h, gm, om)
        b.run()
        for i, (snaps, gm, om) in enumerate(cases):
            lab, Q = b.results(i)
            ol, oq, _ = oracle.leiden(snaps, gm, om)
            assert np.array_equal(lab, ol) and q_close(Q, oq), i
    for h in handles:
        h.close()
