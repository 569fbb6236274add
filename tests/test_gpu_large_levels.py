"""The large levels' kernels, directly: on small graphs every phase of a level runs
inside one launch, so these tests switch that off (MSLICE_RESIDENT_MAX_WORK=0), or
let rounds change hands between the two forms, on graphs with hubs of every degree
tier, tracked and not, dense and hashed, greedy and randomised, and in the
bounds-checked build.  Also the branches of the one-launch aggregation that short
sequences and small communities never take.  Every result must be the oracle's."""
import functools
import os
import subprocess
import sys

import numpy as np
import pytest

import oracle
import paper_2608_03695_gb300 as pkg
from paper_2608_03695_gb300 import synth
from qtol import q_close
from test_gpu_checked import CASES, ROOT

pytestmark = pytest.mark.gpu

COUNTERS = ("iterations", "levels", "lm_rounds", "lm_edges", "lm_moves", "stop_reason", "last_level0_moves")


@pytest.fixture(scope="module", autouse=True)
def built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pkg.build()
    oracle.build()


def same(g, o):
    assert np.array_equal(g[0], o[0])
    assert q_close(g[1], o[1]), (g[1], o[1])
    for k in COUNTERS:
        assert g[2][k] == o[2][k], k


@functools.lru_cache(maxsize=None)
def hubs(n, degrees, extra, T, seed):
    rng = np.random.default_rng(seed)
    us = [np.full(d, i) for i, d in enumerate(degrees)] + [rng.integers(10, n, extra)]
    vs = [rng.choice(np.arange(10, n), size=d, replace=False) for d in degrees] + [rng.integers(10, n, extra)]
    u, v = np.concatenate(us), np.concatenate(vs)
    key = np.unique(np.minimum(u, v) * n + np.maximum(u, v))
    u, v = key // n, key % n
    u, v = u[u != v], v[u != v]
    return [synth.csr_from_edges(n, u, v, rng.integers(1, 5, size=len(u))) for _ in range(T)]


# hubs past the shared tables (9,000 and 5,000 entries), of the block tiers and of the warp tier
GRAPHS = {"top": (12000, (9000, 5000, 1500, 600, 100, 20), 30000, 2, 11), "block": (3000, (1500, 200, 40, 1100), 6000, 3, 3)}


@functools.lru_cache(maxsize=None)
def expected(graph, omega, theta):
    return oracle.leiden(hubs(*GRAPHS[graph]), (1, 1), omega, theta=theta)


@pytest.mark.parametrize("tracked", [None, "0"])
@pytest.mark.parametrize("shared", ["1", "0"])
@pytest.mark.parametrize("dense", [None, "0"])
@pytest.mark.parametrize("graph", sorted(GRAPHS))
def test_hubs(graph, dense, shared, tracked, monkeypatch):
    monkeypatch.setenv("MSLICE_RESIDENT_MAX_WORK", "0")
    monkeypatch.setenv("MSLICE_TIER4_SHARED", shared)
    if dense is not None:
        monkeypatch.setenv("MSLICE_DENSE_LIMIT", dense)
    if tracked is not None:
        monkeypatch.setenv("MSLICE_TRACK_MIN_ENTRIES", tracked)
    for omega in ((1, 2), (3, 1)):
        with pkg.mslice_build(hubs(*GRAPHS[graph])) as h:
            same(h.mslice_leiden(omega=omega), expected(graph, omega, None))


@pytest.mark.parametrize("dense", [None, "0"])
@pytest.mark.parametrize("graph", sorted(GRAPHS))
def test_hubs_randomised(graph, dense, monkeypatch):
    monkeypatch.setenv("MSLICE_RESIDENT_MAX_WORK", "0")
    if dense is not None:
        monkeypatch.setenv("MSLICE_DENSE_LIMIT", dense)
    with pkg.mslice_build(hubs(*GRAPHS[graph])) as h:
        same(h.mslice_leiden(omega=(1, 2), theta=(1, 100)), expected(graph, (1, 2), (1, 100)))


def test_hubs_aggregated(monkeypatch):
    snaps = hubs(*GRAPHS["top"])
    o = oracle.leiden(snaps, omega=(1, 2), stop_level=1, stop_stage=3)
    for bound in ("0", None):
        if bound is None:
            monkeypatch.delenv("MSLICE_RESIDENT_MAX_WORK")
        else:
            monkeypatch.setenv("MSLICE_RESIDENT_MAX_WORK", bound)
        with pkg.mslice_build(snaps) as h:
            g = h.mslice_leiden(omega=(1, 2), stop_level=1, stop_stage=3)
        assert np.array_equal(g[0], o[0])
        for k in ("next_n", "next_nnz", "next_checksum"):
            assert g[2][k] == o[2][k], k


@pytest.mark.parametrize("dense", [None, "0"])
def test_tier_cuts(dense, monkeypatch):
    monkeypatch.setenv("MSLICE_RESIDENT_MAX_WORK", "0")
    if dense is not None:
        monkeypatch.setenv("MSLICE_DENSE_LIMIT", dense)
    with pkg.mslice_build(hubs(*GRAPHS["block"])) as h:
        for cuts in [(0, 0, 0, 0), (4, 8, 16, 32), (16, 16, 64, 64), (0, 32, 256, 1024)]:
            same(h.mslice_leiden(omega=(1, 2), tier_cuts=cuts), expected("block", (1, 2), None))
        same(h.mslice_leiden(omega=(1, 2), autotune=True), expected("block", (1, 2), None))


@pytest.mark.parametrize("dense", [None, "0"])
@pytest.mark.parametrize("bound", ["20000", "60000", "300000"])
def test_rounds_that_change_hands(bound, dense, monkeypatch):
    """Host-driven rounds that pass a level on to resident ones as its lists
    shrink, and get it back when they grow."""
    monkeypatch.setenv("MSLICE_RESIDENT_MAX_WORK", bound)
    monkeypatch.setenv("MSLICE_TRACK_MIN_ENTRIES", "0")
    if dense is not None:
        monkeypatch.setenv("MSLICE_DENSE_LIMIT", dense)
    for omega in ((1, 2), (3, 1)):
        with pkg.mslice_build(hubs(*GRAPHS["top"])) as h:
            same(h.mslice_leiden(omega=omega), expected("top", omega, None))
    snaps = synth.recipe_graph({**synth.RECIPES["powerlaw_t16_n100k"], "n": 4000, "T": 4})
    with pkg.mslice_build(snaps) as h:
        same(h.mslice_leiden(omega=(1, 2), K=3, seed=4), oracle.leiden(snaps, omega=(1, 2), K=3, seed=4))


# ---- the one-launch aggregation


@pytest.mark.parametrize("theta", [None, (1, 100)])
def test_more_null_slices_than_the_strength_table(theta):
    """9,000 snapshots of 3 nodes: communities of more than 256 snapshots are summed
    in a hashed table, those of more than 4,096 by the general path."""
    snaps = synth.random_temporal(3, 9000, p=0.6, w_max=3, seed=1)
    with pkg.mslice_build(snaps) as h:
        same(h.mslice_leiden(theta=theta), oracle.leiden(snaps, theta=theta))


def test_batch_whose_snapshots_sum_past_the_strength_table():
    graphs = [synth.random_temporal(3, 4600, p=0.6, w_max=3, seed=s) for s in (1, 2)]
    handles = [pkg.mslice_build(g) for g in graphs]
    with pkg.Batch() as b:
        for h in handles:
            b.add(h, (1, 1), (3, 1))
        b.run()
        for i, g in enumerate(graphs):
            lab, Q = b.results(i)
            ref, Qref, _ = oracle.leiden(g, (1, 1), (3, 1))
            assert np.array_equal(lab, ref) and q_close(Q, Qref), i
    for h in handles:
        h.close()


@pytest.mark.parametrize("sizes,T,level", [((260, 260), 1, 0), ((300, 200, 150), 2, 1)])
def test_communities_too_long_for_one_block(sizes, T, level):
    """Sub-communities of 67,000 and 109,000 entries (one block sums 32,768)."""
    snaps = synth.cliques_temporal(list(sizes), T)
    o = oracle.leiden(snaps, stop_level=level, stop_stage=3)
    with pkg.mslice_build(snaps) as h:
        g = h.mslice_leiden(stop_level=level, stop_stage=3)
        assert np.array_equal(g[0], o[0])
        for k in ("next_n", "next_nnz", "next_checksum"):
            assert g[2][k] == o[2][k], k
        same(h.mslice_leiden(), oracle.leiden(snaps))


# ---- the bounds-checked build

HUB_CASES = r'''
sys.path.insert(0, os.path.join(ROOT, "tests"))
import test_gpu_large_levels as big
for graph in sorted(big.GRAPHS):
    for dense in (None, "0"):
        os.environ.pop("MSLICE_DENSE_LIMIT", None)
        if dense is not None:
            os.environ["MSLICE_DENSE_LIMIT"] = dense
        for theta in (None, (1, 100)):
            with pkg.mslice_build(big.hubs(*big.GRAPHS[graph])) as h:
                big.same(h.mslice_leiden(omega=(1, 2), theta=theta), big.expected(graph, (1, 2), theta))
print("hubs ok")
'''


@pytest.mark.parametrize("tracked", [False, True])
def test_checked_build(tracked):
    pkg.build(checked=True)
    env = {**os.environ, "MSLICE_LIBRARY": "checked", "MSLICE_RESIDENT_MAX_WORK": "0"}
    if tracked:
        env["MSLICE_TRACK_MIN_ENTRIES"] = "0"
    r = subprocess.run([sys.executable, "-c", "ROOT = %r\n" % ROOT + CASES + HUB_CASES], env=env, capture_output=True,
                       text=True, timeout=900)
    assert r.returncode == 0 and "checked ok" in r.stdout and "hubs ok" in r.stdout, r.stdout[-2000:] + r.stderr[-4000:]
