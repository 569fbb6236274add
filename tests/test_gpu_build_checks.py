"""The builder's check that snapshots are symmetric: only entries above the
diagonal search for their mirror image, and the entries below are counted.
Every way of breaking the symmetry must still be refused, wherever the odd
entry lies and also when two snapshots' errors cancel in the count."""
import numpy as np
import pytest

import paper_2608_03695_gb300 as pkg
from paper_2608_03695_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pkg.build()


def base():
    return synth.random_temporal(40, 3, p=0.2, w_max=5, seed=9)


def without(sn, row, upper):
    """sn less one entry of `row` above (upper) or below the diagonal."""
    a, b = int(sn.indptr[row]), int(sn.indptr[row + 1])
    at = [e for e in range(a, b) if (sn.indices[e] > row) == upper][0]
    ip = sn.indptr.copy()
    ip[row + 1:] -= 1
    return synth.Snapshot(ip, np.delete(sn.indices, at), np.delete(sn.weights, at))


def refused(snaps):
    with pytest.raises(pkg.MsliceError) as e:
        pkg.mslice_build(snaps).close()
    return e.value.code == pkg.MSLICE_EINVAL


def test_the_base_is_accepted():
    for coupling in ("ordinal", "categorical"):
        with pkg.mslice_build(base(), coupling=coupling) as h:
            assert h.N == 120


@pytest.mark.parametrize("upper", [True, False])
@pytest.mark.parametrize("s", [0, 2])
def test_missing_entries(s, upper):
    snaps = base()
    snaps[s] = without(snaps[s], 20, upper)
    assert refused(snaps)


def test_errors_that_cancel_in_the_count():
    snaps = base()
    snaps[0] = without(snaps[0], 20, True)
    snaps[1] = without(snaps[1], 20, False)
    assert refused(snaps)
    snaps = base()
    snaps[1] = without(without(snaps[1], 20, True), 22, False)
    assert refused(snaps)


@pytest.mark.parametrize("upper", [True, False])
def test_weights_that_differ(upper):
    snaps = base()
    a, b = int(snaps[1].indptr[20]), int(snaps[1].indptr[21])
    at = [e for e in range(a, b) if (snaps[1].indices[e] > 20) == upper][0]
    snaps[1].weights[at] += 1
    assert refused(snaps)
