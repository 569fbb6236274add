"""What the Python binding takes as a snapshot's arrays, and what it hands to the
library for them (no GPU and no compiled library needed)."""
import ctypes as C

import numpy as np
import pytest

import paper_2608_03695_gb300 as pkg


class Snap:
    def __init__(self, indptr, indices, weights):
        self.indptr, self.indices, self.weights = indptr, indices, weights


def handed(snaps, **kw):
    """(n, indptr, indices, weights) of every snapshot as the library reads them."""
    arr, keep = pkg._csr_array(snaps, **kw)
    out = []
    for c in C.cast(pkg._ptr(arr), C.POINTER(pkg.Csr))[: len(snaps)]:
        ip = np.ctypeslib.as_array(C.cast(c.indptr, C.POINTER(C.c_int64)), (c.n + 1,)).copy()
        m = int(ip[-1])
        col = [np.ctypeslib.as_array(C.cast(p, C.POINTER(C.c_int32)), (m,)).copy() if m else np.zeros(0, np.int32)
               for p in (c.indices, c.weights)]
        out.append((c.n, ip.tolist(), col[0].tolist(), col[1].tolist()))
    del keep
    return out


PATH = (3, [0, 1, 3, 4], [1, 0, 2, 1], [5, 5, 7, 7])


def forms():
    ip, ix, w = (np.array(x, t) for x, t in zip(PATH[1:], (np.int64, np.int32, np.int32)))
    frozen = [x.copy() for x in (ip, ix, w)]
    for x in frozen:
        x.flags.writeable = False
    return {"arrays": (ip, ix, w), "lists": PATH[1:], "wide": (ip.astype(np.int32), ix.astype(np.int64), w.astype(np.int64)),
            "swapped": (ip.astype(">i8"), ix.astype(">i4"), w.astype(">i4")), "read-only": tuple(frozen),
            "strided": tuple(np.repeat(x, 2)[::2] for x in (ip, ix, w)), "floats": tuple(x.astype(float) for x in (ip, ix, w))}


@pytest.mark.parametrize("form", sorted(forms()))
def test_forms_of_host_arrays(form):
    assert handed([Snap(*forms()[form])] * 2) == [PATH, PATH]


def test_a_scalar_row_pointer_is_an_empty_snapshot():
    empty = Snap(np.array(0), np.zeros(0, np.int32), np.zeros(0, np.int32))
    assert handed([empty]) == [(0, [0], [], [])]
    assert handed([Snap(0, [], [])]) == [(0, [0], [], [])]


def test_arrays_beside_tensors():
    torch = pytest.importorskip("torch")
    ip, ix, w = forms()["arrays"]
    assert handed([Snap(torch.from_numpy(ip), ix, w)], host_tensors=True) == [PATH]
    assert handed([Snap(torch.from_numpy(ip), torch.from_numpy(ix), w)], host_tensors=True) == [PATH]
    arr, _ = pkg._csr_array([Snap(torch.zeros(1, dtype=torch.int64), None, None)], device_ptrs=True)
    assert arr[0, 0] == 0 and arr[0, 2] == 0 and arr[0, 3] == 0
