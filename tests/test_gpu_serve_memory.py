"""The device memory that a request's solve holds stays within the footprint by
which the server admits it (what the library's allocations take from the device's
memory pool at their highest, above the idle server's)."""
import ctypes as C

import pytest

import paper_2608_03695_gb300 as pkg
from paper_2608_03695_gb300 import synth

pytestmark = pytest.mark.gpu

USED_NOW, USED_HIGH = 7, 8  # cudaMemPoolAttr


@pytest.fixture(scope="module", autouse=True)
def built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pkg.build()


class Pool:
    def __init__(self):
        try:
            self.rt = C.CDLL("libcudart.so.13")
        except OSError:
            pytest.skip("libcudart.so.13 cannot be loaded by name")
        self.pool = C.c_void_p()
        assert self.rt.cudaDeviceGetDefaultMemPool(C.byref(self.pool), 0) == 0

    def get(self, attr):
        x = C.c_uint64(0)
        assert self.rt.cudaMemPoolGetAttribute(self.pool, attr, C.byref(x)) == 0
        return x.value

    def restart(self):
        x = C.c_uint64(0)
        assert self.rt.cudaMemPoolSetAttribute(self.pool, USED_HIGH, C.byref(x)) == 0
        return self.get(USED_NOW)


@pytest.mark.parametrize("n,T", [(4000, 8), (12000, 6), (30000, 3)])
def test_a_solve_stays_within_its_footprint(n, T):
    import torch
    pool = Pool()
    snaps, _ = synth.planted_partition_temporal(n, T, 4, 12.0 / n, 1.2 / n, 0.1, 0.05, 8, 50)
    with pkg.Server(window=T, n_slots=1) as srv:
        g = srv.add_graph(n)
        for s in snaps:
            torch.cuda.synchronize()
            idle = pool.restart()
            _, info = srv.wait(srv.submit(g, s))
        # (the last request solves the whole window)
        assert pool.get(USED_HIGH) - idle <= info["footprint"]
