"""A packed batch of one instance holds no more device memory than a system of
the same membrane (whose set-up allocates the same arrays and the k-means
initialisation's besides)."""
import ctypes as C

import pytest

from synth import membranes as M

pytestmark = pytest.mark.gpu

G = pytest.importorskip("paper_1701_02059_gb300")


def pool_used():
    cu, pool, used = C.CDLL("libcuda.so.1"), C.c_void_p(), C.c_uint64(0)
    assert cu.cuCtxSynchronize() == 0
    assert cu.cuDeviceGetDefaultMemPool(C.byref(pool), C.c_int(0)) == 0
    assert cu.cuMemPoolGetAttribute(pool, C.c_int(7), C.byref(used)) == 0    # the bytes in use
    return used.value


@pytest.mark.parametrize("n", [700, 20000])
def test_batch_of_one(n):
    mem = M.vesicle(n, 5, f=max(1, round((n / 1105) ** 0.5)))
    p = G.make_params(kT=mem.kT, n_centroids=mem.n_centroids, box=mem.box, periodic=mem.periodic, seed=3)
    with G.System(p) as g:
        before = pool_used()      # (the handle has made a context)
        g.load_membrane(mem)
        g.init_cells()
        g.integrate(1)
        system = pool_used() - before
    arena = G.Arena(8 << 30)
    try:
        before = pool_used()
        arena.admit(p, mem, 100)
        arena.run(1)
        batch = pool_used() - before
    finally:
        arena.close()
    assert 0 < batch <= system
