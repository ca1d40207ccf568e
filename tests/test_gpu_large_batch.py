"""A batch of more than 2^26 particles (the particle numbers that a neighbour
list's entry holds): its last membranes step as alone, bit for bit."""
import numpy as np
import pytest

from synth import membranes as M

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
G = pytest.importorskip("paper_1701_02059_gb300")


@pytest.mark.parametrize("precision", [G.F32_FORCE_F64_STATE, G.F64_ALL])
def test_last_of_a_large_batch(precision):
    if torch.cuda.mem_get_info()[0] < 90 << 30:
        pytest.skip("wants 90 GB of device memory")
    mem = M.vesicle(900_000, 5)
    n = len(mem.type)
    count = (1 << 26) // n + 2
    p = G.make_params(kT=mem.kT, n_centroids=mem.n_centroids, n_lloyd_init=1, box=mem.box, periodic=mem.periodic, seed=3,
                      precision=precision)
    with G.System(p) as g:
        g.load_membrane(mem)
        g.init_cells()
        g.integrate(2)
        want = g.state()
    arena = G.Arena(150 << 30, precision)
    try:
        # (the others stay in the batch)
        slots = arena.admit_many([(p, mem, 2 if k >= count - 2 else 100) for k in range(count)])
        assert arena.run(2) == 2
        for s in slots[-2:]:
            got = arena.retire(s)
            for k in ("pos", "vel", "ori", "angvel"):
                assert np.array_equal(got[k], want[k]), k
    finally:
        arena.close()
