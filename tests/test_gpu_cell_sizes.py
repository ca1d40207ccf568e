"""The rebuild's sort, gather and cell properties over mean cell sizes from a
few particles to several hundred (cells of up to 64 and 128 particles, larger
ones, and the route of large cells as launches of their own): the forces do
not depend on the cells, bit for bit, the radii are the FP64 definition's and
the cells' order is a permutation that agrees with the offsets."""
import numpy as np
import pytest

from synth import membranes as M

pytestmark = pytest.mark.gpu

G = pytest.importorskip("paper_1701_02059_gb300")


def run(per, precision=None):
    mem = M.vesicle(6000, 11, f=2, chain_beads=10, n_centroids=50)
    n = len(mem.type)
    kw = {} if precision is None else {"precision": precision}
    with G.System(G.make_params(kT=mem.kT, n_centroids=max(n // per, 1), n_lloyd_init=3, box=mem.box,
                                periodic=mem.periodic, seed=3, **kw)) as g:
        g.load_membrane(mem)
        g.init_cells()
        g.integrate(2)
        g.compute_forces()
        return g.state(), g.forces(), g.cells()


@pytest.mark.parametrize("per", [7, 55, 64, 100, 128, 180, 255, 256, 257, 300, 700])
def test_sizes(per):
    s0, f0, _ = run(61)
    s, f, c = run(per)
    for k in ("pos", "vel", "ori", "angvel"):
        assert np.array_equal(s[k], s0[k]), k
    for x, y in zip(f, f0):
        assert np.array_equal(x, y)
    start = c["start"]
    assert start[0] == 0 and start[-1] == len(c["slot_ids"]) and np.array_equal(np.sort(c["slot_ids"]), np.arange(start[-1]))
    cell_of_slot = np.repeat(np.arange(len(start) - 1), np.diff(start))
    assert np.array_equal(c["cell_of_id"][c["slot_ids"]], cell_of_slot)
    d = s["pos"][c["slot_ids"]] - c["centroids"][cell_of_slot]
    r = np.zeros(len(start) - 1)
    np.maximum.at(r, cell_of_slot, np.sqrt((d * d).sum(axis=1)))
    # positions and centroids on the 2^-40 grid: a few FP64 roundings apart
    assert np.allclose(c["radius"], r, rtol=1e-14, atol=0.0)
