"""Nearest centroids of the initialisation against brute force in FP64: input
in id order, at random and striped (a warp's particles in several places),
centroids at random among the particles (uneven cells, searches over several
rings of grid cells), with and without Lloyd rounds, open and periodic."""
import numpy as np
import pytest

from synth import membranes as M

pytestmark = pytest.mark.gpu

G = pytest.importorskip("paper_1701_02059_gb300")


@pytest.mark.parametrize("order", ["ids", "random", "striped"])
@pytest.mark.parametrize("n, K, rounds, shape", [(31, 1, 1, "vesicle"), (33, 3, 0, "vesicle"), (1000, 7, 3, "vesicle"),
                                                 (20000, 350, 4, "vesicle"), (20000, 90, 0, "vesicle"),
                                                 (4608, 80, 3, "patch")])
def test_nearest_centroid(n, K, rounds, shape, order):
    mem = M.vesicle(max(n, 400), 7, f=1, chain_beads=5, n_centroids=50) if shape == "vesicle" else M.patch(3, seed=7)
    rows = np.flatnonzero(mem.type == 0)[:n]
    n = len(rows)
    rng = np.random.default_rng(n + K)
    if order == "random":
        rows = rng.permutation(rows)
    elif order == "striped":
        rows = np.concatenate([rows[k::11] for k in range(11)])
    ids = np.arange(n, dtype=np.uint32)
    pos = mem.pos[rows]
    with G.System(G.make_params(kT=mem.kT, n_centroids=K, n_lloyd_init=rounds, box=mem.box, periodic=mem.periodic)) as g:
        g.set_particles(pos, mem.vel[rows], mem.ori[rows], mem.angvel[rows], np.zeros(n, np.uint8), ids)
        g.init_cells(pos[rng.choice(n, K, replace=False)])
        c = g.cells()
    d = np.rint(pos * 2.0**40)[:, None, :] * 2.0**-40 - c["centroids"][None, :, :]
    for a in range(3):
        if mem.periodic[a]:
            d[:, :, a] -= mem.box[a] * np.rint(d[:, :, a] / mem.box[a])
    r2 = (d * d).sum(axis=2)
    assert np.array_equal(c["cell_of_id"], r2.argmin(axis=1))
