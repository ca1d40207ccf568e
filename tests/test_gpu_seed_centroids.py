"""The first centroids, picked from the members (bilayer particles) in id
order: centroid k is member floor(k M / K).  Against the same positions given
by the caller, the cells after two Lloyd rounds are equal exactly: member
counts that are no multiple of K, ids in any order, sizes on either side of
the chunks the members are counted in, a chunk without members."""
import numpy as np
import pytest

from synth import membranes as M

pytestmark = pytest.mark.gpu

G = pytest.importorskip("paper_1701_02059_gb300")


@pytest.mark.parametrize("n, gap", [(257, (0, 40)), (16383, (0, 0)), (16384, (100, 3000)), (16385, (16384, 16385)),
                                    (40000, (16384, 32768)), (70001, (0, 16390))])
def test_members_in_id_order(n, gap):
    mem = M.vesicle(n, 5, f=1, chain_beads=5, n_centroids=50)
    lip = np.flatnonzero(mem.type == 0)[:n]
    pos, vel, ori, angvel = (x[lip] for x in (mem.pos, mem.vel, mem.ori, mem.angvel))
    rng = np.random.default_rng(n)
    ids = rng.permutation(n).astype(np.uint32)
    typ = np.where((ids >= gap[0]) & (ids < gap[1]), 1, 0).astype(np.uint8)
    typ[rng.random(n) < 0.2] = 2
    by_id = np.empty(n, np.int64)
    by_id[ids] = np.arange(n)
    members = by_id[typ[by_id] == 0]
    K = max(len(members) // 59, 2)
    seeds = members[np.arange(K) * len(members) // K]
    out = []
    for centroids in (None, pos[seeds]):
        with G.System(G.make_params(kT=mem.kT, n_centroids=K, n_lloyd_init=2, box=mem.box, periodic=mem.periodic)) as g:
            g.set_particles(pos, vel, ori, angvel, typ, ids)
            g.init_cells(centroids)
            out.append(g.cells())
    for k in out[0]:
        assert np.array_equal(out[0][k], out[1][k]), k
