"""Energies with FP32 forces from the neighbour lists, against the FP64
oracle with the FP32 bounds of the parity tests: last blocks of every size,
pairs in the overflow list, and more partners than the lists and their
overflow hold (the kernel without lists takes over; stepping such a system
is refused as before)."""
import numpy as np
import pytest

import oracle
from synth import membranes as M

pytestmark = pytest.mark.gpu

G = pytest.importorskip("paper_1701_02059_gb300")

EPS = [[0.0, 1.2, 0.9], [1.2, 1.4, 1.1], [0.9, 1.1, 0.0]]
RC = [[0.0, 2.8, 0.0], [2.8, 2.9, 2.7], [0.0, 2.7, 0.0]]


def check(mem, gkw=None, okw=None, steps_refused=False):
    p = G.make_params(kT=mem.kT, n_centroids=mem.n_centroids, box=mem.box, periodic=mem.periodic, seed=0, **(gkw or {}))
    o = oracle.OracleSystem(oracle.model(box=mem.box, periodic=mem.periodic, **(okw or {})),
                            oracle.run(kT=mem.kT, n_centroids=mem.n_centroids, seed=0))
    o.load(mem)
    o.init_cells()
    eo = o.compute_forces()
    Fo, To = o.forces()
    frms = np.sqrt((Fo ** 2).sum(1).mean())
    with G.System(p) as g:
        g.load_membrane(mem)
        g.init_cells()
        e = g.compute_forces(energies=True)
        again = g.compute_forces(energies=True)
        assert np.array_equal(e, again)
        F, T = g.forces()
        assert (np.linalg.norm(F - Fo, axis=1) / np.maximum(np.linalg.norm(Fo, axis=1), frms)).max() <= 1e-5
        assert abs(e[0] - eo[0]) <= 1e-5 * abs(eo[0]) and abs(e[1] - eo[1]) <= 1e-5 * max(abs(eo[1]), 1.0)
        assert abs(e[4] - eo[4]) <= 1e-5 * max(abs(eo[4]), frms * mem.n)
        if steps_refused:
            with pytest.raises(G.OrbcError):
                g.integrate(1)


@pytest.mark.parametrize("n_lipids", [700, 1279])
def test_vesicle(n_lipids):
    check(M.vesicle(n_lipids, 7, f=1, chain_beads=4, n_centroids=20))


def test_overflow_list():
    # about 35 partners a particle: some pairs beyond the lists' 32 entries
    check(M.vesicle(4000, 7, f=2, chain_beads=4, n_centroids=60), dict(rc_lipid=3.4), dict(rc=3.4))


def test_more_partners_than_the_lists_hold():
    check(M.vesicle(700, 7, f=1, chain_beads=4, n_centroids=9), dict(rc_lipid=4.2), dict(rc=4.2), steps_refused=True)


def test_proteins():
    check(M.with_membrane_proteins(M.vesicle(2000, 3, f=2, chain_beads=6, n_centroids=40), seed=4),
          dict(eps_mem=EPS, rc_mem=RC), dict(mem_eps=EPS, mem_rc=RC))
