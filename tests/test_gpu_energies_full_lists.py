"""Energies of a system with more pairs than the neighbour lists hold: the
first call finds that out, the next ones do not search again; forces alone and
steps stay refused, and a new structure starts afresh."""
import numpy as np
import pytest

from synth import membranes as M

pytestmark = pytest.mark.gpu

G = pytest.importorskip("paper_1701_02059_gb300")


def energies(g):
    n = g.launch_count()
    e = g.compute_forces(energies=True)
    return e, g.launch_count() - n


def test_no_search_in_vain():
    dense, wide = (M.vesicle(700, 7, f=1, chain_beads=4, n_centroids=9) for _ in range(2))
    wide.pos *= 2.0
    with G.System(G.make_params(kT=dense.kT, n_centroids=9, rc_lipid=4.2, seed=0)) as g:
        g.load_membrane(dense)
        g.init_cells()
        first, n0 = energies(g)
        again, n1 = energies(g)
        # search, evaluation, bonds and kinetic energy only once
        assert n0 - n1 == 4 and np.array_equal(first, again)
        for refused in (g.compute_forces, lambda: g.integrate(1)):
            with pytest.raises(G.OrbcError):
                refused()
        assert energies(g)[1] == n1
        # a structure whose lists fit is searched and evaluated from them
        g.load_membrane(wide)
        g.init_cells()
        assert energies(g)[1] == n1 + 1
        g.integrate(1)
        g.rebuild_cells()
        assert energies(g)[1] == n1 + 1
