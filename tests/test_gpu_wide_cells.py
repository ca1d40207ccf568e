"""Cells of up to 32 sigma: particles of neighbouring cells lie up to 96 sigma
from a cell's centre, beyond the mirrors' 64 sigma period.  Pairs, forces,
energies and steps are those of small cells (forces and steps bit for bit): no
particle 64 sigma away is taken for a close one, and no partner is lost."""
import numpy as np
import pytest

from synth import membranes as M

pytestmark = pytest.mark.gpu

G = pytest.importorskip("paper_1701_02059_gb300")


def run(rows, K, precision, **kw):
    n = len(rows[0])
    with G.System(G.make_params(kT=0.2, n_centroids=K, n_lloyd_init=3, seed=4, precision=precision, **kw)) as g:
        g.set_particles(*rows, np.arange(n, dtype=np.uint32))
        g.init_cells()
        radius = g.cells()["radius"].max()
        e = g.compute_forces(energies=True)
        out = [*g.forces(), g.pairs()]
        g.integrate(6)
        s = g.state()
        return out + [s[k] for k in ("pos", "vel", "ori", "angvel")], e, radius


def lipids(mem):
    k = np.flatnonzero(mem.type == 0)
    return [mem.pos[k], mem.vel[k], mem.ori[k], mem.angvel[k], mem.type[k]]


@pytest.mark.parametrize("precision", [G.F32_FORCE_F64_STATE, G.F64_ALL])
@pytest.mark.parametrize("shape, K, least, skin", [("sheet", 30, 20.0, 0.0), ("sheet", 24, 20.0, 0.2), ("sheet", 20, 20.0, 0.0),
                                                   ("vesicle", 2, 30.0, 0.0)])
def test_wide_cells(precision, shape, K, least, skin):
    # an open flat sheet of 107 x 93 sigma, a vesicle of radius 28
    rows = lipids(M.patch(6, seed=7) if shape == "sheet" else M.vesicle(9000, 3, kT=0.3, f=3, chain_beads=6))
    kw = {"rebuild_every": 50, "skin": skin} if skin else {}
    got, e, radius = run(rows, K, precision, **kw)
    assert radius > least
    want, e0, _ = run(rows, len(rows[0]) // 60, precision)
    for x, y in zip(got, want):
        assert np.array_equal(x, y)
    # (energies: sums of rounded parts)
    assert np.allclose(e, e0, rtol=1e-9, atol=1e-6)
