"""FP64 pair forces evaluated from the neighbour lists, against the FP64
oracle: ordinary and long lists (a cutoff with more than 32 partners a
particle sends pairs through the overflow list), last blocks of every size,
separate protein cells, band-3 and glycophorin.  Each term is rounded to
2^-32 once, so forces agree to the fixed-point resolution (the FP64 parity
bounds of the other tests)."""
import numpy as np
import pytest

import oracle
from synth import membranes as M

pytestmark = pytest.mark.gpu

G = pytest.importorskip("paper_1701_02059_gb300")

EPS = [[0.0, 1.2, 0.9], [1.2, 1.4, 1.1], [0.9, 1.1, 0.0]]
RC = [[0.0, 2.8, 0.0], [2.8, 2.9, 2.7], [0.0, 2.7, 0.0]]


def check(mem, gkw=None, okw=None):
    p = G.make_params(kT=mem.kT, n_centroids=mem.n_centroids, box=mem.box, periodic=mem.periodic, seed=0,
                      precision=G.F64_ALL, **(gkw or {}))
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
        for energies in (True, False):
            e = g.compute_forces(energies=energies)
            F, T = g.forces()
            assert (np.linalg.norm(F - Fo, axis=1) / np.maximum(np.linalg.norm(Fo, axis=1), frms)).max() <= 1e-8
            assert np.linalg.norm(T - To, axis=1).max() / max(np.sqrt((To ** 2).sum(1).mean()), frms) <= 1e-8
            if energies:
                assert np.allclose(e[:4], eo[:4], rtol=1e-10, atol=1e-6)
                assert abs(e[4] - eo[4]) <= 1e-9 * max(abs(eo[4]), frms * mem.n)
        before = g.forces()
        g.pairs()
        for x, y in zip(before, g.forces()):
            assert np.array_equal(x, y)


@pytest.mark.parametrize("rc", [2.6, 4.2])
@pytest.mark.parametrize("n_lipids", [700, 1279])
def test_vesicle(n_lipids, rc):
    mem = M.vesicle(n_lipids, 7, f=1, chain_beads=4, n_centroids=9 if rc > 3 else 20)
    check(mem, dict(rc_lipid=rc), dict(rc=rc))


def test_patch():
    check(M.flat_patch_2304())


def test_proteins():
    mem = M.with_membrane_proteins(M.vesicle(2000, 3, f=2, chain_beads=6, n_centroids=40), seed=4)
    check(mem, dict(eps_mem=EPS, rc_mem=RC), dict(mem_eps=EPS, mem_rc=RC))
